"""The Taylor series kernel where a walker's V stays in shared memory and two
CTAs share an SM (up to 128 orbitals in BF16, 80 in TF32), against the float64
replay of tests/test_gpu_taylor.py and within its bounds: the edges of the
route, and more walkers than two per SM, so that CTAs take walkers in turn."""
import numpy as np
import pytest

from test_gpu_taylor import env, operands, reference, round_bf16, round_tf32, run  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,W,N,M", [
    (0, 700, 2, 20),     # one K block
    (0, 5, 32, 128),     # the largest: 64 rows of the term, one full row tile
    (0, 320, 16, 113),   # K blocks that end in padding
    (0, 310, 10, 129),   # the smallest of the other route
    (1, 330, 7, 64),
    (1, 4, 17, 80),
])
def test_matches_reference(env, dtype, W, N, M):  # noqa: F811
    torch, pkg = env
    rnd = round_bf16 if dtype == 0 else round_tf32
    Mp = (M + 15) // 16 * 16
    rng = np.random.default_rng(77 + M)
    dV, dT, Vlo, Tlo = operands(rng, W, N, M, Mp, rnd)
    ref, _ = reference(Vlo, Tlo, N, M, Mp, 6, rnd)
    got = run(torch, pkg, dtype, dV, dT, W, N, M, Mp, Mp, 6, 0)
    err = np.linalg.norm((got - ref)[:, :, :M], axis=(1, 2)) / np.linalg.norm(ref, axis=(1, 2))
    assert err.max() < (3e-3 if dtype == 0 else 6e-4), (int(err.argmax()), err.max())
