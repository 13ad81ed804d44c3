"""The modified Cholesky decomposition in one launch against one launch per
vector (taken above 4096 vectors of room or 64 indices per SM): the same sums in
the same order, so the same pivots, vectors and residual to the last bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,rank,delta", [
    (1, 1, 1e-8),
    (37, 37, 1e-8),       # full rank, one block per eight indices
    (465, 60, 1e-8),
    (1221, 200, 1e-2),    # stops at the threshold
    (1500, 150, 1e-30),   # runs on in the rounding of a deficient matrix
    (3003, 1300, 1e-8),   # more vectors than a block's shared memory holds
])
def test_same_as_one_launch_per_vector(dim, rank, delta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1711_02242_gb300 as pkg

    g = torch.Generator(device="cuda").manual_seed(dim)
    A = torch.randn(rank, dim, generator=g, device="cuda", dtype=torch.float64)
    A *= (0.99 ** torch.arange(rank, device="cuda", dtype=torch.float64))[:, None]
    V = A.T @ A
    V = 0.5 * (V + V.T)
    room = 4096
    if delta < 1e-20:  # past the rank the residual is rounding: bound the vectors instead
        room = rank + 40
        one = pkg.afqmc_modified_cholesky(V, delta, room)
        many = pkg.afqmc_modified_cholesky(V, delta, 4097)
        n = one[0].shape[0]
        assert torch.equal(one[0], many[0][:n]) and torch.equal(one[1], many[1][:n])
        return
    one = pkg.afqmc_modified_cholesky(V, delta, room)
    many = pkg.afqmc_modified_cholesky(V, delta, 4097)
    assert one[0].shape == many[0].shape and one[2] == many[2]
    assert torch.equal(one[0], many[0]) and torch.equal(one[1], many[1])
    assert 1 <= one[0].shape[0] <= rank + 1 and np.isfinite(one[2])
