"""The float64 contractions as products of integer slices (oz.cuh) by
themselves (internal.cu)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

def call(torch, fn, *args):
    """fn(*args, ws, ws_bytes, status, stream); device arrays by their pointers."""
    ws = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    conv = [ctypes.c_void_p(a.data_ptr()) if isinstance(a, torch.Tensor) else a for a in args]
    rc = fn(*conv, ctypes.c_void_p(ws.data_ptr()), ctypes.c_size_t(ws.numel()), ctypes.c_void_p(status.data_ptr()),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == 0 and int(status.item()) == 0


@pytest.mark.parametrize("M,N,W,cw", [(40, 5, 41, 40), (65, 13, 15, 15), (33, 64, 4, 3), (30, 1, 250, 200)])
def test_densities_of_unequal_norms(internal, M, N, W, cw):
    """sum_k conj(Phi_k[p]) Th_k[q] over the walkers and orbitals k of a group: with
    Phi_k times and Th_k divided by a power of two of its own the same bits, and
    within the slices' bound, 2.8 K 2^-56 of the row maxima with those powers taken
    out (maxima below 8 here), of NumPy's sum (K 2^-53)."""
    torch, lib = internal
    rng = np.random.default_rng(M)
    phi, thA, thB = rng.standard_normal((3, W, 2, N, M))
    scale = 2.0 ** rng.integers(-60, 61, (W, 1, N, 1))
    nz = -(-W // cw)
    out = []
    for f in (1.0, scale):
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (phi * f, thA / f, thB / f)]
        D = torch.full((nz, 2 * M, 2 * M), float("nan"), dtype=torch.float64, device="cuda")
        call(torch, lib.sp_densities, *dev, W, N, M, cw, D)
        out.append(D.cpu().numpy())
    # (an orbital's exponent is its largest element's, so the slices see the same numbers)
    assert np.array_equal(out[0], out[1])
    for z in range(nz):
        w = slice(z * cw, min(W, (z + 1) * cw))
        P, A, B = phi[w], thA[w], thB[w]
        top = np.concatenate([P[:, 0], P[:, 1]], 1).reshape(-1, M)      # [Re | Im] per walker
        turn = np.concatenate([-P[:, 1], P[:, 0]], 1).reshape(-1, M)
        cols = [np.concatenate([T[:, 0], T[:, 1]], 1).reshape(-1, M) for T in (A, B)]
        ref = np.block([[top.T @ cols[0], top.T @ cols[1]], [turn.T @ cols[0], turn.T @ cols[1]]])
        K = top.shape[0]
        assert np.abs(out[1][z] - ref).max() < 8 * 8 * K * (2 * 2.8 * 2.0 ** -56 + 2.0 ** -53)
