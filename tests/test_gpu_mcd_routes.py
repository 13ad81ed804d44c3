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


def decompose(internal, dim, rank, delta, wait_cycles, sms):
    torch, lib = internal
    import ctypes

    import paper_1711_02242_gb300 as pkg

    g = torch.Generator(device="cuda").manual_seed(dim)
    A = torch.randn(rank, dim, generator=g, device="cuda", dtype=torch.float64)
    V = A.T @ A
    V = 0.5 * (V + V.T)
    n = ctypes.c_size_t(0)
    pkg._check(pkg.lib().afqmc_mcd_workspace_size(dim, rank + 8, ctypes.byref(n)))
    work = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    L = torch.zeros((rank + 8, dim), dtype=torch.float64, device="cuda")
    piv = torch.zeros(rank + 8, dtype=torch.int32, device="cuda")
    nvec, resid = ctypes.c_int(0), ctypes.c_double(0)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    lib.in_mcd.argtypes = ([ctypes.c_longlong, ctypes.c_void_p, ctypes.c_double, ctypes.c_int] + [ctypes.c_void_p] * 5
                           + [ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p])
    rc = lib.in_mcd(dim, p(V), delta, rank + 8, p(L), p(piv), ctypes.byref(nvec), ctypes.byref(resid), p(work),
                    wait_cycles, sms, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    return rc, L, piv, nvec.value, resid.value


def test_blocks_that_cannot_all_run_at_once(internal):
    """With too few SMs for the one launch a launch per vector does the same."""
    torch, _ = internal
    one = decompose(internal, 1221, 90, 1e-8, 4000000000, 0)
    few = decompose(internal, 1221, 90, 1e-8, 4000000000, 7)
    assert one[0] == 0 and few[0] == 0 and one[3:] == few[3:] and 80 <= one[3] <= 98
    assert torch.equal(one[1], few[1]) and torch.equal(one[2], few[2])


def test_waits_between_the_blocks_end(internal):
    """A wait bound that every first failed poll exceeds: the call returns its
    time-out, and the device goes on working."""
    assert decompose(internal, 3003, 400, 1e-8, -1, 0)[0] == -5  # AFQMC_ETIMEOUT
    assert decompose(internal, 1221, 90, 1e-8, 4000000000, 0)[0] == 0
