"""The float64 contractions as products of integer slices (oz.cuh) by
themselves (internal.cu)."""
import ctypes
import math
from fractions import Fraction

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


def digits(A):
    """Row exponents e and digits v[i][row][k] of the slices: x = 2^(e - 56) X, X
    rounded to nearest (halves up in magnitude), X = sum_i v_i 2^(49 - 7 i), from
    the definition in Python's integers."""
    e, v = [], np.zeros((8, *A.shape))
    for r, row in enumerate(A):
        big = max(abs(float(x)) for x in row)
        # 2^e above every element; subnormals count as the least normal binade
        e.append(max(math.frexp(big)[1], -1021) if big > 0 else 0)
        for k, x in enumerate(row):
            f = abs(Fraction(float(x))) * Fraction(2) ** (56 - e[-1])
            X = math.floor(f + Fraction(1, 2))
            X = -X if x < 0 else X
            for i in range(7, 0, -1):
                d = ((X + 64) & 127) - 64
                v[i, r, k] = d
                X = (X - d) >> 7
            assert abs(X) <= 128
            v[0, r, k] = X
    return e, v


def expected(A, B, alpha):
    """The sum of the products of slices i + j <= 7, rounded to float64 once."""
    (ea, va), (eb, vb) = digits(A), digits(B)
    S = np.zeros((A.shape[0], B.shape[0]), object)
    for i in range(8):
        for j in range(8 - i):
            D = va[i] @ vb[j].T  # integers below 2^53
            S += np.vectorize(int, otypes=[object])(D) << (7 * (7 - i - j))
    def scaled(x, e):
        try:
            return math.ldexp(float(x), e)
        except OverflowError:
            return math.copysign(math.inf, x)

    return np.array([[scaled(S[r, c], ea[r] + eb[c] - 63 + alpha) for c in range(B.shape[0])]
                     for r in range(A.shape[0])])


def extreme(rows, k):
    """Digits at their limits with equal signs: v_0 = -127, all others -64."""
    X = -127 * 2 ** 49 - 64 * sum(2 ** (49 - 7 * i) for i in range(1, 8))
    x = X / 2 ** 56  # 50 bits: exact
    assert Fraction(x) * 2 ** 56 == X
    return np.full((rows, k), x)


def rows_of(kind, rows, k, rng):
    A = rng.standard_normal((rows, k))
    if kind == "binades":  # elements spread over 100 binades
        A = np.ldexp(A, rng.integers(-100, 1, A.shape))
    elif kind == "special":
        A[0] = 0.0
        A[1] = np.ldexp(A[1], -1060)  # subnormals
        A[2] = np.ldexp(A[2], 900)
        A[3, :] = 0.0
        A[3, k // 2] = -5e-324
        A[4] *= -0.0
    elif kind == "extreme":
        A = extreme(rows, k)
    elif kind == "signs":
        A = extreme(rows, k) * rng.choice([-1.0, 1.0], (rows, k))
    return A


@pytest.mark.parametrize("kind", ["plain", "binades", "special", "extreme", "signs"])
@pytest.mark.parametrize("m,n,k", [(5, 9, 1), (7, 5, 16), (6, 65, 400), (129, 5, 401), (6, 7, 800), (5, 6, 1207)])
def test_products_of_slices(internal, kind, m, n, k):
    """Bit for bit what the format says, also with every digit at its limit (one and
    two segments of the sum, and one value more), subnormal, huge and zero rows; and
    within the bound of the product itself."""
    torch, lib = internal
    rng = np.random.default_rng(1000 * m + k)
    A, B = rows_of(kind, m, k, rng), rows_of(kind, n, k, rng)
    for alpha in (0, 1):
        C = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
        call(torch, lib.sp_gemm, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), m, n, k, C, alpha)
        C = C.cpu().numpy()
        assert np.array_equal(C, expected(A, B, alpha))
    for r, c in ((0, 0), (m - 1, n - 1), (2 % m, 3 % n), (4 % m, 2 % n)):
        exact = 2 * sum((Fraction(a) * Fraction(b) for a, b in zip(A[r].tolist(), B[c].tolist())), Fraction(0))
        # 2^e is at most twice a row's largest element, or the least normal number
        top = Fraction(max(np.abs(A[r]).max(), 2.0 ** -1022)) * Fraction(max(np.abs(B[c]).max(), 2.0 ** -1022))
        # (the least subnormal: results there are rounded to its multiples)
        bound = abs(exact) * Fraction(2) ** -53 + 2 * Fraction(112, 10) * k * top * Fraction(2) ** -56 + Fraction(5e-324)
        assert math.isinf(C[r, c]) or abs(Fraction(C[r, c]) - exact) <= bound


def test_rows_that_are_not_finite(internal):
    """An infinity or a NaN in a row makes its results NaN and leaves the others."""
    torch, lib = internal
    rng = np.random.default_rng(0)
    A, B = rng.standard_normal((6, 40)), rng.standard_normal((7, 40))
    want = expected(A, B, 0)
    A[2, 5], A[3, 0], B[4, 39], B[1] = np.inf, np.nan, -np.inf, 0.0
    want[2], want[3], want[:, 1], want[:, 4] = np.nan, np.nan, 0.0, np.nan
    want[2:4, 1] = np.nan
    C = torch.zeros((6, 7), dtype=torch.float64, device="cuda")
    call(torch, lib.sp_gemm, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), 6, 7, 40, C, 0)
    assert np.array_equal(C.cpu().numpy(), want, equal_nan=True)


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
