"""Accuracy of the sliced FP64 product per output, relative to sum |a||b| as a chain of FP64 FMAs has it, on operands that the
digits hold well (no output is left to FMAs, and an error of the lowest level would show) and on operands that they
hold badly: rows graded against each other, zeros where the other operand is large, constant digits whose level sums outgrow
FP32, results below the normal numbers, infinities and NaNs."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U = 2.0 ** -53


def two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def two_prod(a, b):
    def split(x):
        c = 134217729.0 * x
        h = c - (c - x)
        return h, x - h
    p = a * b
    (ah, al), (bh, bl) = split(a), split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def exact_product(A, B):
    """(hi, lo, sum |a||b|) of A B^T: hi + lo to about 2^-100 (Dot2 of Ogita, Rump and Oishi)."""
    hi = np.zeros((A.shape[0], B.shape[0]))
    lo, mag = np.zeros_like(hi), np.zeros_like(hi)
    for j in range(A.shape[1]):
        p, e = two_prod(A[:, j][:, None], B[:, j][None, :])
        hi, f = two_sum(hi, p)
        lo += e + f
        mag += np.abs(p)
    return hi, lo, mag


def product(A, B, mode=0, by_cols=False):
    import device_kernels
    (M, K), N = A.shape, B.shape[0]
    a = torch.from_numpy(np.asfortranarray(A).T.copy() if by_cols else A.copy()).cuda()
    b = torch.from_numpy(B.copy()).cuda()
    z = torch.full((N, M + 3), 7.0, dtype=torch.float64, device="cuda")
    n_fma = ctypes.c_longlong(-1)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    rc = device_kernels.load().t_oz(M, N, K, mode, int(by_cols), p(a), ctypes.c_longlong(a.shape[1]), p(b),
                                    ctypes.c_longlong(K), p(z), ctypes.c_longlong(M + 3), ctypes.byref(n_fma))
    assert rc == 0
    z = z.cpu().numpy()
    assert (z[:, M:] == 7.0).all()
    return z[:, :M].T, n_fma.value


def triangle(A, mode):
    return np.tril(A) if mode == 1 else np.triu(A) if mode == 2 else A


SHAPES = [(128, 64, 256), (129, 65, 257), (300, 33, 300), (64, 1, 320), (387, 130, 387)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("by_cols", [False, True])
def test_flat_rows(shape, by_cols):
    M, N, K = shape
    rng = np.random.default_rng(M + N)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    Z, n_fma = product(A, B, 0, by_cols)
    hi, lo, mag = exact_product(A, B)
    assert n_fma == 0
    assert (np.abs((Z - hi) - lo) <= U * np.abs(Z) + 2.0 ** -58 * mag).all()


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[0] >= s[2]])
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("by_cols", [False, True])
def test_triangles(shape, mode, by_cols):
    M, N, K = shape
    rng = np.random.default_rng(M + mode)
    A = rng.standard_normal((M, K)) * np.exp(-np.abs(np.arange(M)[:, None] - np.arange(K)) / 20.0)   # peaked at the diagonal
    B = rng.standard_normal((N, K))
    B[:, ::3] = 0.0
    Z, _ = product(A, B, mode, by_cols)   # the other triangle is never read as part of A
    hi, lo, mag = exact_product(triangle(A, mode), B)
    assert (np.abs((Z - hi) - lo) <= 2.0 ** -50 * mag).all()


@pytest.mark.parametrize("bits", [5, 20, 40, 200])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("by_cols", [False, True])
def test_rows_graded_against_each_other(bits, mode, by_cols):
    M, N, K = 300, 33, 300
    rng = np.random.default_rng(bits)
    g = 2.0 ** -np.linspace(0.0, bits, K)
    A, B = rng.standard_normal((M, K)) * g, rng.standard_normal((N, K)) * g[::-1]
    A, B = A[:, rng.permutation(K)] if mode == 0 else A, B
    Z, n_fma = product(A, B, mode, by_cols)
    hi, lo, mag = exact_product(triangle(A, mode), B)
    assert (np.abs((Z - hi) - lo) <= 2.0 ** -50 * mag).all()
    if bits >= 20 and mode != 0:
        assert n_fma > 0


def digits(x):
    """The seven 9-bit digits of a row under its exponent, as integers (csrc/oz.cuh)."""
    e = int(np.floor(np.log2(np.abs(x).max()))) + 1
    f = np.rint(np.ldexp(x, 62 - e)).astype(np.int64)
    d = []
    for _ in range(6):
        low = ((f & 511) ^ 256) - 256
        d.append(low)
        f = (f - low) >> 9
    return [f] + d[::-1]


@pytest.mark.parametrize("top", [1.0, 510.0 / 511.0])
def test_level_sums_beyond_fp32(top):
    """Constant digits: with the second value at the head of B's rows all of them are 255, and level 5 sums to 2^24.3."""
    K = 256
    x = 510.0 / 511.0
    A, B = np.full((128, K), x), np.full((64, K), x * 2.0 ** -9)
    B[:, 0] = top
    a, b = digits(A[0]), digits(B[0])
    level = [max(abs(sum((a[i] * b[s - i])[k:k + 64].sum() for i in range(s + 1))) for k in range(0, K, 64)) for s in (4, 5, 6)]
    assert (max(level) >= 1 << 24) == (top == x)
    Z, n_fma = product(A, B)
    hi, lo, mag = exact_product(A, B)
    assert n_fma == (128 * 64 if top == x else 0)
    assert (np.abs((Z - hi) - lo) <= 2.0 ** -50 * mag).all()


def test_outside_the_normal_numbers():
    M, N, K = 130, 66, 256
    rng = np.random.default_rng(5)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    A[3] *= 2.0 ** -1000
    B[5] *= 2.0 ** -60            # products of row 3 and column 5: subnormal results
    A[7, 11], B[9, 2], B[10, 4] = np.inf, np.nan, -np.inf
    A[20] = 0.0
    B[30] = 0.0
    Z, _ = product(A, B)
    with np.errstate(all="ignore"):
        ref = (A[:, :, None] * B.T[None]).sum(axis=1)   # infinities and NaNs where a sum in any order has them
    assert np.array_equal(np.isnan(Z), np.isnan(ref)) and np.array_equal(np.isinf(Z), np.isinf(ref))
    assert np.array_equal(Z[np.isinf(Z)], ref[np.isinf(ref)])
    assert (Z[20, :9] == 0.0).all() and (Z[:7, 30] == 0.0).all()
    fin = np.isfinite(ref)
    # a subnormal sum errs by its last bits as well: K roundings of 2^-1075
    tol = 2.0 ** -50 * (np.abs(np.where(np.isfinite(A), A, 0.0)) @ np.abs(np.where(np.isfinite(B), B, 0.0)).T) + K * 2.0 ** -1074
    assert (np.abs(Z - ref)[fin] <= tol[fin]).all()
    assert Z[3, 5] != 0.0
