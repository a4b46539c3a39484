"""The dense products by exact 8-bit digits against exact sums.

Bound of a Gram entry, from the arithmetic: entries are rounded 55 bits below e, the power of two above their column's
largest entry, products of digits i + j >= 8 are dropped (5 + 4 + .. + 1 pairs of at most 2^14 2^(8 (12 - i - j)), in
units of 2^-110 e_p e_q: below 2^-61 a term), and the sum is rounded once:
    2^-53 |C_pq| + 2^-56 (e_p |b_q|_1 + e_q |a_p|_1) + K 2^-61 e_p e_q.
The same for the update C = A B with the rows of A and the columns of B, whose columns (A) and rows (B) are first
brought to one magnitude by powers of two.
"""
import ctypes
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1902_07041_gb300 as pfe  # noqa: E402

pytestmark = pytest.mark.gpu
P, I, L, D, B = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64, ctypes.c_double, ctypes.c_bool


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    lib = pfe.load()
    sig = {"_ZN3pfe16digit_gram_bytesEliib": (ctypes.c_size_t, [L, I, I, B]),
           "_ZN3pfe18digit_update_bytesElii": (ctypes.c_size_t, [L, I, I]),
           "_ZN3pfe18launch_gram_digitsEliiPKdlS1_lddPdlbPvP11CUstream_st":
               (None, [L, I, I, P, L, P, L, D, D, P, L, B, P, P]),
           "_ZN3pfe20launch_update_digitsEliiPKdlS1_lddPdlbPvP11CUstream_st":
               (None, [L, I, I, P, L, P, L, D, D, P, L, B, P, P])}
    for name, (res, args) in sig.items():
        getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    return lib


def padded(A, extra=3):
    """A on the device with a row stride beyond its width; the gap is NaN."""
    d = torch.full((A.shape[0], A.shape[1] + extra), float("nan"), dtype=torch.float64, device="cuda")
    d[:, :A.shape[1]] = torch.from_numpy(A).cuda()
    return d


def gram(lib, A, Bm=None, alpha=1.0, beta=0.0, C=None, sym=False):
    """alpha A^T B + beta C (m x nn, column-major on the device)."""
    K, m = A.shape
    a, b = padded(A), None if Bm is None else padded(Bm)
    nn = m if Bm is None else Bm.shape[1]
    b = a if b is None else b
    c = torch.full((nn, m + 2), float("nan"), dtype=torch.float64, device="cuda")
    c[:, :m] = 7.0 if C is None else torch.from_numpy(np.ascontiguousarray(C.T)).cuda()
    w = torch.empty(lib._ZN3pfe16digit_gram_bytesEliib(K, m, nn, Bm is None), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    lib._ZN3pfe18launch_gram_digitsEliiPKdlS1_lddPdlbPvP11CUstream_st(
        K, m, nn, a.data_ptr(), a.stride(0), b.data_ptr(), b.stride(0), alpha, beta, c.data_ptr(), m + 2, sym,
        w.data_ptr(), None)
    torch.cuda.synchronize()
    assert c[:, m:].isnan().all()
    return c[:, :m].cpu().numpy().T


def two_product(a, b):
    """a b as an unevaluated sum (Dekker)."""
    def halves(x):
        h = x * 134217729.0
        h = h - (h - x)
        return h, x - h
    (ah, al), (bh, bl) = halves(a), halves(b)
    p = a * b
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def dot(a, b):
    return math.fsum(np.concatenate(two_product(a, b)))


def above(x):
    """The power of two above |x| (1 for 0)."""
    return np.ldexp(1.0, np.frexp(np.where(x == 0, 0.5, np.abs(x)))[1])


def gram_bound(a, b, value):
    ea, eb = above(np.abs(a).max()), above(np.abs(b).max())
    return 2.0**-53 * abs(value) + 2.0**-56 * (ea * np.abs(b).sum() + eb * np.abs(a).sum()) + a.size * 2.0**-61 * ea * eb


def block(kind, K, q, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((K, q))
    if kind == "localised":  # one large entry a column, in a row of its own
        A *= 1e-4
        A[rng.permutation(K)[:q], np.arange(q)] = 1.0
    elif kind == "magnitudes":
        A *= 10.0 ** rng.integers(-140, 140, q)
    elif kind == "digits":  # every digit large and of one sign
        A[:] = sum(100.0 * 2.0 ** -(8 * d + 8) for d in range(6))
    return A


# rows: less than a stage, a stage and a bit, many chunks, more than one slab of digits (18,688 rows at 256 columns)
@pytest.mark.parametrize("kind", ["normal", "localised", "magnitudes", "digits"])
@pytest.mark.parametrize("K,q", [(20, 1), (33, 5), (129, 64), (4000, 65), (20001, 200)])
@pytest.mark.parametrize("sym", [False, True])
def test_gram_within_the_bound(lib, K, q, kind, sym):
    A = block(kind, K, min(q, K), 1)
    G = gram(lib, A, sym=sym)
    rng = np.random.default_rng(2)
    q = A.shape[1]
    for i, j in {(0, 0), (q - 1, 0), (0, q - 1), *map(tuple, rng.integers(0, q, (12, 2)))}:
        exact = dot(A[:, i], A[:, j])
        assert abs(G[i, j] - exact) <= gram_bound(A[:, i], A[:, j], exact), (i, j)
    assert np.array_equal(G, G.T)


def test_gram_of_two_blocks_with_alpha_and_beta(lib):
    A, Bm, C = block("normal", 700, 130, 3), block("localised", 700, 67, 4), block("normal", 130, 67, 5)
    G = gram(lib, A, Bm, alpha=-0.5, beta=2.0, C=C)
    for i, j in np.random.default_rng(6).integers(0, (130, 67), (20, 2)):
        v = dot(A[:, i], Bm[:, j])
        exact = -0.5 * v + 2.0 * C[i, j]
        assert abs(G[i, j] - exact) <= 0.5 * gram_bound(A[:, i], Bm[:, j], v) + 2.0**-52 * (abs(v) + 2.0 * abs(C[i, j]))


def test_gram_of_zero_and_not_finite_columns(lib):
    A = block("normal", 300, 70, 7)
    A[:, 3] = 0.0
    A[5, 10] = np.inf
    A[6, 66] = np.nan
    G = gram(lib, A, sym=True)
    bad = np.isin(np.arange(70), [10, 66])
    assert not np.isfinite(G[bad]).any() and not np.isfinite(G[:, bad]).any()
    assert not G[3, ~bad].any() and np.isfinite(G[np.ix_(~bad, ~bad)]).all()


class DBuf(ctypes.Structure):
    """The library's growing device buffer."""
    _fields_ = [("p", P), ("bytes", ctypes.c_size_t)]


@pytest.mark.parametrize("sym", [False, True])
def test_gram_longer_than_its_sums(lib, sym):
    """More rows than 64-bit sums hold at once: the dispatch adds two parts, each rounded to double."""
    f = lib._ZN3pfe11launch_gramEliiPKdlS1_lddPdlbS2_P11CUstream_stPNS_4DBufE
    f.restype, f.argtypes = None, [L, I, I, P, L, P, L, D, D, P, L, B, P, P, P]
    free = lib._ZN3pfe9dbuf_freeERNS_4DBufE
    free.restype, free.argtypes = None, [P]
    size = lib._ZN3pfe9gram_workEliib
    size.restype, size.argtypes = ctypes.c_size_t, [L, I, I, B]
    K, m = (1 << 22) + 1000, 3
    work = torch.empty(size(K, m, m, sym), dtype=torch.float64, device="cuda")
    A, C = block("normal", K, m, 11), block("normal", m, m, 12)
    C = C + C.T
    a, c, buf = torch.from_numpy(A).cuda(), torch.from_numpy(C.copy()).cuda(), DBuf()
    torch.cuda.synchronize()
    f(K, m, m, a.data_ptr(), m, a.data_ptr(), m, 1.0, 0.5, c.data_ptr(), m, sym, work.data_ptr(), None,
      ctypes.byref(buf))
    torch.cuda.synchronize()
    assert buf.bytes > 0  # the digits' workspace: that path ran
    free(ctypes.byref(buf))
    G = c.cpu().numpy().T
    for i in range(m):
        for j in range(m):
            v = dot(A[:, i], A[:, j])
            bound = gram_bound(A[:, i], A[:, j], v) + 2.0**-51 * (abs(v) + abs(C[i, j]))
            assert abs(G[i, j] - (v + 0.5 * C[i, j])) <= bound, (i, j)


def update(lib, A, Bm, alpha=1.0, beta=0.0, C=None, upper=False):
    """alpha A B + beta C, A and C row-major, B column-major."""
    M, K = A.shape
    N = Bm.shape[1]
    a, b = padded(A), padded(np.ascontiguousarray(Bm.T))
    c = torch.full((M, N + 1), float("nan"), dtype=torch.float64, device="cuda")
    c[:, :N] = 7.0 if C is None else torch.from_numpy(C).cuda()
    w = torch.empty(lib._ZN3pfe18digit_update_bytesElii(M, N, K), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    lib._ZN3pfe20launch_update_digitsEliiPKdlS1_lddPdlbPvP11CUstream_st(
        M, N, K, a.data_ptr(), a.stride(0), b.data_ptr(), b.stride(0), alpha, beta, c.data_ptr(), N + 1, upper,
        w.data_ptr(), None)
    torch.cuda.synchronize()
    assert c[:, N:].isnan().all()
    return c[:, :N].cpu().numpy()


# rows around a tile and beyond a slab (37,376 rows at 128 columns), columns around a tile, an upper triangular B
@pytest.mark.parametrize("kind", ["normal", "localised", "magnitudes"])
@pytest.mark.parametrize("M,N,K,upper", [(1, 1, 1, False), (127, 63, 31, False), (130, 65, 129, False),
                                         (500, 200, 200, True), (40000, 70, 100, False), (3000, 129, 70, True)])
def test_update_within_the_bound(lib, M, N, K, upper, kind):
    rng = np.random.default_rng(8)
    A = block(kind, M, K, 9) if kind != "localised" or M >= K else block("normal", M, K, 9)
    scale = above(np.abs(A).max(0))
    Bm = rng.standard_normal((K, N)) / scale[:, None]  # as R^-1 undoes the columns' magnitudes
    if upper:
        Bm = np.triu(Bm)
    C = rng.standard_normal((M, N))
    Y = update(lib, A, Bm, alpha=-1.0, beta=1.0, C=C, upper=upper)
    for i, j in {(0, 0), (M - 1, N - 1), *map(tuple, rng.integers(0, (M, N), (16, 2)))}:
        v = dot(A[i], Bm[:, j])
        bound = gram_bound(A[i] / scale, Bm[:, j] * scale, v)
        assert abs(Y[i, j] - (C[i, j] - v)) <= bound + 2.0**-52 * (abs(v) + abs(C[i, j])), (i, j)
