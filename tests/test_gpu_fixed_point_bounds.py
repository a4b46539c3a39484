"""The fixed-point filter and adjoint at the edges of what they take, against the FP64 kernels (a forced kernel shape).

Tolerance, as in the tests of the ordinary range: 60 m^2 2^-53 max_c |x_c|_2 sum|g| bounds the rounding of both sides.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import glassgen  # noqa: E402
import paper_1902_07041_gb300 as pfe  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    pfe.load()


def tolerance(X, coef):
    m, top = len(coef) - 1, np.abs(X).max()  # the norm of X / top: the squares of very small entries are 0
    return 60.0 * m * m * 2.0**-53 * top * np.linalg.norm(X / top, axis=0).max() * np.abs(coef).sum()


def context(g, lmax, rank1=1):
    rp, ci, vals = pfe.pfe_springs_to_bsr(g.n_atoms, g.bi, g.bj, g.k, g.rhat)
    ctx = pfe.pfe_create(g.n_atoms, rp, ci, vals, g.mass)
    pfe.pfe_set_param(ctx, pfe.PFE_P_LAMBDA_MAX, lmax)
    pfe.pfe_set_param(ctx, pfe.PFE_P_RANK1, rank1)
    return ctx, ci.size


def adjoint(ctx, nnzb, coef, X, Yb, shape):
    """Xbar and vals_bar with the automatic kernels (shape -1) or a forced shape."""
    n, k = X.shape
    Xd, Yd = (torch.from_numpy(np.ascontiguousarray(v.T)).cuda() for v in (X, Yb))
    Xb, vb = torch.empty_like(Xd), torch.empty(9 * nnzb, dtype=torch.float64, device="cuda")
    pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, shape)
    try:
        pfe.pfe_filter_adjoint(ctx, len(coef) - 1, np.array(coef), k, Xd, n, Yd, n, Xb, n, vb)
        torch.cuda.synchronize()
    finally:
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
    return Xb.cpu().numpy().T, vb.cpu().numpy()


def heat(t, m):
    """Chebyshev coefficients of exp(-t (1 + x)), down to the smallest numbers."""
    def bessel(j):
        return sum((t / 2.0) ** (2 * q + j) / (math.factorial(q) * math.factorial(q + j)) for q in range(12))
    return [(2.0 if j else 1.0) * (-1.0) ** j * math.exp(-t) * bessel(j) for j in range(m + 1)]


# a last coefficient far below the others, by hand and in a converged series; small ones among zeros; growing ones
@pytest.mark.parametrize("rank1", [1, 0])
@pytest.mark.parametrize("coef", [[0.5, 0.25, -0.3, 0.2, 1e-28], [0.5, 0.25, -0.3, 0.2, 1e-60],
                                  [0.5, 0.25, -0.3, 0.2, 1e-280], [0.0, 0.3, 0.0, 1e-70, 0.0, 1e-200],
                                  [1e-200, 1e-100, 1e-30, 1.0, 0.5], [1e-40, 0.5, 1e-40, 0.2, 1e-40],
                                  heat(0.1, 60), heat(0.02, 30)])
def test_adjoint_with_coefficients_of_very_different_size(coef, rank1):
    g = glassgen.generate(150, 9)
    ctx, nnzb = context(g, 0.25, rank1)
    try:
        rng = np.random.default_rng(5)
        X, Yb = rng.standard_normal((g.n, 6)), rng.standard_normal((g.n, 6))
        Yb[:, 3] *= 1e-200
        Yb[4, 4] = np.inf
        Yb[5, 5] = np.nan
        (Xb, vb), (Xr, vr) = (adjoint(ctx, nnzb, coef, X, Yb, s) for s in (-1, 7 if rank1 else 0))
        assert np.array_equal(np.isnan(Xb), np.isnan(Xr)) and np.array_equal(np.isinf(Xb), np.isinf(Xr))
        for c in range(4):
            assert np.max(np.abs(Xb[:, c] - Xr[:, c])) <= tolerance(Yb[:, [c]], coef), c
        (Xb, vb), (Xr, vr) = (adjoint(ctx, nnzb, coef, X[:, :4], Yb[:, :4], s) for s in (-1, 7 if rank1 else 0))
        assert np.max(np.abs(vb - vr)) <= 2.0 / 0.125 * 4 * tolerance(Yb[:, :4], coef) * np.linalg.norm(X, axis=0).max()
    finally:
        pfe.pfe_destroy(ctx)


def bonds_context(n, bi, bj, k, rhat, lmax):
    rp, ci, vals = pfe.pfe_springs_to_bsr(n, np.array(bi, np.int32), np.array(bj, np.int32), np.array(k, float),
                                          np.array(rhat, float))
    ctx = pfe.pfe_create(n, rp, ci, vals, np.ones(n))
    pfe.pfe_set_param(ctx, pfe.PFE_P_LAMBDA_MAX, lmax)
    return ctx


def apply(ctx, coef, X, shape=-1):
    n, k = X.shape
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    Yd = torch.full((k, n), float("nan"), device="cuda", dtype=torch.float64)
    pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, shape)
    try:
        pfe.pfe_filter_apply(ctx, len(coef) - 1, np.array(coef), k, Xd, n, Yd, n, pfe.PFE_F64)
        torch.cuda.synchronize()
    finally:
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
    return Yd.cpu().numpy().T


D = np.ones(3) / np.sqrt(3.0)


# bonds along the diagonals of the axes whose u has |u|_1 = 4.2 (one bond), and two of them in a row of three atoms
@pytest.mark.parametrize("bonds", [([0], [1], [D]), ([0, 0], [1, 2], [D, np.array([1, -1, 0]) / np.sqrt(2)])])
def test_filter_with_a_stiff_bond_far_above_the_bound(bonds):
    """A bound about three times below the spectrum: the operator's entries pass what the products of the fixed-point
    form hold, and the vectors grow, in the FP64 kernels' way.  The difference is relative to the result."""
    bi, bj, rhat = bonds
    n, u = max(bj) + 1, 1.41 * np.sqrt(3.0)
    k = [u * u / 4.0] + [1.4 * 1.4 * 2 / 4.0] * (len(bi) - 1)  # u_r = sqrt(4 k / bound) r
    ctx = bonds_context(n, bi, bj, k, rhat, 1.0)
    try:
        rng = np.random.default_rng(1)
        X = rng.standard_normal((3 * n, 16))
        for m in (12, 40, 41):
            coef = np.ones(m + 1)
            Y, R = apply(ctx, coef, X), apply(ctx, coef, X, 7)
            err = np.linalg.norm(Y - R, axis=0) / np.linalg.norm(R, axis=0)
            assert err.max() <= 60.0 * m * m * 2.0**-53
    finally:
        pfe.pfe_destroy(ctx)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("at", [0, 2, 4])
def test_adjoint_carries_a_non_finite_coefficient(bad, at):
    """The adjoint does not refuse one: its results are not finite, as the FP64 kernels' are."""
    g = glassgen.generate(100, 9)
    ctx, nnzb = context(g, 0.25)
    try:
        coef = [0.5, 0.25, -0.3, 0.2, 0.1]
        coef[at] = bad
        rng = np.random.default_rng(5)
        X, Yb = rng.standard_normal((g.n, 3)), rng.standard_normal((g.n, 3))
        (Xb, vb), (Xr, vr) = (adjoint(ctx, nnzb, coef, X, Yb, s) for s in (-1, 7))
        assert not np.isfinite(Xr).any()
        assert np.array_equal(np.isnan(Xb), np.isnan(Xr)) and np.array_equal(np.isnan(vb), np.isnan(vr))
    finally:
        pfe.pfe_destroy(ctx)


def test_calls_in_flight_on_another_stream_keep_their_operator():
    """Filters on a caller's stream, queued behind one another, with calls in between that use the other form of the
    operator or build its FP32 copy: each result is that of the same call made alone."""
    g = glassgen.generate(8000, 3)
    m, k, n = 150, 32, g.n
    coef = np.cos(np.arange(m + 1.0)) / (1.0 + np.arange(m + 1.0))
    X = torch.randn(k, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    X32 = X.float()

    def calls(ctx, stream, wait):
        out = []
        for rank1, x in ((1, X), (1, X32), (1, X), (0, X), (1, X), (0, X)):
            pfe.pfe_set_param(ctx, pfe.PFE_P_RANK1, rank1)
            out.append(torch.empty_like(x))
            pfe.pfe_filter_apply(ctx, m, coef, k, x, n, out[-1], n, pfe.PFE_F32 if x is X32 else pfe.PFE_F64, stream=stream)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return out

    side = torch.cuda.Stream()
    ctxs = [context(g, 0.25)[0] for _ in range(2)]
    try:
        torch.cuda.synchronize()
        alone, queued = calls(ctxs[0], side, True), calls(ctxs[1], side, False)
        assert all(torch.equal(a, b) for a, b in zip(alone, queued))
    finally:
        for c in ctxs:
            pfe.pfe_destroy(c)


def test_no_room_for_the_fixed_operator():
    """Without device memory for the fixed-point operator the filter runs in FP64, as it did."""
    g = glassgen.generate(60000, 9)
    ctx, nnzb = context(g, 0.25)
    try:
        X = torch.randn(2, g.n, dtype=torch.float64, device="cuda")
        Y, R = torch.empty_like(X), torch.empty_like(X)
        coef = np.array([0.5, 0.25, -0.3, 0.2, 0.1])
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, 7)
        pfe.pfe_filter_apply(ctx, 4, coef, 2, X, g.n, R, g.n, pfe.PFE_F64)  # builds the operator, reserves the buffers
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
        torch.cuda.synchronize()
        hold = []
        size = 1 << 36
        while size >= 1 << 22:
            try:
                hold.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            except torch.OutOfMemoryError:
                size >>= 1
        try:
            pfe.pfe_filter_apply(ctx, 4, coef, 2, X, g.n, Y, g.n, pfe.PFE_F64)
            torch.cuda.synchronize()
        finally:
            del hold
            torch.cuda.empty_cache()
        assert (Y - R).abs().max() <= tolerance(X.cpu().numpy().T, coef)
        pfe.pfe_filter_apply(ctx, 4, coef, 2, X, g.n, Y, g.n, pfe.PFE_F64)  # with the memory back: in fixed point
        torch.cuda.synchronize()
        assert not torch.equal(Y, R)
        assert (Y - R).abs().max() <= tolerance(X.cpu().numpy().T, coef)
    finally:
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
        pfe.pfe_destroy(ctx)


@pytest.mark.parametrize("x,g", [(1e-260, 1e-40), (1e-230, 1e-60), (1.0, 1e-300), (1e-200, 1e-90)])
def test_filter_and_adjoint_keep_tiny_results(x, g):
    net = glassgen.generate(100, 9)
    ctx, nnzb = context(net, 0.25)
    try:
        coef = g * np.array([0.5, 0.25, -0.3, 0.2, 0.1])
        rng = np.random.default_rng(5)
        X, Yb = rng.standard_normal((net.n, 3)), x * rng.standard_normal((net.n, 3))
        Y, R = apply(ctx, coef, Yb), apply(ctx, coef, Yb, 7)
        assert np.abs(R).max() > 0
        (Xb, vb), (Xr, vr) = (adjoint(ctx, nnzb, coef, X, Yb, s) for s in (-1, 7))
        assert np.abs(Y - R).max() <= 1e-12 * np.abs(R).max()
        assert np.abs(Xb - Xr).max() <= 1e-12 * np.abs(Xr).max()
        assert np.abs(vb - vr).max() <= 1e-11 * np.abs(vr).max()
    finally:
        pfe.pfe_destroy(ctx)


def device_adjoint(ctx, nnzb, coef, X, Yb):
    k, n = X.shape
    Xb, vb = torch.empty_like(X), torch.empty(9 * nnzb, dtype=torch.float64, device="cuda")
    pfe.pfe_filter_adjoint(ctx, len(coef) - 1, coef, k, X, n, Yb, n, Xb, n, vb)
    torch.cuda.synchronize()
    return Xb, vb


def test_adjoint_keeps_at_most_a_64th_of_the_device():
    """200 steps of 64 columns keep 12 GB of vectors: more than a 64th of the device, so they are run in segments."""
    g = glassgen.generate(20000, 9)
    ctx, nnzb = context(g, 0.25)
    try:
        k, m = 64, 200
        gen = torch.Generator("cuda").manual_seed(6)
        X, Yb = (torch.randn(k, g.n, dtype=torch.float64, device="cuda", generator=gen) for _ in range(2))
        coef = np.cos(np.arange(m + 1.0)) / (1.0 + np.arange(m + 1.0))
        torch.cuda.synchronize()
        free, total = torch.cuda.mem_get_info()
        Xb, vb = device_adjoint(ctx, nnzb, coef, X, Yb)
        taken = free - torch.cuda.mem_get_info()[0]
        assert taken <= total / 64 + 2**29  # and the operator, Xbar and the gradient
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, 7)
        Xr, vr = device_adjoint(ctx, nnzb, coef, X, Yb)
        tol = tolerance(Yb.cpu().numpy().T, coef)
        assert (Xb - Xr).abs().max() <= tol
        assert (vb - vr).abs().max() <= 2.0 / 0.125 * k * tol * X.norm(dim=1).max().item()
    finally:
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
        pfe.pfe_destroy(ctx)


# segments of one step to several, a short last one, one saved pair to many
@pytest.mark.parametrize("rank1", [1, 0])
@pytest.mark.parametrize("m", [2, 3, 5, 10, 30])
def test_adjoint_in_segments_gives_the_bits_of_one_segment(m, rank1):
    """On a device nearly full the vectors are recomputed from saved pairs: the same vectors, so the same Xbar."""
    g = glassgen.generate(8000, 9)
    ctxs = [context(g, 0.25, rank1) for _ in range(2)]
    hold = None
    try:
        k = 63
        gen = torch.Generator("cuda").manual_seed(6)
        X, Yb = (torch.randn(k, g.n, dtype=torch.float64, device="cuda", generator=gen) for _ in range(2))
        X[5] *= 1e-290  # kept in FP64
        coef = np.cos(np.arange(m + 1.0)) / (1.0 + np.arange(m + 1.0))
        ref = device_adjoint(*ctxs[0], coef, X, Yb)
        small = device_adjoint(*ctxs[1], coef[:2], X[:1], Yb[:1])  # the operator is built
        torch.cuda.empty_cache()
        least = int(np.ceil(np.sqrt(m)))
        room = 8 * g.n * 64 * (2 * least + 2 * -(-m // least) + 5) + 2**27
        hold = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        got = device_adjoint(*ctxs[1], coef, X, Yb)
        assert small[0].isfinite().all() and torch.equal(got[0], ref[0])
        assert (got[1] - ref[1]).abs().max() <= 1e-13 * ref[1].abs().max()  # sums over segments in another order
    finally:
        del hold
        torch.cuda.empty_cache()
        for c, _ in ctxs:
            pfe.pfe_destroy(c)


# rows around the 12 (rank-1) and 16 (full) blocks that a pass over the operator takes, and several passes
@pytest.mark.parametrize("rank1,shape", [(1, 7), (0, 0)])
@pytest.mark.parametrize("n", [2, 12, 13, 14, 17, 18, 40])
def test_springs_between_all_pairs(n, rank1, shape):
    rng = np.random.default_rng(n)
    bi, bj = np.triu_indices(n, 1)
    r = rng.standard_normal((bi.size, 3))
    ctx = bonds_context(n, bi, bj, 1.0 + rng.random(bi.size), r / np.linalg.norm(r, axis=1)[:, None], 0.0)
    try:
        pfe.pfe_set_param(ctx, pfe.PFE_P_RANK1, rank1)
        coef = np.cos(np.arange(8)) / (1.0 + np.arange(8))
        X = rng.standard_normal((3 * n, 5))
        Y, R = apply(ctx, coef, X), apply(ctx, coef, X, shape)
        assert np.max(np.abs(Y - R)) <= tolerance(X, coef)
        assert np.any(Y != R)  # rounded differently: the fixed-point form ran
    finally:
        pfe.pfe_destroy(ctx)


def test_solves_with_a_row_too_long_for_the_fixed_point_step():
    """An atom with 790 weak springs: its row does not fit a CTA's shared memory.  Alone and in a batch beside a network
    that fits, the solves take the FP64 kernels for it and find what LAPACK finds."""
    g = glassgen.generate(800, 12)
    rng = np.random.default_rng(1)
    near = set(g.bj[g.bi == 0]) | set(g.bi[g.bj == 0])
    far = np.array([j for j in range(1, 800) if j not in near], np.int32)
    r = rng.standard_normal((far.size, 3))
    bi, bj = np.r_[g.bi, np.zeros_like(far)], np.r_[g.bj, far]
    ks = np.r_[g.k, 1e-4 * g.k.mean() * np.ones(far.size)]
    rhat = np.r_[g.rhat, r / np.linalg.norm(r, axis=1)[:, None]]
    nets = [(bi, bj, ks, rhat), (g.bi, g.bj, g.k, g.rhat)]
    ctxs = []
    try:
        exact = []
        for t in nets:
            rp, ci, vals = pfe.pfe_springs_to_bsr(800, *t)
            ctxs.append(pfe.pfe_create(800, rp, ci, vals, g.mass))
            H = np.zeros((2400, 2400))
            for i in range(800):
                for p in range(rp[i], rp[i + 1]):
                    blk = vals[9 * p:9 * p + 9].reshape(3, 3) / np.sqrt(g.mass[i] * g.mass[ci[p]])
                    H[3 * i:3 * i + 3, 3 * ci[p]:3 * ci[p] + 3] = blk
            w = np.linalg.eigvalsh(H)
            a, b = 0.5 * (w[40] + w[41]), 0.5 * (w[80] + w[81])
            pfe.pfe_set_interval(ctxs[-1], a, b)
            exact.append(w[41:81])
        assert np.diff(pfe.pfe_springs_to_bsr(800, *nets[0])[0]).max() - 1 > 768
        for batch in (False, True):
            if batch:
                found, status = pfe.pfe_solve_batch(ctxs)
                assert status == pfe.PFE_OK
            else:
                found = [pfe.pfe_solve(c)[0] for c in ctxs]
                shapes = [pfe.pfe_get_stats(c)["filter_shape_f64"] for c in ctxs]
                assert shapes[0] != 12 and shapes[1] == 12
            for c, nf, w in zip(ctxs, found, exact):
                lam, _, _ = pfe.pfe_get_eigenpairs(c, 2400, nf)
                assert nf == 40 and np.allclose(lam, w, rtol=1e-10, atol=0)
    finally:
        for c in ctxs:
            pfe.pfe_destroy(c)
