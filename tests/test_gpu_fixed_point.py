"""The FP64 filter in 64-bit fixed point (the automatic kernel) against the oracle and the FP64 kernels.

Tolerances, from the arithmetic.  A step rounds each entry by at most about 2 units (a half for the sum, a
quarter per dropped low product, a half per rank-1 product times its factor), a unit is at most
2^-60 (||A||_inf + 1) of the column's largest entry < 2^-57 for these networks, and errors of step j reach
y = sum g_j t_j with a factor of at most m - j + 1.  With the FP64 sums of the other side (2^-53 a rounding, up
to 40 a row) a difference of 60 m^2 2^-53 max|t| sum|g| covers both; max|t| <= ||x||_2 bounds every t_j.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import glassgen  # noqa: E402
import oracle  # noqa: E402
import paper_1902_07041_gb300 as pfe  # noqa: E402

pytestmark = pytest.mark.gpu
FIXED = 12  # the fixed-point kernel among the kernel shapes that pfe_get_stats reports


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    pfe.load()


def tolerance(X, coef):
    m = len(coef) - 1
    return 60.0 * m * m * 2.0**-53 * np.linalg.norm(X, axis=0).max() * np.abs(coef).sum()


def context(g, lmax, rank1=1, tension=0.0):
    rp, ci, vals = pfe.pfe_springs_to_bsr(g.n_atoms, g.bi, g.bj, g.k, g.rhat)
    if tension:  # transverse terms: no rank-1 form
        t_rp, t_ci, t_vals = rp, ci, vals.reshape(-1, 3, 3).copy()
        rows = np.repeat(np.arange(g.n_atoms), np.diff(t_rp))
        off = rows != t_ci
        extra = np.zeros_like(t_vals)
        extra[off] = -tension * np.eye(3)
        np.add.at(extra, np.flatnonzero(~off)[rows[off]], tension * np.eye(3))
        vals = (t_vals + extra).reshape(-1)
    ctx = pfe.pfe_create(g.n_atoms, rp, ci, vals, g.mass)
    pfe.pfe_set_param(ctx, pfe.PFE_P_LAMBDA_MAX, lmax)
    pfe.pfe_set_param(ctx, pfe.PFE_P_RANK1, rank1)
    return ctx


def apply(ctx, coef, X, ldx=None, shape=-1):
    n, k = X.shape
    ldx = ldx or n
    Xd = torch.full((k, ldx), float("nan"), dtype=torch.float64)
    Xd[:, :n] = torch.from_numpy(np.ascontiguousarray(X.T))
    Xd = Xd.cuda()
    Yd = torch.full((k, n), float("nan"), device="cuda", dtype=torch.float64)
    pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, shape)
    try:
        pfe.pfe_filter_apply(ctx, len(coef) - 1, coef, k, Xd, ldx, Yd, n, pfe.PFE_F64)
        torch.cuda.synchronize()
    finally:
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
    return Yd.cpu().numpy().T


# columns: one, a pair, odd, one more than a CTA's lanes, two column tiles; atoms: a few, a ragged last CTA, enough
# for two columns a lane and several passes; degrees: first step only, first and last, odd and even ends
@pytest.mark.parametrize("rank1", [1, 0])
@pytest.mark.parametrize("N,k,m", [(60, 1, 1), (61, 2, 2), (333, 3, 5), (500, 33, 8), (300, 257, 7), (300, 1030, 6),
                                   (4001, 64, 9), (4001, 65, 4)])
def test_fixed_point_filter_matches_oracle(N, k, m, rank1):
    g = glassgen.generate(N, 21)
    ctx = context(g, 0.25, rank1)
    try:
        coef = np.cos(np.arange(m + 1)) / (1.0 + np.arange(m + 1))
        X = np.random.default_rng(N + k).standard_normal((g.n, k))
        Y = apply(ctx, coef, X, ldx=g.n + 5)
        ref = oracle.cheb_filter(oracle.csr_from_springs(g), 0.125, 0.125, coef, X)
        assert np.max(np.abs(Y - ref)) <= tolerance(X, coef)
    finally:
        pfe.pfe_destroy(ctx)


@pytest.mark.parametrize("rank1,tension", [(1, 0.0), (0, 0.0), (1, 0.05)])
def test_fixed_point_filter_on_unusual_columns(rank1, tension):
    """Zero columns, columns of very different magnitude, a single atom, Inf and NaN, beside ordinary ones."""
    g = glassgen.generate(700, 3)
    ctx = context(g, 0.3, rank1, tension)
    try:
        coef = np.array([0.3, -0.2, 0.5, 0.1, -0.4, 0.05, 0.2, 0.3])
        X = np.random.default_rng(8).standard_normal((g.n, 12))
        X[:, 1] = 0.0
        X[:, 2] *= 1e-290
        X[:, 3] *= 1e280
        X[:, 4] = 0.0
        X[7, 4] = 1.0
        X[:, 5] *= 1e-150
        X[11, 6] = np.nan
        X[12, 8] = np.inf
        X[:, 10] *= 5e-324
        Y, R = apply(ctx, coef, X), apply(ctx, coef, X, shape=7 if rank1 and not tension else 0)
        assert np.array_equal(np.isnan(Y), np.isnan(R))
        assert np.array_equal(np.isinf(Y), np.isinf(R))
        assert not Y[:, 1].any()
        for c in (0, 2, 3, 4, 5, 7, 9, 11):
            scale = np.abs(X[:, c]).max() * np.sqrt(g.n)
            assert np.max(np.abs(Y[:, c] - R[:, c]) / scale) <= tolerance(X[:, [0]], coef), c
    finally:
        pfe.pfe_destroy(ctx)


@pytest.mark.parametrize("rank1", [1, 0])
def test_fixed_point_filter_rescales_growing_vectors(rank1):
    """A bound below the spectrum: the Chebyshev vectors grow far beyond 60 bits and follow the FP64 kernels.  The
    growth amplifies rounding as it does the vector itself, so the difference is relative to the result: the step
    tolerance of the module, m^2 60 2^-53, with the growth of the early errors inside it."""
    g = glassgen.generate(500, 4)
    ctx = context(g, 0.92 * np.linalg.eigvalsh(oracle.csr_from_springs(g).dense())[-1], rank1)
    try:
        m = 120
        coef = np.ones(m + 1)
        X = np.random.default_rng(2).standard_normal((g.n, 6))
        Y, R = apply(ctx, coef, X), apply(ctx, coef, X, shape=7 if rank1 else 0)
        assert np.abs(R).max() > 2.0**64
        err = np.linalg.norm(Y - R, axis=0) / np.linalg.norm(R, axis=0)
        assert err.max() <= 60.0 * m * m * 2.0**-53
    finally:
        pfe.pfe_destroy(ctx)


def test_atoms_without_neighbours_and_stiff_bonds():
    """A bond far stiffer than the others along (1, 1, 1) (|u|_1 near its bound) and an atom without bonds (a diagonal
    entry of exactly -2): both still fit."""
    g = glassgen.generate(300, 4)
    keep = (g.bi != 17) & (g.bj != 17)
    bi, bj, k, rhat = g.bi[keep], g.bj[keep], g.k[keep].copy(), g.rhat[keep].copy()
    k[40], rhat[40] = 60.0, np.ones(3) / np.sqrt(3.0)
    rp, ci, vals = pfe.pfe_springs_to_bsr(g.n_atoms, bi, bj, k, rhat)
    H = np.zeros((g.n, g.n))
    for i in range(g.n_atoms):
        for p in range(rp[i], rp[i + 1]):
            H[3 * i:3 * i + 3, 3 * ci[p]:3 * ci[p] + 3] = vals[9 * p:9 * p + 9].reshape(3, 3) / np.sqrt(g.mass[i] * g.mass[ci[p]])
    lmax = 1.0001 * np.linalg.eigvalsh(H)[-1]
    ctx = pfe.pfe_create(g.n_atoms, rp, ci, vals, g.mass)
    pfe.pfe_set_param(ctx, pfe.PFE_P_LAMBDA_MAX, lmax)
    try:
        coef = np.array([0.1, 0.2, -0.3, 0.4, 0.5, -0.1])
        X = np.random.default_rng(5).standard_normal((g.n, 7))
        Y = apply(ctx, coef, X)
        T = [X, 2.0 / lmax * (H @ X) - X]
        for _ in coef[2:]:
            T.append(2.0 * (2.0 / lmax * (H @ T[-1]) - T[-1]) - T[-2])
        ref = sum(c * t for c, t in zip(coef, T))
        assert np.max(np.abs(Y - ref)) <= tolerance(X, coef)
        Y2 = apply(ctx, coef, X, shape=7)
        assert np.any(Y != Y2)  # the two kernels round differently: the fixed-point one ran
    finally:
        pfe.pfe_destroy(ctx)


def test_operator_that_does_not_fit_runs_in_fp64():
    """An operator with entries beyond the fixed-point range (a bound far below the spectrum) keeps the FP64 kernels."""
    g = glassgen.generate(200, 4)
    ctx = context(g, 0.01)
    try:
        coef = np.array([0.5, 0.25, 0.125])
        X = np.random.default_rng(1).standard_normal((g.n, 4))
        Y, R = apply(ctx, coef, X), apply(ctx, coef, X, shape=7)
        assert np.allclose(Y, R, rtol=1e-12, atol=0)
    finally:
        pfe.pfe_destroy(ctx)


def test_solver_reports_the_fixed_point_kernel():
    g = glassgen.generate(600, 2)
    ctx = context(g, 0.0)
    try:
        lmax, _ = pfe.pfe_estimate(ctx)
        pfe.pfe_set_interval(ctx, 0.03 * lmax, 0.05 * lmax)
        pfe.pfe_solve(ctx)
        assert pfe.pfe_get_stats(ctx)["filter_shape_f64"] == FIXED
    finally:
        pfe.pfe_destroy(ctx)


# ------------------------------------------------------------------ dense products by exact digits
@pytest.mark.parametrize("width", [48, 63, 64, 65, 127, 128, 129, 200])
def test_solve_at_widths_around_the_product_tiles(width):
    """The Gram matrices, projections and block updates of a solve at block widths around the 64 and 128 column
    tiles: eigenvalues of LAPACK to 1e-10, eigenvectors orthonormal to 1e-12 (a sum of n exact products rounded
    once, 2^-53, with room for the n = 1,200 of the vectors' own rounding), residuals as the tolerance asks."""
    g = glassgen.generate(400, 6)
    ctx = context(g, 0.0)
    try:
        H = oracle.csr_from_springs(g)
        w = np.linalg.eigvalsh(H.dense())
        lmax, _ = pfe.pfe_estimate(ctx)
        a, b = 0.5 * (w[9] + w[10]), 0.5 * (w[39] + w[40])
        pfe.pfe_set_interval(ctx, a, b)
        pfe.pfe_set_param(ctx, pfe.PFE_P_WIDTH, width)
        nf, _ = pfe.pfe_solve(ctx)
        lam, vecs, _ = pfe.pfe_get_eigenpairs(ctx, g.n, nf)
        assert nf == 30
        assert np.allclose(lam, w[10:40], rtol=1e-10, atol=0)
        assert np.max(np.abs(vecs.T @ vecs - np.eye(nf))) <= 1e-12
        assert np.all(oracle.residuals(H, lam, vecs) <= 1e-8 * lmax)
    finally:
        pfe.pfe_destroy(ctx)


# ------------------------------------------------------------------ the adjoint
@pytest.mark.parametrize("rank1", [1, 0])
@pytest.mark.parametrize("N,k,coef", [(60, 1, [0.5, 0.25]), (61, 2, [0.5, 0.25, 1e-17]), (333, 5, [0.0, 0.3, -0.2, 0.1, 0.0]),
                                      (300, 129, [1e-9, 2e-9, -3e-9, 1e-9]), (4001, 52, [0.1, -0.4, 0.3, 0.2, 0.05, 1e-3])])
def test_fixed_point_adjoint_matches_the_checkpointed_one(N, k, coef, rank1):
    """The adjoint that keeps every vector, in fixed point, against the FP64 kernels with checkpoints (a forced kernel
    shape): one step to several, odd and single columns, a last coefficient of 0 or far below the others, columns of
    0, Inf and very small entries beside ordinary ones.  Tolerance as for the filter, with the products' sums of k m
    terms beside it."""
    g = glassgen.generate(N, 9)
    ctx = context(g, 0.25, rank1)
    try:
        coef = np.array(coef)
        m = coef.size - 1
        rng = np.random.default_rng(N)
        X, Yb = rng.standard_normal((g.n, k)), rng.standard_normal((g.n, k))
        if k > 4:
            X[:, 1] = 0.0
            Yb[:, 2] = 0.0
            Yb[:, 3] *= 1e-295
        rp, ci, _ = pfe.pfe_springs_to_bsr(g.n_atoms, g.bi, g.bj, g.k, g.rhat)
        got = []
        for shape in (-1, 7 if rank1 else 0):
            Xd, Yd = (torch.from_numpy(np.ascontiguousarray(v.T)).cuda() for v in (X, Yb))
            Xb, vb = torch.empty_like(Xd), torch.empty(9 * ci.size, dtype=torch.float64, device="cuda")
            pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, shape)
            pfe.pfe_filter_adjoint(ctx, m, coef, k, Xd, g.n, Yd, g.n, Xb, g.n, vb)
            torch.cuda.synchronize()
            pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
            got.append((Xb.cpu().numpy().T, vb.cpu().numpy()))
        tol = tolerance(Yb, coef)
        assert np.max(np.abs(got[0][0] - got[1][0])) <= tol
        assert np.max(np.abs(got[0][1] - got[1][1])) <= 2.0 / 0.125 * k * tol * np.linalg.norm(X, axis=0).max()
        if k > 4:
            assert not got[0][0][:, 2].any()
            small = got[1][0][:, 3]
            assert np.max(np.abs(got[0][0][:, 3] - small)) <= 1e-12 * np.abs(small).max()
    finally:
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F64, -1)
        pfe.pfe_destroy(ctx)


# two columns a lane, with an even and an odd number of columns
@pytest.mark.parametrize("rank1", [1, 0])
@pytest.mark.parametrize("k", [130, 131])
def test_two_columns_a_lane(k, rank1):
    g = glassgen.generate(4001, 22)
    ctx = context(g, 0.25, rank1)
    try:
        coef = np.cos(np.arange(6)) / (1.0 + np.arange(6))
        X = np.random.default_rng(k).standard_normal((g.n, k))
        ref = oracle.cheb_filter(oracle.csr_from_springs(g), 0.125, 0.125, coef, X)
        assert np.max(np.abs(apply(ctx, coef, X) - ref)) <= tolerance(X, coef)
        Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
        rp, ci, _ = pfe.pfe_springs_to_bsr(g.n_atoms, g.bi, g.bj, g.k, g.rhat)
        Xb, vb = torch.empty_like(Xd), torch.empty(9 * ci.size, dtype=torch.float64, device="cuda")
        pfe.pfe_filter_adjoint(ctx, 5, coef, k, Xd, g.n, Xd, g.n, Xb, g.n, vb)  # the filter is symmetric
        torch.cuda.synchronize()
        assert np.max(np.abs(Xb.cpu().numpy().T - ref)) <= tolerance(X, coef)
    finally:
        pfe.pfe_destroy(ctx)
