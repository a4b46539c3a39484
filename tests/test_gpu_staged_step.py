"""The FP32 step with staged blocks (the automatic kernel of the rank-1 form).

The staged step adds a row's terms in the order of kernel shape 7, with the same fused multiply-adds, so the two
give the same bits.
"""
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


def network(N):
    """A glass, or for N < 100 springs between all pairs: rows too long for a CTA's shared memory."""
    if N >= 100:
        g = glassgen.generate(N, 31)
        return g.n_atoms, g.bi, g.bj, g.k, g.rhat, g.mass
    rng = np.random.default_rng(N)
    bi, bj = (v.astype(np.int32) for v in np.triu_indices(N, 1))
    r = rng.standard_normal((bi.size, 3))
    return N, bi, bj, 1.0 + rng.random(bi.size), r / np.linalg.norm(r, axis=1)[:, None], np.ones(N)


# columns: one, odd, a warp, pairs, four a lane, whole rows, two tiles of rows; degrees: every launch mode
@pytest.mark.parametrize("N,k,m", [(60, 1, 3), (60, 70, 4), (333, 7, 1), (333, 33, 2), (333, 64, 5), (1501, 1, 6),
                                   (1501, 45, 7), (1501, 128, 8), (1501, 133, 9), (4001, 260, 4),
                                   (300, 1030, 3), (61, 1024, 2)])
def test_staged_step_equals_shape_7(N, k, m):
    n_atoms, bi, bj, ks, rhat, mass = network(N)
    rp, ci, vals = pfe.pfe_springs_to_bsr(n_atoms, bi, bj, ks, rhat)
    ctx = pfe.pfe_create(n_atoms, rp, ci, vals, mass)
    try:
        lmax, _ = pfe.pfe_estimate(ctx)
        coef = np.cos(np.arange(m + 1)) / (1.0 + np.arange(m + 1))
        X = torch.randn(k, 3 * n_atoms, dtype=torch.float32, device="cuda", generator=torch.Generator("cuda").manual_seed(k))
        got = []
        for shape in (-1, 7):
            Y = torch.full_like(X, float("nan"))
            pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F32, shape)
            pfe.pfe_filter_apply(ctx, m, coef, k, X, 3 * n_atoms, Y, 3 * n_atoms, pfe.PFE_F32)
            torch.cuda.synchronize()
            got.append(Y)
        assert lmax > 0.0 and torch.isfinite(got[0]).all() and torch.equal(got[0], got[1])
    finally:
        pfe.pfe_set_param(ctx, pfe.PFE_P_STEP_SHAPE_F32, -1)
        pfe.pfe_destroy(ctx)
