"""Batches whose samples iterate on their own streams (fixed-point filter), and in the shared FP64 launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import glassgen  # noqa: E402
import oracle  # noqa: E402
import paper_1902_07041_gb300 as pfe  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    pfe.load()


@pytest.mark.parametrize("shape", [-1, 7])  # every sample on its own stream; all in the batched FP64 launches
def test_batch_on_own_streams_and_in_shared_launches(shape):
    gs = [glassgen.generate(n, 60 + i) for i, n in enumerate((210, 95, 260))]
    ctxs = []
    try:
        for g in gs:
            rp, ci, vals = pfe.pfe_springs_to_bsr(g.n_atoms, g.bi, g.bj, g.k, g.rhat)
            ctxs.append(pfe.pfe_create(g.n_atoms, rp, ci, vals, g.mass))
            lmax, _ = pfe.pfe_estimate(ctxs[-1])
            pfe.pfe_set_interval(ctxs[-1], 0.05 * lmax, 0.14 * lmax)
        pfe.pfe_set_param(ctxs[0], pfe.PFE_P_STEP_SHAPE_F64, shape)
        found, status = pfe.pfe_solve_batch(ctxs)
        assert status == pfe.PFE_OK
        for g, ctx, nf in zip(gs, ctxs, found):
            lam, V, _ = pfe.pfe_get_eigenpairs(ctx, g.n, nf)
            stats = pfe.pfe_get_stats(ctx)
            lmax = stats["lambda_max"]
            H = oracle.csr_from_springs(g)
            w, _, _ = oracle.exact_interval(H, 0.05 * lmax, 0.14 * lmax)
            assert nf == w.size and np.allclose(lam, w, rtol=1e-10, atol=0)
            assert np.all(oracle.residuals(H, lam, V) <= 1e-8 * lmax)
            assert stats["batch_replays"] >= stats["iterations"] and stats["seconds_filter"] > 0.0
    finally:
        pfe.pfe_set_param(ctxs[0], pfe.PFE_P_STEP_SHAPE_F64, -1)
        for c in ctxs:
            pfe.pfe_destroy(c)
