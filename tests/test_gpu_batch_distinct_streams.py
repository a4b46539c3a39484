"""Batches of contexts that were each created on a stream of their own, and all on one such stream.  (A context that is
created without a stream uses the legacy default stream: samples of that kind share it.)"""
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


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("method,precision,shape", [(0, 0, -1), (0, 2, -1), (1, 0, -1), (0, 0, 7)])
def test_batch_on_distinct_and_on_one_stream(method, precision, shape, shared):
    gs = [glassgen.generate(n, 70 + i) for i, n in enumerate((210, 95, 260, 150))]
    streams = [torch.cuda.Stream() for _ in range(1 if shared else len(gs))] * (len(gs) if shared else 1)
    ctxs = []
    try:
        for g, s in zip(gs, streams):
            rp, ci, vals = pfe.pfe_springs_to_bsr(g.n_atoms, g.bi, g.bj, g.k, g.rhat)
            ctxs.append(pfe.pfe_create(g.n_atoms, rp, ci, vals, g.mass, stream=s))
            pfe.pfe_set_param(ctxs[-1], pfe.PFE_P_METHOD, method)
            pfe.pfe_set_param(ctxs[-1], pfe.PFE_P_PRECISION, precision)
            lmax, _ = pfe.pfe_estimate(ctxs[-1])
            pfe.pfe_set_interval(ctxs[-1], 0.05 * lmax, 0.14 * lmax)
        pfe.pfe_set_param(ctxs[0], pfe.PFE_P_STEP_SHAPE_F64, shape)
        for _ in range(2):  # the second time with the buffers and operators of the first
            found, status = pfe.pfe_solve_batch(ctxs)
            assert status == pfe.PFE_OK
            for g, ctx, nf in zip(gs, ctxs, found):
                lam, V, _ = pfe.pfe_get_eigenpairs(ctx, g.n, nf)
                lmax = pfe.pfe_get_stats(ctx)["lambda_max"]
                H = oracle.csr_from_springs(g)
                w, _, _ = oracle.exact_interval(H, 0.05 * lmax, 0.14 * lmax)
                assert nf == w.size and np.allclose(lam, w, rtol=1e-10, atol=0)
                assert np.all(oracle.residuals(H, lam, V) <= 1e-8 * lmax)
    finally:
        pfe.pfe_set_param(ctxs[0], pfe.PFE_P_STEP_SHAPE_F64, -1)
        for c in ctxs:
            pfe.pfe_destroy(c)
