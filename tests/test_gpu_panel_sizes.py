"""Panels either side of the size from which a block prepares two phenotypes: the same phenotypes,
bit for bit, and the oracle's."""
import numpy as np
import pytest

import oracle
import paper_2604_21095_gb300 as tg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n_cov", [(1001, 12), (257, 0)])
def test_phenotypes_do_not_depend_on_the_panel_size(tgctx, N, n_cov):
    cov = synth.covariates(8, N, n_cov)
    Yt = synth.phenotypes(9, cov, 457)
    Yt[3] = 2.0  # a constant phenotype: no test
    got = {}
    for P in (1, 4, 456, 457):
        panel = tg.tg_prepare_panel(tgctx, Yt[:P].contiguous().cuda(), N, P,
                                    cov.cuda() if n_cov else None)
        try:
            Yres, s = tg.tg_panel_Yres(panel)
            got[P] = (Yres.cpu().numpy().copy(), s.cpu().numpy().copy())
        finally:
            tg.tg_panel_free(panel)
    for P in (1, 4, 456):
        assert np.array_equal(got[P][0], got[457][0][:P]), P
        assert np.array_equal(got[P][1], got[457][1][:P]), P
    ref = oracle.prepare_panel(Yt.numpy().T.astype(np.float64), cov.numpy().T if n_cov else None)
    scale = np.linalg.norm(ref["Y"] - ref["Y"].mean(0), axis=0).max()
    assert np.allclose(got[457][0].T, ref["Yres"], atol=1e-11 * scale, rtol=0)
