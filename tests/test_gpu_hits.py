"""The FP64 statistics of hits, whose blocks share the hits in two ways (one block per hit up to
8,192 samples, a cluster of blocks per hit above), with fewer and with more hits than clusters,
against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2604_21095_gb300 as tg
import synth
from scan_util import compare_hits, oracle_panel, run_scan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("encoding", ["2bit", "u8"])
@pytest.mark.parametrize("N,M,thr", [(8192, 300, 1.5), (8193, 300, 1.5), (8193, 300, 3.5),
                                     (16_001, 1200, 1.0)])
def test_hit_statistics_either_side_of_the_cluster_form(tgctx, encoding, N, M, thr):
    P = 40
    w = synth.Workload(f"hits_{N}_{M}_{encoding}", N=N, M=M, P=P, n_cov=3, encoding=encoding,
                       missing=0.01 if encoding == "2bit" else 0.0, seed=71, block=M,
                       causal_per_pheno=1)
    pan = synth.make_panel(w)
    blk = synth.make_block(w, 0)
    panel = tg.tg_prepare_panel(tgctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    try:
        res = run_scan(tgctx, panel, blk["G"].cuda(), N, P, encoding, "split", full=False,
                       hit_mlog10p=thr, marker_offset=9)
    finally:
        tg.tg_panel_free(panel)
    assert res["status"] == tg.TG_OK
    ref = oracle.scan(blk["G"].numpy(), encoding, oracle_panel(pan["Yt"], pan["cov_t"]))
    want, _ = compare_hits(res, ref, thr, marker_offset=9)
    assert (want > 200) == (thr < 3)
    # each hit's product is recomputed in FP64: its record is off by half of the marker norm's
    # relative error (norm2 is within 1e-6 of the oracle's in every form) and the rounding to FP32
    j, p = res["hits"]["marker"].astype(int) - 9, res["hits"]["pheno"].astype(int)
    np.testing.assert_allclose(res["hits"]["se"], ref["se"][j, p], rtol=1e-6)
    np.testing.assert_allclose(res["hits"]["t"], ref["t"][j, p], rtol=1e-6)


def test_many_hits_do_not_take_turns(tgctx):
    """Long sample axes share each of a few hits over a cluster of 8 blocks; with many hits every
    block takes its own. Clusters that took 4,800 hits in turn would need more than 60 times as
    long as for one hit each (76 clusters); blocks of their own need about a third of that."""
    N, M, P = 16_001, 1200, 40
    w = synth.Workload("hits_many", N=N, M=M, P=P, n_cov=3, encoding="2bit", missing=0.01, seed=71,
                       block=M, causal_per_pheno=1)
    pan = synth.make_panel(w)
    G = synth.make_block(w, 0)["G"].cuda()
    panel = tg.tg_prepare_panel(tgctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    ms, hits = {}, {}
    try:
        tg.tg_set_profiling(tgctx, True)
        for thr in (4.0, 1.0):
            ms[thr] = 1e9
            for _ in range(6):
                tg.tg_stage_times(tgctx, reset=True)
                hits[thr] = run_scan(tgctx, panel, G, N, P, "2bit", "split", full=False,
                                     hit_mlog10p=thr)["n_hits"]
                ms[thr] = min(ms[thr], tg.tg_stage_times(tgctx, reset=True)["stats"][0])
    finally:
        tg.tg_set_profiling(tgctx, False)
        tg.tg_panel_free(panel)
    assert 0 < hits[4.0] <= 76 and hits[1.0] > 3000, hits
    assert ms[1.0] < 0.7 * (hits[1.0] / 76.0) * ms[4.0], (ms, hits)
