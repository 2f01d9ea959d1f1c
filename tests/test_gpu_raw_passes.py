"""Passes that leave raw products: the joint projection and panel pass on CTA pairs
(128 < P + q - 1 <= 512) and split sample axes, at the edges of their tiles and ranges, against
the FP64 oracle."""
import numpy as np
import pytest

import oracle
import paper_2604_21095_gb300 as tg
import synth
from scan_util import compare_best, compare_full, compare_hits, oracle_panel, run_scan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,P", [
    (1025, 1, 126),     # 129 columns: the narrowest pair tile; one marker; a range of one sample
    (1024, 257, 253),   # 256 columns, one tile; a third 128-row half tile with one marker
    (3073, 300, 254),   # 257 columns, two tiles of 160; four ranges, the last of one sample
    (5000, 31, 509),    # 512 columns, the widest joint pass; five ranges, less than a warp of rows
    (5000, 129, 510),   # 513 columns: the projection and the contraction split on their own
    (23_000, 130, 40),  # one 64-column tile in 23 ranges
    (4099, 5000, 300),  # more tiles than half the pairs: ranges of unequal length
])
@pytest.mark.parametrize("encoding,mode", [("2bit", "projected"), ("u8", "projected"),
                                           ("2bit", "paper")])
def test_raw_passes_at_the_edges(tgctx, encoding, mode, N, M, P):
    w = synth.Workload(f"raw_{N}_{M}_{P}_{encoding}", N=N, M=M, P=P, n_cov=3, encoding=encoding,
                       missing=0.02 if encoding == "2bit" else 0.0, seed=37, block=M,
                       causal_per_pheno=1)
    pan = synth.make_panel(w)
    blk = synth.make_block(w, 0)
    panel = tg.tg_prepare_panel(tgctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    m = tg.TG_MODE_PAPER if mode == "paper" else tg.TG_MODE_PROJECTED
    try:
        full = run_scan(tgctx, panel, blk["G"].cuda(), N, P, encoding, "split", full=True,
                        hit_mlog10p=3.0, marker_offset=5, mode=m)
        hits = run_scan(tgctx, panel, blk["G"].cuda(), N, P, encoding, "split", full=False,
                        hit_mlog10p=3.0, marker_offset=5, mode=m)
    finally:
        tg.tg_panel_free(panel)
    ref = oracle.scan(blk["G"].numpy(), encoding, oracle_panel(pan["Yt"], pan["cov_t"]), mode=mode)
    for res in (full, hits):
        assert res["status"] == tg.TG_OK
        compare_hits(res, ref, 3.0, marker_offset=5)
        compare_best(res, ref, marker_offset=5)
        assert np.array_equal(res["nobs"], ref["decode"]["n_obs"])
    compare_full(full, ref, label=f"raw {encoding}/{mode}/{N}/{M}/{P}")


@pytest.mark.parametrize("encoding,P,M", [("2bit", 300, 1500),   # a CTA-pair pass in five pieces
                                          ("u8", 40, 2000),      # a 64-column pass in ranges
                                          ("2bit", 600, 300)])   # projection and contraction split
def test_scans_beside_a_captured_graph_run_unsplit(encoding, P, M):
    """While a captured graph holds the workspace nothing grows: a scan whose split passes would
    need more room for their partial sums than there is runs unsplit, with the same results."""
    import torch

    N, n_cov = 5000, 3
    w = synth.Workload(f"beside_{encoding}_{P}", N=N, M=M, P=P, n_cov=n_cov, encoding=encoding,
                       missing=0.01 if encoding == "2bit" else 0.0, seed=61, block=M,
                       causal_per_pheno=1)
    pan = synth.make_panel(w)
    blk = synth.make_block(w, 0)
    G = blk["G"].cuda()
    ctx = tg.tg_create(0)
    panel = tg.tg_prepare_panel(ctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    small = tg.tg_prepare_panel(ctx, pan["Yt"][:2].contiguous().cuda(), N, 2, pan["cov_t"].cuda())
    enc = tg.TG_ENC_2BIT if encoding == "2bit" else tg.TG_ENC_U8_DOSAGE
    best = torch.zeros(2, dtype=torch.int64, device="cuda")
    graph = tg.tg_scan_graph_create(ctx, small, [G], N, enc,
                                    tg.tg_scan_opts(tg.TG_PREC_SPLIT_BF16, 0, 0.0),
                                    tg.make_outputs(best=best), [0])
    try:
        res = run_scan(ctx, panel, G, N, P, encoding, "split", full=True, hit_mlog10p=3.0)
        tg.tg_scan_graph_launch(graph)
        torch.cuda.synchronize()
    finally:
        tg.tg_scan_graph_free(graph)
        tg.tg_panel_free(panel)
        tg.tg_panel_free(small)
        tg.tg_destroy(ctx)
    assert res["status"] == tg.TG_OK
    ref = oracle.scan(blk["G"].numpy(), encoding, oracle_panel(pan["Yt"], pan["cov_t"]))
    compare_full(res, ref, label=f"beside a graph {encoding}/{P}/{M}")
    compare_hits(res, ref, 3.0)
    compare_best(res, ref)
    np.testing.assert_array_equal(best.cpu().numpy() & 0xFFFFFFFF, res["best_key"][:2] & 0xFFFFFFFF)
