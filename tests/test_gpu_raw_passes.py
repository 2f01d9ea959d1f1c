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
