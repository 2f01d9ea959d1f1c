"""The routes that read packed rows or split their sample axis, at the sizes where each of their forms
begins, ends inside a stage or is shared by several blocks, against the FP64 oracle:

  - the projection pass that writes the block's operand (P + q - 1 > 512), which 2-bit calls, dosages
    with and without one-pass statistics and small blocks take in forms of their own;
  - the packed-row pass of small panels on blocks of fewer 128-marker tiles than SMs, and on tiles
    that three or more CTAs share;
  - contractions that leave raw products: the tuned split of the one-CTA kernel, panels of at most
    64 phenotypes without covariate columns, and the second wave of the CTA-pair kernel;
  - all of these beside a captured graph that holds the workspace, where nothing is split."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_21095_gb300 as tg
import synth
from scan_util import (compare_best, compare_full, compare_hits, enc_id, oracle_panel, prec_id,
                       run_scan, sample_words)

pytestmark = pytest.mark.gpu

THR = 4.0


def _block(encoding, N, M, P, n_cov, seed):
    w = synth.Workload(f"edges_{encoding}_{N}_{M}_{P}", N=N, M=M, P=P, n_cov=n_cov,
                       encoding=encoding, missing=0.02 if encoding == "2bit" else 0.0, seed=seed,
                       block=M, causal_per_pheno=1)
    pan = synth.make_panel(w)
    G = synth.make_block(w, 0)["G"]
    if encoding == "u8" and G.shape[1] > N:
        G[:, N:] = 0xAB  # row padding: not samples
    return pan, G


def _check(res, ref, label, offset=0):
    assert res["status"] == tg.TG_OK
    compare_full(res, ref, label=label)
    compare_hits(res, ref, THR, marker_offset=offset)
    compare_best(res, ref, marker_offset=offset)
    assert np.array_equal(res["nobs"], ref["decode"]["n_obs"])


def _equal(a, b):
    for k in ("beta", "se", "t", "mlog10p", "best_key", "norm2", "nobs", "mean"):
        assert np.array_equal(a[k], b[k], equal_nan=True), k


@pytest.mark.parametrize("encoding,N,M", [
    ("2bit", 1999, 39_000),  # more 256-marker tiles than SMs
    ("2bit", 1950, 20_000),  # an odd number of 64-sample steps: the last stage ends past the operand
    ("2bit", 1950, 9001),    # fewer 128-marker tiles than SMs, operand above 32 MB
    ("u8", 2000, 39_000),    # one pass: no counting pass
    ("u8", 1950, 39_000),    # one pass, the last stage past the operand
    ("u8", 45, 39_000),      # one pass with fewer samples than the shift is taken from
    ("u8", 1950, 20_000),    # f16 after a counting pass
    ("u8", 1950, 9001),      # bf16 after a counting pass
])
def test_projection_pass_writes_the_operand(encoding, N, M):
    """Each form of the projection pass that also writes the operand. Up to two accumulation chunks a
    tile's partial sums add up in one order whatever the split, so 2-bit calls, which expand to the
    decoded operand's values, agree with the decoded path bit for bit."""
    P, n_cov = 513, 4
    pan, G = _block(encoding, N, M, P, n_cov, 53)
    ctx = tg.tg_create(0)
    panel = tg.tg_prepare_panel(ctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    res = {}
    try:
        for setting in (tg.TG_FUSED_SMALL_PANELS, tg.TG_FUSED_OFF):
            tg.tg_set_fused_decode(ctx, setting)
            res[setting] = run_scan(ctx, panel, G.cuda(), N, P, encoding, "split", full=True,
                                    hit_mlog10p=THR, marker_offset=7)
    finally:
        tg.tg_panel_free(panel)
        tg.tg_destroy(ctx)
    got, off = res[tg.TG_FUSED_SMALL_PANELS], res[tg.TG_FUSED_OFF]
    ref = oracle.scan(G.numpy(), encoding, oracle_panel(pan["Yt"], pan["cov_t"]))
    _check(got, ref, f"operand {encoding}/{N}/{M}", 7)
    assert np.array_equal(got["mean"], off["mean"])
    if encoding == "2bit":
        _equal(got, off)


@pytest.mark.parametrize("N,M,P", [
    (1950, 9000, 40),     # 64 columns, fewer 128-marker tiles than SMs
    (1950, 8999, 100),    # 128 columns
    (60_000, 300, 40),    # two tiles of 59 chunks, each shared by 59 CTAs
    (60_000, 300, 100),
    (5000, 19_456, 16),   # one 128-marker tile per SM: f16; 76 tiles of 5 chunks, 3 CTAs on some
])
def test_packed_pass_on_few_dosage_tiles(tgctx, N, M, P):
    pan, G = _block("u8", N, M, P, 3, 59)
    panel = tg.tg_prepare_panel(tgctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    try:
        res = run_scan(tgctx, panel, G.cuda(), N, P, "u8", "split", full=True, hit_mlog10p=THR)
    finally:
        tg.tg_panel_free(panel)
    ref = oracle.scan(G.numpy(), "u8", oracle_panel(pan["Yt"], pan["cov_t"]))
    _check(res, ref, f"packed {N}/{M}/{P}")


@pytest.mark.parametrize("P", [16, 513])
def test_subset_panel_on_a_one_pass_block(tgctx, P):
    """The subset's norms need the means before the norm kernel makes them from the pass's sums."""
    N, M, n_cov = 1999, 39_000, 3
    pan, G = _block("u8", N, M, P, n_cov, 61)
    keep = np.random.default_rng(3).random(N) < 0.8
    Yt = pan["Yt"].clone()
    Yt[:, ~torch.from_numpy(keep)] = float("nan")
    panel = tg.tg_prepare_panel_subset(tgctx, Yt.cuda(), N, P, pan["cov_t"].cuda(),
                                       sample_words(keep).cuda())
    try:
        res = run_scan(tgctx, panel, G.cuda(), N, P, "u8", "split", full=True, hit_mlog10p=THR)
    finally:
        tg.tg_panel_free(panel)
    ref = oracle.scan(G.numpy(), "u8", oracle_panel(Yt, pan["cov_t"], keep))
    _check(res, ref, f"subset one pass P={P}")
    assert np.array_equal(res["mean"], ref["decode"]["mean_units"])


@pytest.mark.parametrize("encoding", ["2bit", "u8"])
@pytest.mark.parametrize("P,n_cov,mode,splits", [
    (600, 3, "projected", 1), (600, 3, "projected", 2),
    (600, 3, "projected", 4),  # five chunks in four ranges, the last one empty
    (300, 3, "paper", 4),      # a panel with a joint pass, in the mode that has none
    (40, 0, "projected", 0),   # no projection columns: 64-column tiles, ranges by estimate
    (40, 3, "paper", 0),
])
def test_split_contractions(encoding, P, n_cov, mode, splits):
    N, M = 5000, 600
    pan, G = _block(encoding, N, M, P, n_cov, P + 5)
    m = tg.TG_MODE_PAPER if mode == "paper" else tg.TG_MODE_PROJECTED
    ctx = tg.tg_create(0)
    panel = tg.tg_prepare_panel(ctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda() if n_cov else None)
    try:
        if splits:
            tg.tg_set_tuning(ctx, M, "single", 16)
            tg.tg_set_tuning_split(ctx, M, splits)
        res = [run_scan(ctx, panel, G.cuda(), N, P, encoding, "split", full=True, hit_mlog10p=THR,
                        mode=m) for _ in range(2)]
    finally:
        tg.tg_panel_free(panel)
        tg.tg_destroy(ctx)
    _equal(res[0], res[1])  # the same order of additions every run
    ref = oracle.scan(G.numpy(), encoding, oracle_panel(pan["Yt"], pan["cov_t"]), mode=mode)
    _check(res[0], ref, f"split {encoding}/{P}/{mode}/{splits}")


@pytest.mark.parametrize("encoding", ["2bit", "u8"])
def test_second_wave_streams_k_backwards(tgctx, encoding):
    """600 phenotypes are three column tiles of 224: 48 x 3 tiles, more than the CTA pairs, so some
    stream the samples from the end."""
    N, M, P = 2000, 12_288, 600
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    tiles = (M // 256) * 3
    assert pairs < tiles < 2 * pairs
    pan, G = _block(encoding, N, M, P, 4, 17)
    panel = tg.tg_prepare_panel(tgctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    try:
        res = run_scan(tgctx, panel, G.cuda(), N, P, encoding, "split", full=True, hit_mlog10p=THR)
    finally:
        tg.tg_panel_free(panel)
    ref = oracle.scan(G.numpy(), encoding, oracle_panel(pan["Yt"], pan["cov_t"]))
    _check(res, ref, f"second wave {encoding}")


@pytest.mark.parametrize("encoding,precision,N,M,P", [
    ("u8", "split", 23_000, 130, 40),   # 23 ranges of a 64-column pass
    ("u8", "split", 60_000, 300, 100),  # 59 pieces of a packed tile
    ("2bit", "fp32", 5000, 300, 600),   # ranges of the FP32 tiles
])
def test_scans_beside_a_captured_graph_are_not_split(encoding, precision, N, M, P):
    """The graph's workspace has no room for the split's partial sums (pieces x columns x rows floats
    against 512 per marker), so the scan runs unsplit, on whole tiles; with the graph gone it
    splits (into ranges of one accumulation chunk where the pass is on tensor cores, which add up
    as the chunks of a whole tile do). Both are the oracle's."""
    pan, G = _block(encoding, N, M, P, 3, 61)
    ctx = tg.tg_create(0)
    panel = tg.tg_prepare_panel(ctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    small = tg.tg_prepare_panel(ctx, pan["Yt"][:2].contiguous().cuda(), N, 2, pan["cov_t"].cuda())
    best = torch.zeros(2, dtype=torch.int64, device="cuda")
    Gd = G.cuda()
    graph = tg.tg_scan_graph_create(ctx, small, [Gd], N, enc_id(encoding),
                                    tg.tg_scan_opts(prec_id(precision), 0, 0.0),
                                    tg.make_outputs(best=best), [0])
    try:
        res = [run_scan(ctx, panel, Gd, N, P, encoding, precision, full=True, hit_mlog10p=THR)]
        tg.tg_scan_graph_launch(graph)
        torch.cuda.synchronize()
    finally:
        tg.tg_scan_graph_free(graph)
        try:
            res.append(run_scan(ctx, panel, Gd, N, P, encoding, precision, full=True,
                                hit_mlog10p=THR))
        finally:
            tg.tg_panel_free(panel)
            tg.tg_panel_free(small)
            tg.tg_destroy(ctx)
    ref = oracle.scan(G.numpy(), encoding, oracle_panel(pan["Yt"], pan["cov_t"]))
    for r in res:
        _check(r, ref, f"beside a graph {encoding}/{precision}/{N}/{M}/{P}")
