"""The context's workspace: held by captured graphs, and short of device memory."""
import numpy as np
import pytest
import torch

import paper_2604_21095_gb300 as tg
import synth
from scan_util import run_scan

pytestmark = pytest.mark.gpu


def test_fp4_scan_leaves_a_captured_graphs_buffers_alone():
    """An FP4 scan of more markers than the workspace holds is refused while a captured graph has
    pointers into it, before any of its buffers is replaced: the graph replays as before."""
    N, P, M = 2001, 40, 1000
    w = synth.Workload("fp4_beside_graph", N=N, M=M, P=P, n_cov=3, encoding="2bit", missing=0.0,
                       seed=19, block=M, causal_per_pheno=1)
    pan = synth.make_panel(w)
    G = synth.make_block(w, 0)["G"].cuda()
    small = G[:300].contiguous()
    ctx = tg.tg_create(0)
    panel = tg.tg_prepare_panel(ctx, pan["Yt"].cuda(), N, P, pan["cov_t"].cuda())
    best = torch.zeros(P, dtype=torch.int64, device="cuda")
    try:
        first = run_scan(ctx, panel, small, N, P, "2bit", "fp4", full=False)
        graph = tg.tg_scan_graph_create(ctx, panel, [small], N, tg.TG_ENC_2BIT,
                                        tg.tg_scan_opts(tg.TG_PREC_SPLIT_BF16, 0, 0.0),
                                        tg.make_outputs(best=best), [0])
        try:
            tg.tg_scan_graph_launch(graph)
            torch.cuda.synchronize()
            before = best.cpu().numpy().copy()
            with pytest.raises(tg.TgError) as e:
                run_scan(ctx, panel, G, N, P, "2bit", "fp4", full=False)
            assert e.value.status == tg.TG_ERR_INVALID_ARG
            again = run_scan(ctx, panel, small, N, P, "2bit", "fp4", full=False)  # fits: still taken
            best.zero_()
            tg.tg_scan_graph_launch(graph)
            torch.cuda.synchronize()
        finally:
            tg.tg_scan_graph_free(graph)
    finally:
        tg.tg_panel_free(panel)
        tg.tg_destroy(ctx)
    assert before.all() and np.array_equal(best.cpu().numpy(), before)
    assert np.array_equal(again["best_key"], first["best_key"])


def test_scans_and_graphs_run_unsplit_where_memory_is_short():
    """A block whose passes are split would need 362 MB for their partial sums, unsplit half of
    that: with room for the half alone it is scanned, and captured, unsplit. (1,100 samples are two
    accumulation chunks, so an even split over the SMs cuts some tiles in two.)"""
    N, P, M, n_cov = 1100, 110, 400_000, 3
    whole = 4 * (P + n_cov) * M
    gen = torch.Generator(device="cuda").manual_seed(4)
    G = torch.randint(0, 256, (M, 288), generator=gen, dtype=torch.uint8, device="cuda")
    cov = synth.covariates(31, N, n_cov)
    Yt = synth.phenotypes(32, cov, P)
    best = torch.zeros(P, dtype=torch.int64, device="cuda")
    out = tg.make_outputs(best=best)
    opts = tg.tg_scan_opts(tg.TG_PREC_SPLIT_BF16, 0, 0.0)
    filler, res = None, []
    for short in (False, True):
        ctx = tg.tg_create(0)
        panel = tg.tg_prepare_panel(ctx, Yt.cuda(), N, P, cov.cuda())
        graph = None
        try:
            tg.tg_set_fused_decode(ctx, True)  # (a graph then reserves no decoded operand)
            tg.tg_scan_block(ctx, panel, G[:256], N, 256, tg.TG_ENC_2BIT, opts, out)
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            if short:  # room for the marker arrays (under 100 bytes each) and the unsplit products
                room = whole + 100 * M + (32 << 20)
                assert room < 2 * whole
                filler = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8,
                                     device="cuda")
            for captured in (False, True):
                best.zero_()
                if captured:
                    graph = tg.tg_scan_graph_create(ctx, panel, [G], N, tg.TG_ENC_2BIT, opts, out, [0])
                    tg.tg_scan_graph_launch(graph)
                else:
                    tg.tg_scan_block(ctx, panel, G, N, M, tg.TG_ENC_2BIT, opts, out)
                assert tg.tg_status_poll(ctx) == tg.TG_OK
                res.append(best.cpu().numpy().view(np.uint64).copy())
        finally:
            filler = None
            torch.cuda.empty_cache()
            if graph is not None:
                tg.tg_scan_graph_free(graph)
            tg.tg_panel_free(panel)
            tg.tg_destroy(ctx)
    for keys in res[1:]:  # |r| in the upper half; two partial sums of chunks or one, in the same order
        absr = [(k >> 32).astype(np.uint32).view(np.float32) for k in (keys, res[0])]
        np.testing.assert_allclose(absr[0], absr[1], atol=1e-6, rtol=0)


@pytest.mark.parametrize("P,tuned", [(40, False), (300, True)])
def test_autotune_keeps_no_choice_that_the_scans_ignore(tmp_path, P, tuned):
    """A panel of at most 64 phenotypes has no kernel to choose, so tuning it leaves the context's
    choice for the block size as it was; one with a joint pass is tuned for the paper's mode."""
    N, M = 1500, 700
    cov = synth.covariates(85, N, 3)
    ctx = tg.tg_create(0)
    panel = tg.tg_prepare_panel(ctx, synth.phenotypes(85, cov, P).cuda(), N, P, cov.cuda())
    try:
        tg.tg_autotune(ctx, panel, tg.TG_ENC_2BIT, M)
        path = tmp_path / "tuning.json"
        tg.tg_tuning_save(ctx, str(path))
        assert ("min_markers" in path.read_text()) == tuned
        if not tuned:
            tg.tg_set_tuning(ctx, M, "single", 8)
            tg.tg_autotune(ctx, panel, tg.TG_ENC_2BIT, M)
            assert tg.tg_tuning(ctx, M) == {"kernel": "single", "group_m": 8}
    finally:
        tg.tg_panel_free(panel)
        tg.tg_destroy(ctx)


@pytest.mark.parametrize("precision", [tg.TG_PREC_FP32, tg.TG_PREC_SPLIT_BF16])
def test_graph_with_empty_blocks(precision):
    """Empty blocks are accepted and add nothing. (Their plan divided by their number of tiles in the
    FP32 form, which ends the process on hosts whose integer division traps.)"""
    N, P, M = 900, 5, 300
    gen = torch.Generator(device="cuda").manual_seed(6)
    G = torch.randint(0, 256, (M, 240), generator=gen, dtype=torch.uint8, device="cuda")
    cov = synth.covariates(41, N, 2)
    ctx = tg.tg_create(0)
    panel = tg.tg_prepare_panel(ctx, synth.phenotypes(42, cov, P).cuda(), N, P, cov.cuda())
    got = []
    try:
        for blocks, offsets in (([G], [0]), ([G[:0], G[:100], G[100:100], G[100:]], [0, 0, 100, 100])):
            best = torch.zeros(P, dtype=torch.int64, device="cuda")
            graph = tg.tg_scan_graph_create(ctx, panel, blocks, N, tg.TG_ENC_2BIT,
                                            tg.tg_scan_opts(precision, 0, 0.0),
                                            tg.make_outputs(best=best), offsets)
            try:
                tg.tg_scan_graph_launch(graph)
                torch.cuda.synchronize()
            finally:
                tg.tg_scan_graph_free(graph)
            got.append(best.cpu().numpy())
    finally:
        tg.tg_panel_free(panel)
        tg.tg_destroy(ctx)
    assert got[0].all() and np.array_equal(got[0], got[1])
