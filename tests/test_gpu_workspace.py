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
