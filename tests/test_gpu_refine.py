"""Markers in linkage with a marker that is among the covariates: a run of neighbours whose norms are
recomputed in FP64, against the oracle, and without one waiting for the other."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_21095_gb300 as tg
import synth
from scan_util import enc_id, oracle_panel, prec_id, run_scan

pytestmark = pytest.mark.gpu


def _linked(N, M, n_cov, first, run, encoding, seed=5):
    """A block whose markers first .. first + run share 95% of their calls with one, which (with
    noise) is covariate 0: genotypes, covariates, phenotypes."""
    cov = synth.covariates(seed, N, n_cov)
    freq = synth.maf(seed, 0, M)
    freq[first:first + run] = 0.3
    counts, miss = synth.hard_calls(seed, 0, freq, N, 0.01)
    g = torch.Generator().manual_seed(seed)
    lead = counts[first].clone()
    for j in range(first, first + run):
        keep = torch.rand(N, generator=g) < 0.95
        counts[j] = torch.where(keep, lead, counts[j])
    cov[0] = lead.double() + 0.3 * lead.double().std() * cov[0]
    if encoding == "2bit":
        G = synth.pack_2bit(counts, miss)
    else:
        G = torch.zeros(M, synth.round_up(N, 16), dtype=torch.uint8)
        G[:, :N] = (counts.float() * 127.5).round().to(torch.uint8)
    return G, cov


@pytest.mark.parametrize("precision", ["split", "fp32", "static", "fp4"])
@pytest.mark.parametrize("encoding,N,M,first,run", [("2bit", 2000, 700, 40, 64),
                                                    ("u8", 1501, 333, 300, 33),
                                                    ("2bit", 200, 80_000, 79_960, 40)])
def test_linked_neighbours_match_the_oracle(tgctx, precision, encoding, N, M, first, run):
    """Blocks of more markers than the re-projection has blocks, and of more than one of its steps
    over the markers (80,000); 9 covariates are one group of eight columns and one more."""
    if precision == "fp4" and encoding == "u8":
        pytest.skip("the FP4 form scans 2-bit calls")
    if precision == "static" and M > 10_000:
        pytest.skip("larger than the static scratch")
    n_cov, P = 9, 3
    G, cov = _linked(N, M, n_cov, first, run, encoding)
    Yt = synth.phenotypes(6, cov, P)
    panel = tg.tg_prepare_panel(tgctx, Yt.cuda(), N, P, cov.cuda())
    try:
        if precision == "static":
            norm2 = torch.zeros(M, dtype=torch.float64, device="cuda")
            best = torch.zeros(P, dtype=torch.int64, device="cuda")
            tg.tg_scan_block_static(panel, G.cuda(), N, M, enc_id(encoding),
                                    tg.tg_scan_opts(prec_id("split"), 0, 0.0),
                                    tg.make_outputs(best=best, marker_norm2=norm2))
            got = norm2.cpu().numpy()
        else:
            got = run_scan(tgctx, panel, G.cuda(), N, P, encoding, precision, full=False)["norm2"]
    finally:
        tg.tg_panel_free(panel)
    rows = np.r_[0:min(M, 128), first:first + run]
    ref = oracle.scan(G.numpy()[rows], encoding, oracle_panel(Yt, cov))
    g = ref["decode"]["g"]
    gc2 = ((g - g.mean(axis=1, keepdims=True)) ** 2).sum(axis=1)
    close = ref["gres2"] < 0.499 * gc2
    assert close[-run:].all()
    want, got = ref["gres2"], got[rows]
    ok = np.isfinite(want)
    if precision == "fp4":  # markers with a missing call have no test there
        ok &= ref["decode"]["n_obs"] == N
    assert np.array_equal(np.isfinite(got), ok)
    # FP64 from exact codes: k eps |g_c|^2, |g_c|^2 / |g_res|^2 <= 50
    np.testing.assert_allclose(got[close & ok], want[close & ok], rtol=1e-11)
    np.testing.assert_allclose(got[ok], want[ok], rtol=1e-6)


def test_linked_neighbours_do_not_take_turns(tgctx):
    """32 neighbours are re-projected on as many SMs, so that their norms take about as long as those
    of one (one SM for all of them took 27 times as long)."""
    N, M, P, n_cov = 23_000, 1024, 3, 19
    ms = {}
    try:
        for run in (1, 32):
            G, cov = _linked(N, M, n_cov, 64, run, "u8")
            panel = tg.tg_prepare_panel(tgctx, synth.phenotypes(6, cov, P).cuda(), N, P, cov.cuda())
            G = G.cuda()
            tg.tg_set_profiling(tgctx, True)
            ms[run] = 1e9
            for _ in range(6):
                tg.tg_stage_times(tgctx, reset=True)
                run_scan(tgctx, panel, G, N, P, "u8", "split", full=False)
                ms[run] = min(ms[run], tg.tg_stage_times(tgctx, reset=True)["norm"][0])
            tg.tg_set_profiling(tgctx, False)
            tg.tg_panel_free(panel)
    finally:
        tg.tg_set_profiling(tgctx, False)
    assert ms[32] < 4.0 * ms[1], ms
