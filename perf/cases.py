"""The workloads that the genome scan's speed is measured on.

Each case is a plain dict: `listed()` gives the fixed ones, `draw(rng)` one more of the same
ranges, `prepare` makes what a program holds before the call, `run` makes the call through the
package's public entry points and returns its outputs, `work` counts what the call cannot do
without, and `exact` computes the outputs in 64 bits with torch alone.

Fields of a case:
  kind       "scan" (one block on the device), "stream" (a matrix in pinned host memory),
             "graph" (ragged blocks against concatenated panels, one captured graph),
             "prepare" (a panel from phenotypes and covariates)
  enc        "2bit" (PLINK hard calls) or "u8" (8-bit dosages);  missing: rate of missing calls
             (in-band for 2-bit calls, a bit mask for dosages)
  N, M, P    samples, markers, phenotypes;  cov: covariate columns besides the intercept
  prec       "split" or "fp32";  mode "projected" or "paper"
  full       True: every statistic of every test; False: hits and the best marker per phenotype
  observed   share of the samples the phenotypes are observed on (< 1: a subset panel)
  block      markers per streamed block
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2604_21095_gb300 as tg

THRESHOLD = 7.30103   # genome-wide significance, -log10(5e-8)
CHUNK = 4096          # markers drawn at a time
PLANTED = 50          # (marker, phenotype) pairs with an effect, at most 5 per phenotype
H2 = 0.02             # variance explained by a planted marker
HIT_CAPACITY = 4096
EXACT_MAX_FLOPS = 8e12


def _scan(name, enc, N, M, P, cov, missing=0.0, full=False, prec="split", mode="projected",
          observed=1.0):
    return {"name": name, "kind": "scan", "enc": enc, "N": N, "M": M, "P": P, "cov": cov,
            "missing": missing, "full": full, "prec": prec, "mode": mode, "observed": observed}


def listed():
    return [
        # the smallest call: a few hundred typed markers of a pilot cohort, every statistic
        _scan("pilot_2bit_p40_full", "2bit", 777, 300, 40, 2, missing=0.02, full=True),
        # a small cohort's typed chromosome against 16 traits, every statistic
        _scan("cohort2k_2bit_p16_full", "2bit", 2000, 10_000, 16, 4, missing=0.01, full=True),
        # the single-trait association every biobank runs: summary statistics of a dosage block
        _scan("biobank_u8_p1_full", "u8", 23_000, 8192, 1, 19, full=True),
        # a small panel over a full block of imputed dosages: bound by reading the genotypes
        _scan("biobank_u8_p16", "u8", 23_000, 65_536, 16, 19),
        # about a hundred traits over a full block of hard calls with missing ones
        _scan("biobank_2bit_p100", "2bit", 23_000, 65_536, 100, 9, missing=0.005),
        # ragged sizes: masked dosages, phenotypes observed on a subset, every statistic
        _scan("ragged_u8_p300_subset_full", "u8", 10_007, 5003, 300, 7, missing=0.02, full=True,
              observed=0.9),
        # a phenome-wide panel over hard calls
        _scan("phenome_2bit_p2048", "2bit", 23_000, 65_536, 2048, 9, missing=0.005),
        # the largest: a full dosage block against an imaging panel
        _scan("imaging_u8_p20480", "u8", 23_000, 65_536, 20_480, 19),
        # the plain FP32 form, for callers that compare against the split form
        _scan("fp32_u8_p1000_full", "u8", 4099, 3001, 1000, 9, full=True, prec="fp32"),
        # ragged blocks against three concatenated panels, replayed as one graph
        {"name": "graph_2bit_ragged", "kind": "graph", "enc": "2bit", "N": 5001, "M": 11_243,
         "P": 337, "cov": 9, "missing": 0.005, "full": False, "prec": "split",
         "mode": "projected", "observed": 1.0},
        # a genotype matrix in host memory, streamed against a medium panel
        {"name": "stream_2bit_p256", "kind": "stream", "enc": "2bit", "N": 23_000, "M": 65_536,
         "P": 256, "cov": 9, "missing": 0.005, "full": False, "prec": "split",
         "mode": "projected", "observed": 1.0, "block": 16_384},
        # a panel made ready for scanning
        {"name": "prepare_p2048", "kind": "prepare", "N": 23_000, "P": 2048, "cov": 19},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["scan"] * 7 + ["graph", "stream", "prepare"])
    N = _log(rng, 600, 30_000)
    cov = rng.randint(1, 20)
    if kind == "prepare":
        return {"kind": kind, "N": N, "P": _log(rng, 1, 4096), "cov": cov}
    enc = rng.choice(["2bit", "u8"])
    M = _log(rng, 200, 65_536)
    while M * N > 65_536 * 23_000:
        M = _log(rng, 200, 65_536)
    P = _log(rng, 1, 4096)
    missing = rng.choice([0.0, 0.005, 0.02])
    case = {"kind": kind, "enc": enc, "N": N, "M": M, "P": P, "cov": cov, "missing": missing,
            "full": False, "prec": "split", "mode": "projected", "observed": 1.0}
    if kind == "graph":
        case["M"], case["missing"] = max(M, 1000), missing if enc == "2bit" else 0.0
        return case
    if kind == "stream":
        case["missing"] = missing if enc == "2bit" else 0.0
        case["block"] = rng.choice([2048, 4096, 16_384])
        return case
    case["full"] = rng.random() < 0.5
    if rng.random() < 0.15:
        case["prec"] = "fp32"
    if rng.random() < 0.1:
        case["mode"] = "paper"
    if rng.random() < 0.2:
        case["observed"] = 0.9
    while case["full"] and case["M"] * case["P"] > 60_000_000:
        case["P"] = _log(rng, 1, 4096)
    while case["prec"] == "fp32" and case["M"] * case["P"] * N > 2e12:
        case["M"] = _log(rng, 200, 16_384)
        case["P"] = _log(rng, 1, 1024)
    return case


# ------------------------------------------------------------------------------ inputs

def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream * 7919 + 17) & ((1 << 62) - 1))
    return g


def _round_up(x, m):
    return (x + m - 1) // m * m


def _calls(seed, c0, rows, N, missing, masked):
    """Allele counts (uint8, 0..2) of markers c0.. under Hardy-Weinberg with maf ~ U(0.01, 0.5),
    and the missing calls (bool, or None)."""
    g = _generator(seed, 100 + c0 // CHUNK)
    f = 0.01 + 0.49 * torch.rand(rows, 1, generator=g, device="cuda")
    u = torch.rand(rows, N, generator=g, device="cuda")
    counts = (u < f * f).to(torch.uint8) + (u < 2 * f - f * f).to(torch.uint8)
    miss = torch.rand(rows, N, generator=g, device="cuda") < missing if masked else None
    return counts, miss, g


def _dosages(counts, g):
    """Dosage bytes round(127.5 count + U(-8, 8)) within 0..255."""
    e = torch.rand(counts.shape, generator=g, device="cuda").mul_(16.0).sub_(8.0)
    return e.add_(counts, alpha=127.5).round_().clamp_(0, 255).to(torch.uint8)


def _chunk(case, seed, c0):
    """(packed or byte values, missing) of the markers c0 .. c0 + CHUNK of a case."""
    rows = min(CHUNK, case["M"] - c0)
    counts, miss, g = _calls(seed, c0, rows, case["N"], case["missing"], case["missing"] > 0)
    return (counts if case["enc"] == "2bit" else _dosages(counts, g)), miss


def _pack_2bit(counts, miss, ldg):
    """PLINK .bed fields: 2 -> 00, 1 -> 10, 0 -> 11, missing -> 01, four samples to a byte."""
    f = 3 - counts - (counts == 2).to(torch.uint8)
    if miss is not None:
        f = torch.where(miss, torch.ones_like(f), f)
    M, N = f.shape
    f = torch.nn.functional.pad(f, (0, 4 * ldg - N)).view(M, ldg, 4)
    return f[..., 0] | (f[..., 1] << 2) | (f[..., 2] << 4) | (f[..., 3] << 6)


def _pack_mask(miss):
    M, N = miss.shape
    w = (N + 31) // 32
    b = torch.nn.functional.pad(miss, (0, 32 * w - N)).view(M, w, 4, 8).to(torch.uint8)
    byte = torch.zeros(M, w, 4, dtype=torch.uint8, device="cuda")
    for k in range(8):
        byte |= b[..., k] << k
    return byte.view(M, 4 * w).view(torch.int32)


def _ldg(case):
    return _round_up((case["N"] + 3) // 4 if case["enc"] == "2bit" else case["N"], 16)


def _genotypes(case, seed):
    """Packed rows [M][ldg], the bit mask of missing dosages (or None), and the true values of
    the markers that may carry an effect (markers 1 to PLANTED: marker 0 against phenotype 0 would
    read like an empty hit record)."""
    M, N, ldg = case["M"], case["N"], _ldg(case)
    two = case["enc"] == "2bit"
    G = torch.zeros(M, ldg, dtype=torch.uint8, device="cuda")
    mask = None
    if not two and case["missing"] > 0:
        mask = torch.zeros(M, (N + 31) // 32, dtype=torch.int32, device="cuda")
    truth = None
    for c0 in range(0, M, CHUNK):
        v, miss = _chunk(case, seed, c0)
        c1 = c0 + v.shape[0]
        if two:
            G[c0:c1] = _pack_2bit(v, miss, ldg)
        else:
            G[c0:c1, :N] = v
            if mask is not None:
                mask[c0:c1] = _pack_mask(miss)
        if truth is None:
            truth = v[1:PLANTED + 1].to(torch.float32)
            if not two:
                truth *= 2.0 / 255.0
    return G, mask, truth


def _phenotypes(case, seed, truth):
    """Covariates [cov][N] (FP64) and phenotypes [P][N] (FP32): covariate effects, planted marker
    effects and N(0, 1) noise."""
    N, P, cov = case["N"], case["P"], case["cov"]
    g = _generator(seed, 1)
    C = torch.randn(cov, N, generator=g, device="cuda", dtype=torch.float64)
    gam = torch.randn(P, cov + 1, generator=g, device="cuda")
    Y = torch.randn(P, N, generator=g, device="cuda")
    Y += gam[:, :1] + gam[:, 1:] @ C.float()
    if truth is not None:
        var = truth.var(dim=1).clamp_min(1e-3)
        n = min(PLANTED, truth.shape[0], 5 * P)
        for k in range(n):
            Y[k % P] += truth[k] * torch.sqrt(H2 / var[k])
    return C, Y


def _observed(case, seed):
    """Samples the phenotypes are observed on (bool [N]), or None for all of them."""
    if case.get("observed", 1.0) >= 1.0:
        return None
    return torch.rand(case["N"], generator=_generator(seed, 2), device="cuda") < case["observed"]


def _ragged(M):
    """Five block sizes that add up to M, none a multiple of a tile."""
    w = (0.27, 0.11, 0.37, 0.06)
    sizes = [max(1, int(M * x) | 1) for x in w]
    return sizes + [M - sum(sizes)]


def _panel_sizes(P):
    """The panels that a graph case concatenates."""
    a, b = P // 20, P // 5
    return [p for p in (a, b, P - a - b) if p > 0]


# ------------------------------------------------------------------------------ what a program keeps

_ctx = []
_current = []  # the panel that the last "prepare" pass made, kept until the next one replaces it


def _context():
    """A program keeps one context; its workspace grows to the largest block it scans."""
    if not _ctx:
        torch.zeros(1, device="cuda")
        _ctx.append(tg.tg_create(torch.cuda.current_device()))
    return _ctx[0]


class State:
    """Inputs, handles and output buffers of one case; handles are given back with it."""

    def __init__(self, case):
        self.case = case
        self.panels, self.graph, self.own_ctx = [], None, None

    def __del__(self):
        try:
            if self.graph is not None:
                tg.tg_scan_graph_free(self.graph)
            for p in self.panels:
                tg.tg_panel_free(p)
            if self.own_ctx is not None:
                tg.tg_destroy(self.own_ctx)
        except Exception:
            pass


def _options(case):
    prec = tg.TG_PREC_FP32 if case["prec"] == "fp32" else tg.TG_PREC_SPLIT_BF16
    mode = tg.TG_MODE_PAPER if case["mode"] == "paper" else tg.TG_MODE_PROJECTED
    return tg.tg_scan_opts(prec, 1 if case["full"] else 0, 0.0 if case["full"] else THRESHOLD, mode)


def _collect(s, P):
    """One buffer for the hit records, their count and the best keys, so that one fill clears it."""
    hits = HIT_CAPACITY * ctypes.sizeof(tg.tg_hit)
    s.buffer = torch.zeros(hits + 8 + 8 * P, dtype=torch.uint8, device="cuda")
    s.hits = s.buffer[:hits]
    s.n_hits = s.buffer[hits:hits + 8].view(torch.int64)
    s.best = s.buffer[hits + 8:].view(torch.int64)


def prepare(case, seed):
    s = State(case)
    kind, N, P = case["kind"], case["N"], case["P"]
    if kind == "prepare":
        s.ctx = _context()
        s.C, s.Y = _phenotypes(case, seed, None)
        torch.cuda.synchronize()
        return s
    s.enc = tg.TG_ENC_2BIT if case["enc"] == "2bit" else tg.TG_ENC_U8_DOSAGE
    s.G, s.mask, truth = _genotypes(case, seed)
    C, Y = _phenotypes(case, seed, truth)
    s.opts = _options(case)
    if kind in ("graph", "stream"):
        torch.zeros(1, device="cuda")
        s.own_ctx = tg.tg_create(torch.cuda.current_device())
    s.ctx = s.own_ctx if s.own_ctx is not None else _context()
    if kind == "graph":
        at = 0
        for p in _panel_sizes(P):
            s.panels.append(tg.tg_prepare_panel(s.ctx, Y[at:at + p], N, p, C))
            at += p
        s.panel = tg.tg_panel_concat(s.ctx, s.panels)
        s.panels.append(s.panel)
        _collect(s, P)
        s.out = tg.make_outputs(hits=s.hits, n_hits=s.n_hits, best=s.best)
        sizes = _ragged(case["M"])
        s.blocks = list(torch.split(s.G, sizes))
        offsets = [sum(sizes[:i]) for i in range(len(sizes))]
        s.graph = tg.tg_scan_graph_create(s.ctx, s.panel, s.blocks, N, s.enc, s.opts, s.out, offsets)
        torch.cuda.synchronize()
        return s
    seen = _observed(case, seed)
    if seen is None:
        s.panel = tg.tg_prepare_panel(s.ctx, Y, N, P, C)
    else:
        s.seen = _pack_mask(seen.view(1, N)).view(-1)
        s.panel = tg.tg_prepare_panel_subset(s.ctx, Y, N, P, C, s.seen)
    s.panels.append(s.panel)
    if kind == "stream":
        s.G = s.G.cpu().pin_memory()
        s.hits = torch.zeros(HIT_CAPACITY * ctypes.sizeof(tg.tg_hit), dtype=torch.uint8).pin_memory()
        s.best = torch.zeros(P, dtype=torch.int64).pin_memory()
        torch.cuda.synchronize()
        return s
    s.norm2 = torch.zeros(case["M"], dtype=torch.float64, device="cuda")
    s.nobs = torch.zeros(case["M"], dtype=torch.int32, device="cuda")
    s.mean = torch.zeros(case["M"], dtype=torch.float64, device="cuda")
    if case["full"]:
        s.stats = [torch.zeros(case["M"], P, device="cuda") for _ in range(4)]
        b, e, t, m = s.stats
        s.out = tg.make_outputs(beta=b, se=e, t=t, mlog10p=m, ldo=P, marker_norm2=s.norm2,
                                marker_nobs=s.nobs, marker_mean=s.mean)
    else:
        _collect(s, P)
        s.out = tg.make_outputs(hits=s.hits, n_hits=s.n_hits, best=s.best)
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------------------ the pass

def _ranked(s):
    """Hits ordered by phenotype, then marker (they come unordered), and the best markers."""
    rec = s.hits.view(torch.int64).view(-1, 3)
    rec = rec[torch.sort(rec[:, 0]).indices]
    return {"n_hits": s.n_hits, "hit_ids": rec.view(torch.int32)[:, :2],
            "hit_stats": rec.view(torch.float32)[:, 2:],
            "best_marker": s.best.view(torch.int32)[0::2],
            "best_r": s.best.view(torch.float32)[1::2]}


def run(s):
    case = s.case
    kind, N = case["kind"], case["N"]
    if kind == "prepare":
        while _current:  # the panel of the pass before goes
            tg.tg_panel_free(_current.pop())
        _current.append(tg.tg_prepare_panel(s.ctx, s.Y, N, case["P"], s.C))
        yres, norms = tg.tg_panel_Yres(_current[0])  # views of the panel's own memory
        return {"Q": tg.tg_panel_Q(_current[0]), "y_res": yres, "norms": norms}
    if kind == "stream":
        n = tg.tg_scan_host(s.ctx, s.panel, s.G, N, case["M"], s.enc, case["block"], s.opts, s.hits,
                            best_host=s.best)
        rec = tg.hits_to_numpy(s.hits, min(n, HIT_CAPACITY))
        order = np.argsort(rec["pheno"].astype(np.int64) << 32 | rec["marker"])
        table = np.zeros((HIT_CAPACITY, 6), np.float32)  # the ranked hits, as the records they are
        table[HIT_CAPACITY - len(rec):] = rec.view(np.float32).reshape(-1, 6)[order]
        best = s.best.numpy()
        return {"n_hits": n, "hit_ids": table.view(np.int32)[:, :2], "hit_stats": table[:, 2:],
                "best_marker": best.view(np.int32)[0::2].copy(),
                "best_r": best.view(np.float32)[1::2].copy()}
    if kind == "graph":
        s.buffer.zero_()
        tg.tg_scan_graph_launch(s.graph)
        return _ranked(s)
    if not case["full"]:
        s.buffer.zero_()
    tg.tg_scan_block(s.ctx, s.panel, s.G, N, case["M"], s.enc, s.opts, s.out, missing=s.mask)
    if not case["full"]:
        return _ranked(s)
    b, e, t, m = s.stats
    return {"beta": b, "se": e, "t": t, "mlog10p": m, "norm2": s.norm2, "n_obs": s.nobs,
            "mean": s.mean}


def work(case):
    """Inputs read once and outputs written once; the panel counts 4 bytes a value (hi + lo, or
    FP32), the products of Eq. 2 and of the covariate projection 2 flops each."""
    N, P, q = case["N"], case["P"], case["cov"] + 1
    if case["kind"] == "prepare":  # phenotypes in; FP64 residuals, FP32 and hi + lo panel out
        return {"bytes": N * P * (4 + 8 + 4 + 4) + 16 * N * q, "flops": 4.0 * N * P * q}
    M = case["M"]
    packed = (N + 3) // 4 if case["enc"] == "2bit" else N
    b = M * packed + 4 * N * (P + q - 1)
    if case["enc"] == "u8" and case["missing"] > 0:
        b += M * ((N + 31) // 32) * 4
    b += 16 * M * P + 20 * M if case["full"] else 8 * P
    nq = q - 1 if case["mode"] == "projected" else 0
    return {"bytes": b, "flops": 2.0 * N * M * (P + nq)}


# ------------------------------------------------------------------------------ 64 bits

def _ln_beta_half(df):
    return math.lgamma(df / 2) + math.lgamma(0.5) - math.lgamma(df / 2 + 0.5)


def _fraction(a, b, x, terms):
    """Continued fraction of the incomplete beta function (Lentz), elementwise in FP64."""
    tiny = 1e-300
    fix = lambda v: torch.where(v.abs() < tiny, torch.full_like(v, tiny), v)  # noqa: E731
    c = torch.ones_like(x)
    d = 1.0 / fix(1.0 - (a + b) * x / (a + 1.0))
    h = d.clone()
    for m in range(1, terms + 1):
        for e in (m * (b - m) / ((a + 2 * m - 1) * (a + 2 * m)),
                  -(a + m) * (a + b + m) / ((a + 2 * m) * (a + 2 * m + 1))):
            e = e * x
            d = 1.0 / fix(1.0 + e * d)
            c = fix(1.0 + e / c)
            h = h * (d * c)
    return h


def _mlog10p(r, df):
    """-log10 of the two-sided p-value of a correlation, I_{1-r^2}(df/2, 1/2)."""
    a, b = df / 2.0, 0.5
    ar = r.abs().clamp(1e-30, 1.0 - 1e-16)
    y = ar * ar
    x = (1.0 - ar) * (1.0 + ar)
    lnx, lny, lnB = torch.log1p(-y), 2.0 * torch.log(ar), _ln_beta_half(df)
    out = torch.empty_like(r)
    low = x < (a + 1.0) / (a + b + 2.0)
    if low.any():
        v = a * lnx[low] + b * lny[low] - math.log(a) - lnB + torch.log(_fraction(a, b, x[low], 400))
        out[low] = -v / math.log(10.0)
    if (~low).any():
        v = torch.exp(b * lny[~low] + a * lnx[~low] - math.log(b) - lnB +
                      torch.log(_fraction(b, a, y[~low], 60)))
        out[~low] = -torch.log1p(-v.clamp(max=1.0)) / math.log(10.0)
    return out


def _basis(C, N):
    X = np.concatenate([np.ones((N, 1)), C.cpu().numpy().T], axis=1)
    return torch.from_numpy(np.ascontiguousarray(np.linalg.qr(X)[0])).cuda()  # Householder signs


def exact(case, seed):
    kind, N, P = case["kind"], case["N"], case["P"]
    if kind == "prepare":
        C, Y = _phenotypes(case, seed, None)
        Q = _basis(C, N)
        yres = torch.empty(P, N, dtype=torch.float64, device="cuda")
        for p0 in range(0, P, 512):
            y = Y[p0:p0 + 512].double()
            y -= y.mean(dim=1, keepdim=True)
            yres[p0:p0 + 512] = y - (y @ Q) @ Q.T
        return {"Q": Q.T.contiguous(), "y_res": yres, "norms": yres.norm(dim=1)}
    M = case["M"]
    if 2.0 * N * M * P > EXACT_MAX_FLOPS:
        return None
    v, miss = _chunk(case, seed, 0)
    truth = v[1:PLANTED + 1].to(torch.float32)
    if case["enc"] == "u8":
        truth *= 2.0 / 255.0
    C, Y = _phenotypes(case, seed, truth)
    seen = _observed(case, seed)
    keep = slice(None) if seen is None else seen
    C, Y = C[:, keep], Y[:, keep]
    NS = Y.shape[1]
    Q = _basis(C, NS)
    y = Y.double()
    y -= y.mean(dim=1, keepdim=True)
    y -= (y @ Q) @ Q.T
    s = y.norm(dim=1)
    u = (y / s[:, None]).T.contiguous()
    df = float(NS - Q.shape[1] - 1 if case["mode"] == "projected" else NS - 2)
    kappa = 1.0 if case["enc"] == "2bit" else 2.0 / 255.0
    full = case["full"]
    parts, hits = [], []
    top = torch.zeros(P, dtype=torch.float64, device="cuda")
    for c0 in range(0, M, CHUNK):
        v, miss = _chunk(case, seed, c0)
        for r0 in range(0, v.shape[0], 1024):
            g = v[r0:r0 + 1024].double()
            if miss is not None:
                ms = miss[r0:r0 + 1024]
                n_obs = (~ms).sum(dim=1)
                mean = g.masked_fill(ms, 0.0).sum(dim=1) / n_obs
                g = torch.where(ms, mean[:, None], g)
            else:
                n_obs, mean = torch.full((g.shape[0],), N, device="cuda"), g.mean(dim=1)
            g = g[:, keep]
            g = g - g.mean(dim=1, keepdim=True)
            n2 = (g * g).sum(dim=1)
            if case["mode"] == "projected":
                n2 = n2 - ((g @ Q[:, 1:]) ** 2).sum(dim=1)
            r = (g @ u) / n2.sqrt()[:, None]
            if full:
                omr2 = (1.0 - r) * (1.0 + r)
                scale = s[None, :] / (kappa * n2.sqrt()[:, None])
                parts.append((r * scale, scale * (omr2 / df).sqrt(), r * (df / omr2).sqrt(),
                              _mlog10p(r, df), n2 * kappa * kappa, mean))
                continue
            top = torch.maximum(top, r.abs().amax(dim=0))
            # pairs well below the threshold cannot be hits: a normal tail bounds their p-values
            i, p = torch.nonzero(r * r * df > 25.0, as_tuple=True)
            rr = r[i, p]
            m10 = _mlog10p(rr, df) if rr.numel() else rr
            ok = m10 >= THRESHOLD
            i, p, rr, m10 = i[ok], p[ok], rr[ok], m10[ok]
            omr2 = (1.0 - rr) * (1.0 + rr)
            scale = s[p] / (kappa * n2[i].sqrt())
            hits.append((p * (1 << 32) + (c0 + r0 + i), torch.stack(
                [rr * scale, scale * (omr2 / df).sqrt(), rr * (df / omr2).sqrt(), m10], dim=1)))
    if full:
        b, e, t, m, n2, mean = (torch.cat(x) for x in zip(*parts))
        return {"beta": b, "se": e, "t": t, "mlog10p": m, "norm2": n2, "n_obs": None, "mean": mean}
    key, st = torch.cat([h[0] for h in hits]), torch.cat([h[1] for h in hits])
    st = st[torch.sort(key).indices]
    rows = torch.zeros(HIT_CAPACITY, 4, dtype=torch.float64, device="cuda")
    if st.shape[0]:
        rows[HIT_CAPACITY - st.shape[0]:] = st[:HIT_CAPACITY]
    return {"n_hits": None, "hit_ids": None, "hit_stats": rows, "best_marker": None, "best_r": top}
