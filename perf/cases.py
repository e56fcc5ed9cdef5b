"""Timed cases: what programs that use this package have it do, through its public entry points.

A case is a dict of plain values.  ``prepare`` makes the inputs from a seed (case-control genotype
data in Hardy-Weinberg equilibrium with a planted interaction, as the package's synthetic data sets
have it, drawn on the GPU) and the handle or batch a program keeps; ``run`` is one pass; ``exact``
is the answer's scores in 64 bits, from plain torch.

Kinds: ``scan`` a resident handle's exhaustive triplet scan; ``range`` a rank's slice of it;
``oneshot`` create + scan + destroy per data set, from host or device arrays; ``batch`` many cohorts
in one call; ``pairs`` and ``order`` the scans of two and of four to six SNPs; ``noalloc`` the scan
for callers that cannot allocate.
"""
import math
import random

import numpy as np
import torch

import paper_2201_10956_gb300 as epi
from paper_2201_10956_gb300 import epi3

# exact() takes the sets of a case one leading combination at a time; bounds on that work
EXACT_SAMPLE_SETS = 2.0e12
EXACT_PREFIXES = 20000


def _case(name, kind, snps, samples, top_k, case_fraction=0.5, maf_lo=0.05, maf_hi=0.5, **extra):
    return dict(name=name, kind=kind, snps=snps, samples=samples, top_k=top_k,
                case_fraction=case_fraction, maf_lo=maf_lo, maf_hi=maf_hi, **extra)


def listed():
    return [
        # a candidate-gene panel: the smallest scan, where launches and latency count
        _case("scan_panel_64x512", "scan", 64, 512, 10),
        # an ordinary study with odd sizes and fewer cases than controls
        _case("scan_odd_701x5003", "scan", 701, 5003, 10, case_fraction=0.3),
        # the medium workload of the package's benchmark
        _case("scan_medium_1024x8192", "scan", 1024, 8192, 10),
        # its large (headline) workload: many samples, rare variants included
        _case("scan_large_2048x16384", "scan", 2048, 16384, 10, case_fraction=0.4, maf_lo=0.01),
        # its stress workload: many SNPs, few samples, a longer answer
        _case("scan_stress_4096x4096", "scan", 4096, 4096, 64, maf_lo=0.02),
        # a pipeline that opens a small data set already on the GPU, scans it and moves on
        _case("oneshot_device_300x2503", "oneshot", 300, 2503, 10, host=False),
        # the large workload end to end from host memory: copy, pack, scan, read back
        _case("oneshot_host_2048x16384", "oneshot", 2048, 16384, 10, case_fraction=0.4, maf_lo=0.01,
              host=True),
        # many cohorts of uneven size in one call (a third of the benchmark's 48)
        _case("batch_16_cohorts", "batch", 1024, 20000, 5, cohorts=16, snps_lo=96, samples_lo=1000,
              shape_seed=7),
        # the pairwise screen that usually precedes a third-order scan
        _case("pairs_4096x4096", "pairs", 4096, 4096, 64, maf_lo=0.02),
        # fourth- and fifth-order scans of a shortlist of SNPs
        _case("order4_120x2000", "order", 120, 2000, 20, order=4),
        _case("order5_48x1500", "order", 48, 1500, 20, order=5),
        # a caller with a fixed memory budget
        _case("noalloc_400x5003", "noalloc", 400, 5003, 10, case_fraction=0.4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan", "scan", "scan", "range", "oneshot", "oneshot", "batch", "pairs",
                       "order", "order", "noalloc"])
    frac = rng.choice([0.5, round(rng.uniform(0.2, 0.6), 3)])
    maf_lo = rng.choice([0.01, 0.02, 0.05])
    top_k = rng.choice([1, 5, 10, 20, 64])
    extra = {}
    if kind in ("scan", "range", "oneshot"):
        while True:  # no costlier than the largest listed scans
            m, n = _log_int(rng, 48, 4096), _log_int(rng, 300, 20000)
            if math.comb(m, 3) <= 1.15e10 and math.comb(m, 3) * n <= 2.4e13:
                break
        if kind == "range":
            parts = rng.choice([2, 4, 8])
            extra = dict(parts=parts, part=rng.randrange(parts))
        if kind == "oneshot":
            extra = dict(host=rng.random() < 0.5)
    elif kind == "batch":
        m, n = _log_int(rng, 200, 1024), _log_int(rng, 2000, 20000)
        extra = dict(cohorts=rng.randrange(2, 17), snps_lo=min(96, m), samples_lo=1000,
                     shape_seed=rng.randrange(1 << 30))
    elif kind == "pairs":
        m, n = _log_int(rng, 200, 6000), _log_int(rng, 300, 16384)
    elif kind == "order":
        order = rng.choice([4, 5, 6])
        lo, hi = {4: (20, 120), 5: (12, 48), 6: (12, 30)}[order]
        m, n = rng.randrange(lo, hi + 1), _log_int(rng, 200, 3000)
        extra = dict(order=order)
    else:
        m, n = _log_int(rng, 48, 512), _log_int(rng, 300, 8000)
    c = _case("", kind, m, n, top_k, frac, maf_lo, **extra)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------- inputs
def _shapes(case):
    """(SNPs, samples, case fraction) of every data set of the case."""
    if case["kind"] != "batch":
        return [(case["snps"], case["samples"], case["case_fraction"])]
    r = random.Random(case["shape_seed"])
    return [(r.randint(case["snps_lo"], case["snps"]), r.randint(case["samples_lo"], case["samples"]),
             r.uniform(0.2, 0.6)) for _ in range(case["cohorts"])]


def _dataset(case, shape, seed):
    """Genotypes [M, N] and phenotype [N] (uint8, on the GPU): allele frequencies uniform in the
    case's range, genotypes binomial, and three SNPs whose joint heterozygotes have three times the
    odds of being a case; exactly the wanted number of cases."""
    m, n, frac = shape
    gen = torch.Generator(device="cuda").manual_seed(seed)
    maf = case["maf_lo"] + (case["maf_hi"] - case["maf_lo"]) * torch.rand(m, generator=gen, device="cuda")
    planted = torch.randperm(m, generator=gen, device="cuda")[:3]
    maf[planted] = 0.25 + 0.25 * torch.rand(3, generator=gen, device="cuda")
    g = torch.zeros((m, n), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        g += (torch.rand((m, n), generator=gen, device="cuda") < maf[:, None]).to(torch.uint8)
    hit = (g[planted] == 1).all(dim=0)
    gumbel = -torch.log(-torch.log(torch.rand(n, generator=gen, device="cuda").clamp(1e-6, 1 - 1e-6)))
    n1 = max(1, min(n - 1, int(round(frac * n))))
    cases = torch.topk(gumbel + math.log(3.0) * hit, n1).indices
    ph = torch.zeros(n, dtype=torch.uint8, device="cuda")
    ph[cases] = 1
    return g, ph


def _datasets(case, seed):
    return [_dataset(case, s, seed * 1009 + c) for c, s in enumerate(_shapes(case))]


def _pinned(t):
    out = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    out.copy_(t)
    return out


def prepare(case, seed):
    kind = case["kind"]
    data = _datasets(case, seed)
    torch.cuda.synchronize()  # a handle packs its inputs on a stream of its own
    g, ph = data[0]
    state = dict(case=case)
    if kind == "batch":
        state["batch"] = epi.Batch(data)
    elif kind == "oneshot":
        if case["host"]:
            state["keep"] = (_pinned(g), _pinned(ph))
            state["data"] = tuple(t.numpy() for t in state["keep"])
        else:
            state["data"] = (g, ph)
    elif kind == "noalloc":
        state["data"] = (g, ph)
    else:
        state["handle"] = epi.Handle(g, ph)
    return state


def _slice(case):
    """The rank's share of the SNP pairs (equal counts of pairs)."""
    n = epi3.pairs_of(case["snps"])
    return n * case["part"] // case["parts"], n * (case["part"] + 1) // case["parts"]


def run(state):
    case = state["case"]
    kind, k = case["kind"], case["top_k"]
    if kind == "scan":
        return state["handle"].scan(k)
    if kind == "range":
        lo, hi = _slice(case)
        return state["handle"].scan_range(lo, hi, k)
    if kind == "oneshot":
        with epi.Handle(*state["data"]) as h:
            return h.scan(k)
    if kind == "batch":
        return state["batch"].scan(k)
    if kind == "pairs":
        return state["handle"].scan_pairs(k)
    if kind == "order":
        return state["handle"].scan_order(case["order"], k)
    return epi3.scan_noalloc(*state["data"], k)


# ---------------------------------------------------------------------------------- work
def _order(case):
    return {"pairs": 2}.get(case["kind"], case.get("order", 3))


def _counted_share(case):
    """Mean share of the samples that do not have a SNP's most frequent genotype (the one whose
    cells follow from the others)."""
    p = np.linspace(case["maf_lo"], case["maf_hi"], 1001)
    return float(np.mean(1.0 - np.maximum(np.maximum((1 - p) ** 2, 2 * p * (1 - p)), p * p)))


def work(case):
    order, k = _order(case), case["top_k"]
    share = _counted_share(case)
    nbytes = flops = 0.0
    for m, n, _ in _shapes(case):
        sets = float(math.comb(m, order))
        if case["kind"] == "range":
            lo, hi = _slice(case)
            sets = _range_triplets(m, lo, hi)
        # genotypes packed at two bits once resident, a byte each where the call takes the raw arrays
        raw = case["kind"] in ("oneshot", "noalloc")
        nbytes += m * n * (1.0 if raw else 0.25) + k * (4.0 * order + 8.0)
        # four multiply-adds per sample that the leading SNPs do not leave to derivation, and
        # about ten operations per cell of the score
        flops += sets * (8.0 * n * share ** (order - 2) + 10.0 * 3 ** order)
    return {"bytes": nbytes, "flops": flops}


def _range_triplets(m, lo, hi):
    total = 0
    for j in range(1, m - 1):
        a, b = max(lo, j * (j - 1) // 2), min(hi, j * (j - 1) // 2 + j)
        total += max(0, b - a) * (m - 1 - j)
    return float(total)


# ---------------------------------------------------------------------------------- exact
def _best_scores(g, ph, order, k, pair_range=None):
    """The k lowest K2 scores (natural log, sum over the 3^order cells of
    ln (r + 1)! - ln r0! - ln r1!) of all sets of `order` SNPs, in 64 bits: per leading order - 2
    SNPs, the tables of every pair of further SNPs by a matrix product of one-hot genotypes."""
    m, n = g.shape
    lf = torch.lgamma(torch.arange(n + 2, dtype=torch.float64, device=g.device) + 1.0)
    hot = [torch.stack([(g[:, ph == c] == v) for v in range(3)], dim=1).float() for c in range(2)]
    best = torch.empty(0, dtype=torch.float64, device=g.device)

    def visit(prefix, masks):
        nonlocal best
        lo = prefix[-1] + 1 if prefix else 0
        if len(prefix) < order - 2:
            for x in range(lo, m - (order - 1 - len(prefix))):
                visit(prefix + [x],
                      [(masks[c][:, None, :] * hot[c][x][None]).flatten(0, 1) for c in range(2)])
            return
        r = m - lo
        ia, ib = torch.triu_indices(r, r, 1, device=g.device)
        if pair_range is not None:  # pairs (i, j) by index j (j - 1) / 2 + i
            j = ia + lo
            p = torch.div(j * (j - 1), 2, rounding_mode="floor") + prefix[0]
            sel = (p >= pair_range[0]) & (p < pair_range[1])
            ia, ib = ia[sel], ib[sel]
        if ia.numel() == 0:
            return
        counts = []
        for c in range(2):
            rest = hot[c][lo:].flatten(0, 1)
            prod = (masks[c][:, None, :] * rest[None]).flatten(0, 1) @ rest.T
            prod = prod.view(-1, r, 3, r, 3)
            counts.append(prod[:, ia, :, ib, :].reshape(ia.numel(), -1).round().long())
        s = (lf[counts[0] + counts[1] + 1] - lf[counts[0]] - lf[counts[1]]).sum(dim=1)
        both = torch.cat([best, s])
        best = torch.topk(both, min(k, both.numel()), largest=False, sorted=True).values

    visit([], [torch.ones((1, hot[c].shape[2]), device=g.device) for c in range(2)])
    return best.sort().values


def exact(case, seed):
    order = _order(case)
    cost = sum(float(math.comb(m, order)) * n for m, n, _ in _shapes(case))
    lead = sum(math.comb(m, order - 2) for m, _, _ in _shapes(case))
    if cost > EXACT_SAMPLE_SETS or lead > EXACT_PREFIXES:
        return None
    pr = _slice(case) if case["kind"] == "range" else None
    best = [_best_scores(g, ph, order, case["top_k"], pr) for g, ph in _datasets(case, seed)]
    scores = torch.stack(best) if case["kind"] == "batch" else best[0]
    if case["kind"] == "oneshot" and case["host"]:
        scores = scores.cpu().numpy()
    return None, scores
