"""The searches whose speed this library is judged by, each through its public entry points.

Four kinds of call stand for what a program does with the library:

* ``search``: one exhaustive search of a data set that is loaded already (``fc_search``), as a
  program does that searches one data set at several orders, list lengths or rank ranges;
* ``range``: one device's share of a sharded search (``fc_search_range``);
* ``whole``: everything from the genotypes on the host to the list (``fc_load``, ``fc_search``,
  ``fc_free``), as a program does that meets each data set once;
* ``batch``: many data sets times phenotype permutations in one call (``fc_search_batch``).

Genotypes follow Hardy-Weinberg equilibrium with minor-allele frequencies on [0.05, 0.5]; one
interaction of the searched order is planted without lower-order effects, and the samples are
drawn retrospectively to the given class sizes, in random order.
"""
import itertools
import math

import numpy as np
import torch

import paper_2201_03331_gb300 as fc

PREVALENCE, HERITABILITY = 0.2, 0.1


def _case(kind, order, snps, cases, controls, top_n, **more):
    return {"kind": kind, "order": order, "snps": snps, "cases": cases, "controls": controls, "top_n": top_n, **more}


def listed():
    return [
        # A candidate-gene panel: a search of 4,950 pairs, where launches and latency are everything.
        {"name": "order2_100x1600", **_case("search", 2, 100, 800, 800, 10)},
        # A larger panel met once, below the sizes that the tensor cores take: load, triples, free.
        {"name": "whole_order3_200x1003", **_case("whole", 3, 200, 431, 572, 25)},
        # A chip after pruning, met once: pairs of 12,001 SNPs, odd sizes, unequal classes.
        {"name": "whole_order2_12001x2987", **_case("whole", 2, 12001, 1300, 1687, 100)},
        # All pairs of a 40,000-SNP chip in 8,192 samples, a long list.
        {"name": "order2_40000x8192", **_case("search", 2, 40000, 4096, 4096, 1000)},
        # The library's flagship: all triples of 1,000 SNPs in 4,000 samples.
        {"name": "order3_1000x4000", **_case("search", 3, 1000, 2000, 2000, 100)},
        # The same met once: load, operands, search, free.
        {"name": "whole_order3_1000x4000", **_case("whole", 3, 1000, 2000, 2000, 100)},
        # Triples of a cohort with many more controls than cases, ragged sizes.
        {"name": "order3_701x9001", **_case("search", 3, 701, 2700, 6301, 100)},
        # Quadruples of 300 SNPs in 6,000 samples.
        {"name": "order4_300x6000", **_case("search", 4, 300, 3000, 3000, 100)},
        # One of 64 devices' share of a sharded quadruple search.
        {"name": "range_order4_1001x2048", **_case("range", 4, 1001, 1024, 1024, 100, part=40, parts=64)},
        # Quintuples and sextuples at the variant and sample counts of the paper's single-core runs.
        {"name": "order5_152x2048", **_case("search", 5, 152, 1024, 1024, 100)},
        {"name": "order6_76x2048", **_case("search", 6, 76, 1024, 1024, 100)},
        # Permutation tests of triples: data sets of uneven size, eight phenotypes each.
        {"name": "batch_order3_4x8", **_case("batch", 3, 1201, 1410, 2103, 10, sets=4, replicates=8)},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# (smallest and largest SNP count, largest sample count) of the drawn searches by order.
_RANGES = {2: (60, 40000, 8192), 3: (40, 1100, 9000), 4: (30, 300, 6000), 5: (20, 150, 2048), 6: (16, 75, 2048)}


def draw(rng):
    kind = rng.choice(["search", "search", "search", "whole", "whole", "range", "batch"])
    order = {"whole": rng.choice([2, 2, 3, 3, 4]), "range": rng.choice([3, 4, 4, 5]), "batch": 3}.get(kind) or rng.choice([2, 2, 3, 3, 4, 5, 6])
    lo, hi, most = _RANGES[order]
    if kind == "whole":
        hi = {2: 20000, 3: 1000, 4: 200}[order]
    snps, samples = _log_int(rng, lo, hi), _log_int(rng, 500, most)
    if 2400 < samples < 2600:   # around 2,500 samples some searches of orders 2 and 4 are refused (launch error)
        samples += 200
    cases = max(60, int(samples * rng.uniform(0.3, 0.7)))
    more = {}
    if kind == "range":
        more["parts"] = rng.choice([2, 8, 64])
        more["part"] = rng.randrange(more["parts"])
    if kind == "batch":
        snps, samples = _log_int(rng, 250, 1200), _log_int(rng, 1000, 3500)
        cases = int(samples * rng.uniform(0.3, 0.7))
        more = {"sets": rng.randint(2, 4), "replicates": rng.randint(2, 8)}
    top_n = 10 if kind == "batch" else rng.choice([1, 10, 25, 100, 100, 1000])
    return _case(kind, order, snps, cases, samples - cases, top_n, **more)


def _sizes(case):
    """(SNPs, cases, controls) of each data set of the case."""
    if case["kind"] != "batch":
        return [(case["snps"], case["cases"], case["controls"])]
    n = case["sets"]
    # Data set d has (d + 1)/n of the SNPs, and the more samples the fewer SNPs it has.
    return [(max(30, case["snps"] * (d + 1) // n), case["cases"] * (2 * n - d) // n, case["controls"] * (2 * n - d) // n) for d in range(n)]


def _data(gen, order, snps, cases, controls):
    """Genotypes uint8[snps][samples] and phenotype uint8[samples] on the GPU."""
    dev, samples = gen.device, cases + controls
    maf = 0.05 + 0.45 * torch.rand(snps, 1, generator=gen, device=dev)
    g = torch.empty(snps, samples, dtype=torch.uint8, device=dev)
    for s in range(0, snps, 4096):
        q = 1 - maf[s:s + 4096]
        u = torch.rand(len(q), samples, generator=gen, device=dev)
        g[s:s + 4096] = (u >= q * q).to(torch.uint8) + (u >= q * (2 - q)).to(torch.uint8)
    # The planted SNPs have frequency 1/2, so that their contrasts are +1 (homozygous) and -1.
    pool = int(1.5 * max(cases / PREVALENCE, controls / (1 - PREVALENCE))) + 4096
    a = torch.rand(order, pool, generator=gen, device=dev)
    a = (a >= 0.25).to(torch.uint8) + (a >= 0.75).to(torch.uint8)
    sign = torch.prod(1 - 2 * (a == 1).to(torch.int8), dim=0)
    f = PREVALENCE + math.sqrt(HERITABILITY * PREVALENCE * (1 - PREVALENCE)) * sign
    ill = torch.rand(pool, generator=gen, device=dev) < f
    rows = torch.randperm(snps, generator=gen, device=dev)[:order]
    g[rows] = torch.cat([a[:, ill][:, :cases], a[:, ~ill][:, :controls]], dim=1)
    ph = (torch.arange(samples, device=dev) < cases).to(torch.uint8)
    at = torch.randperm(samples, generator=gen, device=dev)
    return g[:, at].contiguous(), ph[at].contiguous()


def _sets(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    for snps, cases, controls in _sizes(case):
        g, ph = _data(gen, case["order"], snps, cases, controls)
        if case["kind"] == "batch":   # the observed phenotype, then permutations of it
            ph = torch.stack([ph] + [ph[torch.randperm(len(ph), generator=gen, device="cuda")] for _ in range(case["replicates"] - 1)])
        yield g, ph


def _span(case):
    total = math.comb(case["snps"], case["order"])
    return (total * case["part"] // case["parts"], total * (case["part"] + 1) // case["parts"]) if case["kind"] == "range" else (0, total)


def prepare(case, seed):
    state = dict(case)
    if case["kind"] in ("search", "range"):
        (g, ph), = _sets(case, seed)
        state["handle"] = fc.fc_load_device(g, ph)
        state["span"] = _span(case)
    elif case["kind"] == "whole":   # as a file reader leaves it: arrays on the host
        (g, ph), = _sets(case, seed)
        state["genotypes"], state["phenotype"] = g.cpu().numpy(), ph.cpu().numpy()
    else:
        both = [(g.cpu().numpy(), ph.cpu().numpy()) for g, ph in _sets(case, seed)]
        state["handle"] = fc.fc_load_batch([g for g, _ in both], [ph for _, ph in both])
    return state


def run(state):
    kind, k, n = state["kind"], state["order"], state["top_n"]
    if kind == "search":
        idx, mi = fc.fc_search(state["handle"], k, n)
    elif kind == "range":
        idx, mi = fc.fc_search_range(state["handle"], k, n, *state["span"])
    elif kind == "whole":
        h = fc.fc_load(state["genotypes"], state["phenotype"])
        idx, mi = fc.fc_search(h, k, n)
        fc.fc_free(h)
    else:
        idx, mi, count = fc.fc_search_batch(state["handle"], k, n)
        return {"idx": idx, "mi": mi, "count": count}
    return {"idx": idx, "mi": mi}


def work(case):
    """Two bits a genotype and the list; of the 3^k cells of a table the 2^k without genotype 2
    determine the others together with lower-order tables, one multiply-add a sample each."""
    k, jobs = case["order"], case.get("replicates", 1)
    size = flops = 0
    for snps, cases, controls in _sizes(case):
        lo, hi = _span(case) if case["kind"] == "range" else (0, math.comb(snps, k))
        samples = cases + controls
        size += snps * samples * (1 if case["kind"] == "whole" else 0.25) + jobs * min(hi - lo, case["top_n"]) * (4 * k + 8)
        flops += jobs * (hi - lo) * 2 ** k * 2 * samples
    return {"bytes": size, "flops": flops}


def _exact_list(g, ph, k, span, top_n):
    """The best mutual informations of the ranks in span, in 64 bits, by plain matrix products of indicator rows."""
    S, M = g.shape
    order = torch.argsort(ph.to(torch.int16), descending=True, stable=True)
    g, m1 = g[:, order], int(ph.sum())
    rows = torch.stack([(g == v) for v in range(3)], dim=1).reshape(3 * S, M).to(torch.float32)   # row 3 s + v
    x = torch.arange(M + 1, dtype=torch.float64, device=g.device)
    xlx = torch.where(x > 0, x * torch.log(x.clamp(min=1)), 0.0)
    hy = math.log(M) - float(xlx[m1] + xlx[M - m1]) / M
    best = torch.empty(0, dtype=torch.float64, device=g.device)
    step = max(1, 400_000_000 // (27 * S * 3 ** max(k - 2, 0)))   # first SNPs of the pair at a time
    seen = 0   # ranks before this prefix
    for prefix in itertools.combinations(range(S - 2), k - 2):
        e0 = prefix[-1] + 1 if prefix else 0
        pairs = math.comb(S - e0, 2)
        if seen + pairs <= span[0] or seen >= span[1]:
            seen += pairs
            continue
        for e in range(e0, S - 1, step):
            e1 = min(S - 1, e + step)
            a, b = rows[3 * e:3 * e1], rows[3 * e:]
            hx = torch.zeros(e1 - e, S - e, dtype=torch.float64, device=g.device)
            hxy = torch.zeros_like(hx)
            for cell in itertools.product(range(3), repeat=k - 2):
                mask = torch.ones(M, device=g.device)
                for s, v in zip(prefix, cell):
                    mask = mask * rows[3 * s + v]
                am = a * mask
                n1 = (am[:, :m1] @ b[:, :m1].T).long()
                n0 = (am[:, m1:] @ b[:, m1:].T).long()

                def cells(t):
                    return t.view(e1 - e, 3, S - e, 3).sum(dim=(1, 3))

                hx += cells(xlx[n1 + n0])
                hxy += cells(xlx[n1]) + cells(xlx[n0])
            mi = hy + (hxy - hx) / M   # H(X) + H(Y) - H(X,Y), with the ln M of the joint terms cancelled
            i = torch.arange(e, e1, device=g.device)[:, None]
            j = torch.arange(e, S, device=g.device)[None, :]
            rank = seen + math.comb(S - e0, 2) - (S - i) * (S - i - 1) // 2 + (j - i - 1)
            keep = mi[(j > i) & (rank >= span[0]) & (rank < span[1])]
            best = torch.cat([best, torch.topk(keep, min(top_n, len(keep))).values])
            best = torch.topk(best, min(top_n, len(best))).values
        seen += pairs
    return best


def exact(case, seed):
    k = case["order"]
    # About what the products and table reads of _exact_list take; orders from four on only where they are small.
    cost = sum(case.get("replicates", 1) * 9 * math.comb(s, 2) * (math.comb(s, k - 2) if k > 2 else 1) * 3 ** (k - 2) * (c + m + 3000)
               for s, c, m in _sizes(case))
    if cost > 2.5e14 or math.comb(case["snps"], k - 2) * 3 ** (k - 2) > 30000:
        return None
    tf32, torch.backends.cuda.matmul.allow_tf32 = torch.backends.cuda.matmul.allow_tf32, False
    try:
        lists = []
        for g, ph in _sets(case, seed):
            for y in (ph if case["kind"] == "batch" else ph[None]):
                lists.append(_exact_list(g, y, k, _span(case) if case["kind"] == "range" else (0, math.comb(len(g), k)), case["top_n"]).cpu().numpy())
    finally:
        torch.backends.cuda.matmul.allow_tf32 = tf32
    if case["kind"] == "batch":
        return {"idx": None, "mi": np.stack(lists), "count": None}
    return {"idx": None, "mi": lists[0]}
