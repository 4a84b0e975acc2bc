"""Timed cases of the framework, each one pass through its public entry points on inputs made from a seed.

The cases are the calls that a user of the library makes: closures of one relation from a few hundred constants up to the
headline graph, partially grounded queries (one row and a batch), compositions, the grouped batch over a knowledge graph's
relations, the composed isForeign program, insertion of new facts and the relation operators, on byte matrices (the
binding's default format) and on packed bit rows. Sizes and graph families are those of bench.py and of the workload
generators (uniform random digraphs, power-law digraphs, grids, a knowledge graph, a place hierarchy).
"""
import math
import random

import torch

from paper_2408_10369_gb300 import bmlp

U8, PACKED = bmlp.BMLP_FMT_U8, bmlp.BMLP_FMT_PACKED64
_FMT = {"u8": U8, "packed": PACKED}
_context = None


def _ctx():
    """The context that a program keeps for all of its calls."""
    global _context
    if _context is None:
        _context = bmlp.Context(0)
    return _context


def listed():
    return [
        # a small database (the paper's examples and unit-sized programs): call latency
        {"name": "rms_er300_u8", "kind": "rms", "family": "er", "n": 300, "degree": 2.0, "fmt": "u8", "variant": "auto", "reflexive": False},
        # the smallest benchmark graph: n = 2,000, p = 2 / n
        {"name": "rms_er2000_u8", "kind": "rms", "family": "er", "n": 2000, "degree": 2.0, "fmt": "u8", "variant": "auto", "reflexive": False},
        # the paper's DG workload: n = 5,000, p_t = 0.1, as a byte matrix
        {"name": "rms_dg5000_u8", "kind": "rms", "family": "er", "n": 5000, "degree": 500.0, "fmt": "u8", "variant": "auto", "reflexive": False},
        # the headline closure
        {"name": "rms_er32768_packed", "kind": "rms", "family": "er", "n": 32768, "degree": 4.0, "fmt": "packed", "variant": "auto", "reflexive": False},
        # a power-law relation of the dispatcher's corpus, by the variant that its model picks there; n is no multiple of 64
        {"name": "frontier_pl20011", "kind": "rms", "family": "powerlaw", "n": 20011, "degree": 2.1, "fmt": "packed", "variant": "smp_packed", "reflexive": False},
        # the paper's DG+partial workload: one query path(c, Y)
        {"name": "smp_dg5000_q1", "kind": "smp", "family": "er", "n": 5000, "degree": 50.0, "fmt": "packed", "q": 1, "sources": 1},
        # the selective query batch: 4,096 rows of 1 to 64 sources
        {"name": "smp_pl65536_q4096", "kind": "smp", "family": "powerlaw", "n": 65536, "degree": 2.1, "fmt": "packed", "q": 4096, "sources": 64},
        # p <- r1 ; p <- r2, p on byte matrices of odd size
        {"name": "compose_er9001_u8", "kind": "compose", "n": 9001, "degree": 2.0, "degree2": 3.0, "fmt": "u8"},
        # every relation's closure and 200 compositions of a knowledge graph of FB15k-237's shape
        {"name": "batch_kg", "kind": "batch", "entities": 15000, "relations": 1345, "triples": 483000, "compositions": 200},
        # the composed program on the place hierarchy
        {"name": "foreign_14541", "kind": "foreign", "n": 14541, "contains": 5993, "adjoins": 1998, "roots": 200, "fmt": "packed"},
        # a growing database: 1,000 new facts into the hierarchy's closure
        {"name": "insert_14541_m1000", "kind": "insert", "n": 14541, "contains": 5993, "roots": 200, "m": 1000, "fmt": "packed"},
        # relation operators: NEG of the symmetric closure of a relation under a type predicate
        {"name": "operators_14541_u8", "kind": "operators", "n": 14541, "degree": 4.0, "fmt": "u8"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rms", "rms", "rms", "frontier", "smp", "smp", "compose", "batch", "foreign", "insert", "operators"])
    fmt = rng.choice(["u8", "packed"])
    if kind == "rms":
        n = _log(rng, 256, 20000)
        if n <= 8192 and rng.random() < 0.3:
            degree = round(n * rng.choice([0.01, 0.1, 0.5]), 3)
        else:
            degree = round(rng.uniform(1.5, 8.0), 3)
        return {"kind": "rms", "family": rng.choice(["er", "er", "powerlaw", "hubs", "grid"]) if degree < 8.0 else "er", "n": n,
                "degree": degree, "fmt": fmt, "variant": "auto", "reflexive": rng.random() < 0.25}
    if kind == "frontier":
        return {"kind": "rms", "family": rng.choice(["er", "powerlaw", "hubs", "grid"]), "n": _log(rng, 1000, 20000),
                "degree": round(rng.uniform(1.8, 3.0), 3), "fmt": fmt, "variant": "smp_packed", "reflexive": False}
    if kind == "smp":
        one = rng.random() < 0.5
        n = _log(rng, 512, 8192) if one else _log(rng, 1000, 65536)
        return {"kind": "smp", "family": "er" if one else rng.choice(["er", "powerlaw", "hubs"]), "n": n,
                "degree": round(n * rng.choice([0.001, 0.01, 0.1]), 3) if one else round(rng.uniform(1.8, 4.0), 3), "fmt": "packed",
                "q": rng.randint(1, 8) if one else _log(rng, 16, 4096), "sources": 1 if one else rng.choice([1, 8, 64])}
    if kind == "compose":
        return {"kind": "compose", "n": _log(rng, 256, 12000), "degree": round(rng.uniform(1.5, 4.0), 3),
                "degree2": round(rng.uniform(1.5, 4.0), 3), "fmt": fmt}
    if kind == "batch":
        e = _log(rng, 1000, 12000)
        return {"kind": "batch", "entities": e, "relations": max(20, e // 11), "triples": 30 * e, "compositions": max(4, e // 75)}
    if kind == "foreign":
        n = _log(rng, 1000, 14541)
        return {"kind": "foreign", "n": n, "contains": int(n * rng.uniform(0.2, 0.6)), "adjoins": max(8, int(n * rng.uniform(0.05, 0.3))),
                "roots": max(4, n // 70), "fmt": fmt}
    if kind == "insert":
        n = _log(rng, 500, 14541)
        return {"kind": "insert", "n": n, "contains": int(n * rng.uniform(0.2, 0.6)), "roots": max(4, n // 70), "m": _log(rng, 4, 1000), "fmt": fmt}
    return {"kind": "operators", "n": _log(rng, 500, 14541), "degree": round(rng.uniform(1.5, 8.0), 3), "fmt": fmt}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(shape, g):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _randint(hi, shape, g):
    return torch.randint(0, hi, shape, generator=g, device="cuda", dtype=torch.int64)


def _distinct(i, j, n, loops=False):
    if not loops:
        keep = i != j
        i, j = i[keep], j[keep]
    key = torch.unique(i * n + j)
    return key // n, key % n


def _er(n, degree, g):
    """Uniform random digraph of that mean out-degree without self-loops. Dense ones are over 95 % of the constants, as a relation over
    a program's shared constant index is (their closure is everything else)."""
    if degree * 64 >= n:
        a = torch.rand((n, n), generator=g, device="cuda") < degree / max(n - 1, 1)
        a.fill_diagonal_(False)
        e = a.nonzero()
        i, j = e[:, 0], e[:, 1]
    else:
        m = int(round(n * degree))
        i, j = _distinct(_randint(n, (m,), g), _randint(n, (m,), g), n)
    if degree >= 10:
        used = _rand((n,), g) < 0.95
        keep = used[i] & used[j]
        i, j = i[keep], j[keep]
    return i, j


def _powerlaw(n, alpha, g, hubs=False):
    """Out-degrees Zipf(alpha) truncated to 1 .. min(1000, n / 4); targets by preferential attachment (an urn with every constant once:
    exponential popularities), or with hubs (popularity ~ rank^-1/2)."""
    top = max(2, min(1000, n // 4))
    w = torch.arange(1, top + 1, device="cuda", dtype=torch.float64) ** -alpha
    cdf = torch.cumsum(w / w.sum(), 0)
    deg = torch.searchsorted(cdf, _rand((n,), g)).clamp_(max=top - 1) + 1
    i = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    if hubs:
        j = torch.randperm(n, generator=g, device="cuda")[(n * _rand((i.numel(),), g) ** 2).long().clamp_(max=n - 1)]
    else:
        popular = torch.cumsum(-torch.log1p(-_rand((n,), g)), 0)
        j = torch.searchsorted(popular, _rand((i.numel(),), g) * popular[-1]).clamp_(max=n - 1)
    return _distinct(i, j, n)


def _grid(n, g):
    """2-D grid (edges right and down) plus round(n / 100) random shortcuts."""
    side = max(1, math.isqrt(n))
    x = torch.arange(n, device="cuda")
    right = x[(x % side != side - 1) & (x + 1 < n)]
    down = x[x + side < n]
    m = max(1, round(n / 100))
    i = torch.cat([right, down, _randint(n, (m,), g)])
    j = torch.cat([right + 1, down + side, _randint(n, (m,), g)])
    return _distinct(i, j, n)


def _edges(family, n, degree, g):
    if family in ("powerlaw", "hubs"):
        return _powerlaw(n, degree, g, family == "hubs")
    return _grid(n, g) if family == "grid" else _er(n, degree, g)


def _words(n):
    return (n + 63) // 64


def _rows(i, j, rows, n):
    """Packed bit rows (rows x ceil(n / 64) words) with the distinct entries (i, j)."""
    w = torch.zeros(rows * _words(n), dtype=torch.int64, device="cuda")
    w.index_add_(0, i * _words(n) + (j >> 6), torch.ones_like(j) << (j & 63))
    return w.view(rows, _words(n))


def _matrix(i, j, n, fmt):
    if fmt == "packed":
        return _rows(i, j, n, n)
    m = torch.zeros((n, n), dtype=torch.uint8, device="cuda")
    m[i, j] = 1
    return m


def _like(n, fmt):
    return torch.empty((n, _words(n)), dtype=torch.int64, device="cuda") if fmt == "packed" else torch.empty((n, n), dtype=torch.uint8, device="cuda")


def _forest(n, facts, roots, g):
    """contains facts of a place hierarchy: constants roots .. roots + facts - 1 each below an earlier one (popular parents first)."""
    facts = min(facts, n - roots)
    child = torch.arange(roots, roots + facts, device="cuda")
    parent = (_rand((facts,), g) ** 2 * child.double()).long()
    label = torch.randperm(n, generator=g, device="cuda")
    return label[parent], label[child]


def _kg_problems(case):
    """(n, [(first constant, constants, triples) of R1, and of R2 for a composition]) of every problem of a knowledge graph: relations of
    Zipf(1.1) frequency, each over the entities that it names; compositions of relation pairs over the entities of both."""
    e, r = case["entities"], case["relations"]
    total = sum(k ** -1.1 for k in range(1, r + 1))
    triples = [max(1, round(case["triples"] * k ** -1.1 / total)) for k in range(1, r + 1)]
    size = [max(2, round(e * (1 - math.exp(-2 * t / e)))) for t in triples]
    problems = [(n, [(0, n, t)]) for n, t in zip(size, triples)]
    pick = random.Random(1)
    for _ in range(case["compositions"]):
        a, b = pick.sample(range(r), 2)
        n = round(size[a] + size[b] - size[a] * size[b] / e)
        problems.append((n, [(0, size[a], triples[a]), (n - size[b], size[b], triples[b])]))
    return problems


def _kg(case, g):
    """The problems' matrices with uniform heads and tails in one buffer, and one buffer for the results."""
    problems = _kg_problems(case)
    mats = [(n, *m) for n, ms in problems for m in ms]
    first_row, first_word, rows, words = [], [], 0, 0
    for n, *_ in mats:
        first_row.append(rows)
        first_word.append(words)
        rows += n
        words += n * _words(n)
    dev = lambda v: torch.tensor(v, dtype=torch.int64, device="cuda")  # noqa: E731
    n, lo, cnt, t = (dev([m[k] for m in mats]) for k in range(4))
    m = torch.repeat_interleave(torch.arange(len(mats), device="cuda"), t)
    i = lo[m] + (_rand((m.numel(),), g) * cnt[m]).long()
    j = lo[m] + (_rand((m.numel(),), g) * cnt[m]).long()
    keep = i != j
    m, i, j = m[keep], i[keep], j[keep]
    key = torch.unique((dev(first_row)[m] + i) * (1 << 20) + j)
    row, j = key >> 20, key & ((1 << 20) - 1)
    m = torch.searchsorted(dev(first_row), row, right=True) - 1
    i = row - dev(first_row)[m]
    data = torch.zeros(words, dtype=torch.int64, device="cuda")
    data.index_add_(0, dev(first_word)[m] + i * ((n[m] + 63) // 64) + (j >> 6), torch.ones_like(j) << (j & 63))
    out = torch.empty(sum(n * _words(n) for n, _ in problems), dtype=torch.int64, device="cuda")
    items, at, k = [], 0, 0
    for n, ms in problems:
        size = n * _words(n)
        it = {"kind": bmlp.BMLP_PROBLEM_CLOSURE if len(ms) == 1 else bmlp.BMLP_PROBLEM_COMPOSE, "n": n, "fmt": PACKED, "out": out[at:at + size]}
        at += size
        for name in ("R1", "R2")[:len(ms)]:
            it[name] = data[first_word[k]:first_word[k] + size]
            k += 1
        items.append(it)
    return items, out, data


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": dict(case), "ctx": _ctx()}
    if kind == "batch":
        # the context holds the batch's instantiated graph, so a program that evaluates a knowledge graph keeps one for it
        s["ctx"] = bmlp.Context(0)
        items, s["out"], s["keep"] = _kg(case, g)
        s["problems"] = bmlp.Context.problems(items)
        return s
    n, fmt = case["n"], case.get("fmt", "packed")
    if kind == "rms":
        s["R"], s["out"] = _matrix(*_edges(case["family"], n, case["degree"], g), n, fmt), _like(n, fmt)
    elif kind == "smp":
        i, j = _edges(case["family"], n, case["degree"], g)
        s["R"] = _matrix(i, j, n, fmt)
        q, most = case["q"], case["sources"]
        count = _randint(most, (q,), g) + 1
        row = torch.repeat_interleave(torch.arange(q, device="cuda"), count)
        # single constants are asked about where they have facts; larger source sets are uniform
        col = i[_randint(i.numel(), (row.numel(),), g)] if most == 1 else _randint(n, (row.numel(),), g)
        s["src"] = _rows(*_distinct(row, col, n, loops=True), q, n)
        s["out"] = torch.empty_like(s["src"])
    elif kind == "compose":
        s["R1"] = _matrix(*_er(n, case["degree"], g), n, fmt)
        s["R2"] = _matrix(*_er(n, case["degree2"], g), n, fmt)
        s["out"] = _like(n, fmt)
    elif kind == "foreign":
        s["contains"] = _matrix(*_forest(n, case["contains"], case["roots"], g), n, fmt)
        s["adjoins"] = _matrix(*_distinct(_randint(n, (case["adjoins"],), g), _randint(n, (case["adjoins"],), g), n), n, fmt)
        s["out"] = _like(n, fmt)
    elif kind == "insert":
        s["closure"], s["out"] = _like(n, fmt), _like(n, fmt)
        s["ctx"].rms(_matrix(*_forest(n, case["contains"], case["roots"], g), n, fmt), n, s["closure"], fmt=_FMT[fmt])
        s["facts"] = torch.stack([_randint(n, (case["m"],), g), _randint(n, (case["m"],), g)], 1).to(torch.int32).contiguous()
    else:
        s["R"], s["out"] = _matrix(*_er(n, case["degree"], g), n, fmt), _like(n, fmt)
        s["t"], s["u"] = _like(n, fmt), _like(n, fmt)
        typed = (_rand((n,), g) < 0.8).nonzero().view(-1)
        s["type"] = _rows(torch.zeros_like(typed), typed, 1, n)
    return s


def run(s):
    c, ctx = s["case"], s["ctx"]
    kind = c["kind"]
    if kind == "batch":
        return {"results": s["out"], "products": torch.tensor(ctx.batch_run(s["problems"]))}
    n, fmt = c["n"], _FMT[c.get("fmt", "packed")]
    if kind == "rms":
        return {"closure": s["out"], "products": ctx.rms(s["R"], n, s["out"], fmt=fmt, variant=c["variant"], reflexive=c["reflexive"])}
    if kind == "smp":
        return {"rows": s["out"], "levels": ctx.smp(s["R"], n, s["src"], c["q"], s["out"], fmt=fmt)}
    if kind == "compose":
        return {"p": s["out"], "products": ctx.compose(s["R1"], s["R2"], n, s["out"], fmt=fmt)}
    if kind == "foreign":
        return {"foreign": s["out"], "products": list(ctx.is_foreign(s["contains"], s["adjoins"], n, s["out"], fmt=fmt))}
    if kind == "insert":
        s["out"].copy_(s["closure"])  # the program keeps the closure that it had
        ctx.insert(s["out"], n, s["facts"], fmt=fmt)
        return {"closure": s["out"]}
    ctx.transpose(s["R"], n, s["t"], fmt=fmt)
    ctx.union(s["R"], s["t"], n, s["u"], fmt=fmt)
    ctx.negate(s["u"], n, s["out"], rows=s["type"], cols=s["type"], fmt=fmt)
    return {"transposed": s["t"], "union": s["u"], "negated": s["out"]}


def work(case):
    """Bytes of the inputs and outputs. The operations depend on the graph and on the method, so none are counted as indispensable."""
    if case["kind"] == "batch":
        return {"bytes": sum((len(ms) + 1) * n * _words(n) * 8 for n, ms in _kg_problems(case)), "flops": 0}
    n = case["n"]
    m = n * (n if case.get("fmt") == "u8" else 8 * _words(n))
    matrices = {"rms": 2, "smp": 1, "compose": 3, "foreign": 3, "insert": 2, "operators": 7}[case["kind"]]
    rows = 2 * case["q"] * 8 * _words(n) if case["kind"] == "smp" else 0
    return {"bytes": matrices * m + rows, "flops": 0}


def exact(case, seed):
    """Every output is bytes, bit words or counts, which stay equal to the bit: there are no floating values."""
    return None
