"""Performance cases: the calls a program that sketches and estimates joins makes.

Six kinds of case, each through the package's public classes:

  update    one batch of one relation added to a running sketch (SketchSet.update)
  estimate  the join size of sketches that are already filled (SketchSet.estimate)
  step      zero the sketches, update every relation, estimate
  plan      zero and refill many relations' sketches in one call each (UpdatePlan)
  many      the estimates of many sketch sets in one call (estimate_many)
  family    zero, update and estimate every sub-query of a star (SketchFamily)

Keys are int64 columns drawn from a Zipf law over [0, domain), the distribution the paper
fits to its databases' columns; "shuffled" keys are dictionary codes in no order of
frequency, the others code 0 as the most frequent value.  Weights are None (inserts),
turnstile (+1, a tenth -1) or amounts (-3 .. 3 without 0).  Every output is a whole number
(int64 counters, 256-bit estimates as four 64-bit words), so there is nothing to compare in
floating point.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

import paper_2402_15953_gb300 as sk


# ---- the listed cases -------------------------------------------------------------------

def listed():
    return [
        # a serving request at the low end: a few thousand tuples with deletions into one
        # relation of a chain, keys of unknown range
        _update("update_request", n=3001, a=2, m=1 << 14, d=9, domain=1_000_000, zipf=1.1, weights="turnstile"),
        # an ordinary ingest batch: a few hundred thousand tuples, a skewed pair of columns
        _update("update_batch", n=200_003, a=2, m=1 << 16, d=9, domain=1_000_000, zipf=1.1, weights="turnstile",
                shuffled=True),
        # the smallest whole query: three relations of ten thousand tuples, sketches of 256 bins
        _step("chain3_step", shape="chain", r=3, n=10_000, n_dim=10_000, m=256, d=5, domain=1000, zipf=1.0,
              declared=False),
        # the headline: a fact table of 1e8 rows joined to five dimension tables, domains known
        _step("star_step", shape="star", r=6, n=100_000_000, n_dim=1_000_000, m=1 << 16, d=9, domain=1_000_000,
              zipf=1.1, declared=True),
        # a fact table's change stream: inserts and deletions, dictionary-coded columns
        _update("star_turnstile", n=20_000_003, a=5, m=1 << 16, d=9, domain=1_000_000, zipf=1.1, declared=True,
                weights="turnstile", shuffled=True),
        # the same table from a source that does not say which keys can occur
        _update("star_undeclared", n=10_000_019, a=5, m=1 << 16, d=9, domain=1_000_000, zipf=1.1),
        # an inner relation of a chain of eight, at a width far beyond one SM's shared memory
        _update("chain8_update", n=10_000_000, a=2, m=1 << 20, d=16, domain=1_000_000, zipf=1.2, declared=True),
        # the largest estimate: eight relations of 1e7 tuples, 2^20 bins, 16 rows
        _estimate("chain8_estimate", shape="chain", r=8, n=10_000_000, m=1 << 20, d=16, domain=1_000_000, zipf=1.2),
        # the paper's own width, which is not a power of two
        _step("wide_odd_step", shape="chain", r=3, n=1_000_000, n_dim=1_000_000, m=1_000_000, d=5, domain=1_000_000,
              zipf=1.2, declared=False),
        # building many sketches of very different sizes at once
        {"name": "plan_build", "kind": "plan", "count": 96, "n": 100_000, "log2m_lo": 10, "log2m_hi": 18, "d": 7},
        # a plan enumerator's estimates over many live sketch sets
        {"name": "many_estimates", "kind": "many", "count": 64, "log2m_lo": 10, "log2m_hi": 18, "d": 7, "n": 20_000},
        # every sub-query of a four-way star: what a join-order search asks for
        {"name": "family_step", "kind": "family", "k": 4, "n": 20_000_000, "n_dim": 1_000_000, "m": 1 << 16, "d": 9,
         "domain": 1_000_000, "zipf": 1.1, "declared": True, "shuffled": False},
    ]


def _update(name, *, n, a, m, d, domain, zipf, declared=False, weights="none", shuffled=False):
    return {"name": name, "kind": "update", "n": n, "a": a, "m": m, "d": d, "domain": domain, "zipf": zipf,
            "declared": declared, "weights": weights, "shuffled": shuffled}


def _estimate(name, *, shape, r, n, m, d, domain, zipf):
    return {"name": name, "kind": "estimate", "shape": shape, "r": r, "n": n, "m": m, "d": d, "domain": domain,
            "zipf": zipf}


def _step(name, *, shape, r, n, n_dim, m, d, domain, zipf, declared, shuffled=False):
    return {"name": name, "kind": "step", "shape": shape, "r": r, "n": n, "n_dim": n_dim, "m": m, "d": d,
            "domain": domain, "zipf": zipf, "declared": declared, "shuffled": shuffled}


# ---- drawn cases ------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """Mostly powers of two, as in every configuration here; a quarter any width."""
    w = _log_int(rng, lo, hi)
    return w if rng.random() < 0.25 else 1 << (w.bit_length() - 1)


def draw(rng):
    kind = rng.choice(["update", "update", "update", "estimate", "step", "plan", "many", "family"])
    zipf = round(rng.uniform(0.8, 1.4), 2)
    domain = _log_int(rng, 1000, 2_000_000)
    d = rng.choice([5, 7, 9, 11, 16])
    declared, shuffled = rng.random() < 0.5, rng.random() < 0.5
    if kind == "update":
        c = _update("", n=_log_int(rng, 1000, 20_000_000), a=rng.randint(1, 5), m=_width(rng, 1 << 8, 1 << 20), d=d,
                    domain=domain, zipf=zipf, declared=declared,
                    weights=rng.choice(["none", "none", "turnstile", "amounts"]), shuffled=shuffled)
    elif kind == "estimate":
        shape = rng.choice(["chain", "star", "shared"])
        r = 4 if shape == "shared" else rng.randint(2, 8 if shape == "chain" else 6)
        c = _estimate("", shape=shape, r=r, n=_log_int(rng, 1000, 1_000_000), m=_width(rng, 1 << 8, 1 << 18), d=d,
                      domain=domain, zipf=zipf)
    elif kind == "step":
        n = _log_int(rng, 3000, 20_000_000)
        c = _step("", shape=rng.choice(["chain", "star"]), r=rng.randint(2, 6), n=n, n_dim=max(1000, n // 20),
                  m=_width(rng, 1 << 8, 1 << 18), d=d, domain=domain, zipf=zipf, declared=declared,
                  shuffled=shuffled)
    elif kind == "plan":
        c = {"kind": "plan", "count": rng.randint(8, 96), "n": _log_int(rng, 3000, 100_000), "log2m_lo": 10,
             "log2m_hi": rng.randint(12, 18), "d": rng.choice([5, 7, 9])}
    elif kind == "many":
        c = {"kind": "many", "count": rng.randint(4, 64), "log2m_lo": 10, "log2m_hi": rng.randint(12, 18),
             "d": rng.choice([5, 7, 9]), "n": _log_int(rng, 3000, 20_000)}
    else:
        n = _log_int(rng, 30_000, 20_000_000)
        c = {"kind": "family", "k": rng.randint(2, 4), "n": n, "n_dim": max(1000, n // 20),
             "m": 1 << rng.randint(10, 16), "d": min(d, 9), "domain": domain, "zipf": zipf, "declared": declared,
             "shuffled": shuffled}
    c.pop("name", None)
    return c


# ---- inputs -----------------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _cdf(zipf, domain):
    # summed on the host: a cumulative sum on the GPU differs in its last bits from run to run
    c = torch.cumsum(torch.arange(1, domain + 1, dtype=torch.float64).pow(-zipf), 0)
    return (c / c[-1]).cuda()


def _keys(gen, n, domain, zipf, shuffled=False):
    """n int64 keys in [0, domain), Zipf for zipf > 0, else uniform."""
    if not zipf:
        return torch.randint(0, domain, (n,), generator=gen, device="cuda")
    u = torch.rand(n, dtype=torch.float64, generator=gen, device="cuda")
    keys = torch.searchsorted(_cdf(zipf, domain), u, right=True).clamp_(max=domain - 1)
    if shuffled:
        keys = torch.randperm(domain, generator=gen, device="cuda")[keys]
    return keys


def _columns(gen, n, a, domain, zipf, shuffled=False):
    cols = torch.empty((a, n), dtype=torch.int64, device="cuda")
    for u in range(a):
        cols[u] = _keys(gen, n, domain, zipf, shuffled)
    return cols


def _weights(gen, n, kind):
    if kind == "none":
        return None
    if kind == "turnstile":
        return 1 - 2 * (torch.rand(n, generator=gen, device="cuda") < 0.1).to(torch.int64)
    w = torch.randint(-3, 3, (n,), generator=gen, device="cuda")
    return w + (w >= 0)


def _query(shape, r):
    """(join attributes per relation, joins) of a chain or star of r relations, or of four
    relations three of which share one attribute."""
    if shape == "chain":
        return ([1] + [2] * (r - 2) + [1] if r > 2 else [1] * r,
                [(k, 0 if k == 0 else 1, k + 1, 0) for k in range(r - 1)])
    if shape == "star":
        return [r - 1] + [1] * (r - 1), [(0, k, 1 + k, 0) for k in range(r - 1)]
    return [1, 2, 1, 1], [(0, 0, 1, 0), (2, 0, 1, 0), (3, 0, 1, 1)]


def _relations(gen, c, attrs):
    """Each relation's columns: the first one of c["n"] rows, in a star the others of
    c["n_dim"] uniform rows (dimension tables), in a chain all of c["n"] Zipf rows."""
    shuffled = c.get("shuffled", False)
    rels = []
    for k, a in enumerate(attrs):
        if k and c.get("shape", "star") == "star":
            rels.append(_columns(gen, c.get("n_dim", c["n"]), a, c["domain"], 0))
        else:
            rels.append(_columns(gen, c["n"], a, c["domain"], c["zipf"], shuffled))
    return rels


def _sizes(c):
    """The sketch sets of a plan or many case: (rows, columns, width, domain, skew) each."""
    rng = np.random.default_rng(7)
    out = []
    for _ in range(c["count"]):
        n = int(np.clip(rng.lognormal(math.log(c["n"]), 1.5), 1000, 100 * c["n"]))
        out.append((min(n, 5_000_000), int(rng.integers(1, 5)),
                    1 << int(rng.integers(c["log2m_lo"], c["log2m_hi"] + 1)), int(10 ** rng.uniform(4, 6.5)),
                    round(float(rng.uniform(0.8, 1.4)), 1)))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    hash_seed = seed * 7919 + 42
    kind = case["kind"]
    if kind == "update":
        attrs, joins = _query("star", case["a"] + 1)
        s = sk.SketchSet(attrs, joins, case["m"], case["d"], hash_seed)
        return {"kind": kind, "set": s,
                "cols": _columns(gen, case["n"], case["a"], case["domain"], case["zipf"], case["shuffled"]),
                "weights": _weights(gen, case["n"], case["weights"]),
                "domain": [case["domain"]] * case["a"] if case["declared"] else None}
    if kind in ("estimate", "step"):
        attrs, joins = _query(case["shape"], case["r"])
        s = sk.SketchSet(attrs, joins, case["m"], case["d"], hash_seed)
        rels = _relations(gen, case, attrs)
        doms = [[case["domain"]] * a if case.get("declared", True) else None for a in attrs]
        if kind == "step":
            return {"kind": kind, "set": s, "rels": rels, "doms": doms}
        for k, cols in enumerate(rels):
            s.update(k, cols, domain=doms[k])
        s.sync()
        return {"kind": kind, "set": s}
    if kind == "plan":
        sizes = _sizes(case)
        words = [(1 + a) * case["d"] * m for _, a, m, _, _ in sizes]
        counters = torch.zeros(sum(words), dtype=torch.int64, device="cuda")
        items, at = [], 0
        for i, ((n, a, m, domain, zipf), w) in enumerate(zip(sizes, words)):
            attrs, joins = _query("star", a + 1)
            s = sk.SketchSet(attrs, joins, m, case["d"], hash_seed + i,
                             counters=counters[at:at + w].view(1 + a, case["d"], m))
            items.append((s, 0, _columns(gen, n, a, domain, zipf), _weights(gen, n, "turnstile")))
            at += w
        return {"kind": kind, "plan": sk.UpdatePlan(items), "counters": counters}
    if kind == "many":
        sets = []
        for i, (_, a, m, domain, zipf) in enumerate(_sizes(case)):
            attrs, joins = _query("star", a + 1)
            s = sk.SketchSet(attrs, joins, m, case["d"], hash_seed + i)
            for k, b in enumerate(attrs):
                s.update(k, _columns(gen, case["n"], b, domain, zipf))
            s.sync()
            sets.append(s)
        return {"kind": kind, "sets": sets}
    k = case["k"]
    attrs, joins = _query("star", k + 1)
    subqueries = [list(c) for size in range(1, k + 1) for c in itertools.combinations(range(k), size)]
    fam = sk.SketchFamily(attrs, joins, subqueries, case["m"], case["d"], hash_seed)
    return {"kind": kind, "family": fam, "rels": _relations(gen, case, attrs),
            "doms": [[case["domain"]] * a if case["declared"] else None for a in attrs]}


# ---- one pass ---------------------------------------------------------------------------

def _words(values):
    """Signed 256-bit integers as rows of four 64-bit words, lowest first."""
    return np.frombuffer(b"".join(v.to_bytes(32, "little", signed=True) for v in values), np.int64).reshape(-1, 4)


def run(state):
    kind = state["kind"]
    if kind == "update":
        state["set"].update(0, state["cols"], state["weights"], state["domain"])
        return state["set"].counters[0]
    if kind == "estimate":
        e = state["set"].estimate()
        return {"rows": _words(e["rows"]), "median": _words([e["median"]])}
    if kind == "step":
        s = state["set"]
        s.reset()
        for k, cols in enumerate(state["rels"]):
            s.update(k, cols, domain=state["doms"][k])
        e = s.estimate()
        return {"counters": s.counters, "rows": _words(e["rows"]), "median": _words([e["median"]])}
    if kind == "plan":
        state["plan"].zero()
        state["plan"].run()
        return state["counters"]
    if kind == "many":
        return {"rows": _words([v for e in sk.estimate_many(state["sets"]) for v in e["rows"]])}
    fam = state["family"]
    fam.reset()
    for k, cols in enumerate(state["rels"]):
        fam.update(k, cols, domain=state["doms"][k])
    return {"rows": _words([v for e in fam.estimate() for v in e["rows"]])}


def exact(case, seed):
    """Every output is a whole number, equal or wrong: none has a nearest 64-bit value."""
    return None


def work(case):
    """Bytes a pass cannot do without: keys and weights read once, counters read by an
    estimate, counters added to by an update read and written (at most one per tuple and
    row), estimates written.  The arithmetic is integer hashing and exact transforms."""
    c = case
    if c["kind"] == "update":
        touched = min(c["n"] * c["d"], c["m"] * c["d"])
        return {"bytes": c["n"] * 8 * (c["a"] + (c["weights"] != "none")) + 16 * touched, "flops": 0}
    if c["kind"] in ("estimate", "step"):
        attrs, _ = _query(c["shape"], c["r"])
        counters = 8 * c["r"] * c["d"] * c["m"]
        if c["kind"] == "estimate":
            return {"bytes": counters + 32 * c["d"], "flops": 0}
        keys = sum(8 * a * (c["n_dim"] if k and c["shape"] == "star" else c["n"]) for k, a in enumerate(attrs))
        return {"bytes": keys + 2 * counters + 32 * c["d"], "flops": 0}
    if c["kind"] == "plan":
        return {"bytes": sum(8 * n * (a + 1) + 8 * c["d"] * m for n, a, m, _, _ in _sizes(c)), "flops": 0}
    if c["kind"] == "many":
        return {"bytes": sum(8 * (1 + a) * c["d"] * m + 32 * c["d"] for _, a, m, _, _ in _sizes(c)), "flops": 0}
    subs = (1 << c["k"]) - 1
    views = subs + c["k"]
    return {"bytes": 8 * c["k"] * (c["n"] + c["n_dim"]) + 2 * 8 * views * c["d"] * c["m"] + 32 * subs * c["d"],
            "flops": 0}
