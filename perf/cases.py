"""The work a user has this library do, as cases that can be timed and compared.

A user builds (or is given) an index file once, loads it once, keeps the handle and
sends batches of queries with ranges. So an index here belongs to a shape, not to a
seed: its base set comes from a fixed seed, the file is built through the public
builder and kept in the cache folder, the handle is kept for the process, and a
case's seed draws what changes from call to call: query vectors, ranges, second
attributes. Construction itself is a case too; its vectors come from the case's seed.

Shapes (the workloads the repository is configured, tested and benchmarked with):
  ints128   1,000,000 x 128, integer-valued mixture in [0, 255], S = 16
  unit96    200,000 x 96, unit-normalised mixture, S = 8
  nonneg960 100,000 x 960, non-negative mixture in [0, 1], S = 8
  gauss     n x d of N(0, 1), attribute a permutation, S = 8 (10,000 x 64 unless the
            case says otherwise)
"""
from __future__ import annotations

import functools
import hashlib
import math
import os
import tempfile

import numpy as np
import torch

import paper_2412_02448_gb300 as U

DEV = "cuda:0"
BASE_SEED = 1234
DTYPES = {"fp32": U.FP32, "bf16": U.BF16, "fp8": U.FP8E4M3}

# n, d, S, efc, attribute domain (None: a permutation of 0..n-1)
SHAPES = {
    "ints128": dict(n=1_000_000, d=128, S=16, efc=100, domain=1_000_000),
    "unit96": dict(n=200_000, d=96, S=8, efc=100, domain=1_000_000),
    "nonneg960": dict(n=100_000, d=960, S=8, efc=32, domain=1_000_000),
    "gauss": dict(n=10_000, d=64, S=8, efc=100, domain=None),
}
M = 16

# Parameters a case may set; the others keep the library's defaults.
PARAMS = ("ef", "ef_post", "m", "cand_cap", "visited_cap", "reg_budget", "tc_scan", "selection", "scan_rows",
          "rerank_mult")

# The benchmark's tuned parameters on the 1M integer shape (tau as fractions of n).
TUNED = dict(ef=16, ef_post=96, m=64, tau_a=0.05, tau_b=0.6, cand_cap=256, visited_cap=1024, reg_budget=80, tc_scan=1)


def listed():
    return [
        # online serving, one request at a time: nothing but latency
        dict(name="one_query", shape="ints128", entry="search", strategy="auto", nq=1, k=10, fracs="0.1", dtype="fp32",
             ef=64, ef_post=128, m=32),
        # a few exact answers over ranges of some thousand rows (ground truth, small tenants)
        dict(name="few_exact", shape="ints128", entry="search", strategy="pre", nq=17, k=10, fracs="0.01,0.02",
             dtype="fp32"),
        # a small table searched through a captured plan, parameters as the tuner leaves them there
        dict(name="small_table_plan", shape="gauss", entry="plan", strategy="auto", nq=200, k=10, fracs="0.01,0.1,0.5",
             dtype="fp32", ef=48, ef_post=384, m=48, tau_a=0.03, tau_b=0.6, cand_cap=768, visited_cap=4096),
        # a service with host buffers in and out, a wide beam, the warp scan
        dict(name="host_service", shape="ints128", entry="host", strategy="auto", nq=1003, k=10,
             fracs="0.001,0.01,0.1,0.5,1.0", dtype="fp32", ef=64, ef_post=128, m=64),
        # the benchmark's batch, tuned, in the three storage formats that serve it
        dict(name="batch_fp32", shape="ints128", entry="search", strategy="auto", nq=10_000, k=10,
             fracs="0.001,0.01,0.1,0.5,1.0", dtype="fp32", **TUNED),
        dict(name="batch_bf16", shape="ints128", entry="search", strategy="auto", nq=10_000, k=10,
             fracs="0.001,0.01,0.1,0.5,1.0", dtype="bf16", **TUNED),
        # log-uniform ranges on FP8 storage with the warp scan
        dict(name="logu_fp8", shape="unit96", entry="search", strategy="auto", nq=5001, k=10, fracs="logu", dtype="fp8",
             ef=16, ef_post=128, m=64, tau_a=0.015, tau_b=0.75, cand_cap=512),
        # many results per query (candidate generation for a later ranking stage)
        dict(name="k100_fp32", shape="unit96", entry="search", strategy="auto", nq=2000, k=100, fracs="0.01,0.1,0.5",
             dtype="fp32", ef=128, ef_post=256, m=32, tc_scan=1),
        # high dimension, short ranges: all pre-filter, on the tensor cores ...
        dict(name="wide_exact_bf16", shape="nonneg960", entry="search", strategy="pre", nq=5000, k=10,
             fracs="0.005,0.02,0.1", dtype="bf16", tc_scan=1),
        # ... and with every distance in FP32
        dict(name="wide_exact_fp32", shape="nonneg960", entry="search", strategy="pre", nq=301, k=10,
             fracs="0.005,0.02,0.1", dtype="fp32"),
        # a second predicate on top of the range
        dict(name="two_attributes", shape="ints128", entry="conj", strategy="auto", nq=999, k=10, fracs="0.01,0.1,0.5",
             dtype="fp32", ef=64, ef_post=128, m=64),
        # construction of a small table's index, the file included
        dict(name="build_small", shape="gauss", entry="build", n=10_000, d=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any entry point, storage format and strategy, batch sizes over
    their range, k up to 100, odd table shapes on the small side."""
    kind = rng.choice(["online", "batch", "batch", "exact", "wide", "small", "small", "conj", "build"])
    if kind == "build":
        return dict(shape="gauss", entry="build", n=_log_int(rng, 2000, 10_000), d=rng.choice([17, 50, 64, 100, 128]))
    c = dict(dtype=rng.choice(["fp32", "fp32", "bf16", "fp8"]), k=rng.choice([1, 5, 10, 10, 20, 33, 100]))
    frac = lambda lo, hi: ",".join("%.5f" % math.exp(rng.uniform(math.log(lo), math.log(hi)))
                                   for _ in range(rng.randint(1, 4)))
    if kind == "online":
        c.update(shape="ints128", entry=rng.choice(["search", "host"]), strategy="auto", nq=_log_int(rng, 1, 300),
                 fracs=frac(0.001, 1.0), ef=rng.choice([32, 64, 100]), m=rng.choice([16, 32, 64]))
    elif kind == "batch":
        c.update(shape=rng.choice(["ints128", "unit96"]), entry=rng.choice(["search", "search", "host"]),
                 strategy=rng.choice(["auto", "auto", "hybrid", "post"]), nq=_log_int(rng, 300, 9000),
                 fracs=rng.choice(["logu", frac(0.002, 1.0)]), ef=rng.choice([16, 32, 64]),
                 ef_post=rng.choice([64, 96, 128]), m=rng.choice([16, 32, 48, 64]), tc_scan=rng.choice([0, 1]),
                 reg_budget=rng.choice([128, 80, 64]), selection=rng.choice([2, 2, 2, 1]))
        if c["k"] > 33:
            c["k"] = 33
    elif kind == "exact":
        c.update(shape=rng.choice(["ints128", "unit96"]), entry="search", strategy="pre", nq=_log_int(rng, 1, 700),
                 fracs=frac(0.0005, 0.03), tc_scan=rng.choice([0, 1]))
    elif kind == "wide":
        c.update(shape="nonneg960", entry="search", strategy="pre", fracs=frac(0.002, 0.1), tc_scan=rng.choice([0, 1, 1]))
        c["nq"] = _log_int(rng, 3, 4000 if c["tc_scan"] else 300)
    elif kind == "small":
        n = _log_int(rng, 2000, 20_000)
        c.update(shape="gauss", n=n, d=rng.choice([17, 50, 64, 100, 128, 200, 333]),
                 entry=rng.choice(["search", "plan"]), strategy=rng.choice(["auto", "hybrid", "post", "pre"]),
                 nq=_log_int(rng, 1, 3000), fracs=frac(0.005, 1.0), ef=rng.choice([48, 100, 200]),
                 m=rng.choice([16, 48]))
    else:
        st = rng.choice(["auto", "pre"])
        c.update(shape="ints128", entry="conj", strategy=st, nq=_log_int(rng, 10, 2000),
                 fracs=frac(0.002, 0.02 if st == "pre" else 1.0))
    if c["entry"] == "host":
        c["strategy"] = "auto"  # the entry point's only one
    return c


# ---- base sets and indexes -------------------------------------------------------

def _gen(*seed):
    g = torch.Generator(device=DEV)
    h = hashlib.sha256(repr(seed).encode()).digest()
    g.manual_seed(int.from_bytes(h[:7], "little"))
    return g


def _spec(case):
    s = dict(SHAPES[case["shape"]])
    s.update({f: int(case[f]) for f in ("n", "d") if f in case})
    return case["shape"], s


def _points(shape, d, count, g):
    """`count` vectors of the shape's distribution, around the shape's own centroids."""
    def normal():
        return torch.randn((count, d), generator=g, device=DEV)

    if shape == "gauss":
        return normal()
    nc = 500 if shape == "unit96" else 1000
    gc = _gen(BASE_SEED, shape, d, "centroids")
    lab = torch.randint(0, nc, (count,), generator=g, device=DEV)
    if shape == "ints128":
        c = torch.rand((nc, d), generator=gc, device=DEV) * 255.0
        return (c[lab] + 20.0 * normal()).round_().clamp_(0.0, 255.0)
    if shape == "unit96":
        c = torch.nn.functional.normalize(torch.randn((nc, d), generator=gc, device=DEV))
        return torch.nn.functional.normalize(c[lab] + (0.35 / math.sqrt(d)) * normal())
    c = torch.rand((nc, d), generator=gc, device=DEV) ** 2
    return (c[lab] + 0.08 * normal()).clamp_(0.0, 1.0)


@functools.lru_cache(maxsize=None)
def _base(shape, n, d, seed=BASE_SEED):
    """(vectors, attributes) on the host."""
    s = SHAPES[shape]
    g = _gen(seed, shape, n, d, "base")
    x = _points(shape, d, n, g).cpu().numpy()
    if s["domain"] is None:
        a = torch.randperm(n, generator=g, device=DEV)
    else:
        a = torch.randint(0, s["domain"], (n,), generator=g, device=DEV)
    return x, a.to(torch.int64).cpu().numpy()


def _cache_dir():
    """The repository's cache folder where it can be written, else a temporary one."""
    d = os.environ.get("UNIFY_CACHE_DIR", os.path.abspath("_cache"))
    try:
        os.makedirs(d, exist_ok=True)
        with tempfile.TemporaryFile(dir=d):
            return d
    except OSError:
        return tempfile.mkdtemp(prefix="hsig_")


def _code_digest():
    """Of the libraries that build an index: another build of either has its own files."""
    h = hashlib.sha256()
    for p in (U.LIB_PATH, os.path.join(os.path.dirname(os.path.dirname(U.LIB_PATH)), "hsig_build", "libhsig_build.so")):
        with open(p, "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:12]


@functools.lru_cache(maxsize=None)
def _index(shape, n, d, tag=""):
    """The handle a program keeps; `tag` gives a case that pins scratch its own."""
    s = SHAPES[shape]
    path = os.path.join(_cache_dir(), "cases_%s_n%d_d%d_%s.idx" % (shape, n, d, _code_digest()))
    if not os.path.exists(path):
        x, a = _base(shape, n, d)
        U.build_index(x, a, path, s["S"], M, s["efc"], seed=7)
    return U.Index(path, device=0)


# ---- cases -----------------------------------------------------------------------

def _queries(case, seed):
    """(q, lo, hi) on the device: vectors of the base set's distribution, inclusive
    ranges of the case's widths (fractions of the attribute domain) at uniform offsets."""
    shape, s = _spec(case)
    nq, domain = int(case["nq"]), s["domain"] or s["n"]
    g = _gen(seed, shape, s["n"], s["d"], nq, "queries")
    q = _points(shape, s["d"], nq, g).contiguous()
    if case["fracs"] == "logu":
        f = 10.0 ** (-4.0 * torch.rand(nq, generator=g, device=DEV, dtype=torch.float64))
    else:
        fl = torch.tensor([float(v) for v in case["fracs"].split(",")], dtype=torch.float64, device=DEV)
        f = fl[torch.arange(nq, device=DEV) % len(fl)]
    w = (f * domain).round().clamp(1, domain).to(torch.int64)
    u = torch.rand(nq, generator=g, device=DEV, dtype=torch.float64)
    lo = torch.minimum((u * (domain - w + 1)).to(torch.int64), domain - w)
    return q, lo, lo + w - 1


def _second(case, seed):
    """Second attribute of every object (fixed, as the table's column) and a range on it
    per query: 20, 50 or 100 % of its domain in turn."""
    _, s = _spec(case)
    nq, domain = int(case["nq"]), 1000
    a2 = torch.randint(0, domain, (s["n"],), generator=_gen(BASE_SEED, "second", s["n"]), device=DEV)
    g = _gen(seed, "second", nq)
    w = torch.tensor([200, 500, 1000], device=DEV)[torch.arange(nq, device=DEV) % 3]
    lo2 = (torch.rand(nq, generator=g, device=DEV, dtype=torch.float64) * (domain - w + 1)).to(torch.int64)
    lo2 = torch.minimum(lo2, domain - w)
    return a2, lo2, lo2 + w - 1


def _params(case, n):
    kw = {f: int(case[f]) for f in PARAMS if f in case}
    kw.update({f: int(case[f] * n) for f in ("tau_a", "tau_b") if f in case})
    p = U.Params.defaults(dtype=DTYPES[case["dtype"]], **kw)
    beam = max(p.ef, p.ef_post)
    if beam > p.cand_cap // 2:
        p.cand_cap = min(4096, 2 * beam)
    return p


def prepare(case, seed):
    shape, s = _spec(case)
    n, d = s["n"], s["d"]
    if case["entry"] == "build":
        x, a = _base.__wrapped__(shape, n, d, ("build", seed))
        return dict(entry="build", x=x, a=a, S=s["S"], efc=s["efc"], dir=tempfile.mkdtemp(prefix="hsig_"))
    q, lo, hi = _queries(case, seed)
    plan = case["entry"] == "plan"
    ix = _index(shape, n, d, repr(sorted(case.items())) if plan else "")
    st = dict(entry=case["entry"], ix=ix, q=q, lo=lo, hi=hi, k=int(case["k"]), strategy=case["strategy"],
              params=_params(case, n))
    if plan:
        st["plan"] = ix.plan(q, lo, hi, st["k"], strategy=st["strategy"], params=st["params"])
    elif case["entry"] == "conj":
        st["a2"], st["lo2"], st["hi2"] = _second(case, seed)
    elif case["entry"] == "host":
        nq, k = int(case["nq"]), st["k"]
        for f in ("q", "lo", "hi"):
            st[f] = st[f].cpu().pin_memory()
        st["out"] = dict(ids=torch.empty((nq, k), dtype=torch.int64).pin_memory(),
                         dist=torch.empty((nq, k), dtype=torch.float32).pin_memory(),
                         count=torch.empty(nq, dtype=torch.int32).pin_memory(),
                         status=torch.empty(nq, dtype=torch.int32).pin_memory())
    return st


def run(st):
    if st["entry"] == "build":
        path = U.build_index(st["x"], st["a"], os.path.join(st["dir"], "table.idx"), st["S"], M, st["efc"], seed=3)
        return np.fromfile(path, dtype=np.uint8)
    if st["entry"] == "plan":
        return st["plan"].launch()
    if st["entry"] == "host":
        return st["ix"].search_auto_host(st["q"], st["lo"], st["hi"], st["k"], params=st["params"], out=st["out"])
    more = dict(attr2=st["a2"], lo2=st["lo2"], hi2=st["hi2"]) if st["entry"] == "conj" else {}
    return st["ix"].search(st["q"], st["lo"], st["hi"], st["k"], strategy=st["strategy"], params=st["params"], **more)


def _fractions(case):
    if case["fracs"] == "logu":
        return [10.0 ** (-4.0 * (i + 0.5) / 64) for i in range(64)]
    return [float(v) for v in case["fracs"].split(",")]


def work(case):
    """Inputs read once, outputs written once, and of the index what a search of that
    kind has to look at: for exact scans the rows of the ranges (their union, at most the
    table) and one distance per query and in-range row; for graph searches the beam's
    expansions, each with its selected neighbours' ids, and about a quarter of these
    neighbours' rows (the others were seen before), taken from the beam's width. For
    construction the vectors, the stored edges, and a beam search per object and segment."""
    _, s = _spec(case)
    n, d = s["n"], s["d"]
    if case["entry"] == "build":
        return {"bytes": n * d * 4.0 + n * s["S"] * M * 4.0 * 2, "flops": 3.0 * d * n * s["S"] * s["efc"] * 2}
    nq, k = int(case["nq"]), int(case["k"])
    row = d * {"fp32": 4, "bf16": 2, "fp8": 1}[case["dtype"]]
    ef, ef_post, m = case.get("ef", 100), case.get("ef_post", case.get("ef", 100)), case.get("m", 16)
    ta, tb = case.get("tau_a", 0.01), case.get("tau_b", 0.5)
    exact_rows = graph_bytes = evals = 0.0
    fr = _fractions(case)
    for f in fr:
        share = nq / len(fr)
        st = case["strategy"]
        if st == "auto":
            st = "pre" if f <= ta else "post" if f >= tb else "hybrid"
        if st == "pre":
            exact_rows += share * f * n
        else:
            beam, ids = (max(ef, k), m) if st == "hybrid" else (max(ef_post, k), M)
            e = share * beam * ids / 4
            evals += e
            graph_bytes += e * row + share * beam * ids * 4
    b = min(exact_rows, n) * row + graph_bytes + nq * (d * 4 + 16) + nq * (k * 12 + 8)
    return {"bytes": b, "flops": 2.0 * d * exact_rows + 3.0 * d * evals}


def exact(case, seed):
    """The distances of the exact answer (the k nearest in-range objects, all of them when
    there are fewer), in 64 bits, where the case asks for the exact strategy. A graph
    search returns what its walk finds, and construction a graph: no such value."""
    shape, s = _spec(case)
    if case.get("strategy") != "pre":
        return None
    x, a = _base(shape, s["n"], s["d"])
    x = torch.from_numpy(x).to(DEV).double()
    a = torch.from_numpy(a).to(DEV)
    q, lo, hi = _queries(case, seed)
    k = int(case["k"])
    if case["entry"] == "conj":
        a2, lo2, hi2 = _second(case, seed)
    xn = (x * x).sum(1)
    out = torch.full((len(lo), k), math.inf, dtype=torch.float64, device=DEV)
    step = max(1, 200_000_000 // s["n"])
    for b in range(0, len(lo), step):
        e = min(len(lo), b + step)
        qb = q[b:e].double()
        dist = torch.addmm(xn[None, :] + (qb * qb).sum(1)[:, None], qb, x.t(), alpha=-2.0)
        inside = (a[None, :] >= lo[b:e, None]) & (a[None, :] <= hi[b:e, None])
        if case["entry"] == "conj":
            inside &= (a2[None, :] >= lo2[b:e, None]) & (a2[None, :] <= hi2[b:e, None])
        dist.masked_fill_(~inside, math.inf)
        kk = min(k, s["n"])
        out[b:e, :kk] = dist.topk(kk, dim=1, largest=False, sorted=True).values.clamp_(min=0.0)
    return {"ids": None, "dist": out, "count": None, "status": None}
