"""What the speed of this framework is judged by: the calls its users make, at the sizes they make them.

Every case is one pass through the public entry points of `paper_2408_10982_gb300.im` (the C ABI of
include/im.h).  Graphs are R-MAT graphs (a/b/c/d = 0.57/0.19/0.19/0.05) in in-CSR form with the weight models
of `paper_2408_10982_gb300.inputs`, made on the GPU from the seed; sizes are those of this repository's
workloads (R-MAT scale 10 to 20, the LiveJournal shape, the batched mix).  All outputs are whole numbers, or
follow from whole numbers by a closed form.

Kinds of case (see `listed` for what each stands for):
  query   reset a kept pool, sample theta RRR sets, select seeds (one or two covers)
  pool    sample and hand the RRR sets and the covering subsets to the caller
  cover   select seeds on a pool that is kept with its index
  imm     im_solve: the theta loop of IMM
  opim    im_opim: the OPIM rounds
  batch   im_solve_batch over many queries on resident graphs
  spread  im_spread: forward simulation of a seed set
  cold    a first query from host arrays: upload, sample, select, read back, free
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2408_10982_gb300 import im

DEV = "cuda"
TWO32 = 1 << 32
LJ_N, LJ_M = 4_847_571, 69_000_000     # the LiveJournal shape

# mean members of an RRR set, and the mean number of their in-edges, by weight model and log2(n): measured on R-MAT graphs of
# edge factor 14 to 16
MEAN_MEMBERS = {
    "lt": {10: 14.7, 12: 19.5, 14: 23.9, 17: 32.4, 20: 40.5, 22.2: 50.2},
    "lt-u0.1": {10: 3.6, 14: 3.7, 17: 3.7, 20: 3.7, 22.2: 3.2},
    "wc": {10: 8.4, 12: 10.3, 14: 12.2, 17: 15.5, 20: 19.5, 22.2: 25.5},
    "ic0.1": {10: 198.0, 12: 567.0, 14: 1744.0, 17: 9488.0, 20: 61031.0},
    "u0.1": {10: 91.7, 12: 271.0, 14: 809.0, 17: 4710.0, 20: 27581.0, 22.2: 113218.0},
    "trivalency": {10: 53.7, 12: 180.0, 14: 535.0, 17: 3353.0, 20: 22090.0, 22.2: 81612.0},
}
MEAN_IN_EDGES = {
    "wc": {10: 589.0, 12: 1282.0, 14: 2669.0, 17: 7867.0, 20: 22570.0, 22.2: 41315.0},
    "ic0.1": {10: 6322.0, 12: 21493.0, 14: 77392.0, 17: 515914.0, 20: 3968338.0},
    "u0.1": {10: 3689.0, 12: 13373.0, 14: 47589.0, 17: 344306.0, 20: 2437558.0, 22.2: 10273734.0},
    "trivalency": {10: 2411.0, 12: 10096.0, 14: 35892.0, 17: 281625.0, 20: 2251501.0, 22.2: 8585247.0},
}


# --- the cases -------------------------------------------------------------------------------------------


def listed():
    return [
        # the smallest call: a plain query on a small network whose pool is kept (launches and latency count)
        dict(name="query_ic_s10", kind="query", n=1024, m=16384, weights="ic0.1", theta=16384, k=16, covers="plain"),
        # an ordinary query of the batched mix asked alone, at an odd size: weighted cascade, RandGreedi
        dict(name="query_wc_s15", kind="query", n=31_337, m=501_393, weights="wc", theta=200_003, k=37, covers="rand64"),
        # the benchmark step: LT on R-MAT scale 20, both covers
        dict(name="step_lt_s20", kind="query", n=1 << 20, m=1 << 24, weights="lt", theta=1 << 22, k=100, covers="plain+rand148"),
        # the paper's own weights (U[0, 0.1]) under IC: sets that percolate, then the greedy on them
        dict(name="query_u01_s20", kind="query", n=1 << 20, m=1 << 24, weights="u0.1", theta=4096, k=100, covers="plain"),
        # the paper's own weights under LT (in-weights of a vertex differ): sets and covering subsets handed over
        dict(name="pool_ltu_s20", kind="pool", n=1_000_003, m=16_000_001, weights="lt-u0.1", theta=1 << 22),
        # trivalency IC on the LiveJournal shape: giant sets, handed over
        dict(name="pool_triv_lj", kind="pool", n=LJ_N, m=LJ_M, weights="trivalency", theta=1024),
        # seed selection on a kept pool (the paper's subject): RandGreedi at 512 parts, alpha = 1/8, and the lazy greedy
        dict(name="cover_wc_s20", kind="cover", n=1 << 20, m=1 << 24, weights="wc", theta=1 << 21, k=100, covers="rand512+lazy"),
        # IMM on the LiveJournal shape, weighted cascade, eps = 0.13, l = 1, k = 200
        dict(name="imm_wc_lj", kind="imm", n=LJ_N, m=LJ_M, weights="wc", k=200, eps=0.13),
        # OPIM at k = 1,000 with truncated RandGreedi, halves up to 2^20 sets
        dict(name="opim_lt_s20", kind="opim", n=1 << 20, m=1 << 24, weights="lt", k=1000, cap=1 << 20, covers="rand148"),
        # many queries at once: the batched mix (R-MAT scale 12 to 18, IC or LT, greedy or RandGreedi)
        dict(name="batch_mix_48", kind="batch", queries=48, lo=12, hi=18, theta_lo=1 << 14, theta_hi=1 << 20),
        # judging a seed set by forward simulation
        dict(name="spread_lt_s20", kind="spread", n=1 << 20, m=1 << 24, weights="lt", k=100, runs=256),
        # a first query, from host arrays to seeds
        dict(name="cold_lt_s20", kind="cold", n=1 << 20, m=1 << 24, weights="lt", theta=1 << 20, k=100, covers="plain"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["query", "query", "query", "pool", "pool", "cover", "imm", "opim", "batch", "spread", "cold"])
    if kind == "batch":
        lo = rng.randint(12, 16)
        a, b = sorted((_log_int(rng, 1 << 14, 1 << 20), _log_int(rng, 1 << 14, 1 << 20)))
        return dict(kind=kind, queries=_log_int(rng, 4, 48), lo=lo, hi=rng.randint(lo, 18), theta_lo=a, theta_hi=b + 1)
    n = _log_int(rng, 1 << 10, 1 << 20)
    m = int(n * rng.uniform(8.0, 16.0))
    light = ["lt", "lt", "wc", "wc", "lt-u0.1"]
    if kind == "spread":
        return dict(kind=kind, n=n, m=m, weights=rng.choice(["lt", "wc", "u0.1"]), k=rng.randint(1, 200), runs=_log_int(rng, 16, 256))
    if kind == "imm":
        return dict(kind=kind, n=max(n, 4096), m=max(m, 40_000), weights=rng.choice(["wc", "lt"]), k=rng.randint(10, 200), eps=rng.choice([0.13, 0.2, 0.3, 0.5]))
    rand = ["rand%d" % p for p in (16, 64, 148) if n <= 18_000 * p]     # a part's candidates fit one block
    if kind == "opim":
        return dict(kind=kind, n=max(n, 4096), m=max(m, 40_000), weights=rng.choice(["wc", "lt"]), k=rng.randint(10, 1000), cap=_log_int(rng, 1 << 14, 1 << 20),
                    covers=rng.choice(["plain"] + rand))
    weights = rng.choice(light + (["ic0.1", "u0.1", "trivalency"] if kind in ("query", "pool") else []))
    if weights in light:
        theta = _log_int(rng, 1 << 10, 1 << 22)
    else:                                              # percolating sets: members, not sets, bound the work
        theta = _log_int(rng, 64, max(128, min(1 << 14, int(3e7 / _mean_members(weights, n)))))
    c = dict(kind=kind, n=n, m=m, weights=weights, theta=theta)
    if kind != "pool":
        c |= dict(k=rng.randint(1, 100), covers=rng.choice(["plain", "plain", "lazy"] + rand))
    return c


# --- inputs ----------------------------------------------------------------------------------------------


def _rmat(n, m, gen):
    """About m distinct R-MAT edges without self-loops as in-CSR (edges sorted by head, then source), on the GPU."""
    levels = max(1, math.ceil(math.log2(n)))
    ta, tb, tc = (int(p * 4096) for p in (0.57, 0.76, 0.95))
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    accept = (n / (1 << levels)) ** 1.3 * 0.9          # candidates with both ends below n, and not seen before
    for _ in range(6):
        want = m - keys.numel()
        if want <= 0:
            break
        cand = min(int(want / accept) + 1024, 6 * m)
        src = torch.zeros(cand, dtype=torch.int32, device=DEV)
        dst = torch.zeros(cand, dtype=torch.int32, device=DEV)
        for lv in range(0, levels, 5):                 # 12 bits of one draw per level
            r = torch.randint(0, 1 << 60, (cand,), generator=gen, device=DEV)
            for _ in range(min(5, levels - lv)):
                q = r & 4095
                r >>= 12
                src = src * 2 + (q >= tb)
                dst = dst * 2 + (((q >= ta) & (q < tb)) | (q >= tc))
            del r
        ok = (src < n) & (dst < n) & (src != dst)
        new = (dst.to(torch.int64) * n + src)[ok]
        del src, dst, ok
        keys = torch.unique(torch.cat([keys, new]))
        del new
    if keys.numel() > m:                               # an even thinning of the sorted edges
        at = torch.arange(m, device=DEV, dtype=torch.float64) * (keys.numel() / m)
        keys = keys[at.to(torch.int64)]
    head = torch.div(keys, n, rounding_mode="floor")
    in_src = (keys - head * n).to(torch.int32)
    deg = torch.bincount(head, minlength=n)
    in_off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(deg, 0, out=in_off[1:])
    return in_off, in_src, deg


def _as_u32(w):
    """int64 values in [0, 2^32) as the bit pattern of uint32."""
    return torch.where(w >= 1 << 31, w - TWO32, w).to(torch.int32)


def _weights(kind, in_off, deg, m, gen):
    if kind in ("lt", "wc"):                           # 1 / in-degree
        per = torch.where(deg > 0, torch.clamp(TWO32 // deg.clamp(min=1), max=TWO32 - 1), torch.zeros_like(deg))
        return _as_u32(torch.repeat_interleave(per, deg))
    if kind == "ic0.1":
        return _as_u32(torch.full((m,), int(0.1 * TWO32 + 0.5), dtype=torch.int64, device=DEV))
    if kind == "trivalency":
        table = torch.tensor([int(p * TWO32 + 0.5) for p in (0.1, 0.01, 0.001)], dtype=torch.int64, device=DEV)
        return _as_u32(table[torch.randint(0, 3, (m,), generator=gen, device=DEV)])
    r = torch.rand(m, generator=gen, device=DEV, dtype=torch.float64) * 0.1
    if kind == "lt-u0.1":                              # scaled so that a vertex's in-weights sum to at most 1
        owner = torch.repeat_interleave(torch.arange(deg.numel(), device=DEV), deg)
        tot = torch.zeros(deg.numel(), dtype=torch.float64, device=DEV)
        tot.index_add_(0, owner, r)
        r = r / tot.clamp(min=1.0)[owner]
    return _as_u32(torch.floor(r * (TWO32 - 1024)).to(torch.int64))


class _Graph:
    """A resident graph of the library."""

    def __init__(self, n, m, weights, seed):
        gen = torch.Generator(DEV)
        gen.manual_seed(seed)
        in_off, in_src, deg = _rmat(n, m, gen)
        w = _weights(weights, in_off, deg, in_src.numel(), gen)
        self.n, self.m, self.top = n, in_src.numel(), torch.argsort(torch.bincount(in_src, minlength=n), descending=True)[:4096]
        self.model = im.IM_LT if weights.startswith("lt") else im.IM_IC
        self.arrays = in_off, in_src, w
        self.handle = None

    def upload(self):
        in_off, in_src, w = self.arrays
        self.handle = im.im_graph_create(in_off, in_src, w, self.n, self.m)
        self.arrays = None
        return self

    def __del__(self):
        if self.handle is not None:
            im.im_graph_destroy(self.handle)


def _covers(text):
    """"plain", "lazy" or "rand<parts>", several joined by "+", as (name, options) of im_max_k_cover."""
    out = []
    for c in text.split("+"):
        if c == "plain":
            out.append((c, None))
        elif c == "lazy":
            out.append((c, im.cover_opts(im.IM_GREEDY_LAZY)))
        else:
            parts = int(c[4:])
            out.append((c, im.cover_opts(im.IM_RANDGREEDI, parts, (1, 8) if parts > 256 else (1, 4), 0.077, 42, fused=False)))
    return out


def _fitting_pool(g, theta, seed, mean):
    """A pool that holds theta sets of this graph: its size from a first sample, as a program finds it out."""
    cap = int(theta * mean * 1.5) + g.n + 4096
    while True:
        pool = im.Pool(g, theta, cap)
        try:
            pool.sample(g.model, seed, 0, theta)
            break
        except im.ImError as e:
            if e.status != im.IM_ERR_CAPACITY:
                raise
            pool.close()
            cap *= 2
    return pool


def _batch(case, seed):
    rng = random.Random(seed)
    scales = list(range(case["lo"], case["hi"] + 1))
    graphs = {s: _Graph(1 << s, 16 << s, "lt", seed * 64 + s).upload() for s in scales}
    queries = []
    for q in range(case["queries"]):
        g = graphs[scales[q % len(scales)]]            # an even mix, so that two seeds cost about the same
        theta = int(case["theta_lo"] + (case["theta_hi"] - case["theta_lo"]) * (q * 0.618034 % 1.0)) + rng.randint(0, 99)
        opts = im.cover_opts(im.IM_RANDGREEDI, 64, (1, 4), 0.077, 42, fused=False) if q // 2 % 2 else None
        queries.append((g.handle, q % 2, rng.randint(5, 100), theta, rng.getrandbits(63), opts))
    return graphs, queries


def prepare(case, seed):
    kind, rs = case["kind"], (seed * 0x9E3779B97F4A7C15 + 1) % (1 << 63)
    st = dict(case=case, seed=rs)
    if kind == "batch":
        st["graphs"], st["queries"] = _batch(case, seed)
        st["handle"] = _Handle(im.im_batch_create(), im.im_batch_destroy)
        return st
    g = _Graph(case["n"], case["m"], case["weights"], seed)
    if kind == "cold":
        st["host"] = [x.cpu().pin_memory() for x in g.arrays]
        st["n"], st["m"], st["model"], st["covers"] = g.n, g.m, g.model, _covers(case["covers"])
        st["cap"] = int(case["theta"] * _mean_members(case["weights"], g.n) * 2) + 2 * g.n + 4096
        g.arrays = None
        return st
    st["graph"] = g.upload()
    if kind == "spread":                               # seeds: some of the vertices with the most out-edges
        gen = torch.Generator(DEV)
        gen.manual_seed(seed + 1)
        k = min(case["k"], g.top.numel())
        top = g.top[: max(k, min(4 * case["k"], g.top.numel()))]
        st["seeds"] = top[torch.randperm(top.numel(), generator=gen, device=DEV)[:k]].to(torch.int32).contiguous()
        st["activated"] = torch.zeros(case["runs"], dtype=torch.int64, device=DEV)
        st["root_hit"] = torch.zeros(case["runs"], dtype=torch.uint8, device=DEV)
        return st
    if kind in ("imm", "opim"):
        if kind == "opim":
            st["opts"] = _covers(case["covers"])[0][1]
        return st
    pool = st["pool"] = _fitting_pool(g, case["theta"], rs, _mean_members(case["weights"], g.n))
    if kind == "pool":
        total = max(pool.info()[1], int(case["theta"] * _mean_members(case["weights"], g.n) * 1.5) + g.n)   # room beyond the last member stays zero
        st["set_off"] = torch.empty(case["theta"] + 1, dtype=torch.int64, device=DEV)
        st["members"] = torch.zeros(total, dtype=torch.int32, device=DEV)
        st["vtx_off"] = torch.empty(g.n + 1, dtype=torch.int64, device=DEV)
        st["set_ids"] = torch.zeros(total, dtype=torch.int32, device=DEV)
        return st
    if kind == "cover":
        im.im_pool_index(pool.handle)
    st["covers"] = _covers(case["covers"])
    return st


class _Handle:
    def __init__(self, handle, destroy):
        self.handle, self.destroy = handle, destroy

    def __del__(self):
        self.destroy(self.handle)


# --- one pass --------------------------------------------------------------------------------------------


def _padded(a, k, fill):
    """Seeds or gains of a selection that may have stopped early, in k places."""
    out = np.full(k, fill, a.dtype)
    out[: a.size] = a
    return out


def _select(pool, k, covers):
    out = {}
    for name, opts in covers:
        c = pool.cover(k, opts)
        out[name] = (_padded(c.seeds, k, -1), _padded(c.gains, k, 0), c.coverage)
    return out


def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "batch":
        out = im.im_solve_batch(state["handle"].handle, state["queries"], 100)
        return dict(seeds=np.stack([_padded(r[0], 100, -1) for r in out]), gains=np.stack([_padded(r[1], 100, 0) for r in out]),
                    coverage=np.array([r[2] for r in out], np.int64), entries=np.array([r[3] for r in out], np.int64))
    if kind == "cold":
        handle = im.im_graph_create(*state["host"], state["n"], state["m"])
        graph = _Handle(handle, im.im_graph_destroy)
        graph.n = state["n"]
        pool = im.Pool(graph, case["theta"], state["cap"])
        pool.sample(state["model"], seed, 0, case["theta"])
        out = _select(pool, case["k"], state["covers"]), pool.info()
        pool.close()
        return out
    g = state["graph"]
    if kind == "spread":
        total = im.im_spread(g.handle, g.model, state["seeds"], seed, 0, case["runs"], state["activated"], state["root_hit"])
        return dict(total=total, activated=state["activated"], root_hit=state["root_hit"])
    if kind == "imm":
        seeds, cov, theta, info = im.im_solve(g.handle, g.model, case["k"], case["eps"], 1.0, seed)
        return dict(seeds=_padded(seeds, case["k"], -1), coverage=cov, theta=theta, lb=info.lb, theta_rounds=np.array(info.theta_rounds), cov_rounds=np.array(info.cov_rounds),
                    entries=(info.round_entries, info.final_entries), examined=info.examined)
    if kind == "opim":
        seeds, info = im.im_opim(g.handle, g.model, case["k"], 0.01, 1.0 / g.n, seed % (1 << 62), case["cap"], state["opts"])
        return dict(seeds=_padded(seeds, case["k"], -1), theta=np.array(info.theta), cov1=np.array(info.cov1), cov2=np.array(info.cov2), upper=np.array(info.cov1_upper),
                    alpha=np.array(info.alpha))
    pool = state["pool"]
    if kind != "cover":
        pool.reset()
        pool.sample(g.model, seed, 0, case["theta"])
    if kind == "pool":
        im.im_pool_export(pool.handle, state["set_off"], state["members"])
        im.im_index_export(pool.handle, state["vtx_off"], state["set_ids"])
        return dict(set_off=state["set_off"], members=state["members"], vtx_off=state["vtx_off"], set_ids=state["set_ids"], info=pool.info())
    return dict(_select(pool, case["k"], state["covers"]), info=pool.info())


# --- what a pass cannot do without -----------------------------------------------------------------------


def _at(table, n):
    """The table's value, interpolated in log2(n)."""
    x, at = math.log2(n), sorted(table)
    x = min(max(x, at[0]), at[-1])
    for a, b in zip(at, at[1:]):
        if x <= b:
            f = (x - a) / (b - a)
            return math.exp(math.log(table[a]) * (1 - f) + math.log(table[b]) * f)
    return table[at[-1]]


def _mean_members(weights, n):
    return _at(MEAN_MEMBERS[weights], n)


def _sample_bytes(weights, n, m, theta):
    """Sampling, from the definition of a set.  LT reads an offset pair and a picked source per member; IC decides over every
    in-edge of every member, whose probability it cannot do without (4 bytes; where all in-edges of a vertex have the same one,
    4 bytes a vertex), and reads an offset pair per member; both write a member and, per set, an offset.  The graph itself is read
    at most once where the sets together cover it (it fits the cache or is shared by the sets in flight)."""
    members = theta * _mean_members(weights, n)
    if weights.startswith("lt"):
        return members * 4 + min(members * 16, 8 * n + 4 * m) + theta * 8
    edges = theta * _at(MEAN_IN_EDGES[weights], n)
    graph = 8 * n + (4 * n if weights in ("wc", "ic0.1") else 4 * m)
    return members * 4 + min(graph, members * 16 + 4 * edges) + theta * 8


def _cover_bytes(members, theta):
    """Seed selection reads each set's members once when the set is first covered, and each seed's subset."""
    return 8 * members + theta / 8


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = 0.0
        scales = list(range(case["lo"], case["hi"] + 1))
        for q in range(case["queries"]):
            s = scales[q % len(scales)]
            theta = case["theta_lo"] + (case["theta_hi"] - case["theta_lo"]) * (q * 0.618034 % 1.0)
            w = "lt" if q % 2 else "wc"
            members = theta * _mean_members(w, 1 << s)
            total += _sample_bytes(w, 1 << s, 16 << s, theta) + 8 * members + _cover_bytes(members, theta)
        return {"bytes": total, "flops": 0}
    n, m, weights = case["n"], case["m"], case["weights"]
    if kind == "spread":                               # the out-edges of what is activated: 16 bytes each, about a tenth of the graph
        return {"bytes": case["runs"] * 0.1 * m * 16, "flops": 0}
    mean = _mean_members(weights, n)
    if kind == "imm":                                  # theta from the bound of IMM with an optimum of about n / 8
        lam = 2.0 * n * (0.63 * math.sqrt(math.log(n)) + math.sqrt(0.63 * case["k"] * math.log(n))) ** 2 / case["eps"] ** 2
        theta, covers = lam / (n / 8), 1
    elif kind == "opim":
        theta, covers = 2 * case["cap"], 1
    else:
        theta, covers = case["theta"], len(case["covers"].split("+")) if "covers" in case else 0
    members = theta * mean
    total = covers * _cover_bytes(members, theta)
    if kind != "cover":
        total += _sample_bytes(weights, n, m, theta) + 8 * members      # the sets, and their transpose read and written
    if kind == "pool":
        total += 16 * members
    if kind == "cold":
        total += 8 * (n + 1) + 8 * m
    return {"bytes": total, "flops": 0}


def exact(case, seed):
    """None: every output is a whole number that two correct programs agree on to the last bit (OPIM's ratios and IMM's
    bound follow from whole numbers by a closed form), so there is nothing that 64 bits would know better."""
    return None
