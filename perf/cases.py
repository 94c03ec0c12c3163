"""The work this framework is used for, as cases that can be timed and checked.

A case is one pass through the public entry points of ``paper_2507_17215_gb300`` on a
synthetic temporal graph of the repository's recipes (``workloads/``: Chung-Lu static
edges with heavy-tailed multiplicities and bursty times, the paper-scale one with
planted communities), drawn here on the GPU so that large inputs are quick to make:

* ``build``:  an edge list in, load + preprocessing + the analyst's queries, results out;
* ``query``:  one query on a resident, preprocessed graph;
* ``batch``:  a mixed batch of queries on a resident graph (what the server runs);
* ``counts``: per-edge counts into the caller's device memory, without allocation.

``exact`` answers the same questions from the definition (every triangle, every temporal
edge, two searches in sorted runs) with plain torch in 64-bit integers.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2507_17215_gb300 as folty

YEAR_S = 31_536_000
OUT, IN, EITHER = folty.DIR_OUT, folty.DIR_IN, folty.DIR_EITHER
HEAD, TAIL, COMMON = folty.U_HEAD, folty.U_TAIL, folty.U_COMMON
EXISTS, FORALL = folty.Q_EXISTS, folty.Q_FORALL_T

INFO = ("n", "m", "m_kept", "static_edges", "max_degree", "degeneracy", "triangles", "probes", "sigma_max",
        "time_sorted")
EXACT_MAX_EDGES = 25_000_000  # larger graphs hold a billion (edge, witness) pairs
CHUNK = 1 << 24               # (edge, witness) pairs handled together by exact()
MAX_PAIRS = 1 << 20           # solution pairs a pass of any case stays below


def _case(name, kind, recipe, m, **kw):
    c = {"name": name, "kind": kind, "recipe": recipe, "m": m, "order": "time", "unit": "s", "source": "device",
         "delta": 3600, "dir": OUT, "quant": FORALL, "universe": HEAD, "rho_num": 1, "rho_den": 2, "queries": 1,
         "edge_counts": False, "certificates": False, "vertices": False, "triples": False}
    c.update(kw)
    return c


def listed():
    return [
        # a small interaction log, analysed once: launches and round trips count
        _case("build_tiny", "build", "light", 20_000, delta=100_000, quant=EXISTS),
        # an export that is not in time order, from the pinned host buffers of a loader
        _case("build_shuffled", "build", "medium", 2_000_003, delta=86_400, dir=IN, order="shuffled", source="pinned"),
        # few messages per pair, as in talk-page logs
        _case("build_light", "build", "light", 6_000_001, delta=20_000, dir=EITHER, quant=EXISTS),
        # event times in milliseconds: a year does not fit 32 bits
        _case("build_milliseconds", "build", "medium", 10_000_003, delta=604_800_000, quant=EXISTS, unit="ms"),
        # the medium benchmark graph and its three windows
        _case("build_medium", "build", "medium", 20_000_000, queries=3),
        # the benchmark's default: the size of the paper's largest graphs
        _case("build_paper", "build", "paper", 70_000_000, rho_num=3, rho_den=10),
        # an interactive query on a small resident graph
        _case("query_small", "query", "light", 100_000, delta=100_000, dir=IN, universe=TAIL, rho_den=10),
        # a query with every optional output on a resident graph
        _case("query_outputs", "query", "medium", 2_000_003, delta=604_800, quant=EXISTS, edge_counts=True,
              certificates=True, vertices=True, triples=True),
        # a day's window in both directions on the medium graph
        _case("query_medium", "query", "medium", 20_000_000, delta=86_400, dir=EITHER, universe=COMMON),
        # the benchmark's query on the resident paper-scale graph
        _case("query_paper", "query", "paper", 70_000_000, rho_num=3, rho_den=10),
        # the benchmark's mixed batch
        _case("batch_medium", "batch", "medium", 20_000_000, queries=256),
        # per-edge counts as device features of a later model, near the entry point's limit
        _case("counts_million", "counts", "medium", 1_000_003, delta=86_400, dir=EITHER),
    ]


def draw(rng: random.Random):
    kind = rng.choice(["build", "build", "query", "query", "batch", "counts"])
    recipe = rng.choice(["light", "medium", "paper"])
    lo, hi = {"light": (5_000, 7_000_000), "medium": (50_000, 20_000_000), "paper": (1_000_000, 60_000_000)}[recipe]
    if kind == "counts":
        lo, hi = min(lo, 500_000), min(hi, 1_040_000)
    elif kind != "build" and recipe == "medium":
        lo = 500_000  # smaller graphs of few dense pairs have hardly a triangle in any window
    order = rng.choice(["time", "time", "shuffled"])
    unit = rng.choice(["s", "s", "s", "ms"])
    if order == "shuffled" or unit == "ms":  # the general paths: no dearer than the largest listed case
        hi = min(hi, 20_000_000)
    m = int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | 1
    # windows of a day to four weeks; the light recipe's times span a million seconds only
    span = (5_000, 100_000) if recipe == "light" else (86_400, 2_419_200)
    delta = int(math.exp(rng.uniform(math.log(span[0]), math.log(span[1])))) * (1000 if unit == "ms" else 1)
    extra = kind == "query" and m < 2_000_000 and rng.random() < 0.5
    return {"kind": kind, "recipe": recipe, "m": m, "order": order, "unit": unit,
            "source": rng.choice(["device", "device", "pinned"]) if kind == "build" else "device",
            "delta": delta, "dir": rng.randrange(3), "quant": rng.choice([EXISTS, EXISTS, FORALL]),
            "universe": rng.randrange(3), "rho_num": rng.randrange(1, 4), "rho_den": 10,
            "queries": int(math.exp(rng.uniform(math.log(2), math.log(256)))) if kind == "batch" else 1,
            "edge_counts": extra, "certificates": extra and rng.random() < 0.5,
            "vertices": extra and rng.random() < 0.5, "triples": extra and rng.random() < 0.5}


# --------------------------------------------------------------------------- inputs

def _truncated(kind, param, cap):
    k = torch.arange(1, cap + 1, dtype=torch.float64, device="cuda")
    pmf = (1.0 - param) ** (k - 1) * param if kind == "geometric" else k ** (-param)
    cdf = torch.cumsum(pmf, 0)
    cdf /= cdf[-1].clone()

    def sample(size, gen):
        u = torch.rand(size, dtype=torch.float64, device="cuda", generator=gen)
        return torch.searchsorted(cdf, u, right=True).clamp_(max=cap - 1) + 1

    return sample


def _cut(keys, sigma, room):
    """The first edges whose multiplicities sum to room (the last one truncated)."""
    total = torch.cumsum(sigma, 0)
    if int(total[-1]) <= room:
        return keys, sigma
    last = int(torch.searchsorted(total, room))
    keys, sigma = keys[:last + 1], sigma[:last + 1].clone()
    sigma[-1] -= total[last] - room
    return keys, sigma


def _communities(n, count, size, p, gen):
    """count groups of size vertices of the highest ids, each pair with probability p."""
    pool = n - 1 - torch.randperm(count * size, device="cuda", generator=gen).view(count, size)
    group = pool.sort(dim=1).values
    i, j = torch.triu_indices(size, size, 1, device="cuda")
    keep = torch.rand(count, i.shape[0], device="cuda", generator=gen) < p
    return (group[:, i] * n + group[:, j])[keep]


def _edge_list(case, seed):
    """(n, src, dst, t) on the GPU; src and dst int32, t int64."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1_000_003 + case["m"])
    m, recipe = case["m"], case["recipe"]
    if recipe == "light":
        n, gamma, sample = max(m // 10, 8), 2.3, _truncated("geometric", 0.5, 16)
    elif recipe == "medium":
        n, gamma, sample = max(m // 20, 8), 2.1, _truncated("zipf", 1.5, 1000)
    else:
        n, gamma, sample = max(m // 14, 1000), 2.0, _truncated("zipf", 1.3, 10_000)
    weight = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (gamma - 1.0))
    cdf = torch.cumsum(weight, 0)
    cdf /= cdf[-1].clone()
    parts, total = [], 0
    seen = torch.empty(0, dtype=torch.int64, device="cuda")
    if recipe == "paper":
        scale = math.sqrt(m / 70_000_000)
        keys = _communities(n, max(2, round(50 * scale)), max(10, int(300 * scale)), 0.7, gen)
        keys = keys[torch.randperm(keys.shape[0], device="cuda", generator=gen)]
        parts.append(_cut(keys, _truncated("zipf", 1.3, 16)(keys.shape[0], gen), m))
        seen, total = keys, int(parts[0][1].sum())
    mean = float(sample(1 << 16, gen).double().mean())
    while total < m:
        want = int(1.4 * (m - total) / mean) + 1024
        ends = torch.searchsorted(cdf, torch.rand(2, want, dtype=torch.float64, device="cuda", generator=gen),
                                  right=True).clamp_(max=n - 1)
        a, b = ends.amin(0), ends.amax(0)
        keys = torch.unique((a * n + b)[a != b])
        keys = keys[~torch.isin(keys, seen)]
        if keys.numel() == 0:
            continue
        keys = keys[torch.randperm(keys.shape[0], device="cuda", generator=gen)]
        parts.append(_cut(keys, sample(keys.shape[0], gen), m - total))
        total += int(parts[-1][1].sum())
        seen = torch.cat([seen, parts[-1][0]])
    keys = torch.cat([p[0] for p in parts])
    sigma = torch.cat([p[1] for p in parts])
    key = torch.repeat_interleave(keys, sigma)
    lo, hi = key // n, key % n
    flip = torch.rand(m, device="cuda", generator=gen) < 0.5
    src, dst = torch.where(flip, hi, lo).int(), torch.where(flip, lo, hi).int()
    if recipe == "light":
        t = torch.randint(0, 1_000_001, (m,), device="cuda", generator=gen)
    else:  # bursts: a start per static edge, then lognormal gaps, wrapped at a year
        gap = torch.empty(m, dtype=torch.float64, device="cuda").log_normal_(6.0, 2.0, generator=gen)
        gap = gap.round_().clamp_(max=YEAR_S).long()
        start = torch.cumsum(sigma, 0) - sigma
        gap[start] = 0
        run = torch.cumsum(gap, 0)
        first = torch.randint(0, YEAR_S, (keys.shape[0],), device="cuda", generator=gen)
        t = (run + torch.repeat_interleave(first - run[start], sigma)) % YEAR_S
    if case["unit"] == "ms":
        t = t * 1000 + torch.randint(0, 1000, (m,), device="cuda", generator=gen)
    if case["order"] == "time":
        t, order = torch.sort(t, stable=True)
    else:
        order = torch.randperm(m, device="cuda", generator=gen)
        t = t[order]
    return n, src[order].contiguous(), dst[order].contiguous(), t.contiguous()


def _query(case, **kw):
    q = dict(delta=case["delta"], rho_num=case["rho_num"], rho_den=case["rho_den"], quant=case["quant"],
             dir=case["dir"], universe=case["universe"], want_edge_counts=case["edge_counts"],
             want_certificates=case["certificates"], outer=int(case["vertices"]), outer_rho_num=1, outer_rho_den=10,
             want_triples=case["triples"])
    q.update(kw)
    return SimpleNamespace(**q)


def _queries(case, seed):
    """The case's queries: one, the medium benchmark's three windows, or a random mix."""
    if case["kind"] == "build" and case["queries"] == 3:
        return [_query(case, delta=d) for d in (600, 3600, 86_400)]
    if case["kind"] != "batch":
        return [_query(case)]
    rng = random.Random(seed)
    unit = 1000 if case["unit"] == "ms" else 1
    longest = 20_000 if case["recipe"] == "light" else 604_800
    return [_query(case, delta=unit * round(math.exp(rng.uniform(math.log(60), math.log(longest)))),
                   rho_num=rng.randrange(1, 10), rho_den=10, quant=rng.randrange(2), dir=rng.randrange(3),
                   universe=HEAD) for _ in range(case["queries"])]


def _tables(case):
    """The arrays a program collects its results in, sized once for its workload."""
    pairs = min(case["queries"] * 2 * case["m"], MAX_PAIRS)
    tables = {"sizes": np.zeros((case["queries"], 2), np.int64), "pairs": np.zeros((4, pairs), np.int32)}
    if case["vertices"]:
        tables["vertices"] = np.zeros((2, pairs), np.int32)
    if case["certificates"]:
        tables["certificates"] = np.zeros(case["m"], np.int64)
    if case["triples"]:
        tables["triples"] = np.zeros((MAX_PAIRS, 3), np.int32)
    return tables


def _collect(results, tables):
    """The solution pairs (u, v, count, ncert) of all queries one after another, with each
    query's number of pairs and of certificates, and the optional lists of a single query."""
    n = 0
    for i, r in enumerate(results):
        k = len(r["u"])
        tables["sizes"][i] = k, r["n_cert_edges"]
        if k:
            rows = tables["pairs"][:, n:n + k]
            rows[0], rows[1], rows[2], rows[3] = r["u"], r["v"], r["count"], r["ncert"]
            n += k
        if "vertices" in tables:
            tables["vertices"][0, :len(r["vertex"])] = r["vertex"]
            tables["vertices"][1, :len(r["vertex"])] = r["vertex_count"]
        if "certificates" in tables:
            tables["certificates"][:len(r["certificates"])] = r["certificates"]
        if "triples" in tables:
            tables["triples"][:len(r["triples"])] = r["triples"]
    out = dict(tables)
    if r.get("edge_count") is not None:
        out["edge_count"] = r["edge_count"]
    return out


def prepare(case, seed):
    n, src, dst, t = _edge_list(case, seed)
    state = {"kind": case["kind"], "queries": _queries(case, seed)}
    if case["kind"] == "counts":
        state["out"] = torch.empty(case["m"], dtype=torch.int32, device="cuda")
    else:
        state["tables"] = _tables(case)
    if case["kind"] == "build":
        edges = (src, dst, t)
        if case["source"] == "pinned":
            edges = tuple(x.cpu().pin_memory() for x in edges)
        state.update(n=n, edges=edges)
    else:
        state["graph"] = folty.TemporalGraph(n, src, dst, t)
    return state


# --------------------------------------------------------------------------- a pass

def run(state):
    kind, queries = state["kind"], state["queries"]
    if kind == "build":
        with folty.TemporalGraph(state["n"], *state["edges"]) as graph:
            results = [graph.query(q) for q in queries]
            info = graph.info()
        return _collect(results, state["tables"]) | {k: info[k] for k in INFO}
    graph = state["graph"]
    if kind == "counts":
        folty.folty_edge_counts_noalloc(graph.handle, queries[0].delta, queries[0].dir, state["out"])
        return state["out"]
    results = graph.query_batch(queries) if kind == "batch" else [graph.query(queries[0])]
    return _collect(results, state["tables"])


def work(case):
    """What a pass cannot do without. A build reads the edge list (16 B per edge). A pass
    over a resident graph reads its timestamps (4 or 8 B per edge); per-edge counts are 4 B
    per edge more. The results are small beside them; there is no floating arithmetic."""
    m = case["m"]
    per_edge = 16 if case["kind"] == "build" else (8 if case["unit"] == "ms" else 4)
    if case["kind"] == "counts" or case["edge_counts"]:
        per_edge += 4
    return {"bytes": per_edge * m, "flops": 0}


# --------------------------------------------------------------------------- the definition

class _Exact:
    """The answers for one edge list, from the definition."""

    def __init__(self, n, src, dst, t):
        self.n, self.m = n, src.shape[0]
        self.time_sorted = int(bool((t[1:] >= t[:-1]).all()))
        kept = torch.nonzero(src != dst).flatten()
        x, y, t = src[kept].long(), dst[kept].long(), t[kept]
        a, b = torch.minimum(x, y), torch.maximum(x, y)
        self.keys, s = torch.unique(a * n + b, return_inverse=True)
        self.ea, self.eb = self.keys // n, self.keys % n
        run = 2 * s + (x > y)
        by_t = torch.sort(t, stable=True).indices
        order = by_t[torch.sort(run[by_t], stable=True).indices]
        self.input_index = kept[order]
        self.run, self.t = run[order], t[order]
        self.tmin = int(t.min()) if t.numel() else 0
        self.span = (int(t.max()) - self.tmin + 1) if t.numel() else 1
        self.key = self.run * self.span + (self.t - self.tmin)
        S = self.S = self.keys.shape[0]
        self.start = torch.searchsorted(self.run, torch.arange(2 * S + 1, device="cuda"))
        self.deg = torch.bincount(torch.cat([self.ea, self.eb]), minlength=n)
        self._triangles()
        self.common = torch.bincount(torch.cat(self.tri), minlength=S)
        self.gaps = {}

    def _triangles(self):
        """Each triangle's static edges (uv, uw, vw) and vertices, u < v < w by (degree, id)."""
        n, S = self.n, self.S
        order = torch.sort(self.deg, stable=True).indices
        rank = torch.empty_like(order)
        rank[order] = torch.arange(n, device="cuda")
        up = rank[self.ea] < rank[self.eb]
        u, v = torch.where(up, self.ea, self.eb), torch.where(up, self.eb, self.ea)
        u, e = torch.sort(u, stable=True)
        v = v[e]
        ptr = torch.searchsorted(u, torch.arange(n + 1, device="cuda"))
        out = ptr[1:] - ptr[:-1]
        found, vertices = [[], [], []], [[], [], []]
        reps = out[u]
        ends = torch.cumsum(reps, 0)
        lo = 0
        while lo < S:
            base = int(ends[lo - 1]) if lo else 0
            hi = max(lo + 1, int(torch.searchsorted(ends, base + CHUNK)))
            r = reps[lo:hi]
            i = torch.repeat_interleave(torch.arange(lo, hi, device="cuda"), r)
            j = ptr[u[i]] + torch.arange(i.shape[0], device="cuda") - (ends[i] - reps[i] - base)
            ok = rank[v[i]] < rank[v[j]]
            i, j = i[ok], j[ok]
            want = torch.minimum(v[i], v[j]) * n + torch.maximum(v[i], v[j])
            at = torch.searchsorted(self.keys, want).clamp_(max=S - 1)
            ok = self.keys[at] == want
            i, j, at = i[ok], j[ok], at[ok]
            for parts, value in zip(found, (e[i], e[j], at)):
                parts.append(value)
            for parts, value in zip(vertices, (u[i], v[i], v[j])):
                parts.append(value)
            lo = hi
        empty = torch.empty(0, dtype=torch.int64, device="cuda")
        self.tri = [torch.cat(p) if p else empty for p in found]
        self.corner = [torch.cat(p) if p else empty for p in vertices]

    def info(self):
        deg, core = self.deg.clone(), 0  # the degeneracy, by removing the vertices of least degree
        ends = torch.stack([torch.cat([self.ea, self.eb]), torch.cat([self.eb, self.ea])])
        alive, k = deg > 0, 0
        ends = ends[:, alive[ends[0]]]
        while ends.shape[1]:
            gone = alive & (deg <= k)
            if not bool(gone.any()):
                k = int(deg[alive].min())
                continue
            core = k
            alive &= ~gone
            leaves = ends[:, gone[ends[0]]]
            deg -= torch.bincount(leaves[1], minlength=self.n)
            ends = ends[:, alive[ends[0]] & alive[ends[1]]]
            deg[~alive] = 0
            if not ends.shape[1]:
                break
        size = self.start[2::2] - self.start[:-2:2]
        return {"n": self.n, "m": self.m, "m_kept": self.run.shape[0], "static_edges": self.S,
                "max_degree": int(self.deg.max()), "degeneracy": core, "triangles": self.tri[0].shape[0],
                "probes": int(sum(size[e].sum() for e in self.tri)), "sigma_max": int(size.max()),
                "time_sorted": self.time_sorted}

    def _first(self, run, t):
        """First timestamp >= t of each run (span when there is none); t relative to tmin."""
        at = torch.searchsorted(self.key, run * self.span + t)
        at_c = at.clamp(max=self.key.shape[0] - 1)
        return torch.where((at < self.start[run + 1]) & (t < self.span), self.t[at_c] - self.tmin, self.span)

    def matches(self, direction):
        """(sorted edge, witness, gap t3 - t) of every edge and witness with t <= t2 <= t3."""
        if direction in self.gaps:
            return self.gaps[direction]
        parts = [[], [], []]
        for e, z in zip(self.tri, reversed(self.corner)):  # uv has witness w, uw v, vw u
            for d in (0, 1):
                x, y = (self.ea[e], self.eb[e]) if d == 0 else (self.eb[e], self.ea[e])
                n1 = self.start[2 * e + d + 1] - self.start[2 * e + d]
                ends = torch.cumsum(n1, 0)
                lo, total = 0, e.shape[0]
                while lo < total:
                    base = int(ends[lo - 1]) if lo else 0
                    hi = max(lo + 1, int(torch.searchsorted(ends, base + CHUNK)))
                    i = torch.repeat_interleave(torch.arange(lo, hi, device="cuda"), n1[lo:hi])
                    pos = self.start[2 * e[i] + d] + torch.arange(i.shape[0], device="cuda") - (ends[i] - n1[i] - base)
                    t = self.t[pos] - self.tmin
                    t3 = t
                    for end in (x, y):
                        vertex, w = end[i], z[i]
                        s = torch.searchsorted(self.keys, torch.minimum(vertex, w) * self.n + torch.maximum(vertex, w))
                        forward = (vertex > w).long()  # the run of edges vertex -> w
                        if direction == OUT:
                            t3 = self._first(2 * s + forward, t3)
                        elif direction == IN:
                            t3 = self._first(2 * s + 1 - forward, t3)
                        else:
                            t3 = torch.minimum(self._first(2 * s, t3), self._first(2 * s + 1, t3))
                    ok = t3 < self.span
                    parts[0].append(pos[ok])
                    parts[1].append(z[i][ok])
                    parts[2].append((t3 - t)[ok])
                    lo = hi
        self.gaps[direction] = tuple(torch.cat(p) if p else torch.empty(0, dtype=torch.int64, device="cuda")
                                     for p in parts)
        return self.gaps[direction]

    def counts(self, q):
        pos, _, gap = self.matches(q.dir)
        return torch.bincount(pos[gap <= q.delta], minlength=self.run.shape[0])

    def in_input_order(self, c):
        out = torch.zeros(self.m, dtype=torch.int32, device="cuda")
        out[self.input_index] = c.int()
        return out

    def query(self, q):
        c = self.counts(q)
        hit = torch.nonzero(c).flatten()
        run, ch = self.run[hit], c[hit]
        s, d = run // 2, run % 2
        x, y = torch.where(d == 0, self.ea[s], self.eb[s]), torch.where(d == 0, self.eb[s], self.ea[s])
        size = self.common[s] if q.universe == COMMON else self.deg[x if q.universe == HEAD else y]
        ok = torch.ones_like(hit, dtype=torch.bool) if q.quant == EXISTS else ch * q.rho_den >= q.rho_num * size
        most = torch.zeros(2 * self.S, dtype=torch.int64, device="cuda").scatter_reduce_(0, run, ch, "amax")
        ncert = torch.bincount(run[ok], minlength=2 * self.S)
        r = torch.nonzero(ncert).flatten()
        u = torch.where(r % 2 == 0, self.ea[r // 2], self.eb[r // 2])
        v = self.ea[r // 2] + self.eb[r // 2] - u
        order = torch.sort(u * self.n + v).indices
        res = {"u": u[order].int(), "v": v[order].int(), "count": most[r][order].int(),
               "ncert": ncert[r][order].int(), "n_cert_edges": int(ok.sum())}
        if q.want_edge_counts:
            res["edge_count"] = self.in_input_order(c)
        if q.outer:
            heads = torch.bincount(u, minlength=self.n)
            vertex = torch.nonzero((heads >= 1) & (heads * q.outer_rho_den >= q.outer_rho_num * self.deg)).flatten()
            res["vertex"], res["vertex_count"] = vertex.int(), heads[vertex].int()
        if q.want_certificates:
            res["certificates"] = torch.sort(self.input_index[hit[ok]]).values
        if q.want_triples:
            pos, z, gap = self.matches(q.dir)
            pos, z = pos[gap <= q.delta], z[gap <= q.delta]
            rz = torch.unique(torch.stack([self.run[pos], z], 1), dim=0)
            s = rz[:, 0] // 2
            x = torch.where(rz[:, 0] % 2 == 0, self.ea[s], self.eb[s])
            xyz = torch.stack([x, self.ea[s] + self.eb[s] - x, rz[:, 1]], 1)
            res["triples"] = torch.unique(xyz, dim=0).int()
        return {k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for k, v in res.items()}


def exact(case, seed):
    if case["m"] > EXACT_MAX_EDGES or (case["recipe"] == "paper" and case["m"] > 8_000_000):
        return None
    graph = _Exact(*_edge_list(case, seed))
    queries = _queries(case, seed)
    if case["kind"] == "counts":
        return graph.in_input_order(graph.counts(queries[0]))
    out = _collect([graph.query(q) for q in queries], _tables(case))
    return out | graph.info() if case["kind"] == "build" else out
