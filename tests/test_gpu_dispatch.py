"""The sizes at which the library changes from one kernel or table size to another, against
the CPU oracle (bit-exact: all arithmetic is integer)."""
import numpy as np
import pytest

import oracle
import workloads as W

from _support import pairs_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_17215_gb300 as F
    return F


def _check(F, g, queries, device=False):
    if device:
        import torch
        arrays = [torch.from_numpy(x).cuda() for x in (g.src, g.dst, g.t)]
    else:
        arrays = [g.src, g.dst, g.t]
    with F.TemporalGraph(g.n, *arrays) as G, oracle.OracleGraph.of(g) as og:
        for q in queries:
            got, want = G.query(q), og.query(q)
            if q.want_edge_counts:
                np.testing.assert_array_equal(got["edge_count"], want["edge_count"], err_msg=str(q))
            assert pairs_of(got) == pairs_of(want), str(q)
            assert got["n_cert_edges"] == want["n_cert_edges"], str(q)
        return G.info()


def _distinct_pairs_graph(pairs, repeats, seed):
    """A time-ordered graph of exactly `pairs` distinct pairs, `repeats` of them twice: a
    block of 120 vertices with every pair (triangles), the rest random pairs."""
    rng = np.random.default_rng(seed)
    n, b = 400_000, 120
    i, j = np.triu_indices(b, 1)
    keys = i.astype(np.int64) * n + j
    while keys.shape[0] < pairs:
        x, y = rng.integers(b, n, (2, pairs))
        more = np.unique(np.minimum(x, y) * n + np.maximum(x, y))
        more = more[more // n != more % n]
        keys = np.unique(np.concatenate([keys, rng.permutation(more)[: pairs - keys.shape[0]]]))
    keys = np.concatenate([keys, keys[:repeats]])
    a, c = keys // n, keys % n
    flip = rng.random(keys.shape[0]) < 0.5
    t = rng.integers(0, 1000, keys.shape[0])
    o = np.argsort(t, kind="stable")
    return W.TemporalGraph(n, np.where(flip, c, a)[o].astype(np.int32), np.where(flip, a, c)[o].astype(np.int32),
                           t[o].astype(np.int64))


# the first table of 524,289 to 12.5M edges has 2^20 slots: it serves up to 2^19 pairs, is
# retried when it turns out fuller, and is abandoned on the way past 9/16 of its slots
@pytest.mark.parametrize("pairs", [(1 << 19) - 1, 1 << 19, (1 << 19) + 1, 560_000, 590_000, 700_000, 1_100_000])
@pytest.mark.parametrize("device", [False, True])
def test_pair_table_sizes(F, pairs, device):
    g = _distinct_pairs_graph(pairs, 30_000, pairs)
    info = _check(F, g, [W.Query(300, 1, 4, W.Q_FORALL_T, W.DIR_EITHER, W.U_COMMON, True)], device)
    assert info["static_edges"] == pairs


def _plain(deltas):
    return [W.Query(d, num, 4, quant, dr, uni, False) for d in deltas
            for num, quant, dr, uni in ((1, W.Q_FORALL_T, W.DIR_OUT, W.U_HEAD), (1, W.Q_EXISTS, W.DIR_EITHER, W.U_TAIL),
                                        (3, W.Q_FORALL_T, W.DIR_IN, W.U_COMMON))]


# one group of 32 edges, one word of 32 groups, and their edges; a plain query leaves its
# counters and bits zero for the next one, so every query runs twice, in both orders
@pytest.mark.parametrize("m", [1, 31, 32, 33, 1023, 1024, 1025, 33_000])
def test_plain_queries_leave_their_workspace_clear(F, m):
    g = W.random_small_graph(np.random.default_rng(m), 12 if m < 2000 else 90, m, 500)
    qs = _plain((0, 20, 500))
    _check(F, g, qs + qs[::-1])


def test_plain_query_with_32_bit_counters_and_hit_groups_everywhere(F):
    """A hub of degree past 16 bits (32-bit counters) in a graph whose hits spread over more
    32-edge groups than one block lists."""
    rng = np.random.default_rng(3)
    n, extra = 66_000, 200_000
    leaves = np.arange(1, n, dtype=np.int32)
    a = rng.integers(1, n, extra).astype(np.int32)
    b = np.minimum(a + rng.integers(1, 4, extra), n - 1).astype(np.int32)
    src = np.concatenate([np.zeros(2 * (n - 1), np.int32), a])
    dst = np.concatenate([leaves, leaves, b])
    t = rng.integers(0, 1000, src.shape[0]).astype(np.int64)
    qs = _plain((100, 900))
    info = _check(F, W.TemporalGraph(n, src, dst, t), qs + qs[:3])
    assert info["max_degree"] >= 65_535


def _triangles_of_sizes(sizes, t_max, seed, scale=1):
    """One triangle per ordered choice of three sizes: each side holds that many edges, about
    a third of them against the side's direction."""
    import itertools
    rng = np.random.default_rng(seed)
    src, dst = [], []
    n = 0
    for combo in sorted(set(itertools.permutations(sizes, 3))):
        v = rng.permutation(3) + n
        n += 3
        for (a, b), c in zip(((0, 1), (0, 2), (1, 2)), combo):
            flip = rng.random(c) < 0.33
            src.append(np.where(flip, v[b], v[a]))
            dst.append(np.where(flip, v[a], v[b]))
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    t = rng.integers(0, t_max, src.shape[0]).astype(np.int64) * scale
    o = np.argsort(t, kind="stable")
    return W.TemporalGraph(n, src[o], dst[o], t[o])


# the probes of a role are driven by its shortest list: lists around the sizes at which L2 or
# L3 takes over from L1 (half the slots, 64 entries of L1 per slot) and at which L1 is cut
# into chunks (16384); many equal times, all of them, few; 32- and 64-bit stores
@pytest.mark.parametrize("sizes", [(1, 1, 2, 3, 4, 5), (1, 2, 63, 64, 65, 129), (3, 40, 500, 520), (2, 300, 16_384, 16_385),
                                   (5, 1, 60_000)])
@pytest.mark.parametrize("t_max,scale", [(1, 1), (30, 1), (5000, 1), (10 ** 6, 1), (10 ** 6, 10 ** 7)])
def test_probes_from_every_list(F, sizes, t_max, scale):
    g = _triangles_of_sizes(sizes, t_max, sum(sizes) + t_max, scale)
    qs = [W.Query(d * scale, 1, 2, W.Q_EXISTS, dr, W.U_HEAD, True) for d in (0, 1, max(t_max // 50, 2), t_max)
          for dr in (W.DIR_OUT, W.DIR_IN, W.DIR_EITHER)]
    _check(F, g, qs)
    batch = [W.Query(q.delta, 1, 2, W.Q_EXISTS, q.dir, W.U_HEAD, False) for q in qs]
    with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G, oracle.OracleGraph.of(g) as og:
        for q, r in zip(batch, G.query_batch(batch)):
            assert pairs_of(r) == pairs_of(og.query(q)), str(q)


def _cliques_and_hubs(cliques, hubs, spread, seed, scale=1):
    """Cliques of the given sizes; per hub size one vertex pair joined to that many others (its
    triangles share one edge); a sparse remainder. Every edge repeated until the graph is past
    the allocation-free counts' limit, so that its triangles are listed in one pass."""
    rng = np.random.default_rng(seed)
    pairs, n = [], 0
    for k in cliques:
        i, j = np.triu_indices(k, 1)
        pairs.append(np.stack([i + n, j + n], 1))
        n += k
    for k in hubs:
        leaf = np.arange(k) + n + 2
        pairs += [np.stack([np.full(k, n + h), leaf], 1) for h in (0, 1)] + [np.array([[n, n + 1]])]
        n += k + 2
    a = rng.integers(0, n + spread, (spread, 2))
    pairs.append(a[a[:, 0] != a[:, 1]])
    n += spread
    pairs = np.concatenate(pairs)
    pairs = np.concatenate([pairs] * (1_100_000 // len(pairs) + 1))
    order = rng.permutation(n).astype(np.int32)  # degeneracy order and id order differ
    flip = rng.random(len(pairs)) < 0.4
    src = order[np.where(flip, pairs[:, 1], pairs[:, 0])]
    dst = order[np.where(flip, pairs[:, 0], pairs[:, 1])]
    return W.TemporalGraph(n, src, dst, np.sort(rng.integers(0, 20_000, len(pairs))) * scale)


# the one-pass listing: stretches of out-lists up to, at and past the table's 256 entries, lists
# of a whole step of 32 and around it, a warp's chunk filled exactly and overrun, triangles so few
# that most of a chunk stays empty, none; 32- and 64-bit stores; against the counting pass
@pytest.mark.parametrize("cliques,hubs,spread", [((3,), (), 1000), ((31, 32, 33, 34), (31, 33), 0), ((255, 257), (700,), 9),
                                                 ((300,), (), 50_000), ((), (), 900_000), ((), (40_000,), 0),
                                                 ((5,) * 4000, (), 0)])
@pytest.mark.parametrize("scale", [1, 10 ** 6])
def test_one_pass_listing(F, monkeypatch, cliques, hubs, spread, scale):
    g = _cliques_and_hubs(cliques, hubs, spread, 17 * len(cliques) + len(hubs) + spread, scale)
    qs = [W.Query(d * scale, 1, 2, W.Q_EXISTS, dr, W.U_HEAD, True) for d in (0, 40, 20_000)
          for dr in (W.DIR_IN, W.DIR_OUT, W.DIR_EITHER)]
    got = []
    for layout in ("", "counted"):
        monkeypatch.setenv("FOLTY_TRI_LAYOUT", layout)
        with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G:
            assert G.info()["m_kept"] > F.NOALLOC_MAX_EDGES
            got.append((G.info(), [G.query(q) for q in qs], G.query_batch([W.Query(q.delta, 1, 2, W.Q_EXISTS, q.dir, W.U_HEAD)
                                                                          for q in qs])))
    (info, res, batch), (info2, res2, batch2) = got
    keys = ("triangles", "probes", "sigma_max", "degeneracy", "max_out_degree")
    assert [info[k] for k in keys] == [info2[k] for k in keys]
    n_clique = sum(k * (k - 1) * (k - 2) // 6 for k in cliques) + sum(hubs)
    assert info["triangles"] >= n_clique
    for x, y in zip(res, res2):
        np.testing.assert_array_equal(x["edge_count"], y["edge_count"])
        assert pairs_of(x) == pairs_of(y)
    for x, y in zip(batch, batch2):
        assert pairs_of(x) == pairs_of(y)


def test_triples_of_a_one_pass_listing(F):
    """The exists-triples output, which numbers roles by the triangle array's entries."""
    g = _cliques_and_hubs((9, 4), (20,), 200, 5)
    q = W.Query(3, 1, 2, W.Q_EXISTS, W.DIR_OUT, W.U_HEAD, False, want_triples=True)
    with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G, oracle.OracleGraph.of(g) as og:
        got, want = G.query(q)["triples"], og.triples(q.delta, q.dir)
    assert len(want) > 0
    np.testing.assert_array_equal(got, want)


# the sorts at the edges of their tiles (4096 pairs of 64-bit keys, 8192 ids) and with one digit
# holding every key; in time order (the store's passes) and not (the time sort)
@pytest.mark.parametrize("m", [4095, 4096, 4097, 8191, 8192, 8193, 16_385, 24_576])
@pytest.mark.parametrize("n", [2, 700])
def test_sorts_at_tile_edges(F, m, n):
    rng = np.random.default_rng(m + n)
    g = W.random_small_graph(rng, n, m, 10 ** 6)
    p = rng.permutation(len(g.src))
    for x in (g, W.TemporalGraph(g.n, g.src[p], g.dst[p], g.t[p])):
        _check(F, x, [W.Query(d, 1, 2, W.Q_FORALL_T, W.DIR_OUT, W.U_HEAD, True) for d in (1000, 10 ** 6)])


def _core_numbers(n, pairs):
    """Core numbers by the bucket algorithm: remove a vertex of least degree, one at a time."""
    adj = [[] for _ in range(n)]
    for a, b in pairs.tolist():
        adj[a].append(b)
        adj[b].append(a)
    deg = [len(x) for x in adj]
    buckets = [[] for _ in range(max(deg) + 1)]
    for v in range(n):
        buckets[deg[v]].append(v)
    core, level, d = [-1] * n, 0, 0
    while d < len(buckets):
        if not buckets[d]:
            d += 1
            continue
        v = buckets[d].pop()
        if core[v] >= 0 or deg[v] != d:
            continue
        level = max(level, d)
        core[v] = level
        for w in adj[v]:
            if core[w] < 0:
                deg[w] -= 1
                buckets[deg[w]].append(w)
                d = min(d, deg[w])
    return np.array(core)


# adjacency rows at the lengths where the work on a row changes hands (a lane, a warp, a block,
# several), hubs past the longest histogram, cores of every size up to the largest clique
@pytest.mark.parametrize("rows,cliques", [((8, 9, 64, 65), (5, 9)), ((511, 512, 513), (33,)), ((8192, 8193), (65, 130)),
                                          ((16_384, 16_385, 40_000), (10,)), ((), (520,))])
def test_core_numbers_at_row_edges(F, rows, cliques):
    rng = np.random.default_rng(sum(rows) + len(cliques))
    n = max((0,) + rows) + len(rows) + sum(cliques) + 50
    pairs = [rng.integers(0, n, (n, 2))]
    at = 0
    for k in cliques:
        i, j = np.triu_indices(k, 1)
        pairs.append(np.stack([i + at, j + at], 1))
        at += k
    for k in rows:
        others = rng.choice(np.setdiff1d(np.arange(n), [at]), k, replace=False)
        pairs.append(np.stack([np.full(k, at), others], 1))
        at += 1
    pairs = np.concatenate(pairs)
    pairs = np.unique(np.sort(pairs[pairs[:, 0] != pairs[:, 1]], axis=1), axis=0)
    ids = rng.permutation(n)
    pairs = ids[pairs]
    want = _core_numbers(n, pairs)
    with F.TemporalGraph(n, pairs[:, 0].astype(np.int32), pairs[:, 1].astype(np.int32),
                         np.zeros(len(pairs), np.int64)) as G:
        np.testing.assert_array_equal(G.core_numbers(), want)
        assert G.info()["degeneracy"] == want.max()


# the tile of the small sorts and the size at which the larger tiles take over
@pytest.mark.parametrize("m", [1023, 1024, 1025, 3072, (1 << 18) - 1, 1 << 18, (1 << 18) + 1])
def test_small_sorts(F, m):
    rng = np.random.default_rng(m)
    n = 60 if m < 5000 else 60_000
    src, dst = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    dst = np.where(src == dst, (dst + 1) % n, dst).astype(np.int32)
    _check(F, W.TemporalGraph(n, src, dst, rng.integers(0, 10 ** 6, m)),
           [W.Query(10 ** 5, 1, 2, W.Q_FORALL_T, W.DIR_EITHER, W.U_HEAD, True)])
