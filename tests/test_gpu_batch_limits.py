"""Batches whose solutions fill their buffer, against single queries."""
import numpy as np
import pytest

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


def _dense_graph(n, seed, t_max=1000):
    """Every pair of n vertices in both directions: most directed pairs have a triangle."""
    rng = np.random.default_rng(seed)
    i, j = np.triu_indices(n, 1)
    src, dst = np.concatenate([i, j]).astype(np.int32), np.concatenate([j, i]).astype(np.int32)
    return W.TemporalGraph(n, src, dst, np.sort(rng.integers(0, t_max, len(src))))


def _mix(count, windows, rng):
    return [W.Query(int(windows[k]), int(num), 10, int(quant), int(dr), int(uni), False)
            for k, num, quant, dr, uni in zip(rng.integers(0, len(windows), count), rng.integers(0, 4, count),
                                              rng.integers(0, 2, count), rng.integers(0, 3, count),
                                              rng.integers(0, 3, count))]


# buffers that take one pass's solutions but not the next one's, none, all but the last; several
# windows per chunk and more of them (200 distinct) than one pass holds; queries with per-edge
# counts between them
@pytest.mark.parametrize("cap", [1, 3000, 20_000, 60_000, 150_000])
@pytest.mark.parametrize("windows", [np.array([0, 7, 400]), np.arange(300, 500)])
def test_solution_buffers_of_several_passes(F, monkeypatch, cap, windows):
    g = _dense_graph(45, cap + len(windows))
    rng = np.random.default_rng(cap + len(windows))
    qs = _mix(900, windows, rng)
    qs += [W.Query(int(windows[-1]), 1, 2, W.Q_EXISTS, dr, W.U_HEAD, True) for dr in range(3)]
    qs = [qs[i] for i in rng.permutation(len(qs))]
    monkeypatch.setenv("FOLTY_BATCH_SOLUTION_CAP", str(cap))
    with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G:
        got = G.query_batch(qs)
        want = {q: G.query(q) for q in set(qs)}
    for q, r in zip(qs, got):
        assert pairs_of(r) == pairs_of(want[q]), str(q)
        assert r["n_cert_edges"] == want[q]["n_cert_edges"], str(q)
        if q.want_edge_counts:
            np.testing.assert_array_equal(r["edge_count"], want[q]["edge_count"])
    assert sum(len(r["u"]) for r in got) > 150_000


# most probes hit, the others none; lists below and above the length from which they have a plan
@pytest.mark.parametrize("n, mult", [(64, 1), (40, 20), (24, 150)])
def test_marked_edges_where_most_probes_hit(F, n, mult):
    one = _dense_graph(n, mult)
    g = W.TemporalGraph(n, np.repeat(one.src, mult), np.repeat(one.dst, mult),
                        np.sort(np.random.default_rng(n).integers(0, 1000, mult * one.m)))
    p = np.random.default_rng(mult).permutation(g.m)
    g = W.TemporalGraph(n, g.src[p], g.dst[p], g.t)
    qs = [W.Query(d, k, 10, quant, dr, W.U_COMMON, True) for d in (0, 30, 1000) for dr in range(3)
          for quant, k in ((W.Q_EXISTS, 0), (W.Q_FORALL_T, 9))]
    with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G:
        for q, r in zip(qs, G.query_batch(qs)):
            want = G.query(q)
            np.testing.assert_array_equal(r["edge_count"], want["edge_count"], err_msg=str(q))
            assert pairs_of(r) == pairs_of(want), str(q)


class _Watched:
    """A graph whose device memory is PyTorch's, with the largest amount held at a time."""

    def __init__(self, F, g):
        import ctypes
        import torch
        self.F, self.live, self.peak = F, {}, 0

        @F.ALLOC_FN
        def alloc(nbytes, stream, ctx):
            p = torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))
            self.live[p] = int(nbytes)
            self.peak = max(self.peak, sum(self.live.values()))
            return p

        @F.FREE_FN
        def free(ptr, stream, ctx):
            del self.live[int(ptr)]
            torch.cuda.caching_allocator_delete(int(ptr))

        self.allocator, h = F.folty_allocator(alloc, free, None), ctypes.c_void_p()
        st = F.lib.folty_load_temporal_graph(g.n, g.m, g.src.ctypes.data, g.dst.ctypes.data, g.t.ctypes.data,
                                             ctypes.byref(self.allocator), F.current_stream(), ctypes.byref(h))
        assert st == F.FOLTY_OK, F.folty_last_error()
        self.handle = h.value
        F.folty_preprocess(self.handle)

    def batch(self, qs):
        """The results, and what the call took at its peak."""
        before = self.peak = sum(self.live.values())
        got = self.F.folty_query_batch(self.handle, qs)
        return got, self.peak - before

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.F.folty_free(self.handle)


def test_memory_of_a_batch_does_not_grow_with_its_queries(F):
    """3000 queries of some 8,000 solutions each: the batch's 24M would take 1.4 GB together (56
    B each with their sort and results); the 2.1M of the 256 queries of a pass fit the buffer
    of 2^22 and take 235 MB."""
    with _Watched(F, _dense_graph(128, 5)) as G:
        qs = [W.Query(900 + i % 3, 1, 10, W.Q_EXISTS, W.DIR_OUT, W.U_HEAD, False) for i in range(3000)]
        want = [F.folty_query(G.handle, q) for q in qs[:3]]
        got, grown = G.batch(qs)
    assert sum(len(r["u"]) for r in got) > 20_000_000
    for i, r in enumerate(got):
        np.testing.assert_array_equal(r["u"], want[i % 3]["u"])
        np.testing.assert_array_equal(r["ncert"], want[i % 3]["ncert"])
    # the buffer and its sort, the bins and marks of 16,256 edges and the allocator's blocks
    assert grown < 56 * (1 << 22) + (64 << 20), grown


# budgets below a row's least size, between two, in the middle of a 16-byte chunk of bins
@pytest.mark.parametrize("bins", [1, 7, 8, 13, 30])
def test_bin_rows_within_a_budget(F, monkeypatch, bins):
    """40 windows over 250,000 edges with a hit: rows of 80 bytes, in chunks of windows whose
    padded rows fit the budget (of `bins` 16-bit bins a row; one 16-byte chunk at least)."""
    rng = np.random.default_rng(bins)
    i, j = np.triu_indices(64, 1)
    base = np.repeat(np.arange(62) * 64, len(i))
    i, j = np.tile(i, 62) + base, np.tile(j, 62) + base
    src, dst = np.concatenate([i, j]).astype(np.int32), np.concatenate([j, i]).astype(np.int32)
    g = W.TemporalGraph(62 * 64, src, dst, np.sort(rng.permutation(len(src)) % 1000))

    windows = range(2, 1002, 25)
    queries = [W.Query(d, 1, 2, quant, W.DIR_EITHER, W.U_COMMON, False) for d in windows
               for quant in (W.Q_EXISTS, W.Q_FORALL_T)]

    def without_solutions(windows):  # no edge has every neighbour of its head as a witness
        return [W.Query(d, 1, 1, W.Q_FORALL_T, W.DIR_EITHER, W.U_HEAD, False) for d in windows]

    with _Watched(F, g) as G:
        want = [F.folty_query(G.handle, q) for q in queries]
        monkeypatch.setenv("FOLTY_BATCH_SOLUTION_CAP", "1000")
        G.batch(without_solutions((2, 999)))  # allocates what the graph keeps for batches
        _, least = G.batch(without_solutions((2, 999)))  # rows of one 16-byte chunk
        monkeypatch.setenv("FOLTY_BATCH_BIN_BUDGET", str(bins * 2 * g.m))
        _, grown = G.batch(without_solutions(windows))
        got = F.folty_query_batch(G.handle, queries)
    for q, r, w in zip(queries, got, want):
        assert pairs_of(r) == pairs_of(w), str(q)
    chunks = max(bins * 2 // 16, 1)
    assert grown <= least + (chunks - 1) * 16 * g.m + (1 << 20), (grown, least)
