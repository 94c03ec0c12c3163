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


def test_memory_of_a_batch_does_not_grow_with_its_queries(F):
    """3000 queries of some 8,000 solutions each: the batch's 24M would take 1.4 GB together (56
    B each with their sort and results); the 2.1M of the 256 queries of a pass fit the buffer
    of 2^22 and take 235 MB."""
    import torch
    g = _dense_graph(128, 5)
    live, peak = {}, [0]

    @F.ALLOC_FN
    def alloc(nbytes, stream, ctx):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))
        live[p] = int(nbytes)
        peak[0] = max(peak[0], sum(live.values()))
        return p

    @F.FREE_FN
    def free(ptr, stream, ctx):
        del live[int(ptr)]
        torch.cuda.caching_allocator_delete(int(ptr))

    import ctypes
    a, h = F.folty_allocator(alloc, free, None), ctypes.c_void_p()
    st = F.lib.folty_load_temporal_graph(g.n, g.m, g.src.ctypes.data, g.dst.ctypes.data, g.t.ctypes.data,
                                         ctypes.byref(a), F.current_stream(), ctypes.byref(h))
    assert st == F.FOLTY_OK, F.folty_last_error()
    try:
        F.folty_preprocess(h.value)
        qs = [W.Query(900 + i % 3, 1, 10, W.Q_EXISTS, W.DIR_OUT, W.U_HEAD, False) for i in range(3000)]
        want = [F.folty_query(h.value, q) for q in qs[:3]]
        before, peak[0] = sum(live.values()), 0
        got = F.folty_query_batch(h.value, qs)
        grown = peak[0] - before
        solutions = sum(len(r["u"]) for r in got)
    finally:
        F.folty_free(h.value)
    assert solutions > 20_000_000
    for i, r in enumerate(got):
        np.testing.assert_array_equal(r["u"], want[i % 3]["u"])
        np.testing.assert_array_equal(r["ncert"], want[i % 3]["ncert"])
    # the buffer and its sort, the bins and marks of 16,256 edges and the allocator's blocks
    assert grown < 56 * (1 << 22) + (64 << 20), grown
