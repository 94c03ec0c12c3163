"""Calls whose allocator runs out once, at every allocation in turn: the call says so, and the
same call on the same graph succeeds afterwards with the results of an undisturbed one."""
import ctypes

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


class _Failing:
    """A graph on PyTorch's memory whose allocator refuses its `fail`-th request from now on."""

    def __init__(self, F, g):
        import torch
        self.F, self.left, self.live, self.peak, self.fill = F, -1, {}, 0, None

        @F.ALLOC_FN
        def alloc(nbytes, stream, ctx):
            if self.left == 0:
                self.left = -1
                return None
            self.left -= self.left > 0
            p = torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))
            self.live[p] = int(nbytes)
            self.peak = max(self.peak, sum(self.live.values()))
            if self.fill is not None:  # what the memory holds before its first use, on its own stream
                view = type("Bytes", (), {"__cuda_array_interface__": {"shape": (int(nbytes),), "typestr": "|u1",
                                                                       "data": (p, False), "version": 3}})()
                own = torch.cuda.ExternalStream(int(stream)) if stream else torch.cuda.default_stream()
                with torch.cuda.stream(own):
                    torch.as_tensor(view, device="cuda").fill_(self.fill)
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

    def refused(self, fail, call):
        """Whether call ran out at its fail-th request (else it made fewer)."""
        self.left = fail
        try:
            call()
        except self.F.FoltyError as e:
            assert e.status == self.F.FOLTY_ENOMEM, e
            assert self.left == -1
            return True
        finally:
            self.left, reached = -1, self.left == -1
        assert not reached, "a refused request went unnoticed"
        return False

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.F.folty_free(self.handle)


def _graph(kind):
    if kind == "small":  # within the allocation-free counts' limit
        return W.config_graph(2, scale=0.01)
    return W.config_graph(2, scale=0.06)


QUERIES = [W.Query(86400, 1, 10, W.Q_FORALL_T, W.DIR_EITHER, W.U_COMMON, False),
           W.Query(3600, 1, 2, W.Q_EXISTS, W.DIR_OUT, W.U_HEAD, False)]


@pytest.mark.parametrize("kind", ["small", "large"])
def test_first_query_after_one_that_ran_out_of_memory(F, kind):
    g = _graph(kind)
    with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G:
        want = [pairs_of(G.query(q)) for q in QUERIES]
    fail = 0
    while True:
        with _Failing(F, g) as G:
            F.folty_preprocess(G.handle)
            refused = G.refused(fail, lambda: F.folty_query(G.handle, QUERIES[0]))
            for q, w in zip(QUERIES + QUERIES, want + want):
                assert pairs_of(F.folty_query(G.handle, q)) == w, (fail, str(q))
        if not refused:
            break
        fail += 1
    assert fail > 8  # the plan's buffers, at least


@pytest.mark.parametrize("kind", ["small", "large", "shuffled"])
def test_preprocessing_repeated_after_it_ran_out_of_memory(F, kind):
    g = _graph(kind)
    if kind == "shuffled":
        p = np.random.default_rng(1).permutation(g.m)
        g = W.TemporalGraph(g.n, g.src[p], g.dst[p], g.t[p])
    counts = W.Query(86400, 1, 10, W.Q_EXISTS, W.DIR_IN, W.U_HEAD, True)
    with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G:
        want, edges, info = [pairs_of(G.query(q)) for q in QUERIES], G.query(counts)["edge_count"], G.info()
    fail = 0
    while True:
        with _Failing(F, g) as G:
            refused = G.refused(fail, lambda: F.folty_preprocess(G.handle))
            if refused:
                F.folty_preprocess(G.handle)
            assert [pairs_of(F.folty_query(G.handle, q)) for q in QUERIES] == want, fail
            np.testing.assert_array_equal(F.folty_query(G.handle, counts)["edge_count"], edges)
            got = F.folty_graph_get_info(G.handle)
            assert {k: v for k, v in got.items() if k != "device_bytes"} == {k: v for k, v in info.items() if k != "device_bytes"}
        if not refused:
            break
        fail += 1
    assert fail > 10


@pytest.mark.parametrize("kind", ["small", "large"])
def test_preprocessing_that_ran_out_of_memory_leaves_nothing(F, kind):
    """A refused call gives back what it had taken, and the repeated one computes everything
    anew, whatever the memory it is given held (255: a triangle of no window)."""
    g = _graph(kind)
    with F.TemporalGraph(g.n, g.src, g.dst, g.t) as G:
        want = [pairs_of(G.query(q)) for q in QUERIES]
    fail, refused = 0, True
    while refused:
        with _Failing(F, g) as G:
            loaded = dict(G.live)
            refused = G.refused(fail, lambda: F.folty_preprocess(G.handle))
            if refused:
                assert G.live == loaded, fail
                G.fill = 255
                F.folty_preprocess(G.handle)
                G.fill = None
            assert [pairs_of(F.folty_query(G.handle, q)) for q in QUERIES] == want, fail
        fail += 1
    assert fail > 10


def _sparse_bounds_graph():
    """1.2M static edges between two sides of 20,000 vertices, without a triangle: the listing's
    bound (the sum of the shorter out-lists) has tens of millions of entries, all empty."""
    rng = np.random.default_rng(4)
    n, m = 20_000, 1_200_000
    src, dst = rng.integers(0, n, m), rng.integers(n, 2 * n, m)
    return W.TemporalGraph(2 * n, src.astype(np.int32), dst.astype(np.int32), np.sort(rng.integers(0, 1000, m)))


def test_liveness_rows_have_the_triangles_size(F, monkeypatch):
    """The array of a one-pass listing has room for its bound, 16 B an entry; the rows of
    liveness bytes (3 B an entry) have that of the triangles."""
    g = _sparse_bounds_graph()
    held, largest = [], []
    for layout in ("", "counted"):
        monkeypatch.setenv("FOLTY_TRI_LAYOUT", layout)
        with _Failing(F, g) as G:
            F.folty_preprocess(G.handle)
            info = F.folty_graph_get_info(G.handle)
            assert info["triangles"] == 0 and info["m_kept"] > F.NOALLOC_MAX_EDGES
            held.append(sum(G.live.values()))
            largest.append(max(G.live.values()))
    entries = largest[0] // 16
    assert entries > 5_000_000 and largest[0] > 2 * largest[1]
    assert held[0] - largest[0] - held[1] < entries // 2


def test_tuning_takes_one_set_of_selection_buffers(F):
    """The first query of a graph with 16M triangles times its probe shapes before it allocates
    its plan, which holds one set of selection buffers (17 B a triangle) and little else: the
    trials must not need more."""
    k, size = 100, 100
    i, j = np.triu_indices(size, 1)
    base = np.repeat(np.arange(k) * size, len(i))
    src, dst = np.tile(i, k) + base, np.tile(j, k) + base
    src, dst = np.tile(src, 3).astype(np.int32), np.tile(dst, 3).astype(np.int32)
    g = W.TemporalGraph(k * size, src, dst, np.sort(np.random.default_rng(2).integers(0, 1000, len(src))))
    F.folty_tuning_clear_cache()
    with _Failing(F, g) as G:
        F.folty_preprocess(G.handle)
        assert F.folty_graph_get_info(G.handle)["triangles"] == k * size * (size - 1) * (size - 2) // 6
        before = G.peak = sum(G.live.values())
        F.folty_query(G.handle, QUERIES[1])
        assert F.folty_graph_tuning(G.handle)["probe_source"] == "timed trials"
        kept, peak = sum(G.live.values()) - before, G.peak - before
    assert kept > 17 * 16_000_000 and peak < 1.2 * kept, (kept, peak)


def test_a_query_that_ran_out_of_memory_holds_no_result(F):
    """A query with every optional output, whose host arrays exist before its last device
    buffers: the call that fails leaves nothing for the caller to release."""
    g = _graph("large")  # its per-edge counts are allocated after the result
    q = F._params(W.Query(86400, 1, 10, W.Q_EXISTS, W.DIR_EITHER, W.U_COMMON, True, outer=W.OUTER_FORALL_T,
                          want_certificates=True, want_triples=True))
    with _Failing(F, g) as G:
        F.folty_preprocess(G.handle)
        fail = 0
        while True:
            r = F.folty_result()
            G.left = fail
            st = F.lib.folty_query(G.handle, ctypes.byref(q), ctypes.byref(r), F.current_stream())
            G.left, reached = -1, G.left == -1
            if st == F.FOLTY_OK:
                F._take_results(r, 1)
                break
            assert st == F.FOLTY_ENOMEM and reached, F.folty_last_error()
            assert r.tag != 0x464F4C5459525354 and not r.u and not r.certificate and not r.edge_count and not r.triple_x, fail
            fail += 1
        assert fail > 2
