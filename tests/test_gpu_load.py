"""What the load keeps of its input: list in device memory, pinned and pageable host memory,
on and off 16-byte boundaries, with a pair table that serves or not, and with timestamps whose
range passes 32 bits visibly, by one timestamp, or not at all; against the CPU oracle."""
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


def _place(x, where):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(x))
    kind, _, shift = where.partition("+")
    if kind == "pageable":
        return x
    room = torch.empty(len(x) + 1, dtype=t.dtype, pin_memory=kind == "pinned", device="cuda" if kind == "device" else "cpu")
    view = room[int(shift or 0):][:len(x)]
    view.copy_(t)
    return view


def _graph(pairs, m, times):
    """m edges over at most `pairs` pairs of 700 vertices (and one block of 40), in time order."""
    rng = np.random.default_rng(pairs + m)
    x, y = rng.integers(0, 700, (2, pairs))
    i, j = np.triu_indices(40, 1)
    x, y = np.concatenate([x, i]), np.concatenate([y, j])
    k = rng.integers(0, len(x), m)
    t = np.sort(rng.integers(0, 10 ** 6, m))
    if times == "wide":
        t = t * 10 ** 5
    elif times == "one outlier":
        t[-1] = (1 << 32) + 7
    elif times == "largest offsets":  # the last range that 32 bits hold, not from 0
        t = t + (1 << 40)
        t[-1] = t[0] + (1 << 32) - 2
    return W.TemporalGraph(700, x[k].astype(np.int32), y[k].astype(np.int32), t)


def _check(F, g, where, scale):
    q = W.Query(3000 * scale, 1, 10, W.Q_EXISTS, W.DIR_EITHER, W.U_COMMON, True)
    arrays = [_place(a, w) for a, w in zip((g.src, g.dst, g.t), where)]
    with F.TemporalGraph(g.n, *arrays) as G, oracle.OracleGraph.of(g) as og:
        got, want = G.query(q), og.query(q)
    np.testing.assert_array_equal(got["edge_count"], want["edge_count"])
    assert pairs_of(got) == pairs_of(want)
    assert want["edge_count"].any()


@pytest.mark.parametrize("where", [("device",) * 3, ("device+1",) * 3, ("pinned",) * 3, ("pinned+1",) * 3,
                                   ("pageable",) * 3, ("pinned", "device", "device"), ("device", "device", "pinned"),
                                   ("device", "pageable", "pinned+1")])
@pytest.mark.parametrize("times", ["narrow", "wide", "one outlier", "largest offsets"])
@pytest.mark.parametrize("table", ["serves", "keys"])
def test_list_in_any_memory(F, monkeypatch, where, times, table):
    if table == "keys":
        monkeypatch.setenv("FOLTY_PAIR_SORT", "keys")
    _check(F, _graph(3000, 20_003, times), where, 10 ** 5 if times == "wide" else 1)


# lists of so many edges whose times the load looks at first (2^22 and up), and just too few
@pytest.mark.parametrize("m", [(1 << 22) - 1, 1 << 22, (1 << 22) + 2])
@pytest.mark.parametrize("times", ["narrow", "wide", "one outlier", "largest offsets"])
def test_long_lists_in_device_memory(F, m, times):
    g = _graph(60_000, m, times)
    scale = 10 ** 5 if times == "wide" else 1
    queries = [W.Query(d * scale, 1, 10, W.Q_EXISTS, W.DIR_OUT, W.U_HEAD, False) for d in (1, 50)]
    arrays = [_place(a, "device") for a in (g.src, g.dst, g.t)]
    results = []
    for xs in (arrays, (g.src, g.dst, g.t)):
        with F.TemporalGraph(g.n, *xs) as G:
            results.append([pairs_of(G.query(q)) for q in queries])
            info = G.info()
        assert info["m"] == m and info["time_sorted"] == 1
    assert results[0] == results[1] and len(results[0][1]) > 0


# pinned lists whose times the load looks at first (2^20 edges and up), and just too few; a look
# that misses the one late edge
@pytest.mark.parametrize("m", [(1 << 20) - 1, 1 << 20, (1 << 20) + 3])
@pytest.mark.parametrize("times", ["narrow", "wide", "one outlier", "largest offsets", "outlier unseen"])
def test_long_lists_in_pinned_memory(F, m, times):
    g = _graph(30_000, m, times.replace("outlier unseen", "one outlier"))
    if times == "outlier unseen":
        g.t[[-1, m // 2 + 5]] = g.t[[m // 2 + 5, -1]]
    scale = 10 ** 5 if times == "wide" else 1
    queries = [W.Query(d * scale, 1, 10, W.Q_EXISTS, W.DIR_OUT, W.U_HEAD, False) for d in (1, 50)]
    results = []
    for xs in ([_place(a, "pinned") for a in (g.src, g.dst, g.t)], (g.src, g.dst, g.t)):
        with F.TemporalGraph(g.n, *xs) as G:
            results.append([pairs_of(G.query(q)) for q in queries])
            assert G.info()["time_sorted"] == (times != "outlier unseen")
    assert results[0] == results[1] and len(results[0][1]) > 0


def test_pinned_lists_cross_the_link_once(F):
    """4M edges of 64-bit times whose pair table does not serve: read once, the 64 MB take about a
    third of a millisecond; read twice, as much again. The load must stay within 1.6 times
    that of one the table serves with 32-bit times, which reads every array once too."""
    import time

    import torch
    rng = np.random.default_rng(3)
    m, n = 4_000_000, 600_000

    def load_time(pairs, scale):
        x, y = rng.integers(0, n, (2, pairs))
        k = rng.integers(0, pairs, m)
        t = np.sort(rng.integers(0, 10 ** 6, m)) * scale
        arrays = [_place(a, "pinned") for a in (x[k].astype(np.int32), y[k].astype(np.int32), t)]
        best = np.inf
        for _ in range(12):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            h = F.folty_load_temporal_graph(n, *arrays)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
            F.folty_free(h)
        return best

    assert load_time(2_000_000, 10 ** 5) < 1.6 * load_time(50_000, 1)
