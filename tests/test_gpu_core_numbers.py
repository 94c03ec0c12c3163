"""Core numbers of graphs whose hubs' rows are shortened more than once, and given up again,
while the values fall, against the bucket algorithm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_17215_gb300 as F
    return F


def core_numbers(n, pairs):
    """By the bucket algorithm: remove a vertex of least degree, one at a time."""
    ends = np.concatenate([pairs, pairs[:, ::-1]])
    ends = ends[np.argsort(ends[:, 0], kind="stable")]
    row = np.searchsorted(ends[:, 0], np.arange(n + 1)).tolist()
    adj = ends[:, 1].tolist()
    deg = [row[v + 1] - row[v] for v in range(n)]
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
        for w in adj[row[v]:row[v + 1]]:
            if core[w] < 0:
                deg[w] -= 1
                buckets[deg[w]].append(w)
                d = min(d, deg[w])
    return np.array(core)


def hub_graph(groups, cliques, hubs=1):
    """Hubs (ids from 0) joined to groups of members and to cliques, (n, pairs). A group is
    (members, degree, supports, share): members of that degree, `supports` of their neighbours
    vertices of a degree near it that `share` members have in common, the rest leaves. The
    supports' values fall to `share` after the first round and the members' after the second.
    A clique is (size, joined): the first `joined` of its vertices are the hubs' neighbours."""
    parts, n = [], hubs
    if hubs > 1:
        parts.append(np.stack(np.triu_indices(hubs, 1), 1))
    every = np.arange(hubs)

    def join(a, b):
        parts.append(np.stack(np.broadcast_arrays(a, b), -1).reshape(-1, 2))

    for members, degree, supports, share in groups:
        w = np.arange(members) + n
        n += members
        join(w[:, None], every[None, :])
        if supports:
            cohorts = -(-members // share)
            s = np.arange(cohorts * supports).reshape(cohorts, supports) + n
            n += s.size
            join(np.repeat(w, supports), s[np.arange(members) // share].ravel())
            leaves = max(supports - share, 0)
            join(np.repeat(s.ravel(), leaves), np.arange(s.size * leaves) + n)
            n += s.size * leaves
        leaves = degree - supports - hubs
        join(np.repeat(w, leaves), np.arange(members * leaves) + n)
        n += members * leaves
    for size, joined in cliques:
        i, j = np.triu_indices(size, 1)
        parts.append(np.stack([i + n, j + n], 1))
        join((np.arange(joined) + n)[:, None], every[None, :])
        n += size
    return n, np.concatenate(parts)


# a row cut at 65 (an eighth of 520), cut again at 34 (a third of 100) while its value falls to
# between the two: the 60-clique's members went with the first cut. Falls in more stages, with
# cliques around the cut values. Several hubs at once. A cut row that fits a warp and has to be
# given up for a whole row that does not, once and after a second cut.
@pytest.mark.parametrize("groups,cliques,hubs", [
    ([(520, 521, 100, 10)], [(60, 60), (70, 40)], 1),
    ([(520, 700, 150, 30)], [(64, 64), (90, 51), (50, 50)], 1),
    ([(900, 700, 300, 60)], [(110, 110), (150, 105), (34, 34)], 3),
    ([(520, 521, 0, 1)], [(60, 60), (70, 40)], 1),
    ([(520, 521, 100, 10)], [(62, 62), (80, 40)], 2),
])
def test_core_numbers_with_rows_shortened_twice(F, groups, cliques, hubs):
    n, pairs = hub_graph(groups, cliques, hubs)
    want = core_numbers(n, pairs)
    ids = np.random.default_rng(n).permutation(n)
    with F.TemporalGraph(n, ids[pairs[:, 0]].astype(np.int32), ids[pairs[:, 1]].astype(np.int32),
                         np.zeros(len(pairs), np.int64)) as G:
        np.testing.assert_array_equal(G.core_numbers()[ids], want)
        info = G.info()
    assert info["degeneracy"] == want.max()
    assert info["max_out_degree"] <= info["degeneracy"]


def test_long_stretches_of_rounds_are_no_timeout(F, monkeypatch):
    """A path of 60,000 vertices: 30,000 rounds by one block, while the others wait for longer
    than their bound."""
    monkeypatch.setenv("FOLTY_CORE_TIMEOUT_MS", "5")
    n = 60_000
    a = np.arange(n - 1, dtype=np.int32)
    with F.TemporalGraph(n, a, a + 1, np.zeros(n - 1, np.int64)) as G:
        assert (G.core_numbers() == 1).all()
        assert G.info()["peel_rounds"] == n // 2


def removal_rounds(n, pairs):
    """Rounds of the peeling that removes, level by level, every vertex of at most the level's
    remaining degree at once."""
    ends = np.concatenate([pairs, pairs[:, ::-1]])
    ends = ends[np.argsort(ends[:, 0], kind="stable")]
    row = np.searchsorted(ends[:, 0], np.arange(n + 1))
    deg = np.diff(row)
    left, rounds, level = n, 0, 0
    out = np.zeros(n, bool)
    while left:
        front = np.flatnonzero(~out & (deg <= level))
        if len(front) == 0:
            level = int(deg[~out].min())
            continue
        while len(front):
            rounds += 1
            out[front] = True
            left -= len(front)
            told = np.concatenate([ends[row[v]:row[v + 1], 1] for v in front])
            np.subtract.at(deg, told, 1)
            told = np.unique(told)
            front = told[~out[told] & (deg[told] <= level)]
    return rounds


def _paths(lengths, first=0):
    """Paths of the given numbers of vertices, (pairs, their first vertices, vertices in all)."""
    start = first + np.concatenate([[0], np.cumsum(lengths)])
    a = np.concatenate([np.arange(s, e - 1) for s, e in zip(start, start[1:])])
    return np.stack([a, a + 1], 1), start[:-1], int(start[-1])


def _chain_graph(kind):
    rng = np.random.default_rng(7)
    if kind == "path":
        return 5001, _paths([5001])[0]
    if kind in ("few paths", "many paths"):  # 2 vertices a round each: through 32 and through 96
        pairs, _, n = _paths(rng.integers(2, 900, 21 if kind == "few paths" else 55))
        return n, pairs
    if kind == "caterpillar":  # rows of 3 to 12, too long for one warp from 9 on
        pairs, _, n = _paths([1200])
        feet = np.repeat(np.arange(n), rng.integers(0, 11, n))
        return n + len(feet), np.concatenate([pairs, np.stack([feet, np.arange(len(feet)) + n], 1)])
    if kind == "hubs":  # chains from leaves to two hubs of long rows, which clique members hold
        i, j = np.triu_indices(40, 1)
        pairs, ends, n = _paths(rng.integers(1, 400, 1400), 42)
        clique = np.stack([np.repeat([40, 41], 40), np.tile(np.arange(40), 2)], 1)
        return n, np.concatenate([np.stack([i, j], 1), clique, pairs,
                                  np.stack([ends, np.where(rng.random(len(ends)) < 0.5, 40, 41)], 1)])
    if kind == "ladder":
        a = np.arange(3000)
        return 6000, np.concatenate([np.stack([a[:-1], a[1:]], 1), np.stack([a[:-1], a[1:]], 1) + 3000, np.stack([a, a + 3000], 1)])
    if kind == "binary tree":
        a = np.arange(1, (1 << 13) - 1)
        return (1 << 13) - 1, np.stack([(a - 1) // 2, a], 1)
    a = np.arange(1, 20_000)  # every vertex joined to one of the 30 before it
    return 20_000, np.stack([np.maximum(a - rng.integers(1, 31, len(a)), 0), a], 1)


# rounds of few vertices: by one warp up to 32 with rows of up to 8, by one block up to 96
# (192 once it runs), between the two as the frontier shrinks, grows and meets long rows
@pytest.mark.parametrize("kind", ["path", "few paths", "many paths", "caterpillar", "hubs", "ladder", "binary tree",
                                  "long tree"])
def test_core_numbers_of_chains(F, kind):
    n, pairs = _chain_graph(kind)
    ids = np.random.default_rng(n).permutation(n)
    with F.TemporalGraph(n, ids[pairs[:, 0]].astype(np.int32), ids[pairs[:, 1]].astype(np.int32),
                         np.zeros(len(pairs), np.int64)) as G:
        np.testing.assert_array_equal(G.core_numbers()[ids], core_numbers(n, pairs))
        assert G.info()["peel_rounds"] == removal_rounds(n, pairs)
