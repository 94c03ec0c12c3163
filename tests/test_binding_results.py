"""How the binding takes results over from the library's memory: lists past 2^31 bytes, an
error on the way, and what an array of per-edge counts keeps alive. Results are made here as
the library makes them (host memory of malloc, released by folty_free)."""
import ctypes

import numpy as np
import pytest

RESULT_TAG, FREED_TAG = 0x464F4C5459525354, 0x464F4C5459465245


@pytest.fixture(scope="module")
def F():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_17215_gb300 as F
    return F


@pytest.fixture(scope="module")
def libc():
    libc = ctypes.CDLL(None)
    libc.calloc.restype = ctypes.c_void_p
    libc.calloc.argtypes = [ctypes.c_size_t, ctypes.c_size_t]
    return libc


def _set_pairs(F, libc, r, k, m=0):
    """k pairs (0 so far) in one block, and with m > 0 that many per-edge counts."""
    r.tag, r.n_pairs = RESULT_TAG, k
    block = libc.calloc(4 * k, 4)
    for i, name in enumerate(("u", "v", "count", "ncert")):
        setattr(r, name, ctypes.cast(block + 4 * k * i, ctypes.POINTER(ctypes.c_int32)))
    if m:
        r.m = m
        r.edge_count = ctypes.cast(libc.calloc(m, 4), ctypes.POINTER(ctypes.c_int32))


@pytest.mark.parametrize("count", [(1 << 28) + 2])
def test_certificates_past_two_gigabytes(F, libc, count):
    r = F.folty_result()
    r.tag, r.n_cert_edges = RESULT_TAG, count
    r.certificate = ctypes.cast(libc.calloc(count, 8), ctypes.POINTER(ctypes.c_int64))
    r.certificate[count - 1] = 7
    got = F._take_results(r, 1)[0]["certificates"]
    assert got.shape == (count,) and got.dtype == np.int64 and got[-1] == 7 and got[0] == 0
    assert r.tag == FREED_TAG


@pytest.mark.parametrize("k", [(1 << 27) + 1])
def test_pairs_past_two_gigabytes(F, libc, k):
    r = F.folty_result()
    _set_pairs(F, libc, r, k)
    r.u[k - 1], r.ncert[k - 1] = 5, 9
    got = F._take_results(r, 1)[0]
    assert [got[x].shape for x in ("u", "v", "count", "ncert")] == [(k,)] * 4
    assert got["u"][-1] == 5 and got["v"][0] == 0 and got["ncert"][-1] == 9
    assert r.tag == FREED_TAG


def test_edge_counts_keep_their_own_memory_only(F, libc):
    rs = (F.folty_result * 2)()
    for i, r in enumerate(rs):
        _set_pairs(F, libc, r, 3, 5 + i)
        r.edge_count[4] = 11 + i
    got = F._take_results(rs, 2)
    # the lists have been released, the counts live on with their arrays
    assert [r.tag for r in rs] == [FREED_TAG] * 2
    assert [bool(r.u) for r in rs] == [False] * 2
    counts = [x["edge_count"] for x in got]
    del got
    assert [c.tolist() for c in counts] == [[0, 0, 0, 0, 11], [0, 0, 0, 0, 12, 0]]
    assert all(c.flags["WRITEABLE"] for c in counts)


def test_an_error_releases_every_result(F, libc, monkeypatch):
    rs = (F.folty_result * 4)()
    for r in rs:
        _set_pairs(F, libc, r, 3, 5)
    real, calls = F._block, []

    def failing(*args):
        calls.append(args)
        if len(calls) == 2:
            raise MemoryError
        return real(*args)

    monkeypatch.setattr(F, "_block", failing)
    with pytest.raises(MemoryError):
        F._take_results(rs, 4)
    assert [r.tag for r in rs] == [FREED_TAG] * 4
