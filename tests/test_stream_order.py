"""What the library prepares for a stream's traversals is ordered on that stream.

A non-blocking stream does not wait for the legacy default stream, and device
fills and pageable copies on the latter may still be outstanding when the call
returns.  So a call on stream S puts its fills and its copies to the device on
S, or waits for them.  Run on the stand-in CUDA runtime (no GPU).
"""
import ctypes

import pytest

from fake_cuda import FakeLibrary

S = 0x5150  # a stream handle


def unordered(log, stream):
    """Fills and copies that neither run on `stream` nor are waited for before the next launch."""
    pending, bad = [], []
    for e in log:
        if e.what in ("memset", "memcpy") and e.stream != stream:
            pending.append(e)
        elif e.what == "device sync" or (e.what == "stream sync" and e.stream != stream):
            pending = [p for p in pending if e.what != "device sync" and p.stream != e.stream]
        elif e.what == "launch" and e.stream == stream:
            bad += pending
            pending = []
    return bad + pending


@pytest.fixture()
def lib():
    return FakeLibrary()


def test_first_run_on_a_stream(lib):
    g = lib.graph()
    log = lib.taken(lambda: lib.run(g, 100, S))
    assert [e for e in log if e.what == "launch"] and [e for e in log if e.what == "memset"]
    assert not unordered(log, S)


def test_first_batch_on_a_stream(lib):
    n = 100
    g = lib.graph(n)
    out = (ctypes.c_int32 * (4 * n))()
    base = ctypes.addressof(out)
    log = lib.taken(lambda: lib.c.bfs_run_batch(g, (ctypes.c_int32 * 2)(0, 1), 2, ctypes.c_void_p(base),
                                                ctypes.c_void_p(base + 8 * n), None, ctypes.c_void_p(S)))
    assert [e for e in log if e.what == "launch"]
    assert not unordered(log, S)


def test_ragged_run_and_its_union(lib):
    n = 50
    parts = (ctypes.c_void_p * 2)(lib.graph(n), lib.graph(n))
    u = ctypes.c_void_p()
    log = lib.taken(lambda: lib.c.bfs_graph_union(parts, 2, ctypes.c_void_p(S), ctypes.byref(u)))
    table = [e for e in log if e.what == "memcpy" and e.bytes == 8 * 3][-1]  # where the parts start
    assert table.stream == S or any(e.what == "stream sync" and e.stream == table.stream for e in log[log.index(table):])
    outs = [(ctypes.c_int32 * n)() for _ in range(4)]
    ptr = [ctypes.addressof(o) for o in outs]
    log = lib.taken(lambda: lib.c.bfs_run_ragged(u, (ctypes.c_int32 * 2)(0, 0), (ctypes.c_void_p * 2)(*ptr[:2]),
                                                 (ctypes.c_void_p * 2)(*ptr[2:]), None, ctypes.c_void_p(S)))
    assert [e for e in log if e.what == "launch"]
    assert not unordered(log, S)


def test_first_learned_run_on_a_stream(lib):
    import paper_1104_4518_gb300 as bfs
    g = lib.graph()
    assert lib.c.bfs_selector_set_params((ctypes.c_float * bfs.BFS_MLP_PARAMS)()) == 0
    o = bfs.bfs_opts(selector=bfs.BFS_SELECT_LEARNED)
    log = lib.taken(lambda: lib.run(g, 100, S, ctypes.byref(o)))
    assert [e for e in log if e.what == "memcpy" and e.bytes == 4 * bfs.BFS_MLP_PARAMS]
    assert not unordered(log, S)


def test_first_static_run_on_a_stream(lib):
    off, adj = (ctypes.c_int64 * 3)(0, 1, 2), (ctypes.c_int32 * 2)(1, 0)
    out = (ctypes.c_int32 * 4)()
    base = ctypes.addressof(out)
    log = lib.taken(lambda: lib.c.bfs_run_static(off, adj, 2, ctypes.c_int64(2), 0, ctypes.c_void_p(base),
                                                 ctypes.c_void_p(base + 8), ctypes.c_void_p(S)))
    assert [e for e in log if e.what == "launch"] and [e for e in log if e.what == "memset"]
    assert not unordered(log, S)


def test_clearing_a_reported_error(lib):
    n = 100
    g = lib.graph(n)
    log = lib.taken(lambda: lib.run(g, n, S))
    status = [e for e in log if e.what == "memset" and e.bytes == 16][0].ptr
    ctypes.c_int.from_address(status).value = 5  # as a traversal whose wait ran out leaves it
    log = lib.taken(lambda: lib.c.bfs_sync(g, ctypes.c_void_p(S)))
    fills = [e for e in log if e.what == "memset"]
    assert status in [e.ptr for e in fills] and ctypes.c_int.from_address(status).value == 0
    assert all(e.stream == S for e in fills)


def test_copying_the_rows_out_waits_for_the_copies(lib):
    """bfs_graph_copy_csr is synchronous, to device memory too (cudaMemcpy between device arrays does not wait)."""
    n = 100
    g = lib.graph(n)
    off, adj = (ctypes.c_int64 * (n + 1))(), (ctypes.c_int32 * (2 * n))()
    log = lib.taken(lambda: lib.c.bfs_graph_copy_csr(g, off, adj, 0))
    copies = [i for i, e in enumerate(log) if e.what == "memcpy"]
    assert len(copies) == 2
    assert any(e.what == "stream sync" and e.stream == log[copies[-1]].stream for e in log[copies[-1]:])


def test_first_run_on_a_captured_stream(lib):
    """Work on a captured stream happens when the graph is launched, if ever; what a workspace and the selector's
    parameters start from has to be there for every later run as well."""
    import paper_1104_4518_gb300 as bfs
    g = lib.graph()
    assert lib.c.bfs_selector_set_params((ctypes.c_float * bfs.BFS_MLP_PARAMS)()) == 0
    o = bfs.bfs_opts(selector=bfs.BFS_SELECT_LEARNED)
    lib.c.fake_set_captured(ctypes.c_void_p(S))
    log = lib.taken(lambda: setattr(lib, "rc", lib.run(g, 100, S, ctypes.byref(o))))
    lib.c.fake_set_captured(None)
    assert lib.rc == 0, lib.c.bfs_last_error()
    done = [(i, e) for i, e in enumerate(log) if e.what in ("memset", "memcpy")]
    assert {16, 128 * 2} <= {e.bytes for _, e in done} and 4 * bfs.BFS_MLP_PARAMS in {e.bytes for _, e in done}
    for i, e in done:
        assert e.stream != S and any(x.what == "stream sync" and x.stream == e.stream for x in log[i:])
