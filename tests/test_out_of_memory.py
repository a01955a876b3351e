"""A call that runs out of device memory says so, and the next call starts again.

The buffers that a workspace gets on first use come in several allocations, and
any of them can be the one that fails.  Run on the stand-in CUDA runtime (no
GPU), which records a launch instead of running it on null pointers.
"""
import ctypes

import pytest

import paper_1104_4518_gb300 as bfs
from fake_cuda import FakeLibrary

N = 1000


def batch(lib, g):
    out = (ctypes.c_int32 * (4 * N))()
    base = ctypes.addressof(out)
    return lib.c.bfs_run_batch(g, (ctypes.c_int32 * 2)(0, 1), 2, ctypes.c_void_p(base), ctypes.c_void_p(base + 8 * N),
                               None, None)


def host_outputs(flags):
    return lambda lib, g: lib.run(g, N, 0, ctypes.byref(bfs.bfs_opts(flags=flags)))


CALLS = {"batched": batch, "host outputs": host_outputs(bfs.BFS_HOST_PTRS),
         "asynchronous host outputs": host_outputs(bfs.BFS_HOST_PTRS | bfs.BFS_HOST_ASYNC)}


@pytest.mark.parametrize("name", CALLS)
def test_every_allocation_of_a_call_may_fail(name):
    """Memory ends at the call's i-th allocation, for every i: the call and its repeat return BFS_ERR_OOM and launch
    nothing; with memory again it runs; and nothing is left once the graph is destroyed."""
    for i in range(100):
        lib = FakeLibrary()
        lib.c.fake_set_reported_total(ctypes.c_size_t(0))  # nothing is kept for later: live bytes are the graph's
        g = lib.graph(N)
        lib.c.fake_set_mallocs_left(ctypes.c_longlong(i))
        log = lib.taken(lambda: setattr(lib, "rc", CALLS[name](lib, g)))
        if lib.rc == 0:
            break
        assert lib.rc == bfs.BFS_ERR_OOM, lib.c.bfs_last_error()
        log += lib.taken(lambda: setattr(lib, "rc", CALLS[name](lib, g)))
        assert lib.rc == bfs.BFS_ERR_OOM, f"repeat after allocation {i} failed"
        assert not [e for e in log if e.what == "launch"]
        lib.c.fake_set_mallocs_left(ctypes.c_longlong(-1))
        log = lib.taken(lambda: setattr(lib, "rc", CALLS[name](lib, g)))
        assert lib.rc == 0 and [e for e in log if e.what == "launch"]
        lib.c.bfs_graph_destroy(g)
        assert lib.c.fake_live_bytes() == 0
    assert i > 3
