"""The cache that the library's device memory goes back through (csrc/api.cu),
on the stand-in CUDA runtime: what it may keep, when it gives it back, and that
a block it hands out is idle and still the library's.  No GPU."""
import ctypes
import threading
import time

import pytest

from fake_cuda import FakeLibrary

N = 1000


@pytest.fixture()
def lib():
    return FakeLibrary()


def whats(log):
    return [e.what for e in log]


def cycle(lib, n=N):
    lib.c.bfs_graph_destroy(lib.graph(n))


def test_a_block_is_not_reused_after_a_wait_that_failed(lib):
    """A release whose wait for the device fails (a capture in another thread forbids it, say) cannot know that the
    block is idle: it goes to the driver, which knows."""
    cycle(lib)
    assert "malloc" not in whats(lib.taken(lambda: cycle(lib)))  # (a wait that succeeded keeps them)
    g = lib.graph(N)
    lib.c.fake_sync_error(700)
    log = lib.taken(lambda: lib.c.bfs_graph_destroy(g))
    lib.c.fake_sync_error(0)
    assert "free" in whats(log)
    assert "malloc" in whats(lib.taken(lambda: lib.graph(N)))


def test_waiting_for_a_stream_frees_nothing(lib):
    """bfs_sync waits for its stream; a cudaFree there would wait for the whole device."""
    cycle(lib)
    g = lib.graph(7)
    time.sleep(1.1)  # the cached blocks have waited for more than a second
    log = lib.taken(lambda: lib.c.bfs_sync(g, ctypes.c_void_p(0x5150)))
    assert "stream sync" in whats(log)
    assert not {"free", "device sync"} & set(whats(log))
