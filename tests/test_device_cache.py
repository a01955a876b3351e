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


def test_bound(lib):
    """At most 1/64 of the device's memory is kept."""
    lib.c.fake_set_reported_total(ctypes.c_size_t(64 * 10000))
    log = lib.taken(lambda: cycle(lib))
    assert "free" in whats(log)
    assert 0 < lib.c.fake_live_bytes() <= 10000


def test_blocks_go_back_after_a_second_and_on_request(lib):
    cycle(lib)
    assert lib.c.fake_live_bytes() > 0
    time.sleep(1.1)
    lib.c.bfs_graph_destroy(lib.graph(3))
    assert lib.c.fake_live_bytes() <= 16 * 512  # what the small graph left
    cycle(lib)
    assert lib.c.bfs_memory_trim() == 0
    assert lib.c.fake_live_bytes() == 0
    lib.c.fake_set_device(1)  # blocks of any device
    cycle(lib)
    lib.c.fake_set_device(0)
    cycle(lib)
    assert lib.c.bfs_memory_trim() == 0
    assert lib.c.fake_live_bytes() == 0


def test_request_leaves_blocks_in_use_alone(lib):
    g = lib.graph(N)
    cycle(lib)
    used = lib.c.fake_live_bytes()
    assert lib.c.bfs_memory_trim() == 0
    assert 0 < lib.c.fake_live_bytes() < used
    assert lib.run(g, N) == 0 and lib.c.bfs_sync(g, None) == 0


def test_a_failed_allocation_takes_the_idle_blocks_first(lib):
    cycle(lib, 20 * N)
    assert lib.c.fake_live_bytes() > 300000
    lib.c.fake_set_total(ctypes.c_size_t(700000))  # not for both graphs
    g = None

    def create():
        nonlocal g
        g = lib.graph(40 * N)
    log = whats(lib.taken(create))
    at = log.index("malloc failed")
    assert log[at + 1] == "free" and "malloc" in log[at:]


def test_a_failed_first_allocation_of_a_thread_takes_the_idle_blocks_too(lib):
    """No context is current in a thread before its first call; the allocation makes it so, and then the idle blocks
    can be told to be its own."""
    cycle(lib, 20 * N)
    lib.c.fake_set_total(ctypes.c_size_t(400000))
    lib.c.fake_set_context(ctypes.c_ulonglong(0))
    log = whats(lib.taken(lambda: lib.graph(20 * N)))
    at = log.index("malloc failed")
    assert log[at + 1] == "free" and "malloc" in log[at:]


def test_request_leaves_the_current_context_alone(lib):
    """With all idle blocks on the current device there is no need to make another context current."""
    cycle(lib)
    log = lib.taken(lambda: lib.c.bfs_memory_trim())
    assert "set device" not in whats(log) and lib.c.fake_live_bytes() == 0
    cycle(lib)
    lib.c.fake_set_context(ctypes.c_ulonglong(0))  # in a thread that has made no call yet
    assert lib.c.bfs_memory_trim() == 0 and lib.c.fake_live_bytes() == 0


def test_release_with_another_device_current(lib):
    """A block of another device is not idle after a wait for the current one; and a device gets its own blocks only."""
    g = lib.graph(N)
    lib.c.fake_set_device(1)
    before = lib.c.fake_live_bytes()
    lib.c.bfs_graph_destroy(g)
    assert lib.c.fake_live_bytes() < before
    lib.c.fake_set_device(0)
    cycle(lib)
    lib.c.fake_set_device(1)
    kept = lib.c.fake_live_bytes()
    g = lib.graph(N)
    assert lib.c.fake_live_bytes() > kept
    lib.c.bfs_graph_destroy(g)


def test_two_threads(lib):
    """Graphs made, run and destroyed by two threads at once: no block has two owners."""
    owned, mu, bad = set(), threading.Lock(), []

    def work(seed):
        n = 50 + seed
        for i in range(200):
            g = lib.graph(n)
            off, adj = ctypes.c_void_p(), ctypes.c_void_p()
            lib.c.bfs_graph_csr(g, ctypes.byref(off), ctypes.byref(adj))
            with mu:
                if off.value in owned or adj.value in owned:
                    bad.append((seed, i))
                owned.update((off.value, adj.value))
            ok = lib.run(g, n, 0x1000 + seed) == 0 and lib.c.bfs_sync(g, ctypes.c_void_p(0x1000 + seed)) == 0
            rows = (ctypes.c_int64 * (n + 1)).from_address(off.value)
            if not ok or rows[n] != 2 * (n - 1) or rows[1] != 1:
                bad.append((seed, i))
            with mu:
                owned.difference_update((off.value, adj.value))
            lib.c.bfs_graph_destroy(g)
            if i % 50 == 49:
                lib.c.bfs_memory_trim()

    threads = [threading.Thread(target=work, args=(s,)) for s in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    assert lib.c.bfs_memory_trim() == 0
    assert lib.c.fake_live_bytes() == 0


def test_the_selectors_parameters_may_take_an_idle_block(lib):
    """With no memory left but what the library holds unused, a learned run still runs the network."""
    import paper_1104_4518_gb300 as bfs
    g = lib.graph(N)
    assert lib.run(g, N) == 0
    cycle(lib, 20 * N)
    lib.c.fake_set_total(ctypes.c_size_t(lib.c.fake_live_bytes()))
    assert lib.c.bfs_selector_set_params((ctypes.c_float * bfs.BFS_MLP_PARAMS)()) == 0
    o = bfs.bfs_opts(selector=bfs.BFS_SELECT_LEARNED)
    log = lib.taken(lambda: lib.run(g, N, 0, ctypes.byref(o)))
    assert [e for e in log if e.what == "memcpy" and e.bytes == 4 * bfs.BFS_MLP_PARAMS]


def test_blocks_of_a_context_that_was_reset_are_forgotten(lib):
    """cudaDeviceReset frees everything: what the cache held then is neither handed out nor freed again (its address
    may belong to someone else by then)."""
    cycle(lib)
    old = {e.ptr for e in lib.taken(lambda: cycle(lib, 20 * N)) if e.what == "malloc"}
    g = lib.graph(N)
    lib.c.fake_set_context(2)
    log = lib.taken(lambda: cycle(lib))
    assert "malloc" in whats(log) and "free" not in whats(log)
    assert not old & {e.ptr for e in log if e.what in ("memset", "memcpy")}
    time.sleep(1.1)
    log = lib.taken(lambda: (cycle(lib), lib.c.bfs_memory_trim()))
    assert not old & {e.ptr for e in log if e.what == "free"}
    kept = lib.c.fake_live_bytes()
    lib.c.bfs_graph_destroy(g)  # a graph of the old context: its blocks are not kept either
    lib.c.bfs_memory_trim()
    assert lib.c.fake_live_bytes() <= kept
