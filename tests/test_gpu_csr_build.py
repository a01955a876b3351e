"""Device CSR construction at the edges of its tiles, digits and row gaps.

Key counts one below, at and one above the sort's and the emission's tile of
8,192 keys and the key emission's tile of 2,048 edges, vertex counts whose ids
need one to 31 bits (each width splits into other digits), repeats of every
key, loops only, and long runs of rows without entries.  The rows equal those
of a NumPy construction."""
import numpy as np
import pytest
import torch

import paper_1104_4518_gb300 as bfs
from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu


def numpy_csr(src, dst, n, directed):
    keep = src != dst
    u, v = src[keep].astype(np.int64), dst[keep].astype(np.int64)
    if not directed:
        u, v = np.concatenate([u, v]), np.concatenate([v, u])
    key = np.unique(u * n + v)
    rows, cols = key // n, key % n
    off = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=off[1:])
    return off, cols.astype(np.int32)


def check(src, dst, n, directed=False):
    src, dst = np.asarray(src, np.int32), np.asarray(dst, np.int32)
    g = bfs.bfs_graph_create_from_edges(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n, directed=directed)
    off, adj = bfs.bfs_graph_copy_csr(g)
    want_off, want_adj = numpy_csr(src, dst, n, directed)
    assert g.nnz == want_adj.size
    assert np.array_equal(off.cpu().numpy(), want_off)
    assert np.array_equal(adj.cpu().numpy(), want_adj)
    g.destroy()


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("keys", [2, 2046, 2048, 2050, 4094, 4096, 4098, 8190, 8192, 8194, 16384, 40962, 3000002])
def test_key_counts_around_the_tiles(keys, directed):
    require_cuda()
    m = keys if directed else keys // 2
    rng = np.random.default_rng(keys)
    n = max(3, m // 9)
    src = rng.integers(0, n, m)
    check(src, (src + 1 + rng.integers(0, n - 1, m)) % n, n, directed)  # no loops: exactly `keys` keys


@pytest.mark.parametrize("bits", list(range(1, 25)))
def test_id_widths(bits):
    require_cuda()
    rng = np.random.default_rng(bits)
    n = (1 << bits) - (1 if bits > 1 else 0)
    check(rng.integers(0, n, 5000), rng.integers(0, n, 5000), n)


@pytest.mark.parametrize("directed", [False, True])
def test_repeats_loops_and_gaps(directed):
    require_cuda()
    rng = np.random.default_rng(4)
    n = 200003
    one = rng.integers(0, n, 3)
    check(np.repeat(one, 30000), np.repeat(one[::-1], 30000), n, directed)    # few values, many repeats, long gaps
    check(rng.integers(0, n, 50), rng.integers(0, n, 50), n, directed)        # gaps of thousands of rows
    loops = rng.integers(0, n, 9000)
    check(loops, loops, n, directed)                                          # loops only
    check([0], [n - 1], n, directed)
    check([n - 1], [0], n, directed)
    check([], [], n, directed)
    star = np.arange(1, 30000)
    check(np.zeros(star.size), star, 30000, directed)                         # one long row


def test_endpoint_outside_the_range_is_refused():
    require_cuda()
    for bad in (-1, 100, 2**31 - 1):
        src = torch.zeros(5000, dtype=torch.int32, device="cuda")
        dst = torch.ones(5000, dtype=torch.int32, device="cuda")
        dst[4321] = bad
        with pytest.raises(bfs.BfsError) as e:
            bfs.bfs_graph_create_from_edges(src, dst, 100)
        assert e.value.code == bfs.BFS_ERR_INVALID_ARG
