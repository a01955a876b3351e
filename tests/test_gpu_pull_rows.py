"""Pull levels whose rows end at every depth of the scan: at the probe record
(up to three entries), inside or at the edge of an aligned group of four or a
step of eight, and past the length from which a whole warp scans a row.

Root 0 joins H hubs; row vertex i joins one hub and L_i leaves with larger ids,
so with the hubs as frontier its scan has to pass all L_i leaves before the hub,
its largest frontier neighbour, at the very end of its row.  The frontier is
tested in shared memory exactly (n up to 65,536), through the summary (few
hubs) and in the bitmap (many hubs).  Levels and parents equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
import paper_1104_4518_gb300 as bfs
from gpu_helpers import assert_same, device_graph_from_edges, require_cuda, run_gpu
from paper_1104_4518_gb300 import inputs

pytestmark = pytest.mark.gpu

LENGTHS = list(range(0, 22)) + list(range(60, 68)) + list(range(124, 136)) + [300, 1023, 1024, 1025, 3000]


def deep_rows(hubs: int, repeat: int, pad: int = 0):
    rng = np.random.default_rng(hubs * 31 + repeat)
    lens = rng.permutation(np.repeat(LENGTHS, repeat)).astype(np.int64)
    rows = 1 + hubs + np.arange(lens.size)
    leaves = 1 + hubs + lens.size + np.arange(lens.sum())
    src = np.concatenate([np.zeros(hubs, np.int64), rows, np.repeat(rows, lens)])
    dst = np.concatenate([np.arange(1, hubs + 1), rng.integers(1, hubs + 1, lens.size), leaves])
    n = 1 + hubs + lens.size + int(lens.sum()) + pad
    return inputs.EdgeList(n, src.astype(np.int32), dst.astype(np.int32), f"deep-{hubs}-{repeat}-{pad}")


# n: 19 K and 46 K (exact), 65,536 and 65,537 (its last and the first summarised), 139 K with few and many hubs
@pytest.mark.parametrize("hubs,repeat,n", [(1, 2, 0), (40, 5, 0), (3, 6, 65536), (3, 6, 65537), (7, 15, 0), (3000, 15, 0)])
def test_rows_of_every_depth(hubs, repeat, n):
    require_cuda()
    el = deep_rows(hubs, repeat)
    if n:
        assert n >= el.n
        el.n = n
    og = oracle.csr_of(el)
    ref = oracle.bfs(og, 0)
    g = device_graph_from_edges(el)
    for opts in (bfs.RunOptions(selector=bfs.BFS_SELECT_FORCED, forced_variant=bfs.BFS_VARIANT_PULL), None):
        assert_same(ref, run_gpu(g, 0, opts), f"{el.name} {'pull' if opts else 'heuristic'}")
    bfs.bfs_set_tuning(g, pull_thread_degree=1)
    assert_same(ref, run_gpu(g, 0, bfs.RunOptions(selector=bfs.BFS_SELECT_FORCED, forced_variant=bfs.BFS_VARIANT_PULL)),
                f"{el.name} one probe")
    g.destroy()


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_rows_without_probe_records_at_any_alignment(shift):
    """The static entry point has no probe records and scans the caller's adjacency where it lies."""
    require_cuda()
    og = oracle.csr_of(deep_rows(2000, 4))
    ref = oracle.bfs(og, 0)
    adj = torch.empty(og.adj.shape[0] + shift, dtype=torch.int32, device="cuda")[shift:]
    adj.copy_(torch.from_numpy(og.adj))
    off = torch.from_numpy(og.offsets).cuda()
    parent = torch.empty(og.n, dtype=torch.int32, device="cuda")
    level = torch.empty(og.n, dtype=torch.int32, device="cuda")
    bfs.bfs_run_static(off, adj, 0, parent, level)
    assert_same(ref, (level.cpu().numpy(), parent.cpu().numpy()), f"static, adjacency {4 * shift} bytes off")
