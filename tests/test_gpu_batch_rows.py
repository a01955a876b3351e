"""Batched traversals at the edges of their row steps, word widths and level planes.

Rows end their scan inside and at the edges of the packed steps (8 and 40
entries), of the warp's row scan, and of the chunks of 1,024 entries; the number
of roots sits below, at and above each word width; levels need up to nine bit
planes.  Levels and parents equal the oracle's with every level pulled and with
every level expanded top-down."""
import numpy as np
import pytest

import oracle
import paper_1104_4518_gb300 as bfs
from gpu_helpers import assert_same, device_graph_from_edges, require_cuda
from paper_1104_4518_gb300 import inputs

pytestmark = pytest.mark.gpu

LENGTHS = list(range(0, 12)) + list(range(36, 46)) + [103, 104, 105, 167, 168, 169, 1022, 1023, 1024, 1025, 2047, 2500]


def check(el, roots, topdown_limit):
    og = oracle.csr_of(el)
    g = device_graph_from_edges(el)
    bfs.bfs_set_tuning(g, batch_topdown_limit=topdown_limit)
    parent, level = bfs.run_batch(g, [int(r) for r in roots])
    bfs.bfs_sync(g)
    refs = {}
    for i, r in enumerate(roots):
        if int(r) not in refs:
            refs[int(r)] = oracle.bfs(og, int(r))
        assert_same(refs[int(r)], (level[i].cpu().numpy(), parent[i].cpu().numpy()), f"{el.name} root {i} = {r}")
    g.destroy()


def deep_rows(hubs):
    """Root 0 joins the hubs; row vertex i joins one hub and L_i leaves with larger ids."""
    rng = np.random.default_rng(hubs)
    lens = rng.permutation(np.repeat(LENGTHS, 2)).astype(np.int64)
    rows = 1 + hubs + np.arange(lens.size)
    leaves = 1 + hubs + lens.size + np.arange(lens.sum())
    src = np.concatenate([np.zeros(hubs, np.int64), rows, np.repeat(rows, lens)])
    dst = np.concatenate([np.arange(1, hubs + 1), rng.integers(1, hubs + 1, lens.size), leaves])
    return inputs.EdgeList(1 + hubs + lens.size + int(lens.sum()), src.astype(np.int32), dst.astype(np.int32),
                           f"deep-{hubs}")


@pytest.mark.parametrize("topdown_limit", [1, 1 << 30])
@pytest.mark.parametrize("hubs", [1, 5])
def test_rows_of_every_depth(hubs, topdown_limit):
    require_cuda()
    el = deep_rows(hubs)
    check(el, [0, 1, hubs, 1 + hubs, el.n - 1, el.n // 2, 0], topdown_limit)


@pytest.mark.parametrize("topdown_limit", [1, 1 << 30])
@pytest.mark.parametrize("k", [1, 7, 8, 9, 16, 17, 31, 32, 33, 63, 64, 65, 129])
def test_root_counts_around_the_word_widths(k, topdown_limit):
    require_cuda()
    el, _ = inputs.disjoint_union([inputs.rmat(9, 8, seed=77), inputs.path(6)])
    check(el, inputs.roots(el, 400, 5)[np.arange(k) % 150], topdown_limit)


@pytest.mark.parametrize("topdown_limit", [1, 1 << 30])
@pytest.mark.parametrize("n", [2, 3, 5, 9, 17, 33, 257, 300])
def test_levels_of_every_plane(n, topdown_limit):
    """A path from its end, its middle and the other end: levels up to n - 1."""
    require_cuda()
    check(inputs.path(n), [0, n // 2, n - 1], topdown_limit)
