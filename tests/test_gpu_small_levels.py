"""Top-down levels whose edges are dealt flat over the grid, at the edges of the rule.

A root joins K children and child i joins L_i leaves that the children share, so
that level 1 has K frontier vertices: below, at and above the 2,048 that a flat
level may have, with empty, single-entry and chunk-length rows, and with 16 edges
per thread of the grid, one fewer and one more.  Levels and parents equal the
oracle's for the variant forced and for the heuristic."""
import numpy as np
import pytest
import torch

import oracle
import paper_1104_4518_gb300 as bfs
from gpu_helpers import assert_same, device_graph_from_edges, require_cuda
from paper_1104_4518_gb300 import inputs

pytestmark = pytest.mark.gpu

POOL = 60_000
LENGTHS = {"empty": lambda k: np.zeros(k), "single": lambda k: np.ones(k),
           "mixed": lambda k: np.resize([0, 1, 31, 32, 33, 255, 256, 257, 1023, 1024, 1025, 3000], k)}


def children(k, lens, seed):
    rng = np.random.default_rng(seed)
    lens = np.asarray(lens, np.int64)
    start = np.repeat(rng.integers(0, POOL, k), lens)
    at = np.arange(lens.sum()) - np.repeat(np.cumsum(lens) - lens, lens)
    # ids of the children in the middle, so that parents are not simply the last child
    base, leaf = POOL // 2, (start + at) % POOL
    leaf = np.where(leaf < base, leaf, leaf + k)
    kids = base + np.arange(k)
    root = POOL + k
    src = np.concatenate([np.full(k, root), np.repeat(kids, lens)]).astype(np.int32)
    dst = np.concatenate([kids, leaf]).astype(np.int32)
    return inputs.EdgeList(POOL + k + 1, src, dst, f"children-{k}"), root


def check(el, root):
    g = device_graph_from_edges(el)
    want = oracle.bfs(oracle.csr_of(el), root)
    for o in (bfs.RunOptions(), bfs.RunOptions(selector=bfs.BFS_SELECT_FORCED, forced_variant=bfs.BFS_VARIANT_TD_BINNED)):
        parent, level = bfs.run(g, root, o)
        bfs.bfs_sync(g)
        assert_same(want, (level.cpu().numpy(), parent.cpu().numpy()), el.name)
    g.destroy()


@pytest.mark.parametrize("lengths", LENGTHS)
@pytest.mark.parametrize("k", [1, 2, 511, 512, 513, 2047, 2048, 2049, 5000])
def test_frontiers_around_the_flat_limit(k, lengths):
    require_cuda()
    check(*children(k, LENGTHS[lengths](k), k))


@pytest.mark.parametrize("more", [-1, 0, 1])
def test_edges_around_the_flat_limit(more):
    require_cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edges = 16 * 2 * sms * 512 + more  # of the frontier, the arcs back to the root included
    lens = np.full(2048, edges // 2048 - 1)
    lens[: edges - 2048 * (edges // 2048)] += 1
    check(*children(2048, lens, 7))
