"""Batched pull over a directed graph's long in-rows whose out-rows are short.

A chunk list has room for the chunks of all rows longer than 1,024 entries.  A
vertex that a pull reaches through a long in-row gets chunk items only if its
own out-row is long: an item for each of them regardless (which the short rows
are also expanded without) would need more room than that on this graph, in
one level.  Checked against the oracle, in the normal and in the
bounds-checking build.
"""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import paper_1104_4518_gb300 as bfs
from gpu_helpers import assert_same, require_cuda
from paper_1104_4518_gb300 import inputs

pytestmark = pytest.mark.gpu

CHUNK = 1024
M = 8000  # vertices A (long in-row, one out-arc) and as many B (out-row of 1,025 arcs to vertices A)


def graph():
    """Two roots point at every A and B, so that one pull level reaches them all."""
    a, b = np.arange(M), M + np.arange(M)
    roots, sink = np.array([2 * M, 2 * M + 1]), 2 * M + 2
    src = [np.repeat(b, CHUNK + 1), np.repeat(roots, 2 * M), a]
    dst = [((np.arange(M)[:, None] + np.arange(CHUNK + 1)) % M).ravel(), np.tile(np.arange(2 * M), 2), np.full(M, sink)]
    n = 2 * M + 3
    return inputs.EdgeList(n, np.concatenate(src), np.concatenate(dst), "long-in-rows"), roots


def test_items_regardless_of_the_out_row_would_not_fit():
    el, _ = graph()
    out = np.bincount(el.src, minlength=el.n)
    into = np.bincount(el.dst, minlength=el.n)
    cap = 2 * (el.src.size // CHUNK) + 4096 + 1024  # entries of a workspace's chunk list
    chunks = -(-out // CHUNK)
    reached = np.arange(el.n) < 2 * M
    assert chunks[reached & ((into > CHUNK) | (out > CHUNK))].sum() > cap
    assert chunks[out > CHUNK].sum() <= cap


@pytest.mark.parametrize("k", [2, 17, 64])
def test_batched_pull_of_long_in_rows(k):
    require_cuda()
    el, roots = graph()
    og = oracle.digraph_of(el)
    g = bfs.bfs_graph_create_from_edges(torch.from_numpy(el.src).cuda(), torch.from_numpy(el.dst).cuda(), el.n, directed=True)
    sources = [int(roots[i % 2]) for i in range(k)]
    refs = {s: oracle.bfs_directed(og, s) for s in set(sources)}
    for limit in (1, 0):  # pull from the first level on; the default
        bfs.bfs_set_tuning(g, batch_topdown_limit=limit)
        parent, level = bfs.run_batch(g, sources)
        bfs.bfs_sync(g)
        pa, lv = parent.cpu().numpy(), level.cpu().numpy()
        for i, s in enumerate(sources):
            assert_same(refs[s], (lv[i], pa[i]), f"root {s}, row {i}, limit {limit}")
    g.destroy()


def test_the_same_in_the_bounds_checking_build():
    from paper_1104_4518_gb300 import build as b
    b.build_checked()
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", __file__, "-k", "test_batched_pull_of_long_in_rows"],
                       env=dict(os.environ, BFS_BOUNDS_CHECK="1"), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:]
