"""Ragged traversals of parts whose borders fall anywhere among a warp's vertices.

The outputs are dealt to the parts in one pass over the union: single-vertex
parts, parts around a warp's 32 vertices, many small ones beside a large one.
Every part's levels and parents equal the oracle's, in each part's own array."""
import pytest
import torch

import oracle
import paper_1104_4518_gb300 as bfs
from gpu_helpers import assert_same, device_graph_from_edges, require_cuda
from paper_1104_4518_gb300 import inputs

pytestmark = pytest.mark.gpu

PARTS = {"one": [1], "singles": [1] * 70, "warp edges": [31, 32, 33, 1, 63, 64, 65, 2],
         "small beside large": [3, 200_000, 1, 1, 700_000, 5] + [2] * 300}


@pytest.mark.parametrize("name", PARTS)
def test_parts_of_every_size(name):
    require_cuda()
    graphs = [inputs.path(n) for n in PARTS[name]]
    for i in [i for i, n in enumerate(PARTS[name]) if n >= 1000]:
        n = PARTS[name][i]
        graphs[i] = inputs.erdos_renyi(n, 4, seed=800 + i)
    sources = [(7 * i) % n for i, n in enumerate(PARTS[name])]
    parts = [device_graph_from_edges(el) for el in graphs]
    u = bfs.bfs_graph_union(parts)
    levels = [torch.full((el.n + 2,), -7, dtype=torch.int32, device="cuda") for el in graphs]
    parents = [torch.full((el.n + 2,), -7, dtype=torch.int32, device="cuda") for el in graphs]
    bfs.bfs_run_ragged(u, sources, [t[1:-1] for t in parents], [t[1:-1] for t in levels])
    bfs.bfs_sync(u)
    for i, (el, s) in enumerate(zip(graphs, sources)):
        lv, pa = levels[i].cpu().numpy(), parents[i].cpu().numpy()
        assert_same(oracle.bfs(oracle.csr_of(el), s), (lv[1:-1], pa[1:-1]), f"{name} part {i}")
        assert lv[0] == lv[-1] == pa[0] == pa[-1] == -7  # nothing beside the part's array
    u.destroy()
    for g in parts:
        g.destroy()
