"""The tables that a graph's creation makes of its rows, from a CSR whose offsets
leave the adjacency: without BFS_VALIDATE it is accepted, as before there were
probe records, and no entry that is not there is read; with it the CSR is
refused.  (Nothing traverses the graph: that may read out of bounds.)"""
import pytest
import torch

import paper_1104_4518_gb300 as bfs
from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offsets", [[0, 1, 2, 900], [-700, 1, 2, 4], [0, 800, 802, 4], [-900, -700, 2, 4]])
def test_rows_outside_the_adjacency(offsets):
    require_cuda()
    if bfs.lib().bfs_bounds_checked():
        pytest.skip("the bounds-checking build refuses such offsets")
    off = torch.tensor(offsets, dtype=torch.int64, device="cuda")
    adj = torch.tensor([1, 0, 2, 1], dtype=torch.int32, device="cuda")
    g = bfs.bfs_graph_create(off, adj)
    assert g.n == 3
    g.destroy()
    with pytest.raises(bfs.BfsError):
        bfs.bfs_graph_create(off, adj, validate=True)
