"""Traversals in a captured CUDA graph (relaxed mode: the first run on a stream
allocates), with the first run on the stream inside the capture: the graph's
replays and eager runs on the same stream, before and after them, are all right."""
import numpy as np
import pytest
import torch

import oracle
import paper_1104_4518_gb300 as bfs
from gpu_helpers import device_graph_from_edges, require_cuda
from paper_1104_4518_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("selector", [bfs.BFS_SELECT_HEURISTIC, bfs.BFS_SELECT_LEARNED])
def test_first_run_on_a_stream_is_captured(selector):
    require_cuda()
    el = inputs.rmat(14, 16, seed=91)
    og = oracle.csr_of(el)
    roots = [int(r) for r in inputs.roots(el, 2, 92)]
    refs = oracle.bfs_many(og, roots)
    g = device_graph_from_edges(el)
    if selector == bfs.BFS_SELECT_LEARNED:
        bfs.bfs_selector_set_params(np.random.default_rng(7).normal(size=bfs.BFS_MLP_PARAMS).astype(np.float32) * 0.2)
    parent = torch.empty(g.n, dtype=torch.int32, device="cuda")
    level = torch.empty_like(parent)
    opts = bfs.RunOptions(selector=selector)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def check(ref):
        bfs.bfs_sync(g, stream)
        torch.cuda.synchronize()
        assert np.array_equal(level.cpu().numpy(), ref[0]) and np.array_equal(parent.cpu().numpy(), ref[1])

    try:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
            bfs.bfs_run(g, roots[0], parent, level, opts)
        for _ in range(2):
            with torch.cuda.stream(stream):
                bfs.bfs_run(g, roots[1], parent, level, opts)
            check(refs[1])
            parent.fill_(7)
            level.fill_(7)
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                graph.replay()
            check(refs[0])
    finally:
        bfs.bfs_selector_set_params(None)
        torch.cuda.synchronize()
        g.destroy()
