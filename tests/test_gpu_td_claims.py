"""Claims of the thread and warp variants around the ends of a CTA's buffers.

A two-level tree: one row per warp of the grid in level 1, whose children make
each CTA claim just under, exactly and just over what its buffer holds,
what the long buffer of these variants holds, and more."""
import numpy as np
import pytest
import torch

import paper_1104_4518_gb300 as bfs
from gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

WARPS = 16                # rows that a CTA of 512 threads expands
BUFFER = 4352             # entries of its own buffer
LONG = 15040              # entries with the phases' area behind it


def edges(ends):
    return sorted({e // WARPS + d for e in ends for d in (-1, 0, 1)}) + [1000]


def want_parent_of(inner, of):
    return torch.cat([torch.zeros_like(inner[:1]), torch.zeros_like(inner), of])


def level_of(inner, of):
    return torch.cat([torch.zeros_like(inner[:1]), torch.ones_like(inner), torch.full_like(of, 2)])


def check(g, want_parent, want_level):
    for variant in (bfs.BFS_VARIANT_TD_THREAD, bfs.BFS_VARIANT_TD_WARP, bfs.BFS_VARIANT_TD_BINNED):
        opts = bfs.RunOptions(selector=bfs.BFS_SELECT_FORCED, forced_variant=variant, want_counts=True)
        parent, level = bfs.run(g, 0, opts)
        bfs.bfs_sync(g)
        name = bfs.VARIANT_NAMES[variant]
        assert torch.equal(level, want_level), name
        assert torch.equal(parent, want_parent), name
        assert opts.edges == int((want_level > 0).sum()) and opts.nlevels == 3, name
    g.destroy()


@pytest.mark.parametrize("children", edges((BUFFER, LONG)))
@pytest.mark.parametrize("large", [False, True])
def test_claims_at_the_ends_of_the_buffers(children, large):
    """large: with isolated vertices up to a size whose forced runs have the long buffer."""
    require_cuda()
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    rows = WARPS * ctas
    n = 1 + rows + rows * children
    inner = torch.arange(1, rows + 1, dtype=torch.int32, device="cuda")
    leaves = torch.arange(rows + 1, n, dtype=torch.int32, device="cuda")
    of = inner.repeat_interleave(children)
    more = max(0, 3000000 - n) if large else 0
    g = bfs.bfs_graph_create_from_edges(torch.cat([torch.zeros_like(inner), of]), torch.cat([inner, leaves]), n + more)
    none = torch.full((more,), -1, dtype=torch.int32, device="cuda")
    check(g, torch.cat([want_parent_of(inner, of), none]), torch.cat([level_of(inner, of), none]))


def test_chunked_rows_beside_overflowing_ones():
    """Rows split into chunks in the same level: the CTA's warps claim from chunk items and from rows at once."""
    require_cuda()
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    rows, hubs = 2 * WARPS * ctas, ctas
    children = torch.full((rows,), 700, dtype=torch.int64, device="cuda")
    children[::rows // hubs] = 1025 + 64
    inner = torch.arange(1, rows + 1, dtype=torch.int32, device="cuda")
    of = inner.repeat_interleave(children)
    n = 1 + rows + of.numel()
    leaves = torch.arange(rows + 1, n, dtype=torch.int32, device="cuda")
    g = bfs.bfs_graph_create_from_edges(torch.cat([torch.zeros_like(inner), of]), torch.cat([inner, leaves]), n)
    check(g, want_parent_of(inner, of), level_of(inner, of))


def test_edges_cover_what_they_should():
    assert {d * WARPS for d in edges((BUFFER, LONG))} >= {BUFFER, BUFFER + 16, LONG - 16,
                                                                        LONG, LONG + 16, 16000}
    assert np.all(np.array(edges((BUFFER, LONG))) <= 1024)  # no row is split into chunks
