"""What a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public entry points of paper_1104_4518_gb300.  Five
kinds of work, each over the sizes that the repository's own configurations,
tests and benchmark use:

  run     traversals from single roots, one after another (bfs_run): R-MAT
          scales 12 to 26, Erdos-Renyi graphs and 3D grids; undirected or
          directed; the threshold heuristic or the learned variant selector
  batch   1 to 64 roots in one traversal (bfs_run_batch)
  ragged  one traversal of each part of a union of small graphs (bfs_run_ragged)
  build   edge list -> graph -> its CSR (bfs_graph_create_from_edges,
          bfs_graph_copy_csr)
  grad    loss and gradient of the selector network over a training set
          (bfs_mlp_loss_grad), the backward half of training it

Graphs are drawn on the GPU from the seed alone, with the distributions of
paper_1104_4518_gb300/inputs: R-MAT with (A, B, C) = (0.57, 0.19, 0.19),
self-loops and repeats left in and the vertices relabelled at random, uniform
pairs, and the 7-point grid in row-major order.  Roots are uniform over the
vertices of degree >= 1 (a grid's root lies near one of its corners).
"""
import os

import torch

import paper_1104_4518_gb300 as bfs

RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(bfs.__file__)), "selector_weights.bin")


def listed():
    return [
        # the smallest call: one root of a graph whose whole state sits in L2
        {"name": "run_rmat16", "kind": "run", "graph": "rmat", "scale": 16, "ef": 16, "directed": False,
         "selector": "heuristic", "roots": 1},
        # ordinary traversals of a mid-size social-network-like graph, several roots in a row
        {"name": "run_rmat22", "kind": "run", "graph": "rmat", "scale": 22, "ef": 16, "directed": False,
         "selector": "heuristic", "roots": 4},
        # the benchmark's graph: 8.4 GB of adjacency
        {"name": "run_rmat26", "kind": "run", "graph": "rmat", "scale": 26, "ef": 16, "directed": False,
         "selector": "heuristic", "roots": 4},
        # high diameter: 382 narrow levels, a road-network- or mesh-like graph
        {"name": "run_grid128", "kind": "run", "graph": "grid", "n": 128, "directed": False,
         "selector": "heuristic", "roots": 1},
        # no hubs, a vertex count that is no power of two, the learned selector
        {"name": "run_er_learned", "kind": "run", "graph": "er", "n": 1000003, "degree": 9, "directed": False,
         "selector": "learned", "roots": 2},
        # arcs followed one way (a web crawl, a follower graph)
        {"name": "run_rmat20_directed", "kind": "run", "graph": "rmat", "scale": 20, "ef": 16, "directed": True,
         "selector": "heuristic", "roots": 4},
        # the batched configuration: 64 roots at once (all-pairs samples, centrality estimates)
        {"name": "batch_rmat24", "kind": "batch", "graph": "rmat", "scale": 24, "ef": 16, "directed": False,
         "k": 64},
        # a few roots, not a power of two, of a smaller and sparser graph
        {"name": "batch_rmat19_k17", "kind": "batch", "graph": "rmat", "scale": 19, "ef": 8, "directed": False,
         "k": 17},
        # 32 independent graphs of scales 12 to 20 in one launch
        {"name": "ragged32", "kind": "ragged", "parts": 32, "lo": 12, "hi": 20, "ef": 16},
        # graph construction, small and at the size of the mid-size traversals (67 M edges)
        {"name": "build_rmat16", "kind": "build", "graph": "rmat", "scale": 16, "ef": 16, "directed": False},
        {"name": "build_rmat22", "kind": "build", "graph": "rmat", "scale": 22, "ef": 16, "directed": False},
        # one full-batch gradient of the selector network, at its training set's size
        {"name": "selector_grad", "kind": "grad", "rows": 1379},
    ]


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "batch", "ragged", "build", "grad"])
    if kind == "grad":
        return {"kind": "grad", "rows": int(2 ** rng.uniform(5, 14)) + rng.randrange(2)}
    if kind == "ragged":
        lo = rng.randrange(12, 17)
        return {"kind": "ragged", "parts": rng.randrange(3, 33), "lo": lo, "hi": rng.randrange(lo, 21),
                "ef": rng.choice([8, 16])}
    graph = rng.choice(["rmat", "rmat", "er", "grid"]) if kind == "run" else rng.choice(["rmat", "rmat", "er"])
    c = {"kind": kind, "graph": graph, "directed": graph != "grid" and rng.random() < 0.25}
    if graph == "rmat":
        top = {"run": 25, "batch": 23, "build": 21}[kind]
        c["scale"] = rng.randrange(12, top + 1)
        c["ef"] = rng.choice([8, 16, 32]) if c["scale"] < top else rng.choice([4, 8, 16])
    elif graph == "er":
        c["n"] = int(2 ** rng.uniform(12, 22)) | 1
        c["degree"] = rng.randrange(4, 33)
    else:
        c["n"] = rng.randrange(20, 129)
    if kind == "run":
        c["selector"] = rng.choice(["heuristic", "heuristic", "learned"])
        c["roots"] = rng.randrange(1, 5) if graph != "grid" else 1
    elif kind == "batch":
        c["k"] = min(64, int(2 ** rng.uniform(0, 6.2)))
    return c


# ---------------- graphs ----------------

def _vertices(case):
    return {"rmat": lambda: 1 << case["scale"], "er": lambda: case["n"], "grid": lambda: case["n"] ** 3}[case["graph"]]()


def _edges(case):
    return {"rmat": lambda: case["ef"] << case["scale"], "er": lambda: case["n"] * case["degree"] // 2,
            "grid": lambda: 3 * case["n"] ** 2 * (case["n"] - 1)}[case["graph"]]()


def _scales(case):
    """The scales of a ragged batch's parts: lo to hi in turn, in no sorted order."""
    spread = case["hi"] - case["lo"] + 1
    return [case["lo"] + (5 * i + i // spread) % spread for i in range(case["parts"])]


def _rmat(scale, ef, gen):
    n, m = 1 << scale, ef << scale
    src = torch.empty(m, dtype=torch.int32, device="cuda")
    dst = torch.empty(m, dtype=torch.int32, device="cuda")
    perm = torch.randperm(n, generator=gen, device="cuda", dtype=torch.int32)
    step = 1 << 26
    for lo in range(0, m, step):
        c = min(step, m - lo)
        s = torch.zeros(c, dtype=torch.int32, device="cuda")
        d = torch.zeros(c, dtype=torch.int32, device="cuda")
        r = torch.empty(c, dtype=torch.float32, device="cuda")
        for _ in range(scale):  # one bit of both ends per step: the quadrant of the matrix
            r.uniform_(generator=gen)
            low = r >= RMAT_A + RMAT_B
            right = ((r >= RMAT_A) ^ low) | (r >= RMAT_A + RMAT_B + RMAT_C)
            s.mul_(2).add_(low)
            d.mul_(2).add_(right)
        src[lo:lo + c] = perm.index_select(0, s)
        dst[lo:lo + c] = perm.index_select(0, d)
    return src, dst


def _grid(n):
    ids = torch.arange(n ** 3, dtype=torch.int32, device="cuda").view(n, n, n)
    pairs = [(ids[:-1], ids[1:]), (ids[:, :-1], ids[:, 1:]), (ids[:, :, :-1], ids[:, :, 1:])]
    return (torch.cat([a.reshape(-1) for a, _ in pairs]).contiguous(),
            torch.cat([b.reshape(-1) for _, b in pairs]).contiguous())


def _edge_list(case, gen):
    if case["graph"] == "rmat":
        return _rmat(case["scale"], case["ef"], gen)
    if case["graph"] == "er":
        m = _edges(case)
        return tuple(torch.randint(0, case["n"], (m,), generator=gen, device="cuda", dtype=torch.int32)
                     for _ in range(2))
    return _grid(case["n"])


def _graph(case, gen):
    src, dst = _edge_list(case, gen)
    return bfs.bfs_graph_create_from_edges(src, dst, _vertices(case), directed=case["directed"])


def _roots(g, k, gen):
    """k vertices of degree >= 1, uniform (repeats possible, as in a user's sample)."""
    off, _ = bfs.bfs_graph_copy_csr(g)
    cand = torch.randint(0, g.n, (4096,), generator=gen, device="cuda")
    good = cand[off[cand + 1] > off[cand]].tolist()
    while len(good) < k:
        good.append(good[0] if good else 0)
    return good[:k]


def _corner(n, gen):
    """A grid vertex within n / 16 of a corner: nearly the longest traversal."""
    at = torch.randint(0, max(1, n // 16), (3,), generator=gen, device="cuda")
    far = torch.randint(0, 2, (3,), generator=gen, device="cuda")
    x, y, z = torch.where(far == 1, n - 1 - at, at).tolist()
    return x + n * (y + n * z)


def _ints(*shape):
    return torch.empty(shape, dtype=torch.int32, device="cuda")


# ---------------- the interface ----------------

def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "grad":
        b = case["rows"]
        w = torch.randn(bfs.BFS_MLP_PARAMS, generator=gen, device="cuda")
        w[:832] *= (2.0 / 12) ** 0.5   # W1, b1 of 12 -> 64
        w[832:4992] *= (2.0 / 64) ** 0.5  # W2, b2 of 64 -> 64
        w[4992:] *= (2.0 / 64) ** 0.5  # W3, b3 of 64 -> 4
        st["params"] = w
        st["x"] = torch.rand((b, bfs.BFS_MLP_IN), generator=gen, device="cuda")   # level features lie in [0, 1]
        st["t"] = torch.randn((b, bfs.BFS_MLP_OUT), generator=gen, device="cuda") * 2 + 4  # log2 of times in us
        st["grad"] = torch.empty(bfs.BFS_MLP_PARAMS, device="cuda")
        st["loss"] = torch.empty(1, device="cuda")
        return st
    if kind == "ragged":
        parts = []
        st["sources"], st["parents"], st["levels"] = [], [], []
        for scale in _scales(case):
            part = {"graph": "rmat", "scale": scale, "ef": case["ef"], "directed": False}
            g = _graph(part, gen)
            st["sources"].append(_roots(g, 1, gen)[0])
            st["parents"].append(_ints(g.n))
            st["levels"].append(_ints(g.n))
            parts.append(g)
        st["graph"] = bfs.bfs_graph_union(parts)
        for g in parts:
            g.destroy()
        return st
    if kind == "build":
        st["src"], st["dst"] = _edge_list(case, gen)
        st["n"], st["directed"] = _vertices(case), case["directed"]
        st["offsets"] = torch.empty(st["n"] + 1, dtype=torch.int64, device="cuda")
        # room for every arc; the rows of a graph with repeats or loops end earlier
        st["adj"] = torch.full((_edges(case) * (1 if case["directed"] else 2),), -1, dtype=torch.int32, device="cuda")
        return st
    g = st["graph"] = _graph(case, gen)
    k = case["k"] if kind == "batch" else case["roots"]
    st["sources"] = [_corner(case["n"], gen)] * k if case["graph"] == "grid" else _roots(g, k, gen)
    st["parent"], st["level"] = _ints(k, g.n), _ints(k, g.n)
    if kind == "run":
        st["opts"] = None
        if case["selector"] == "learned":
            bfs.bfs_selector_load(WEIGHTS)
            st["opts"] = bfs.RunOptions(selector=bfs.BFS_SELECT_LEARNED)
    return st


def run(st):
    kind = st["kind"]
    if kind == "run":
        for i, s in enumerate(st["sources"]):
            bfs.bfs_run(st["graph"], s, st["parent"][i], st["level"][i], st["opts"])
        return st["parent"], st["level"]
    if kind == "batch":
        bfs.bfs_run_batch(st["graph"], st["sources"], st["parent"], st["level"])
        return st["parent"], st["level"]
    if kind == "ragged":
        bfs.bfs_run_ragged(st["graph"], st["sources"], st["parents"], st["levels"])
        return st["parents"] + st["levels"]
    if kind == "build":
        g = bfs.bfs_graph_create_from_edges(st["src"], st["dst"], st["n"], directed=st["directed"])
        bfs.lib().bfs_graph_copy_csr(g.handle, st["offsets"].data_ptr(), st["adj"].data_ptr(), 0)
        g.destroy()
        return st["offsets"], st["adj"]
    bfs.bfs_mlp_loss_grad(st["params"], st["x"], st["t"], st["grad"], st["loss"])
    return st["grad"], st["loss"]


def work(case):
    """Each input read once, each output written once (repeats in the edge list not deducted)."""
    if case["kind"] == "grad":
        b, p = case["rows"], bfs.BFS_MLP_PARAMS
        return {"bytes": 4 * (2 * p + b * (bfs.BFS_MLP_IN + bfs.BFS_MLP_OUT) + 1),
                "flops": 2 * b * (3 * (64 * 64 + 64 * 4) + 2 * 12 * 64)}
    if case["kind"] == "ragged":
        n = sum(1 << s for s in _scales(case))
        return {"bytes": 8 * n + 4 * 2 * case["ef"] * n + 8 * n, "flops": 0}
    n, m = _vertices(case), _edges(case)
    arcs = m if case["directed"] else 2 * m
    if case["kind"] == "build":  # the edge list in, the rows out
        return {"bytes": 8 * m + 8 * (n + 1) + 4 * arcs, "flops": 0}
    if case["kind"] == "batch":  # the rows once, a level and a parent per root and vertex
        return {"bytes": 8 * (n + 1) + 4 * arcs + 8 * n * case["k"], "flops": 0}
    return {"bytes": case["roots"] * (8 * (n + 1) + 4 * arcs + 8 * n), "flops": 0}


def exact(case, seed):
    """Loss and gradient in float64; traversals and rows are whole numbers, which have to be equal."""
    if case["kind"] != "grad":
        return None
    st = prepare(case, seed)
    p, x, t = st["params"].double(), st["x"].double(), st["t"].double()
    w1, b1 = p[:768].view(12, 64), p[768:832]
    w2, b2 = p[832:4928].view(64, 64), p[4928:4992]
    w3, b3 = p[4992:5248].view(64, 4), p[5248:]
    z1 = x @ w1 + b1
    h1 = z1.clamp(min=0)
    z2 = h1 @ w2 + b2
    h2 = z2.clamp(min=0)
    diff = h2 @ w3 + b3 - t
    dy = 2 * diff / diff.numel()
    dz2 = (dy @ w3.T) * (z2 > 0)
    dz1 = (dz2 @ w2.T) * (z1 > 0)
    grads = [x.T @ dz1, dz1.sum(0), h1.T @ dz2, dz2.sum(0), h2.T @ dy, dy.sum(0)]
    return torch.cat([g.reshape(-1) for g in grads]), (diff * diff).mean().reshape(1)
