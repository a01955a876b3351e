"""Construction after cudaDeviceReset, in a child process: the memory that the
library held unused went with the old context, so nothing of it may be handed
out.  (The child goes on only once it has seen that the new context's identity
differs from the old one's.)"""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, sys
import numpy as np
from paper_1104_4518_gb300 import build
lib = ctypes.CDLL(build.LIB)
lib.bfs_last_error.restype = ctypes.c_char_p
cuda = ctypes.CDLL("libcuda.so.1")
rt = ctypes.CDLL(sys.argv[1])

def context():
    i = ctypes.c_ulonglong(0)
    assert cuda.cuCtxGetId(None, ctypes.byref(i)) == 0
    return i.value

def construct(n, seed):
    rng = np.random.default_rng(seed)
    src, dst = (rng.integers(0, n, 8 * n, dtype=np.int32) for _ in range(2))
    g = ctypes.c_void_p()
    rc = lib.bfs_graph_create_from_edges(src.ctypes.data_as(ctypes.c_void_p), dst.ctypes.data_as(ctypes.c_void_p),
                                         ctypes.c_int64(src.size), n, 1, None, ctypes.byref(g))
    assert rc == 0, lib.bfs_last_error()
    nnz = ctypes.c_int64()
    lib.bfs_graph_info(g, None, ctypes.byref(nnz), None)
    off, adj = np.empty(n + 1, np.int64), np.empty(nnz.value, np.int32)
    assert lib.bfs_graph_copy_csr(g, off.ctypes.data_as(ctypes.c_void_p), adj.ctypes.data_as(ctypes.c_void_p), 1) == 0
    lib.bfs_graph_destroy(g)
    keep = src != dst
    keys = np.unique(np.concatenate([src[keep].astype(np.int64) * n + dst[keep], dst[keep].astype(np.int64) * n + src[keep]]))
    assert np.array_equal(off, np.searchsorted(keys, np.arange(n + 1) * n)) and np.array_equal(adj, keys % n)

construct(50000, 1)
construct(50000, 2)
before = context()
assert rt.cudaDeviceReset() == 0
assert rt.cudaFree(None) == 0  # the new context
after = context()
print("contexts", before, after, flush=True)
assert after != before
construct(50000, 3)
construct(50000, 4)
assert lib.bfs_memory_trim() == 0
print("done")
"""


def test_construction_after_a_device_reset():
    import torch  # (finds the runtime library; the child does without)
    assert torch.cuda.is_available()
    runtime = next(line.split()[-1] for line in open("/proc/self/maps") if "libcudart.so" in line)
    r = subprocess.run([sys.executable, "-c", CHILD, runtime], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr[-3000:]
