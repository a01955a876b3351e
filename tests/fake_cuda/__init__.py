"""The library's objects linked to the stand-in CUDA runtime of fake_cudart.cpp."""
import ctypes
import os
import shutil
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
_linked = None


def _link():
    global _linked
    if _linked is None:
        from paper_1104_4518_gb300 import build as b
        b.build()
        objs = [os.path.join(b.BUILD_DIR, os.path.basename(s)[:-3] + ".o") for s in b.sources()]
        include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b.nvcc()))), "include")
        _linked = os.path.join(tempfile.mkdtemp(prefix="fake_cuda"), "libbfs_fake.so")
        r = subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", include,
                            os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", _linked, "-ldl", "-lpthread"],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    return _linked


class Entry:
    def __init__(self, what, ptr, nbytes, stream):
        self.what, self.ptr, self.bytes, self.stream = what, ptr, nbytes, stream

    def __repr__(self):
        return f"{self.what}(ptr={self.ptr:#x}, bytes={self.bytes}, stream={self.stream:#x})"


class FakeLibrary:
    """A fresh copy of the library (its own cache and other static state) on the stand-in."""

    def __init__(self):
        path = os.path.join(tempfile.mkdtemp(prefix="fake_cuda"), "libbfs_fake.so")
        shutil.copy(_link(), path)
        self.c = ctypes.CDLL(path)
        self.c.fake_log_entry.restype = ctypes.c_char_p
        self.c.fake_live_bytes.restype = ctypes.c_size_t
        self.c.bfs_last_error.restype = ctypes.c_char_p

    def log(self):
        out = []
        for i in range(self.c.fake_log_size()):
            p, n, s = ctypes.c_void_p(), ctypes.c_size_t(), ctypes.c_void_p()
            what = self.c.fake_log_entry(i, ctypes.byref(p), ctypes.byref(n), ctypes.byref(s))
            out.append(Entry(what.decode(), p.value or 0, n.value, s.value or 0))
        return out

    def taken(self, call):
        """The log of what `call` did."""
        self.c.fake_log_clear()
        call()
        return self.log()

    def graph(self, n=100, flags=0x1):
        """A path 0 - 1 - ... - (n - 1) from host arrays."""
        off = [0] + [1 + 2 * i for i in range(n - 1)] + [2 * (n - 1)]
        adj = [x for i in range(n) for x in (i - 1, i + 1) if 0 <= x < n]
        g = ctypes.c_void_p()
        rc = self.c.bfs_graph_create((ctypes.c_int64 * len(off))(*off), (ctypes.c_int32 * max(1, len(adj)))(*adj), n,
                                     ctypes.c_int64(len(adj)), flags, ctypes.byref(g))
        assert rc == 0, self.c.bfs_last_error()
        return g

    def run(self, g, n, stream=0, opts=None):
        out = (ctypes.c_int32 * (2 * n))()
        base = ctypes.addressof(out)
        return self.c.bfs_run(g, 0, ctypes.c_void_p(base), ctypes.c_void_p(base + 4 * n), opts, ctypes.c_void_p(stream))
