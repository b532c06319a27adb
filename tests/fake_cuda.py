"""The library's host side on a stand-in CUDA runtime (fake_cuda.cpp): builds and loads it, and
calls it through the C ABI with numpy buffers."""
import ctypes
import os
import subprocess

import numpy as np

from paper_2603_05381_gb300 import _capi, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
P = ctypes.c_void_p


def build_fake(out_dir):
    """Links capi.cu's and host_graph.cpp's objects with the stand-ins into a library of its own."""
    build.build()
    so = os.path.join(str(out_dir), "libbp4m_fake.so")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-pthread", "-Wl,-Bsymbolic", "-I", cuda, "-I", build.CSRC,
                    "-I", build.INCLUDE, os.path.join(ROOT, "tests", "fake_cuda.cpp"), os.path.join(build.BUILD, "capi.cu.o"),
                    os.path.join(build.BUILD, "host_graph.cpp.o"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for name, (res, args) in _capi.SIGNATURES.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    lib.fake_enqueue_write.argtypes = [P, P, P, ctypes.c_size_t]
    return lib


class Fake:
    def __init__(self, lib):
        self.lib = lib
        self._graphs = {}

    def graph(self, d=13, model=_capi.CIRCUIT, p=0.005):
        """A graph, kept for the life of the library (building one takes a second)."""
        key = (d, model, p)
        if key not in self._graphs:
            self._graphs[key] = self.new_graph(d, model, p)
        return self._graphs[key]

    def new_graph(self, d=5, model=_capi.CIRCUIT, p=0.005):
        h = P()
        assert self.lib.bp4m_build_graph(ctypes.byref(_capi.Code(0, d, 0, 0)), ctypes.byref(_capi.Noise(model, p, 0, 0)), ctypes.byref(h)) == 0
        return h

    def words(self, g, type=0):
        info = _capi.GraphInfo()
        assert self.lib.bp4m_graph_info(g, ctypes.byref(info)) == 0
        return info.n_words[type], info.n_det[type]

    def stream(self, nonblocking=True, prio=0):
        s = P()
        assert self.lib.cudaStreamCreateWithPriority(ctypes.byref(s), 1 if nonblocking else 0, prio) == 0
        return s

    def buffer(self, n, dtype, where):
        """n elements of host ("pageable"), pinned or "device" memory as a numpy array."""
        if where == "pageable":
            return np.zeros(n, dtype=dtype)
        p = P()
        fn = self.lib.cudaMallocHost if where == "pinned" else self.lib.cudaMalloc
        nb = max(n * np.dtype(dtype).itemsize, 1)
        assert fn(ctypes.byref(p), ctypes.c_size_t(nb)) == 0
        a = np.frombuffer((ctypes.c_char * nb).from_address(p.value), dtype=dtype, count=n)
        a[:] = 0
        return a

    def syndromes(self, g, sizes, seed, type=0):
        """Rows of the given defect counts."""
        nw, nd = self.words(g, type)
        rng = np.random.default_rng(seed)
        bits = np.zeros((len(sizes), nw * 32), dtype=np.uint8)
        for r, s in enumerate(sizes):
            bits[r, rng.choice(nd, size=s, replace=False)] = 1
        return np.packbits(bits, axis=1, bitorder="little").view(np.uint32)

    @staticmethod
    def expected(synd):
        """(obs, converged, iterations) that the stand-in kernels give."""
        h = np.zeros(synd.shape[0], dtype=np.uint64)
        for k in range(synd.shape[1]):
            h = ((h ^ synd[:, k]) * np.uint64(2654435761)) & np.uint64(0xFFFFFFFF)
        s = np.unpackbits(synd.view(np.uint8), axis=1).sum(axis=1).astype(np.int16)
        return (np.where(s > 0, h >> np.uint64(31), 0).astype(np.uint8), ((s % 5 != 0) | (s == 0)).astype(np.uint8), s)

    def decode(self, g, synd, out, stream=None, iters=5, opts=None):
        opts = opts or _capi.Opts(_capi.FP32, 1, 0, 1.0, 0, 0, 0, 0)
        return self.lib.bp4m_decode_batch(g, synd.ctypes.data, synd.shape[0], iters, ctypes.byref(opts),
                                          *[None if o is None else o.ctypes.data for o in out], stream)

    def launches(self):
        n = self.lib.fake_launches(None, 0)
        buf = (ctypes.c_int * (4 * max(n, 1)))()
        self.lib.fake_launches(buf, n)
        return np.array(buf, dtype=np.int64)[:4 * n].reshape(n, 4)


CLASSIFY, LIST, GLOBAL, PARTITION, OTHER = range(5)
