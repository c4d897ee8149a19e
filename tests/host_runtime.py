"""libmw's host code without a GPU: its objects linked with tests/fake_cudart.cpp, which
records the launches and grants shared memory by device.  Operands are addresses that
nothing reads."""
import ctypes
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PACKAGE = os.path.join(ROOT, "paper_2606_20863_gb300")


class HostLibrary:
    def __init__(self, mw, path):
        self.mw = mw
        self.lib = ctypes.CDLL(path)
        for name in mw.EXPORTED:
            f, g = getattr(self.lib, name), getattr(mw._lib, name)
            f.argtypes, f.restype = g.argtypes, g.restype
        self.lib.fake_launch.restype = ctypes.c_char_p

    def device(self, dev):
        self.lib.fake_set_device(dev)

    def launches(self, call):
        """(kernel name, grid, block, shared memory, stream) of the launches of call()."""
        self.lib.fake_clear()
        rc = call()
        assert rc == 0, self.lib.mw_last_error().decode()
        out = []
        for i in range(self.lib.fake_launches()):
            _, name, grid, block, smem, stream = self.lib.fake_launch(i).decode().split()
            out.append((name, int(grid), int(block), int(smem), int(stream)))
        return out

    def plan(self, m, mode, M, N, K, ra, rb, w=0):
        p = self.mw.mw_plan(w=w)
        rc = self.lib.mw_plan_gemm(m, self.mw._MODES[mode], M, N, K, ra, rb, ctypes.byref(p))
        assert rc == 0, self.lib.mw_last_error().decode()
        return p

    def gemm(self, p, M, N, K, ta=0, tb=0):
        ws = ctypes.c_size_t()
        assert self.lib.mw_gemm_workspace_size(ctypes.byref(p), M, N, K, ctypes.byref(ws)) == 0
        a, b, c, w = (0x100000000 * (i + 1) for i in range(4))
        lda, ldb = (M if ta else K), (K if tb else N)
        return self.lib.mw_gemm(ctypes.byref(p), ta, tb, M, N, K, a, lda, M * K, b, ldb, K * N,
                                c, N, M * N, w, ws.value, None)

    def measure(self, m, M, N, K, ta=0, tb=0):
        ra, rb = ctypes.c_int(), ctypes.c_int()
        a, b, w = (0x100000000 * (i + 1) for i in range(3))
        return self.lib.mw_measure_spread(m, ta, tb, M, N, K, a, M if ta else K, M * K, b,
                                          K if tb else N, K * N, w, 1 << 40, ctypes.byref(ra),
                                          ctypes.byref(rb), None)

    def convolve(self, p, count, n):
        a, b, c = (0x100000000 * (i + 1) for i in range(3))
        return self.lib.mw_convolve_batched(ctypes.byref(p), count, n, a, n, count * n, b, n,
                                            count * n, c, n, count * n, None)

    def dot(self, p, count, K):
        a, b, c = (0x100000000 * (i + 1) for i in range(3))
        return self.lib.mw_dot_batched(ctypes.byref(p), count, K, a, K, count * K, b, K, count * K,
                                       c, count, None)

    def batch(self, p, shapes):
        sh = (ctypes.c_int64 * (3 * len(shapes)))(*[x for s in shapes for x in s])
        b, ws = self.mw.mw_batch(), ctypes.c_size_t()
        assert self.lib.mw_batch_describe(len(shapes), sh, ctypes.byref(b)) == 0
        assert self.lib.mw_gemm_batched_workspace_size(ctypes.byref(p), ctypes.byref(b),
                                                       ctypes.byref(ws)) == 0
        return self.lib.mw_gemm_batched(ctypes.byref(p), ctypes.byref(b), 0x100000000, 0x200000000,
                                        ws.value, None)


def link(mw, folder):
    """The host library, linked in `folder`; None without a C++ compiler or CUDA's headers."""
    import importlib.util
    spec = importlib.util.spec_from_file_location("_mw_build", os.path.join(PACKAGE, "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    cxx = shutil.which("g++") or shutil.which("c++")
    include = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    if not cxx or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        return None
    path = os.path.join(folder, "libmwhost.so")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include,
                    "-o", path, os.path.join(ROOT, "tests", "fake_cudart.cpp")] + objs, check=True)
    return HostLibrary(mw, path)
