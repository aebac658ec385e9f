"""Builds tests/native/probes.cu against the library's objects and binds it."""
import ctypes as C
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))


def load(directory):
    """The probes, compiled into `directory`."""
    from paper_2403_04946_gb300 import build
    build.build()
    out = os.path.join(str(directory), "probes.so")
    objs = [os.path.join(build.BUILD, os.path.splitext(s)[0] + ".o") for s in build.SOURCES if s != "noalloc.cu"]
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-I" + build.CSRC, "-shared", "-cudart", "static", "-o", out,
           os.path.join(HERE, "native", "probes.cu"), *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return Probes(C.CDLL(out))


def _p(a):
    return a.ctypes.data_as(C.POINTER(C.c_double))


class Probes:
    def __init__(self, lib):
        self.lib = lib
        d, i, ll = C.POINTER(C.c_double), C.c_int, C.c_longlong
        lib.probe_product.argtypes = [i, i, i, d, d, d, ll, ll, ll, C.c_double, i, i, i, ll]
        lib.probe_gemm.argtypes = [i, i, i, d, d, d, i, i, i]
        lib.probe_part_bytes.argtypes = [i, i, i, i]
        lib.probe_part_bytes.restype = ll
        lib.probe_reciprocals.argtypes = [i, d, d, d]
        lib.probe_house.argtypes = [i, d, d, d]

    def wide_product(self, A, B, C0=None, alpha=1.0, transposed=False, balance=False, digits=0, max_part=0):
        """alpha A B^T (+ C0) for complex A (M x K), B (N x K), by the wide digits or by `digits`."""
        A, B = np.ascontiguousarray(A, np.complex128), np.ascontiguousarray(B, np.complex128)
        (M, K), N = A.shape, B.shape[0]
        pad = 3  # unused rows of the leading dimension, which must stay
        rso, ldo, shape = (N + pad, 1, (M, N + pad)) if transposed else (1, M + pad, (N, M + pad))
        out = np.full(shape, 7.0 - 3.0j)
        view = out[:, :N] if transposed else out[:, :M].T
        if C0 is not None:
            view[...] = C0
        st = self.lib.probe_product(M, N, K, _p(A.view(np.float64)), _p(B.view(np.float64)),
                                    _p(out.view(np.float64)), out.size, rso, ldo, alpha, C0 is not None, balance, digits,
                                    max_part)
        assert st == 0, st
        rest = out[:, N:] if transposed else out[:, M:]
        assert (rest == 7.0 - 3.0j).all()
        return view.copy()

    def gemm(self, A, R, coff=0, uh=False, mixed=False):
        """A R^H for the upper trapezoid of R's columns from coff on, or A^H R."""
        A, R = np.asfortranarray(A, np.complex128), np.asfortranarray(R, np.complex128)
        K, M = A.shape if uh else A.shape[::-1]
        N = R.shape[1] if uh else R.shape[0]
        out = np.empty((M, N), np.complex128, order="F")
        p = lambda x: x.ctypes.data_as(C.POINTER(C.c_double))
        st = self.lib.probe_gemm(M, N, K, p(A), p(R), p(out), coff, uh, mixed)
        assert st == 0, st
        return out

    def reciprocals(self, x):
        x = np.ascontiguousarray(x, np.float64)
        a, b = np.empty_like(x), np.empty_like(x)
        assert self.lib.probe_reciprocals(x.size, _p(x), _p(a), _p(b)) == 0
        return a, b

    def house(self, alpha, s2):
        alpha, s2 = np.ascontiguousarray(alpha, np.complex128), np.ascontiguousarray(s2, np.float64)
        out = np.empty((alpha.size, 3), np.complex128)
        assert self.lib.probe_house(alpha.size, _p(alpha.view(np.float64)), _p(s2), _p(out.view(np.float64))) == 0
        return out[:, 0], out[:, 1], out[:, 2].real
