"""The elimination tree's level code (csrc/lhaf_tree.cuh) built for the host and compared with
the definition: every size with its odd paddings, every way to cut the tree into a breadth-
first part, walks and units, or all breadth first, matrices of several kinds, with canaries around the buffers."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from oracle import lhaf as L
from paper_2010_15595_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2010_15595_gb300", "csrc")
# Fixed point keeps 2^-81 absolute where the scaled result is above 2^-28 (smaller ones go to
# the subset sum): 2^-53 relative, times a few ulps of the rounding to double and of the
# reference (the definition in complex128, up to ~1e-15 sqrt(matchings) at N = 18). An ulp of a
# subnormal result is 2^-1074 whatever its size (the 1e-40 matrix at N = 16 and 18).
TOL = 1e-13
ULP = 4 * 2.0 ** -1074


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("tree") / "tree_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fwrapv", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "tree_host.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.tree_host_lhaf.restype = ctypes.c_int

    def run(A, m1, top):
        A = np.ascontiguousarray(A, dtype=np.complex128)
        N = A.shape[0]
        off = A - np.diag(np.diag(A))
        f = np.linalg.norm(off)
        rho = np.linalg.norm(off.conj().T @ off) / f if f > 0 else 0.0
        v = np.diag(A)
        den = max(rho, (np.abs(v) ** 2).sum() / 8, 1.25 * max(np.abs(off).max(), (np.abs(v) ** 2).max()))
        mant, ex = math.frexp(1 / math.sqrt(den))
        out = (ctypes.c_double * 2)()
        rc = lib.tree_host_lhaf(A.ctypes.data_as(ctypes.c_void_p), N, int(mant * 32), ex - 1, m1, top, out)
        assert rc == 0
        return complex(out[0], out[1])

    return run


def _pairs(N):
    return max(4, N + (N & 1)) // 2


@pytest.mark.parametrize("N", list(range(1, 19)))
def test_every_size_and_cut(host, N):
    rng = np.random.default_rng(400 + N)
    n = _pairs(N)
    mats = [W.single_lhaf_mid(N), W.random_complex_symmetric(N, rng)]
    if N % 2 == 0:
        mats += [W.all_ones(N), W.random_complex_symmetric(N, rng) * 1e-40]
        H = W.single_lhaf_mid(N)
        np.fill_diagonal(H, 0)
        mats.append(H)
    for A in mats:
        ref = L.lhaf_brute(A) if N <= 12 else L.lhaf_dp(A)
        m1 = n if n == 2 else n - 1
        first = host(A, m1, min(3, m1))
        assert abs(first - ref) <= TOL * abs(ref) + ULP, (N, first, ref)
        # exact sums: the way the tree is cut cannot change a bit
        for cut in {(m1, 2), (m1, m1), (max(2, m1 - 2), 2), (max(2, m1 - 2), max(2, m1 - 3)), (2, 2), (0, 0)}:
            assert host(A, *cut) == first, (N, cut)
