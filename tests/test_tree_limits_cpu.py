"""Overflow of the elimination tree's sums (csrc/lhaf_tree.cuh, built for the host). A sum of
products is accumulated modulo 1024, so one that ends near a multiple of it would pass for a small
number; what a level may hold is limited such that no sum of its products gets there. And the cluster
sizes of the small problems."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2010_15595_gb300", "csrc")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("phase") / "tree_phase_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fwrapv", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "tree_phase_host.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def step(host):
    def run(n, M, polys):
        """polys: {pair (j, k): coefficients}; the + child's polynomial of pair (0, 1), and the flag."""
        L, P, Pc = n - M + 1, M * (2 * M + 1), (M - 1) * (2 * M - 1)
        src = np.zeros((L, P), complex)
        for (j, k), c in polys.items():
            src[:, k * (k - 1) // 2 + j] = c
        dst = np.zeros((L + 1, Pc), complex)
        vp = ctypes.c_void_p
        bad = host.tree_host_step(n, M, vp(src.ctypes.data), vp(dst.ctypes.data))
        return dst[:, 0], bad

    return run


def _complementary(L):
    """Two +-1 sequences whose aperiodic autocorrelations cancel (Golay) but for shift 0."""
    a, b = np.array([1]), np.array([1])
    if L % 10 == 0:
        a = np.array([1, 1, -1, 1, -1, 1, -1, -1, 1, 1])
        b = np.array([1, 1, -1, 1, 1, 1, 1, 1, -1, -1])
    while len(a) < L:
        a, b = np.concatenate([a, b]), np.concatenate([a, -b])
    assert len(a) == L
    return a, b


def _peak(step, n, L, x):
    """A step whose product A_0a A_1b + A_0b A_1a has a single coefficient, the last, 4 L x^2."""
    M = n - L + 1
    a, b = _complementary(L)
    r = 2 * M
    return step(n, M, {(0, r - 2): x * (1 + 1j) * a, (1, r - 1): x * (1 - 1j) * a[::-1],
                       (0, r - 1): x * (1 + 1j) * b, (1, r - 2): x * (1 - 1j) * b[::-1]})


@pytest.mark.parametrize("n,L", [(12, 8), (13, 10), (20, 16), (22, 20), (30, 20), (30, 16)])
def test_no_accepted_level_wraps(step, n, L):
    wrap = math.sqrt(1024 / (4 * L))  # factors of that size: the peak is 1024, 0 in the sum
    if wrap < 4:
        got, bad = _peak(step, n, L, wrap)
        assert not bad and abs(got[L]) < 1e-3  # the products alone do not show it ...
    # ... but no level that long takes such numbers: the step that would make them is flagged
    M = n - L + 1
    for x, want in ((min(wrap, 4.0), 1), (min(wrap, 4.0) * 0.995, 0)):
        old = np.full(L - 1, x)
        old[0] = 0.5  # the lowest coefficient is the matrix entry, below 1
        for sign in (1, -1, 1j, -1j):
            got, bad = step(n, M + 1, {(0, 1): sign * old})
            assert bad == want, (n, L, x)
    # the largest that are taken: a sum of theirs is either right or flagged
    got, bad = _peak(step, n, L, min(wrap, 4.0) * 0.995)
    assert bad
    got, bad = _peak(step, n, L, 0.9 / math.sqrt(L))
    assert not bad and abs(got[L] - 4 * 0.81) < 1e-9 and np.abs(got[:L]).max() < 1e-9


def test_flags_at_the_limit_of_short_levels(step):
    """Up to 15 coefficients a level takes everything below 4, at any n."""
    for n, M in ((6, 4), (15, 4), (30, 20)):
        for x, want in ((3.999, 0), (4.0, 1)):
            old = np.full(n - M + 1, x)
            old[0] = 0.5
            assert step(n, M, {(0, 1): old})[1] == want


@pytest.mark.parametrize("most", [1, 2, 4, 8, 16])
def test_clusters_that_the_device_can_hold(host, most):
    for slots in (2, 64, 304):
        for n in range(2, 9):
            for count in (1, 2, 5, 19, 38, 100, 1000, 2**31 // 16 + 1):
                c = host.tree_host_cluster(n, count, slots, most)
                assert 1 <= c <= most and c & (c - 1) == 0
                assert c == 1 or c * count <= slots
    assert host.tree_host_cluster(8, 1, 304, most) == most
