"""Evaluation by the elimination tree (csrc/lhaf_tree.cu): edges of its range against the
definition, agreement of all entry points, and the cases it hands back to the subset sum."""
import numpy as np
import pytest

from oracle import lhaf as L
from paper_2010_15595_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# Fixed point keeps 2^-81 absolute and results above 2^-28 of the scale: 2^-53 relative; the rest
# is the reference (the definition in complex128).
TOL = 1e-13


def _dev(A):
    import torch
    return torch.from_numpy(np.ascontiguousarray(A)).to("cuda")


def _async(gbsh, A, prec, nbytes=None):
    import torch
    out = torch.zeros(1, dtype=torch.complex128, device="cuda")
    ws = torch.empty(nbytes or gbsh.workspace_size(A.shape[0], prec), dtype=torch.uint8, device="cuda")
    gbsh.lhaf_async(_dev(A), out, ws, precision=prec)
    return complex(out.item())


# 1..6: padding to four vertices, no signed pair, one signed pair; 13..16 and 19, 20: units
# above and at the breadth-first level; 23: odd
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 13, 14, 16, 19, 20, 23])
def test_sizes_and_entry_points(gbsh, N):
    rng = np.random.default_rng(700 + N)
    for A in (W.single_lhaf_mid(N), W.random_complex_symmetric(N, rng)):
        ref = L.lhaf_brute(A) if N <= 12 else L.lhaf_dp(A)
        got = gbsh.lhaf(A, precision=gbsh.PREC_TF)
        assert abs(got - ref) <= TOL * abs(ref), (N, got, ref)
        assert gbsh.lhaf(_dev(A), precision=gbsh.PREC_TF) == got
        assert _async(gbsh, A, gbsh.PREC_TF) == got
        big = np.zeros((N, N + 3), complex)
        big[:, :N] = A
        assert gbsh.lhaf(_dev(big)[:, :N], precision=gbsh.PREC_TF) == got  # leading dimension


def test_batch_equals_single(gbsh):
    """Every size 0..31 in one batch and alone: the limb sums are exact, so the bits agree."""
    rng = np.random.default_rng(71)
    mats = [W.random_complex_symmetric(N, rng) for N in list(range(32)) + [7, 7, 30, 1]]
    got = gbsh.lhaf_batch(mats, precision=gbsh.PREC_TF)
    for A, g in zip(mats, got):
        if A.shape[0] == 0:
            assert g == 1
        else:
            assert g == gbsh.lhaf(A, precision=gbsh.PREC_TF), A.shape


@pytest.mark.parametrize("N", [6, 11, 20])
def test_handed_back_to_the_subset_sum(gbsh, N):
    """Graded, nearly vanishing and huge-weight matrices, zeros and NaN: the result of the
    subset sum in the same entry point."""
    rng = np.random.default_rng(72)
    graded = np.zeros((N, N), complex)
    h = N // 2
    graded[:h, :h] = W.random_complex_symmetric(h, rng) * 1e-9
    graded[h:, h:] = W.random_complex_symmetric(N - h, rng)
    weights = W.single_lhaf_mid(N)
    weights[0, 0] = 1e12
    nan = W.single_lhaf_mid(N)
    nan[1, 1] = np.nan
    for A in (graded, weights, np.zeros((N, N), complex), nan, W.single_lhaf_mid(N)):
        single, _ = gbsh.lhaf(A, precision=gbsh.PREC_TF, return_error=True)
        batch = gbsh.lhaf_batch([A, A], precision=gbsh.PREC_TF, return_abs_sum=True)[0][1]
        for v, subset in ((gbsh.lhaf(A, precision=gbsh.PREC_TF), single), (_async(gbsh, A, gbsh.PREC_TF), single),
                          (gbsh.lhaf_batch([A, A], precision=gbsh.PREC_TF)[1], batch)):
            if np.isnan(subset):
                assert np.isnan(v)
            else:
                assert abs(v - subset) <= 1e-12 * abs(subset), (v, subset)


def test_workspace_of_the_subset_sum_is_still_taken(gbsh):
    """A workspace too small for the tree but large enough for the subset sum is accepted."""
    A = W.single_lhaf_mid(18)
    small = gbsh.workspace_size(18)  # the FP64 subset sum's, which the triple-float one fits too
    v = _async(gbsh, A, gbsh.PREC_TF, nbytes=max(small, 1 << 16))
    assert abs(v - gbsh.lhaf(A, precision=gbsh.PREC_TF)) <= 1e-13 * abs(v)


def test_graph_capture(gbsh):
    """lhaf_async inside a CUDA graph: replays read the matrix that is there at replay time."""
    import torch
    N = 20
    A, B = W.single_lhaf_mid(N), W.single_lhaf_mid(N, seed=1)
    dA = _dev(A)
    out = torch.zeros(1, dtype=torch.complex128, device="cuda")
    ws = torch.empty(gbsh.workspace_size(N, gbsh.PREC_TF), dtype=torch.uint8, device="cuda")
    gbsh.lhaf_async(dA, out, ws, precision=gbsh.PREC_TF)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gbsh.lhaf_async(dA, out, ws, precision=gbsh.PREC_TF)
    for M in (A, B, A):
        dA.copy_(_dev(M))
        g.replay()
        torch.cuda.synchronize()
        assert complex(out.item()) == gbsh.lhaf(M, precision=gbsh.PREC_TF)
