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


# 1..6: padding to four vertices, no signed pair, one signed pair; 8, 10, 12, 16: cluster sizes of
# the small kernel, 16 its last size; 18 on: the other kernels; 24, 25: the last FP64 size and after
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 13, 16, 18, 19, 23, 24, 25, 26])
def test_sizes_and_entry_points(gbsh, N):
    rng = np.random.default_rng(700 + N)
    for A in (W.single_lhaf_mid(N), W.random_complex_symmetric(N, rng)):
        tol = TOL
        if N <= 24:
            ref = L.lhaf_brute(A) if N <= 12 else L.lhaf_dp(A)
        else:  # the long-double subset sum and its own rounding floor
            ref = L.lhaf_subset_ld(A)
            tol = max(TOL, 512 * 2.0 ** -64 * L.lhaf_subset_stats(A)[2] ** 0.5 / abs(ref))
        got = gbsh.lhaf(A, precision=gbsh.PREC_TF)
        assert abs(got - ref) <= tol * abs(ref), (N, got, ref)
        assert gbsh.lhaf(_dev(A), precision=gbsh.PREC_TF) == got
        assert _async(gbsh, A, gbsh.PREC_TF) == got
        big = np.zeros((N, N + 3), complex)
        big[:, :N] = A
        assert gbsh.lhaf(_dev(big)[:, :N], precision=gbsh.PREC_TF) == got  # leading dimension
        if N <= 24:  # FP64 entry points: the same evaluation
            assert gbsh.lhaf(A) == got and _async(gbsh, A, gbsh.PREC_FP64) == got
            B = np.zeros((N + 2, N + 2), complex)
            B[:N, :N] = A
            g = np.concatenate([np.diag(A), [3, 4]])
            pattern = [1] * N + [0, 0]
            assert gbsh.gbs_prob(B, g, pattern, return_lhaf=True)[1] == got
            assert gbsh.gbs_prob_batch(B, g, [pattern, pattern])[1][1] == got


def test_batch_equals_single(gbsh):
    """Every size 0..31 in one batch and alone, a batch of small problems large enough for
    one-CTA clusters, and a mixed-precision one: the limb sums are exact, so the bits agree."""
    rng = np.random.default_rng(71)
    mats = [W.random_complex_symmetric(N, rng) for N in list(range(32)) + [7, 7, 30, 1]]
    many = [W.random_complex_symmetric(1 + i % 18, rng) for i in range(330)]
    for batch in (mats, many, mats[:25]):
        got = gbsh.lhaf_batch(batch, precision=gbsh.PREC_TF)
        for A, g in zip(batch, got):
            if A.shape[0] == 0:
                assert g == 1
            else:
                assert g == gbsh.lhaf(A, precision=gbsh.PREC_TF), A.shape
    fp64 = gbsh.lhaf_batch(mats)
    mixed = gbsh.lhaf_batch(mats, precision=gbsh.PREC_MIXED)
    tf = gbsh.lhaf_batch(mats, precision=gbsh.PREC_TF)
    for i in range(25):  # N <= 24
        assert fp64[i] == tf[i]
        assert mixed[i] == fp64[i] if i > gbsh.C32_MAX_N else abs(mixed[i] - fp64[i]) <= 1e-5 * abs(fp64[i])


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
    A = W.single_lhaf_mid(24)
    small = gbsh.workspace_size(26)  # FP64 above N = 24: the subset sum's alone, larger than N = 24's
    assert small < gbsh.workspace_size(24, gbsh.PREC_TF)
    for prec in (gbsh.PREC_FP64, gbsh.PREC_TF):
        v = _async(gbsh, A, prec, nbytes=small)
        subset, _ = gbsh.lhaf(A, precision=prec, return_error=True)
        assert v == subset


def test_more_large_problems_than_a_grid_has_rows(gbsh):
    """A level's launch has a row of CTAs per problem, at most 65535."""
    A = W.single_lhaf_mid(18)[:17, :17]
    v = gbsh.lhaf_batch([A] * 65540, precision=gbsh.PREC_TF)
    assert np.all(v == gbsh.lhaf(A, precision=gbsh.PREC_TF))


def test_graph_capture(gbsh):
    """lhaf_async inside a CUDA graph: replays read the matrix that is there at replay time."""
    import torch
    N = 26
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


def test_synchronous_batch_during_a_capture(gbsh):
    """While a thread captures an evaluation of several launch classes, which takes the library's
    side streams into the capture, synchronous batches of both kinds of problems go on."""
    import torch
    A = W.single_lhaf_mid(40)
    mats = [W.single_lhaf_mid(N) for N in (8, 20)]
    st = torch.cuda.Stream()
    want = gbsh.lhaf_batch(mats, precision=gbsh.PREC_TF, stream=st)  # and everything is allocated
    dA = _dev(A)
    out = torch.zeros(1, dtype=torch.complex128, device="cuda")
    ws = torch.empty(gbsh.workspace_size(40, gbsh.PREC_TF), dtype=torch.uint8, device="cuda")
    gbsh.lhaf_async(dA, out, ws, precision=gbsh.PREC_TF)
    ref = complex(out.item())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        gbsh.lhaf_async(dA, out, ws, precision=gbsh.PREC_TF)
        got = gbsh.lhaf_batch(mats, precision=gbsh.PREC_TF, stream=st)
    assert np.all(got == want)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert complex(out.item()) == ref
