"""Strongly displaced states by the elimination tree: loop weights up to several times the matrix
entries, of one size or many, in and out of phase."""
import numpy as np
import pytest

from oracle import lhaf as L
from paper_2010_15595_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# as in test_gpu_tree.py: results are kept where the tree's error is 2^-53 of them; the rest is the
# reference (the definition in complex128)
TOL = 1e-13


def _matrices(N, seed):
    rng = np.random.default_rng(4000 + 10 * N + seed)
    B = W.squeezed_kernel(W.haar_unitary(N, rng), rng.uniform(0.4, 0.9, N))
    for sigma in (0.4, 0.7, 1.0, 2.0):
        yield W.with_diagonal(B, W.complex_normal(N, sigma, rng))
    for amplitude in (0.3, 1.0, 2.0):
        yield W.with_diagonal(B, np.full(N, amplitude * np.exp(0.3j)))
    heavy = W.complex_normal(N, 0.2, rng)
    heavy[N // 3] = 1e3
    heavy[0] = 1e8
    yield W.with_diagonal(B, heavy)
    yield np.diag(rng.standard_normal(N)).astype(complex)
    yield W.with_diagonal(B * 1e-24, W.complex_normal(N, 1e-10, rng))
    yield W.with_diagonal(B * 1e20, W.complex_normal(N, 1e10, rng))


@pytest.mark.parametrize("N", [2, 3, 8, 15, 16, 17, 20, 22, 23])
def test_displaced_states_stay_on_the_tree(gbsh, N):
    """Within the tree's tolerance (the FP64 subset sum is not at N = 20 and above), with the
    same bits in both precisions (the subset sum's differ)."""
    for A in _matrices(N, 0):
        ref = L.lhaf_brute(A) if N <= 12 else L.lhaf_dp(A)
        got = gbsh.lhaf(A)
        assert abs(got - ref) <= TOL * abs(ref), (N, got, ref)
        assert got == gbsh.lhaf(A, precision=gbsh.PREC_TF)
    mats = list(_matrices(N, 1))
    assert np.array_equal(gbsh.lhaf_batch(mats), [gbsh.lhaf(A) for A in mats])


@pytest.mark.parametrize("N", [26, 32, 36])
def test_displaced_states_against_the_subset_sum(gbsh, N):
    """Above the definition's reach: the triple-float subset sum, where its words of FP32 hold the
    polynomials' coefficients (which grow as powers of the largest entry)."""
    for A in _matrices(N, 0):
        if not 0.01 < np.abs(A).max() < 100:
            continue
        ref, err = gbsh.lhaf(A, precision=gbsh.PREC_TF, return_error=True)
        got = gbsh.lhaf(A, precision=gbsh.PREC_TF)
        assert abs(got - ref) <= max(TOL, err) * abs(ref), (N, got, ref, err)
