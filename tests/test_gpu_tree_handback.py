"""What the elimination tree hands back to the subset sum where the way back is longest: gated
evaluations of several launch classes, captured or not, mixed batches, and the sampler."""
import numpy as np
import pytest

from paper_2010_15595_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _dev(A):
    import torch
    return torch.from_numpy(np.ascontiguousarray(A)).to("cuda")


def _graded(N, seed=0):
    """Two blocks, the entries of one a thousandth of the other's: below the fixed point's resolution, and
    within the FP32 range of the triple-float words."""
    rng = np.random.default_rng(3000 + 10 * N + seed)
    h = N // 2
    A = np.zeros((N, N), complex)
    A[:h, :h] = W.random_complex_symmetric(h, rng) * 1e-3
    A[h:, h:] = W.random_complex_symmetric(N - h, rng)
    A[np.arange(h), np.arange(h)] *= 0.1
    return A


@pytest.mark.parametrize("N", [18, 25, 32, 36])
def test_asynchronous(gbsh, N):
    """One class and several; a captured evaluation whose replays meet both kinds of matrices."""
    import torch
    prec = gbsh.PREC_TF
    A, B = _graded(N), W.single_lhaf_mid(N)
    subset, tree = gbsh.lhaf(A, precision=prec, return_error=True)[0], gbsh.lhaf(B, precision=prec)
    assert (gbsh.plan(N, precision=prec)["nclass"] > 1) == (N >= 32)
    assert subset != 0 and gbsh.lhaf(A, precision=prec) == subset  # handed back
    dA = _dev(A)
    out = torch.zeros(1, dtype=torch.complex128, device="cuda")
    ws = torch.empty(gbsh.workspace_size(N, prec), dtype=torch.uint8, device="cuda")
    for M, want in ((A, subset), (B, tree), (A, subset)):
        dA.copy_(_dev(M))
        gbsh.lhaf_async(dA, out, ws, precision=prec)
        assert complex(out.item()) == want
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gbsh.lhaf_async(dA, out, ws, precision=prec)
    for M, want in ((B, tree), (A, subset), (A, subset), (B, tree)):
        dA.copy_(_dev(M))
        g.replay()
        torch.cuda.synchronize()
        assert complex(out.item()) == want


@pytest.mark.parametrize("prec_name", ["PREC_FP64", "PREC_TF"])
def test_in_a_mixed_batch(gbsh, prec_name):
    """Small and large problems, every other one handed back, and an empty one."""
    prec = getattr(gbsh, prec_name)
    sizes = [11, 14, 18, 20, 23] + ([28, 31] if prec == gbsh.PREC_TF else [])
    mats, back = [np.zeros((0, 0), complex)], [False]
    for N in sizes:
        mats += [_graded(N), W.single_lhaf_mid(N)]
        back += [True, False]
    got = gbsh.lhaf_batch(mats, precision=prec)
    assert got[0] == 1
    for A, b, v in list(zip(mats, back, got))[1:]:
        if not b:
            assert v == gbsh.lhaf(A, precision=prec), A.shape
        else:
            subset = gbsh.lhaf_batch([A, A], precision=prec, return_abs_sum=True)[0][1]
            assert subset != 0 and abs(v - subset) <= 1e-12 * abs(subset), (A.shape, v, subset)


def test_in_the_sampler(gbsh):
    """Strongly displaced modes: about half of the loop hafnians above N = 28 come back. The photon
    numbers are those of a sampler whose budget leaves everything above N = 18 to the subset sum."""
    from paper_2010_15595_gb300 import sampler
    rng = np.random.default_rng(5)
    M = 16
    U = W.haar_unitary(M, rng)
    alpha = 1.3 * np.exp(0.2j) * np.ones(M)
    state = sampler.pure_state(U, rng.uniform(0.3, 0.6, M), alpha)

    def run(**kw):
        with sampler.Sampler(state, cutoff=6, n_cap=32, **kw) as s:
            ids = [s.submit(i, 1) for i in range(3)]
            return np.concatenate([s.wait(i)[0] for i in ids])

    want = run(mem_budget=1 << 20)
    assert want.sum(axis=1).max() >= 28
    back = 0
    for row in want:
        if 28 <= row.sum() <= 32:
            idx = np.repeat(np.arange(M), row)
            A = W.with_diagonal(state.B[np.ix_(idx, idx)], np.asarray(state.gamma)[idx])
            back += gbsh.lhaf(A, precision=gbsh.PREC_TF) == gbsh.lhaf(A, precision=gbsh.PREC_TF, return_error=True)[0]
    assert back > 0
    assert np.array_equal(run(), want)
    assert np.array_equal(run(batching=False), want)
