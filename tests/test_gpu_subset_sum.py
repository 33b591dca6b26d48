"""The triple-float and FP64 subset sums where the elimination tree serves the plain calls: reached by
asking for the error estimate or sum |p_Z|. References and tolerances are those of
test_gpu_accurate.py and test_gpu_tuning.py."""
import json
import os

import numpy as np
import pytest

from oracle import lhaf as L
from paper_2010_15595_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _dev(A):
    import torch
    return torch.from_numpy(np.ascontiguousarray(A)).to("cuda")


def _subset(gbsh, A, prec):
    return gbsh.lhaf(A, precision=prec, return_error=True)[0]


def telephone(n):
    t = [1, 1]
    for k in range(2, n + 1):
        t.append(t[-1] + (k - 1) * t[-2])
    return t[n]


@pytest.mark.parametrize("N", list(range(1, 25)))
def test_sizes_against_the_definition(gbsh, N):
    rng = np.random.default_rng(2000 + N)
    A = W.random_complex_symmetric(N, rng)
    ref = L.lhaf_brute(A) if N <= 12 else L.lhaf_dp(A)
    got = _subset(gbsh, _dev(A), gbsh.PREC_TF)
    assert abs(got - ref) <= 1e-9 * abs(ref), (N, got, ref)
    batch, _ = gbsh.lhaf_batch([A, A], precision=gbsh.PREC_TF, return_abs_sum=True)
    assert np.all(np.abs(batch - ref) <= 1e-9 * abs(ref)), (N, batch, ref)


@pytest.mark.parametrize("n", [2, 9, 20, 30, 36, 40, 46])
def test_all_ones(gbsh, n):
    """The per-subset rescaling: the terms grow to 2^120 at n = 46."""
    got = _subset(gbsh, W.all_ones(n), gbsh.PREC_TF)
    assert abs(got - telephone(n)) / telephone(n) <= 1e-12, (n, got)


@pytest.mark.parametrize("name", ["lhaf_n50", "lhaf_n50_block"])
def test_long_double_references(gbsh, name):
    from tests.golden.make_golden import read_matrix
    with open(os.path.join(HERE, "golden", name + ".json")) as f:
        rec = json.load(f)
    if "lhaf_ld" not in rec:
        pytest.skip("fixture has no long-double value")
    ref = complex(*rec["lhaf_ld"])
    got = _subset(gbsh, _dev(read_matrix(os.path.join(HERE, "golden", name + ".matrix.txt"))), gbsh.PREC_TF)
    assert abs(got - ref) <= 1e-7 * abs(ref), (got, ref)


def test_deterministic_and_launch_shape_independent(gbsh):
    A = _dev(W.single_lhaf_mid(28))
    vals = {_subset(gbsh, A, gbsh.PREC_TF) for _ in range(3)}
    assert len(vals) == 1
    a = vals.pop()
    try:
        gbsh.set_tuning(4, 0)
        b = _subset(gbsh, A, gbsh.PREC_TF)
        gbsh.set_tuning(8, 6)
        c = _subset(gbsh, A, gbsh.PREC_TF)
    finally:
        gbsh.set_tuning(0, 0)
    assert a == b
    assert abs(c - a) < 1e-15 * abs(a)


def test_tuned_plans_agree(gbsh):
    N = 30
    dA = _dev(W.single_lhaf_mid(N, seed=5))
    base = _subset(gbsh, dA, gbsh.PREC_TF)
    try:
        for cfg in [(8, gbsh.LADDER_FINE, 18), (16, gbsh.LADDER_FINE, 12), (10, gbsh.LADDER_COARSE, 9)]:
            gbsh.set_lhaf_tuning(gbsh.PREC_TF, N, *cfg)
            a, b = _subset(gbsh, dA, gbsh.PREC_TF), _subset(gbsh, dA, gbsh.PREC_TF)
            assert a == b
            assert abs(a - base) <= 1e-13 * abs(base)
    finally:
        gbsh.set_lhaf_tuning(gbsh.PREC_TF, N)
    assert _subset(gbsh, dA, gbsh.PREC_TF) == base


@pytest.mark.parametrize("prec_name", ["PREC_FP64", "PREC_TF"])
def test_batch_graphs_of_equal_count_and_another_layout(gbsh, prec_name):
    """Batches of equal count, largest size and chunk total whose small problems differ in size: each
    is captured on its second use and replayed from then on, with its own offsets."""
    prec = getattr(gbsh, prec_name)
    rng = np.random.default_rng(22)
    batches = [[W.random_complex_symmetric(N, rng) for N in sizes] for sizes in ([14, 14, 6, 6], [14, 14, 4, 8])]

    def run(mats):
        return gbsh.lhaf_batch(mats, precision=prec, return_abs_sum=True)[0]

    try:
        gbsh.set_batch_graphs(False)
        direct = [run(m) for m in batches]
        gbsh.set_batch_graphs(True)
        s0 = gbsh.batch_graph_stats()
        runs = [run(batches[i % 2]) for i in range(6)]
        s1 = gbsh.batch_graph_stats()
    finally:
        gbsh.set_batch_graphs(True)
    assert s1["captures"] == s0["captures"] + 2
    assert s1["replays"] == s0["replays"] + 4
    for i, r in enumerate(runs):
        assert np.array_equal(r, direct[i % 2]), i
