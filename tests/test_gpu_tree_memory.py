"""Device memory of the elimination tree: where its scratch cannot be had the subset sum serves the
call, and a sampler's stays within its budget."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2010_15595_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# A process of its own: the library's scratch must be small when the memory becomes scarce. The
# kernels are loaded before that.
SCARCE = """
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
from paper_2010_15595_gb300 import lib, workloads as W
A = W.single_lhaf_mid(40)
subset = lib.lhaf(A, precision=lib.PREC_TF, return_error=True)[0]
batch = lib.lhaf_batch([A, A[:8, :8]], precision=lib.PREC_TF, return_abs_sum=True)[0]
S = A[:26, :26]
small = lib.lhaf(S, precision=lib.PREC_TF)
lib.lhaf_batch([S, S[:8, :8]], precision=lib.PREC_TF)
keep = []
while torch.cuda.mem_get_info()[0] > 300 << 20:  # less than the 740 MB of the tree at N = 40
    free = torch.cuda.mem_get_info()[0] - (200 << 20)
    keep.append(torch.empty(min(free, 32 << 30), dtype=torch.uint8, device="cuda"))
assert lib.lhaf(A, precision=lib.PREC_TF) == subset
assert np.array_equal(lib.lhaf_batch([A, A[:8, :8]], precision=lib.PREC_TF), batch)
assert lib.lhaf(S, precision=lib.PREC_TF) == small
keep.clear()
torch.cuda.empty_cache()
tree = lib.lhaf(A, precision=lib.PREC_TF)
assert tree != subset and abs(tree - subset) < 1e-10 * abs(subset)
print("ok")
"""


def test_subset_sum_where_memory_is_scarce(gbsh):
    out = subprocess.run([sys.executable, "-c", SCARCE, ROOT], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stderr[-2000:]


def test_sampler_stays_within_its_budget(gbsh):
    """Some 25 photons in 24 modes: the tree takes 15 MB for one loop hafnian of N = 26, 75 for N = 30."""
    import torch
    from paper_2010_15595_gb300 import sampler
    U, r, alpha = W.serving_state(0, M=24, n_squeezed=24, r=1.1)
    state = sampler.pure_state(U, r, alpha)

    def run(budget):
        with sampler.Sampler(state, cutoff=3, n_cap=30, mem_budget=budget) as s:
            before = torch.cuda.mem_get_info()[0]
            ids = [s.submit(i, 1) for i in range(3)]
            out = np.concatenate([s.wait(i)[0] for i in ids])
            return out, before - torch.cuda.mem_get_info()[0]

    run(1 << 20)  # the kernels are loaded
    want, large = run(2 << 30)
    assert want.sum(axis=1).max() >= 26 and large > 32 << 20
    for budget in (1 << 20, 4 << 20, 16 << 20):  # N = 18, 22 and 24 at most
        got, used = run(budget)
        assert np.array_equal(got, want)
        assert used <= max(budget, 4 << 20) + (4 << 20), (budget, used)
