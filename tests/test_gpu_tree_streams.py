"""Streams of the elimination tree's callers: nobody's work waits for what another caller's stream
still has to do."""
import threading
import time

import numpy as np
import pytest

from paper_2010_15595_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_sampler_does_not_wait_for_a_batch(gbsh):
    """A batch of small and large problems stands behind a long kernel on its stream; a sampler
    whose ticks are of both kinds too runs meanwhile."""
    import torch
    from paper_2010_15595_gb300 import sampler
    mats = [W.single_lhaf_mid(N) for N in (8, 12, 20, 22)]
    U, r, alpha = W.serving_state(0, M=32, n_squeezed=14, sigma=0.2)
    s = sampler.Sampler(sampler.pure_state(U, r, alpha), cutoff=4, n_cap=24)
    st = torch.cuda.Stream()

    def sample():
        ids = [s.submit(i, 1) for i in range(8)]
        return np.concatenate([s.wait(i)[0] for i in ids])

    want = gbsh.lhaf_batch(mats, precision=gbsh.PREC_TF, stream=st)  # everything is allocated
    alone = sample()
    assert alone.sum(axis=1).max() > 16 and alone.sum(axis=1).min() < 16
    got, end = [], []

    def batch():
        got.append(gbsh.lhaf_batch(mats, precision=gbsh.PREC_TF, stream=st))
        end.append(time.perf_counter())

    with torch.cuda.stream(st):
        torch.cuda._sleep(4_000_000_000)  # about two seconds
    t = threading.Thread(target=batch)
    t.start()
    time.sleep(0.3)  # the batch is launched
    beside = sample()
    sampled = time.perf_counter()
    t.join()
    assert sampled < end[0] - 0.2, "the sampler waited for the batch's stream"
    assert np.array_equal(beside, alone)
    assert np.array_equal(got[0], want)
