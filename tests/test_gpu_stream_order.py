"""Host matrices are read in stream order: after what was queued on the call's stream before."""
import ctypes
import time

import numpy as np
import pytest

from paper_2010_15595_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _rt():
    import torch
    torch.cuda.init()
    return ctypes.CDLL("libcudart.so.13")


# 2..60: staged through page-locked memory; FP64 above N = 24 is copied by the subset sum's path
@pytest.mark.parametrize("N,prec_name", [(2, "PREC_FP64"), (16, "PREC_FP64"), (16, "PREC_TF"), (30, "PREC_FP64"),
                                         (30, "PREC_TF")])
@pytest.mark.parametrize("legacy", [False, True])
def test_matrix_written_by_the_stream(gbsh, N, prec_name, legacy):
    """A host function fills the matrix a while after the call; on the legacy default stream it
    runs on a stream that the default one waits for."""
    rt, prec = _rt(), getattr(gbsh, prec_name)
    before, after = W.single_lhaf_mid(N), W.single_lhaf_mid(N, seed=1)
    want = gbsh.lhaf(after, precision=prec)  # everything is allocated
    assert want != gbsh.lhaf(before, precision=prec)
    A = before.copy()
    st = ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(st)) == 0

    def fill(_):
        time.sleep(0.2)
        A[:] = after

    cb = ctypes.CFUNCTYPE(None, ctypes.c_void_p)(fill)
    try:
        assert rt.cudaLaunchHostFunc(st, cb, None) == 0
        got = gbsh.lhaf(A, precision=prec, stream=0 if legacy else st.value)
        assert rt.cudaStreamSynchronize(st) == 0
    finally:
        rt.cudaStreamDestroy(st)
    assert got == want
