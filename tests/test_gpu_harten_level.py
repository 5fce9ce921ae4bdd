"""mr_run_static takes any regularity guess mu_bar >= 0.  From 2^(mu_bar + 1)
eps_l above every detail on, a larger one changes nothing: no pair is refined
by the Harten rule, whatever the exponent range of the level."""
import ctypes

import numpy as np
import pytest

from paper_2102_12163_gb300 import MR_FP32_MIXED, MR_FP64, capi, workloads as W
from paper_2102_12163_gb300 import _desc as desc_of

pytestmark = pytest.mark.gpu


def _run(d, inst, precision):
    import torch

    m = torch.as_tensor(np.ascontiguousarray(inst.m0)).cuda()
    out = torch.full((inst.nf, 1 << inst.Jmax), float("nan"), dtype=torch.float64, device="cuda")
    upd = ctypes.c_ulonglong()
    capi.check(None, capi.load().mr_run_static(ctypes.byref(d), precision, ctypes.c_void_p(m.data_ptr()), 6,
                                               ctypes.c_void_p(out.data_ptr()), ctypes.byref(upd),
                                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return out.cpu().numpy(), upd.value


@pytest.mark.parametrize("precision", [MR_FP64, MR_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("mu_bar", [31, 500, 1022, 1023, 1024, 1100, 2047, 2 ** 31 - 1])
def test_large_regularity_guess(mu_bar, precision):
    inst = W.random_smooth(9, W.EQ_BURGERS, seed=3, eps=1e-3)
    d = desc_of(inst)
    d.mu_bar = 30
    want, updates = _run(d, inst, precision)
    d.mu_bar = mu_bar
    got, n = _run(d, inst, precision)
    assert n == updates
    assert np.array_equal(got, want)


@pytest.mark.parametrize("mu_bar", [30, 1023, 1100])
def test_zero_threshold_keeps_the_whole_tree(mu_bar):
    inst = W.random_smooth(7, W.EQ_BURGERS, seed=3, eps=0.0)
    d = desc_of(inst)
    d.mu_bar = mu_bar
    assert _run(d, inst, MR_FP64)[1] == 6 << inst.Jmax
