"""Default threads per block (host rule, 152 SMs): a batch of equal instances
that fits one wave of narrower blocks is not sent through two waves of wider
ones; uneven batches keep the line by instances per SM."""
import ctypes

import pytest

from paper_2102_12163_gb300 import MR_FP32_MIXED, MR_FP64, capi, workloads as W
from paper_2102_12163_gb300 import _desc as desc_of

SMS = 152


def _block(insts, precision):
    f = capi.load().mrg_default_block
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int]
    arr = (capi.mr_instance_desc * len(insts))(*[desc_of(i) for i in insts])
    return f(ctypes.byref(arr), len(insts), precision, SMS)


@pytest.mark.parametrize("precision", [MR_FP64, MR_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("eq", [W.EQ_BURGERS, W.EQ_SW, W.EQ_EULER, W.EQ_SW_D1Q5])
@pytest.mark.parametrize("n", [1, 20, 152, 153, 200, 304, 305, 400, 600, 608])
def test_equal_instances_run_in_one_wave(n, eq, precision):
    b = _block([W.random_smooth(9, eq, seed=1, eps=1e-3)] * n, precision)
    # blocks an SM that the variants are compiled for; the scalar one fits three of 512 in FP32
    resident = 3 if (b, eq, precision) == (512, W.EQ_BURGERS, MR_FP32_MIXED) else 1024 // b
    assert n <= SMS * resident
    assert b >= 256


@pytest.mark.parametrize("precision", [MR_FP64, MR_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("n,block", [(32, 512), (152, 512), (200, 1024), (300, 1024), (450, 512), (800, 512), (1100, 256), (4096, 256)])
def test_uneven_instances_by_instances_per_sm(n, block, precision):
    assert _block(W.batch(n=n, Jmax_range=(8, 14)), precision) == block


def test_a_lone_whole_tree_takes_the_widest_block():
    for precision in (MR_FP64, MR_FP32_MIXED):
        assert _block([W.random_smooth(14, W.EQ_BURGERS, seed=1, eps=0.0)], precision) == 1024
        assert _block([W.random_smooth(14, W.EQ_BURGERS, seed=1, eps=1e-4)], precision) == 512
        assert _block([W.random_smooth(10, W.EQ_BURGERS, seed=1, eps=0.0)], precision) == 512
