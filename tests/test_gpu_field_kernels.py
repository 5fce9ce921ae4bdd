"""The whole-field kernels against the oracle: the reconstruction of deep
instances by runs of 512 finest cells (1e-12 of each moment), and the decisions
of the initial state dropped when a step comes before the first adaptation (the
trees bit for bit), with the bit arrays in shared and in global memory."""
import numpy as np
import pytest

from oracle_helpers import oracle_of, params_of
import oracle as O
from test_gpu_parity import assert_finest_close, gpu_state
from paper_2102_12163_gb300 import MR_FP64, MRLBM, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eq,gamma,bc", [(W.EQ_EULER, 1, W.BC_PERIODIC), (W.EQ_EULER, 3, W.BC_COPY), (W.EQ_SW, 2, W.BC_PERIODIC),
                                         (W.EQ_SW_D1Q5, 1, W.BC_COPY)])
def test_finest_of_a_deep_instance(eq, gamma, bc):
    inst = W.random_smooth(17, eq, seed=31, eps=1e-3, bc=bc).with_(gamma=gamma)
    s = MRLBM(inst, precision=MR_FP64)
    s.set_initial()
    s.advance(3)
    R, vals, (lv, _, _) = gpu_state(s)
    assert lv.min() < 12  # most of the finest level is predicted
    o = O.Oracle(params_of(inst))
    o.set_state(R, vals)
    assert_finest_close(s.finest(), o.finest_moments())


# Jmax 17 beside another instance: its bit arrays exceed a batch's share of shared memory
@pytest.mark.parametrize("depths", [(10,), (15,), (17, 8)])
def test_step_before_the_first_adaptation(depths):
    insts = [W.random_smooth(J, W.EQ_BURGERS, seed=40 + J, eps=1e-3) for J in depths]
    s = MRLBM(insts, precision=MR_FP64)
    s.set_initial()
    s.lbm_step()
    s.advance(2)
    for i, inst in enumerate(insts):
        o = oracle_of(inst)
        o.lbm_step()
        o.step(2)
        R, _, (lv, ix, f) = gpu_state(s, i)
        assert np.array_equal(R, o.get_state()[0])
        _, _, of = o.leaves()
        assert np.max(np.abs(f - of)) <= 1e-12 * np.max(np.abs(of))
