"""A constant state is its own reconstruction: the weights of every window sum
to one, so with the wide stencils (gamma = 2, 3) every leaf of every level keeps,
in a collide and stream, the value that the collision gives one cell, to the
last bit, next to refined cells and at both boundaries."""
import numpy as np
import pytest

from oracle_helpers import params_of, random_graded_tree
import oracle as O
from paper_2102_12163_gb300 import MR_FP32_MIXED, MR_FP64, MRLBM, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [MR_FP64, MR_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_COPY], ids=["periodic", "copy"])
@pytest.mark.parametrize("gamma", [2, 3])
@pytest.mark.parametrize("Jmin,Jmax", [(2, 5), (2, 10), (4, 14)])
def test_constant_state_stays_constant(gamma, bc, precision, Jmin, Jmax):
    rng = np.random.default_rng(17 * gamma + Jmax)
    inst = W.random_smooth(Jmax, W.EQ_SW, seed=9, Jmin=Jmin, bc=bc).with_(gamma=gamma)
    s = MRLBM(inst, precision=precision)
    s.set_initial()
    S = O.level_offsets(Jmin, Jmax)[Jmax + 1]
    for trial in range(4):
        R = random_graded_tree(Jmin, Jmax, rng, density=0.05, bc=bc, gamma=gamma)
        base = O.equilibrium(params_of(inst), np.array([[0.5 + rng.random()], [rng.random()]]))
        s.set_state(0, R, np.repeat(base, S, axis=1))
        s.lbm_step()
        lv, _, f = s.leaves()
        assert len(np.unique(lv)) > 1
        assert np.array_equal(f, np.repeat(f[:, :1], f.shape[1], axis=1)), trial
