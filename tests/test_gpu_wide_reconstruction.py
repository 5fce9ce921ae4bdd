"""Reconstruction tables of the wide stencils (gamma = 2, 3) on random graded
trees, whose leaves lie next to refined cells on either side, near both copy
boundaries and on levels smaller than the window: one collide + stream against
the oracle, 1e-12 of the largest population."""
import numpy as np
import pytest

from oracle_helpers import params_of, random_graded_tree
import oracle as O
from test_gpu_parity import gpu_state
from paper_2102_12163_gb300 import MR_FP64, MRLBM, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("density", [0.02, 0.3])
@pytest.mark.parametrize("Jmin,Jmax", [(2, 4), (2, 9), (3, 11), (5, 8)])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_COPY], ids=["periodic", "copy"])
@pytest.mark.parametrize("gamma", [2, 3])
def test_one_step_on_a_random_tree(gamma, bc, Jmin, Jmax, density):
    rng = np.random.default_rng(1000 * gamma + 10 * Jmax + Jmin)
    inst = W.random_smooth(Jmax, W.EQ_SW, seed=9, Jmin=Jmin, bc=bc).with_(gamma=gamma)
    s = MRLBM(inst, precision=MR_FP64)
    s.set_initial()
    o = O.Oracle(params_of(inst))
    for trial in range(3):
        R = random_graded_tree(Jmin, Jmax, rng, density=density, bc=bc, gamma=gamma)
        base = O.equilibrium(params_of(inst), np.array([[1.0], [0.1]]))[:, :1]
        vals = base + 0.05 * rng.normal(size=(inst.q, o.S))
        s.set_state(0, R, vals)
        o.set_state(R, vals)
        o.lbm_step()
        s.lbm_step()
        _, _, (lv, ix, f) = gpu_state(s)
        _, _, of = o.leaves()
        assert np.max(np.abs(f - of)) <= 1e-12 * np.max(np.abs(of)), trial
