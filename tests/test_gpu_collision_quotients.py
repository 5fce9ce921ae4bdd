"""The FP64 collision's quotients come from one reciprocal and, for a lattice
velocity that is no power of two, from its stored reciprocal: states at rest
(zero numerators), tiny and huge scales (which take the division) and relaxation
rates at and beside 1 against the oracle, 1e-12 of the largest population."""
import numpy as np
import pytest

from oracle_helpers import params_of
import oracle as O
from test_gpu_parity import gpu_state
from paper_2102_12163_gb300 import MR_FP64, MRLBM, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eq,lam", [(W.EQ_EULER, 3.0), (W.EQ_EULER, 4.0), (W.EQ_SW, 3.0), (W.EQ_SW_D1Q3, 2.0), (W.EQ_SW_D1Q5, 3.0),
                                    (W.EQ_BURGERS, 1.5)])
@pytest.mark.parametrize("s", [1.0, 1.25])
@pytest.mark.parametrize("scale,u", [(1.0, 0.0), (1.0, 0.1), (2.0 ** -420, 0.1), (2.0 ** 300, 0.1)])
def test_one_collision(eq, lam, s, scale, u):
    if eq not in (W.EQ_EULER,) and scale != 1.0:
        pytest.skip("gravity and Burgers' flux are not homogeneous of degree one")
    inst = W.random_smooth(7, eq, seed=5, eps=1e-3).with_(lam=lam, s=(s, s, s))
    rng = np.random.default_rng(3)
    n = 1 << inst.Jmax
    if inst.nf == 3:
        rho = 0.5 + rng.random(n)
        inst.m0 = scale * np.stack([rho, u * rng.standard_normal(n), 1.0 + rng.random(n)])
    elif inst.nf == 2:
        inst.m0 = np.stack([0.5 + rng.random(n), u * rng.standard_normal(n)])
    else:
        inst.m0 = u * rng.standard_normal((1, n))
    g = MRLBM(inst.with_(eps=0.0), precision=MR_FP64)
    g.set_initial()
    o = O.Oracle(params_of(inst.with_(eps=0.0)))
    R, vals, _ = gpu_state(g)
    o.set_state(R, vals)
    o.lbm_step()
    g.lbm_step()
    _, _, (lv, ix, f) = gpu_state(g)
    olv, oix, of = o.leaves()
    assert np.array_equal(ix, oix)
    assert np.max(np.abs(f - of)) <= 1e-12 * np.max(np.abs(of))
