"""Data whose powers or quotients leave the exponent range although every moment
is in it: the populations of the initial state equal the plain IEEE evaluation
of the equilibria, infinities where it has them and no NaN where it has none."""
import numpy as np
import pytest

from oracle_helpers import params_of
import oracle as O
from paper_2102_12163_gb300 import MR_FP64, MRLBM, workloads as W

pytestmark = pytest.mark.gpu

# equilibrium, exponents of the conserved moments (None: zero)
DATA = [
    (W.EQ_EULER, (600, 300, 600)),    # rho^2 overflows
    (W.EQ_EULER, (520, None, 520)),   # the same at rest
    (W.EQ_EULER, (-520, None, -520)), # rho^2 underflows, at rest
    (W.EQ_EULER, (-540, -545, -530)),
    (W.EQ_EULER, (-300, 290, 0)),     # quotients near the top of the range
    (W.EQ_SW, (-400, 400)),           # (hu)^2 / h overflows
    (W.EQ_SW, (-480, 0)),
    (W.EQ_SW_D1Q3, (-400, 400)),
]


@pytest.mark.parametrize("lam", [2.0, 3.0])
@pytest.mark.parametrize("eq,exps", DATA)
def test_initial_state_at_the_ends_of_the_range(eq, exps, lam):
    rng = np.random.default_rng(11)
    inst = W.random_smooth(6, eq, seed=1, eps=0.0).with_(lam=lam)
    n = 1 << inst.Jmax
    inst.m0 = np.stack([np.zeros(n) if e is None else np.ldexp(1.0 + rng.random(n), e) for e in exps])
    s = MRLBM(inst, precision=MR_FP64)
    s.set_initial()
    _, ix, f = s.leaves()
    want = O.equilibrium(params_of(inst), inst.m0)[:, ix]
    if eq == W.EQ_SW_D1Q3:  # products with the inverse moment matrix may be fused
        assert np.array_equal(np.isfinite(f), np.isfinite(want)) and not np.isnan(f).any()
    else:
        assert np.array_equal(f, want, equal_nan=True)
