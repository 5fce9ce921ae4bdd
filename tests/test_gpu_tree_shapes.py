"""Level ranges at the edges of the bit arrays' words: one level, levels inside
one word, the coarsest level at and past a word, one word and many words per
level, every stencil width and both boundaries.  Lock-step against the oracle:
the tree bit for bit, the populations within 1e-12 of the largest."""
import numpy as np
import pytest

from oracle_helpers import params_of
import oracle as O
from test_gpu_parity import gpu_state
from paper_2102_12163_gb300 import MR_FP64, MRLBM, workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 1), (2, 3, 1), (3, 5, 1), (5, 5, 1), (2, 6, 1), (6, 7, 1), (6, 11, 1), (10, 12, 1), (11, 14, 1), (7, 15, 1),
          (2, 4, 2), (3, 6, 2), (6, 9, 2), (11, 13, 2), (3, 5, 3), (4, 8, 3), (7, 12, 3)]


@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_COPY], ids=["periodic", "copy"])
@pytest.mark.parametrize("Jmin,Jmax,gamma", SHAPES)
def test_lockstep_tree(Jmin, Jmax, gamma, bc):
    eq = W.EQ_BURGERS if Jmax > 12 else W.EQ_SW
    inst = W.random_smooth(Jmax, eq, seed=200 + 20 * Jmin + Jmax, Jmin=Jmin, eps=2e-3, bc=bc).with_(gamma=gamma)
    s = MRLBM(inst, precision=MR_FP64)
    s.set_initial()
    o = O.Oracle(params_of(inst))
    for n in range(4):
        R, vals, _ = gpu_state(s)
        o.set_state(R, vals)
        o.step()
        s.advance(1)
        R2, _, (lv, ix, f) = gpu_state(s)
        assert np.array_equal(R2, o.get_state()[0]), n
        olv, oix, of = o.leaves()
        assert np.array_equal(lv, olv) and np.array_equal(ix, oix)
        assert np.max(np.abs(f - of)) <= 1e-12 * np.max(np.abs(of))
