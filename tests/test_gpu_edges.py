"""Edges of the launch rules and of the node update: block edges of the
two-lane FP64 conduction step, compared with the general path."""
import numpy as np
import pytest

from paper_1701_00702_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_1701_00702_gb300 import lbm as m
    return m


def twin(lbm, s, form=0):
    t = lbm.Solver(s.params).set_step_form(form)
    t.load(s.save())
    return t


@pytest.mark.parametrize("nx", [3, 15, 16, 17, 31, 32, 33, 47, 48, 49, 65, 200])
def test_conduction_lanes_beyond_the_grid(lbm, nx):
    """Widths whose last block has lanes beyond the grid: in the last node's warp,
    in the block's other warp (nx mod 32 from 1 to 16: a whole warp without a
    node, which may touch no history) and none.  Hundreds of steps, graph
    replays among them, equal those of one thread per node."""
    p = inputs.conduction_1d(nx, 37, wall_kind=[0, 0, 1, 1], wall_T=[1.0, 0.0, 0.4, 0.7], T_solidus=0.29,
                             T_liquidus=0.31, L_char=100.0)
    _, G, H, dT = inputs.random_state(nx, 37, 5, seed=nx, H_range=(0.0, 1.6))
    s = lbm.Solver(p)
    s.set_state(None, G, H, dT)
    t = twin(lbm, s)
    b = lbm.Batch([t], autotune=False).configure(128, 0)
    s.step(197)
    b.step(197)
    assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()
