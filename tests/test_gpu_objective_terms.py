"""The TNE term of the objective alone is the gradient's: the same Delta, summed in another order. In a
uniform gas at rest Delta is nothing but rounding, so any other way of forming it gives another value.
Sums of n terms of one sign agree to n 2^-53: 96 cells, 12 moments and 20 steps, 2.6e-12."""
import numpy as np
import pytest

from paper_1411_6697_gb300 import lbkm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [0.93, 1.07, 1.31])
def test_rounding_level_delta_is_the_gradient_s(T):
    nx, steps = 96, 20
    s = lbkm.Solver(nx=nx, ny=1, precision=lbkm.F64, gamma=1.4, S=np.full(16, 3e4), T_ig=9.0, dx=1e-3, dy=1e-3,
                    dt=1e-5, bc=(0, 0))
    one = np.ones(nx)
    s.init_fields(1.13 * one, 0.21 * one, 0 * one, T * one, 0 * one)
    v = s.objective(one, steps, w_tne=1.0, checkpoint_every=8)
    g = s.grad(one, steps, w_tne=1.0, checkpoint_every=8)
    s.close()
    assert v["J_tne"] > 0.0
    assert abs(v["J_tne"] - g["J_tne"]) <= 2.6e-12 * g["J_tne"], (v["J_tne"], g["J_tne"])
