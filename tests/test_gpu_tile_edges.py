"""Tile edges of an FP64 grid leave no trace in the result: a velocity has the same bits in the tile that owns the
cell and in the rims of the tiles around it."""
import numpy as np
import pytest

from paper_1411_6697_gb300 import lbkm
from test_gpu_parity import mixed_2d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ux,uy", [(0.3, -0.17), (-0.041, 0.26)])
def test_a_uniform_fp64_flow_stays_uniform(ux, uy):
    params, _ = mixed_2d(65, 17)
    s = lbkm.Solver(nx=65, ny=17, precision=lbkm.F64, bc=(0, 0), dy=params["dx"],
                    **{k: params[k] for k in ("gamma", "orbit_kind", "orbit_speed", "orbit_eta", "S", "dx", "dt")})
    one = np.ones((17, 65))
    s.init_fields(1.07 * one, ux * one, uy * one, 0.93 * one, 0 * one)
    s.step(40)
    f = s.f_planes()
    s.close()
    assert np.all(f == f[:, :1, :1])
