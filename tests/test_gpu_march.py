"""The marching FP32 step on wide grids, whose inner strips touch no x side: per-side
conditions at odd and even heights against the FP64 oracle (2e-5 per plane, the tolerance of
the parity tests)."""
import pytest

from gpu_common import TOL, rel_l2
from paper_1411_6697_gb300 import lbkm
from test_gpu_parity import SIDES, WALLS, mixed_2d, start

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rec", [0, 1], ids=["f64", "df"])
@pytest.mark.parametrize("kind", sorted(SIDES))
@pytest.mark.parametrize("nx,ny", [(1000, 125), (1030, 130), (2111, 61)])
def test_inner_strips_take_the_y_sides(nx, ny, kind, rec):
    """At an odd height the second ghost row above the grid shares its row pair with a row that
    is not needed; a Dirichlet lid has to fill it there too."""
    params, fields = mixed_2d(nx, ny, bc=(5, 5), seed=nx)
    params["sides"], params["walls"] = SIDES[kind], WALLS
    s, ob, f, lam = start(params, fields, lbkm.F32, rec, noise_seed=ny)
    s.step(5)
    f_ref, lam_ref = ob.run(f, lam, 5)
    got = s.f_planes()
    for i in range(16):
        assert rel_l2(got[i], f_ref[i]) <= TOL[lbkm.F32], ("f", i + 1, rel_l2(got[i], f_ref[i]))
    assert rel_l2(got[16], lam_ref) <= TOL[lbkm.F32]
