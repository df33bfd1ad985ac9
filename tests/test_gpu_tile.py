"""The 2-D tile step (FP64 grids, FP32 grids of few tiles) and the marching FP32 step at the
sizes where either begins or its index rules change: single cells and columns, one cell more
or less than a tile, and on both sides of the line where FP32 grids change kernels (1000 tiles
of 32 x 4 cells, 400 with the double-float recovery). Tolerances are those of the parity tests
(1e-12 in FP64, 2e-5 in FP32 per plane)."""
import numpy as np
import pytest

from gpu_common import TOL, rel_l2
from paper_1411_6697_gb300 import lbkm
from test_gpu_parity import PID, PRECS, SIDES, WALLS, mixed_2d, start

pytestmark = pytest.mark.gpu


def check(nx, ny, prec, rec, bc, kind=None, steps=9):
    params, fields = mixed_2d(nx, ny, bc=(5, 5) if kind else bc, seed=nx)
    if kind:
        params["sides"], params["walls"] = SIDES[kind], WALLS
    s, ob, f, lam = start(params, fields, prec, rec, noise_seed=ny)
    s.step(steps)
    f_ref, lam_ref = ob.run(f, lam, steps)
    got = s.f_planes()
    for i in range(16):
        assert rel_l2(got[i], f_ref[i]) <= TOL[prec], ("f", i + 1, rel_l2(got[i], f_ref[i]))
    assert rel_l2(got[16], lam_ref) <= TOL[prec]


@pytest.mark.parametrize("prec,rec", PRECS, ids=PID)
@pytest.mark.parametrize("bc", [(0, 0), (1, 1), "inflow", "mixed"], ids=str)
@pytest.mark.parametrize("nx,ny", [(31, 5), (32, 8), (33, 9), (64, 4), (65, 17), (7, 130)])
def test_tile_step_parity(prec, rec, bc, nx, ny):
    check(nx, ny, prec, rec, bc, bc if isinstance(bc, str) else None)


@pytest.mark.parametrize("rec", [0, 1], ids=["f64", "df"])
@pytest.mark.parametrize("bc", [(0, 0), (1, 1), "inflow", "mixed"], ids=str)
@pytest.mark.parametrize("nx,ny", [(1000, 125), (1001, 127), (131, 845), (2111, 61)])
def test_fp32_step_parity_on_both_sides_of_the_line(rec, bc, nx, ny):
    check(nx, ny, lbkm.F32, rec, bc, bc if isinstance(bc, str) else None, steps=5)


@pytest.mark.parametrize("nx,ny", [(33, 9), (65, 17)])
def test_fp64_tile_records_leave_the_state_alone(nx, ny):
    params, fields = mixed_2d(nx, ny, seed=1)
    a, _, _, _ = start(params, fields, lbkm.F64, 0, noise_seed=1, tne_every=2, tne_capacity=8)
    b, _, _, _ = start(params, fields, lbkm.F64, 0, noise_seed=1)
    a.step(7)
    b.step(7)
    assert np.array_equal(a.f_planes(), b.f_planes())
    assert [r["step"] for r in a.tne_history()] == [0, 2, 4, 6]
