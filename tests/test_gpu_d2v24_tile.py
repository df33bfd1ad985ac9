"""The D2V24 step's tiles (32 x 8 cells in FP32, 32 x 4 in FP64, 32 cells in 1-D) at their edges:
one cell more or less than a tile, ragged last rows and columns, every kind of side. Tolerances
are those of the D2V24 parity tests (1e-12 in FP64; 4e-5 in FP32, whose Dirichlet ghost states
are rounded to FP32)."""
import numpy as np
import pytest

from paper_1411_6697_gb300 import lbkm
from test_gpu_d2v24 import PID, PRECS, SIDES, check_state, mixed_2d, start

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", PRECS, ids=PID)
@pytest.mark.parametrize("bc", [(0, 0), (1, 1), (5, 5)], ids=str)
@pytest.mark.parametrize("nx,ny", [(31, 9), (32, 8), (33, 7), (64, 17), (97, 4), (65, 1), (96, 1)])
def test_tile_edges(prec, bc, nx, ny):
    cfg = mixed_2d(nx, ny, bc=bc if ny > 1 else (bc[0], 0), seed=nx)
    if bc == (5, 5):
        for key in ("params", "lib_params"):
            cfg[key]["sides"] = SIDES if ny > 1 else SIDES[:2] + [SIDES[1]] * 2
    s, ob, f, lam = start(cfg, prec, noise_seed=ny)
    s.step(7)
    f_ref, lam_ref = ob.run(f, lam, 7)
    check_state(s, ob, f_ref, lam_ref, prec, floor=0.0 if prec == lbkm.F64 else 4e-5)


@pytest.mark.parametrize("prec", PRECS, ids=PID)
@pytest.mark.parametrize("nx,ny", [(33, 9), (97, 1)])
def test_records_leave_the_state_alone(prec, nx, ny):
    cfg = mixed_2d(nx, ny, seed=2)
    a, _, _, _ = start(cfg, prec, noise_seed=1, tne_every=2, tne_capacity=8)
    b, _, _, _ = start(cfg, prec, noise_seed=1)
    a.step(7)
    b.step(7)
    assert np.array_equal(a.f_planes(), b.f_planes())
    assert [r["step"] for r in a.tne_history()] == [0, 2, 4, 6]
