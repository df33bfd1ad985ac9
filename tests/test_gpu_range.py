"""Densities far from one. Without a reaction the model is linear in f, so a run whose density is
scaled by a power of two has the bits of the unscaled one, scaled, in every form of the FP64 step:
windows, short grids (four warps to a window), tiles, with records."""
import numpy as np
import pytest

from paper_1411_6697_gb300 import lbkm
from test_gpu_parity import mixed_2d

pytestmark = pytest.mark.gpu


def run(nx, ny, tne, scale, precision=lbkm.F64):
    params, fields = mixed_2d(nx, ny, bc=(1, 0), seed=nx, reactive=False)
    kw = {k: params[k] for k in ("gamma", "orbit_kind", "orbit_speed", "orbit_eta", "S", "dx", "dt")}
    s = lbkm.Solver(nx=nx, ny=ny, precision=precision, dy=params["dx"], bc=(1, 0), T_ig=1e3, tne_every=tne,
                    tne_capacity=8, **kw)
    s.init_fields(scale * fields["rho"], fields["ux"], fields["uy"], fields["T"], 0.0 * fields["lam"])
    s.step(9)
    f, h = s.f_planes(), s.tne_history()
    s.close()
    return f, [np.concatenate([np.ravel(r[k]) for k in ("sum", "abs_sum", "min", "max")]) for r in h]


@pytest.mark.parametrize("power", [-400, -127, 130, 400])
@pytest.mark.parametrize("nx,ny,tne", [(300, 1, 0), (300, 1, 2), (20000, 1, 0), (70, 37, 0), (70, 37, 2)])
def test_fp64_step_scales_with_the_density(nx, ny, tne, power):
    scale = 2.0 ** power
    f, h = run(nx, ny, tne, 1.0)
    g, hs = run(nx, ny, tne, scale)
    assert np.array_equal(g[:16], scale * f[:16])
    for a, b in zip(h, hs):
        assert np.array_equal(b, scale * a)


@pytest.mark.parametrize("power", [-85, -60, 60, 90])
@pytest.mark.parametrize("nx,ny", [(300, 1), (20000, 1), (70, 37), (700, 300)])
def test_fp32_step_scales_with_the_density(nx, ny, power):
    """Exact conserved sums at any density that leaves f and the sums' low parts (2^-24 of it) normal."""
    scale = 2.0 ** power
    f, _ = run(nx, ny, 0, 1.0, lbkm.F32)
    g, _ = run(nx, ny, 0, scale, lbkm.F32)
    assert np.array_equal(g[:16], np.float32(scale) * f[:16])
