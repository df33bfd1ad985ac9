"""FP64 1-D steps whose windows of 32 cells are shared by four warps (short grids without
records), at the lengths where the number of steps per launch or the kernel changes. A run that
keeps records takes the kernel with one thread per cell; both do the same operations in the same
order, so their states must be equal bit for bit."""
import numpy as np
import pytest

from paper_1411_6697_gb300 import lbkm
from test_gpu_d2v24 import SIDES
from test_gpu_d2v24 import mixed_2d as mixed24
from test_gpu_d2v24 import start as start24
from test_gpu_line import ENDS
from test_gpu_parity import mixed_2d, start

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ends", sorted(ENDS))
@pytest.mark.parametrize("nx", [3, 28, 29, 400, 2432, 2433, 3648, 3649, 4256, 4257, 4864, 4865, 7297,
                                8512, 8513])
def test_line_split_same_bits(nx, ends):
    kw = dict(ENDS[ends])
    params, fields = mixed_2d(nx, 1, bc=kw.pop("bc"), seed=nx)
    params.update(kw)
    a, _, _, _ = start(params, fields, lbkm.F64, 0, noise_seed=5)
    b, _, _, _ = start(params, fields, lbkm.F64, 0, noise_seed=5, tne_every=64, tne_capacity=4)
    for n in (37, 1, 3):  # a replayed chunk of 32, and launches shorter than the plan's
        a.step(n)
        b.step(n)
    assert np.array_equal(a.f_planes(), b.f_planes())
    assert a.steps_taken == b.steps_taken == 41


def outcome(s):
    try:
        return s.f_planes()
    except lbkm.LbkmError as e:
        return e.code


@pytest.mark.parametrize("bc", [0, 1, 5])
@pytest.mark.parametrize("nx", [3, 28, 29, 2432, 2433, 3648, 3649, 12768, 12769])
def test_d2v24_split_same_bits(nx, bc):
    cfg = mixed24(nx, 1, bc=(bc, 0), seed=nx)
    if bc == 5:
        for key in ("params", "lib_params"):
            cfg[key]["sides"] = SIDES[:2] + [SIDES[1]] * 2
    a, _, _, _ = start24(cfg, lbkm.F64, noise_seed=5)
    b, _, _, _ = start24(cfg, lbkm.F64, noise_seed=5, tne_every=64, tne_capacity=4)
    a.step(7)
    b.step(7)
    assert np.array_equal(a.f_planes(), b.f_planes())
    for n in (30, 1, 3):
        a.step(n)
        b.step(n)
    # the run of 28 cells diverges between steps 15 and 37 (the oracle's too): both must say so
    assert np.array_equal(outcome(a), outcome(b))
