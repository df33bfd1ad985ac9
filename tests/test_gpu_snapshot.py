"""A state snapshot into device memory (one packing kernel; copies where the destination is not
aligned to an element) against the snapshot into host memory: the same bytes, for row lengths
that do and do not allow 16-byte vectors, grids of one row and of more rows than the launch has
blocks in a column, and destinations at every alignment; the bytes around it stay."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1411_6697_gb300 import lbkm
from test_gpu_d2v24 import mixed_2d as mixed24
from test_gpu_d2v24 import start as start24
from test_gpu_parity import mixed_2d, start

pytestmark = pytest.mark.gpu


def check(s):
    n = s.state_bytes()
    host = s.get_state()
    for off in (0, 1, 4, 8, 16):
        buf = torch.full((n + 32,), 171, dtype=torch.uint8, device="cuda")
        s._check(s._api.get_state(s._h, ctypes.c_void_p(buf.data_ptr() + off), 1))
        got = buf.cpu().numpy()
        assert np.array_equal(got[off:off + n], host)
        assert (got[:off] == 171).all() and (got[off + n:] == 171).all()
    assert np.array_equal(s.get_state(device=True).cpu().numpy(), host)


@pytest.mark.parametrize("prec", [lbkm.F64, lbkm.F32], ids=["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 1), (4100, 1), (37, 11), (64, 5), (8, 2048)])
def test_device_snapshot(prec, nx, ny):
    params, fields = mixed_2d(nx, ny, bc=(0, 0), seed=nx)
    s, _, _, _ = start(params, fields, prec, 0, noise_seed=1)
    s.step(3)
    check(s)


@pytest.mark.parametrize("prec", [lbkm.F64, lbkm.F32], ids=["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(33, 1), (33, 7)])
def test_device_snapshot_d2v24(prec, nx, ny):
    s, _, _, _ = start24(mixed24(nx, ny, seed=nx), prec, noise_seed=1)
    s.step(3)
    check(s)
