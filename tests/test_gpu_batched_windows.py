"""The batched step's windows (64 or 128 cells carried through two time steps, 8 cells of them
shared with the neighbours) at their edges: instances shorter than a stencil, one group of cells
more or less than a window's own cells, and step counts that leave a last pass of one step.
Tolerance: the FP32 parity tests' 2e-5 per plane."""
import numpy as np
import pytest

import lbkm_inputs as li
from gpu_common import make_oracle, rel_l2
from test_gpu_batched import make_batched, split

pytestmark = pytest.mark.gpu

NX = [4, 8, 52, 56, 60, 64, 112, 116, 120, 124, 128, 236, 240, 244, 480, 484]


@pytest.mark.parametrize("recovery", [0, 1], ids=["f64rec", "df32"])
@pytest.mark.parametrize("steps", [1, 2, 5, 33])
def test_batched_windows(recovery, steps):
    inst = []
    for i, nx in enumerate(NX):
        S = np.full(16, 1e5)
        S[4:7] = 1e4 * (1 + 0.02 * i)
        inst.append(li.detonation(nx=nx, steps=steps, driver=max(1, nx // 8), Q=1 + 0.01 * i,
                                  S=S, ripple=1e-2))
    cfg = dict(instances=inst, nx=NX, S=[d["params"]["S"] for d in inst],
               Q=[d["params"]["Q"] for d in inst])
    s = make_batched(cfg, recovery)
    s.step(steps)
    assert s.steps_taken == steps
    planes = split(s.f_planes(), NX)
    for i, d in enumerate(inst):
        ob, fl = make_oracle(d["params"]), d["fields"]
        f0 = ob.init(fl["rho"], fl["ux"], fl["uy"], fl["T"]).astype(np.float32).astype(np.float64)
        f, lam = ob.run(f0, fl["lam"], steps)
        assert rel_l2(planes[i][:16], f) <= 2e-5, NX[i]
        assert rel_l2(planes[i][16], lam) <= 2e-5, NX[i]
