"""The 1-D step (several time steps per launch, blocks of overlapping windows) against the
FP64 oracle where its index rules change: grids shorter than a stencil, one cell more or less
than a block's own cells, several blocks, every kind of end. Tolerances are those of the
parity tests (1e-12 in FP64, 2e-5 in FP32 per plane; the records of an FP64 run to 1e-10 of
the largest entry)."""
import numpy as np
import pytest

from gpu_common import TOL, rel_l2
from oracle.oracle import unpack_tne
from paper_1411_6697_gb300 import lbkm
from test_gpu_parity import PID, PRECS, mixed_2d, start

pytestmark = pytest.mark.gpu

ENDS = {"periodic": dict(bc=(0, 0)), "zero-gradient": dict(bc=(1, 0)),
        "dirichlet": dict(bc=(5, 0), sides=((3, 1.05, 0.15, 0.0, 1.1, 0.2), (1, 1, 0, 0, 1, 0),
                                            (1, 1, 0, 0, 1, 0), (1, 1, 0, 0, 1, 0)))}


@pytest.mark.parametrize("prec,rec", PRECS, ids=PID)
@pytest.mark.parametrize("ends", sorted(ENDS))
@pytest.mark.parametrize("nx", [1, 2, 5, 31, 33, 64, 129, 1000, 5003])
def test_line_step_parity(prec, rec, ends, nx):
    kw = dict(ENDS[ends])
    params, fields = mixed_2d(nx, 1, bc=kw.pop("bc"), seed=nx)
    params.update(kw)
    steps = 43  # a replayed chunk of 32 steps and launches of fewer steps than the plan's
    s, ob, f, lam = start(params, fields, prec, rec, noise_seed=3, tne_every=3, tne_capacity=32)
    s.step(steps)
    plain, _, _, _ = start(params, fields, prec, rec, noise_seed=3)
    plain.step(steps)
    f_ref, lam_ref, tne_ref = ob.run(f, lam, steps, tne=True)
    got = s.f_planes()
    for i in range(16):
        assert rel_l2(got[i], f_ref[i]) <= TOL[prec], ("f", i + 1, rel_l2(got[i], f_ref[i]))
    assert rel_l2(got[16], lam_ref) <= TOL[prec]
    assert np.array_equal(got, plain.f_planes())  # records do not touch the state
    hist = s.tne_history()
    assert [r["step"] for r in hist] == list(range(0, steps, 3))
    if prec == lbkm.F64:
        for r in hist:
            ref = unpack_tne(tne_ref[r["step"]])
            for k in ("sum", "abs_sum", "min", "max", "d_sum", "d2_sum"):
                scale = np.abs(ref["abs_sum"]).max() if "sum" in k else np.abs(ref["max"]).max()
                assert np.abs(np.asarray(r[k]) - ref[k]).max() <= 1e-10 * scale, (k, r["step"])
