"""The reverse sweep's overlapping windows against the reverse-mode oracle: grids shorter than a
stencil, one cell more or less than a block's own cells, several blocks, both kinds of ends,
launches of fewer steps than the plan's. Tolerance 1e-9, that of the adjoint tests."""
import pytest

from test_gpu_adjoint import compare, gpu_grad, oracle_grad, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periodic", [False, True], ids=["zero-gradient", "periodic"])
@pytest.mark.parametrize("nx", [5, 6, 19, 28, 29, 60, 61, 121, 150])
def test_reverse_windows(nx, periodic):
    steps = 19
    c, p, m, rho_t = problem(nx, steps, omega1=2e3, driver=max(2, min(16, nx // 3)), periodic=periodic)
    r = oracle_grad(c, p, m, rho_t, steps, w_tne=1.0)
    for ck in (19, 7):
        g = gpu_grad(c, p, rho_t, steps, w_tne=1.0, ck=ck, bc=(0 if periodic else 1, 0))
        compare(g, r, 1e-9)
