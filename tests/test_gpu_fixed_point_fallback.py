"""Nodes that the fixed-point step of FP64 storage leaves to its FP64 form: nu above what the integer weights allow,
weights that do not fit them, projections |u| / theta beyond 2^10. Their results are checked against the oracle in
test_gpu_fixed_point.py; here, that a grid full of them stays within 2.5 times the fixed-point step. That is 1.75 times
what every step took in FP64 arithmetic; with f_eq and the weights formed again for each direction it was 5.7."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402


def _time(lam, tau, theta):
    nx, ny = 1024, 768
    rng = np.random.default_rng(1)
    s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, tau * 1e-5, lam, [F.FDLBM_BC_OUTFLOW] * 4, F.FDLBM_FP64)
    s.set_macro(rng.uniform(0.8, 1.2, (ny, nx)), rng.uniform(-1, 1, (ny, nx)), rng.uniform(-1, 1, (ny, nx)),
                rng.uniform(*theta, (ny, nx)))
    f, best = s.get_f(), np.inf
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for _ in range(8):
        s.set_f(f)
        a.record()
        s.step(1)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    s.close()
    return best


@pytest.mark.parametrize("lam,tau,theta", [(600.0, 1.0, (0.4, 3.0)), (2.0, 0.1, (0.4, 3.0)), (2.0, 1.0, (5e-4, 6e-4))])
def test_a_grid_in_the_fp64_form_is_not_much_slower(lam, tau, theta):
    assert _time(lam, tau, theta) <= 2.5 * _time(2.0, 1.0, (0.4, 3.0))
