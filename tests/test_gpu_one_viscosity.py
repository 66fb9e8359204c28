"""FP64 storage: a node's nu has one value for all its velocities, the integer weights' one. Two lambdas whose nu round to
the same integer give the same bits, the rest velocity's too: its five operations are in FP64, and with nu itself instead
of the rounded one it stepped with another viscosity than the moving velocities."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402


@pytest.mark.parametrize("variant", [9, 8, 0, 1, 2])
def test_velocities_share_the_rounded_viscosity(variant):
    nx, ny, u, dt_dx = 301, 203, 0.5, 0.01
    n = np.random.default_rng(5).uniform(0.5, 1.5, (ny, nx))
    ak = u * dt_dx
    out = []
    for part in (0.1, 0.4):  # of a unit of 2^-59 above a multiple of 2^-50: the units are 2^-55 to 2^-59
        nu = 137 * 2.0 ** -20 + part * 2.0 ** -59
        s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, nu / (0.5 * ak * (1 - ak)), (0, 0, 0, 0), F.FDLBM_FP64,
                     flags=F.FDLBM_SWITCH_CONST)
        s.set_variant(variant)
        s.set_macro(n, np.full((ny, nx), u), np.zeros((ny, nx)), np.ones((ny, nx)))
        s.step(1)
        assert s.sync() == F.FDLBM_OK
        out.append(s.get_f())
        s.close()
    assert np.array_equal(out[0][1:], out[1][1:])
    assert np.array_equal(out[0][0], out[1][0])
