"""One step of the kernels that form f_eq in fixed point, against the oracle from the same f, at the edges of
their tiles and of their number range; and every launch shape against the others, bit for bit.

Tolerance. FP32 storage rounds each value of f_eq's pair, the pair and the products of Eq. 17 (at most nine,
weights of sum below 4) to 2^-24 relative: 16 x 2^-24 of the largest value that the result is formed from.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fdlbm as O  # noqa: E402
from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402

PER, OUT, WALL = F.FDLBM_BC_PERIODIC, F.FDLBM_BC_OUTFLOW, F.FDLBM_BC_WALL
# name: scale of n, theta's range, |u|, lambda, tau / dt, dt / dx
STATES = {
    "rough": (1.0, (0.4, 3.0), 1.0, 2.0, 1.0, 0.01),         # f changes sign and class from node to node
    "relaxed": (1.0, (0.9, 1.1), 0.3, 2.0, 2.5, 0.01),       # the node's own value keeps 1 - dt/tau
    "viscous": (1.0, (0.4, 3.0), 1.0, 60.0, 1.0, 0.01),      # a switch of order one
    "large": (1e30, (0.9, 1.1), 0.3, 2.0, 1.0, 0.01),        # FP32 storage: weights beyond 2^40
    "small": (1e-25, (0.9, 1.1), 0.3, 2.0, 1.0, 0.01),       # ... below 2^-60
}
BCS = {"periodic": [PER] * 4, "mixed": [OUT, WALL, WALL, OUT]}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    F.lib()


def _step(nx, ny, state, bc, prec, variants):
    scale, (lo, hi), u, lam, tau, k = STATES[state]
    rng = np.random.default_rng(nx * 1000 + ny)
    m = [scale * rng.uniform(0.8, 1.2, (ny, nx)), u * rng.uniform(-1, 1, (ny, nx)), u * rng.uniform(-1, 1, (ny, nx)),
         rng.uniform(lo, hi, (ny, nx))]
    dt, dx = 1e-3, 1e-3 / k
    out, f0 = [], None
    for v in variants:
        s = F.Solver(nx, ny, dx, dx, dt, tau * dt, lam, BCS[bc], prec)
        s.set_variant(v)
        s.set_macro(*m)
        f0 = s.get_f()
        s.step(1)
        assert s.sync() == F.FDLBM_OK
        out.append(s.get_f())
        s.close()
    o = O.Sim(nx, ny, dx, dx, dt, tau * dt, lam, BCS[bc])
    o.set_f(f0)
    assert o.step(1) == 0
    return f0, out, o.get_f()


def _check(f0, out, ref):
    for g in out[1:]:
        assert np.array_equal(out[0], g)
    top = np.abs(np.concatenate([f0, ref])).max()
    assert np.abs(out[0] - ref).max() <= 16 * 2.0**-24 * top


FP32_SMALL, FP32_LARGE = (9, 8, 0, 2, 3, 5, 6, 12), (0, 1, 2, 4, 6, 7, 12)


@pytest.mark.parametrize("bc", sorted(BCS))
@pytest.mark.parametrize("nx,ny,state", [
    (2, 2, "rough"), (7, 3, "rough"), (9, 5, "large"), (33, 9, "small"), (31, 17, "rough"),
    (65, 33, "relaxed"), (37, 13, "viscous"),
])
def test_fp32_storage_step(nx, ny, state, bc):
    _check(*_step(nx, ny, state, bc, F.FDLBM_FP32_STORE, FP32_SMALL))


@pytest.mark.parametrize("nx,ny", [(300, 210), (129, 521)])
def test_fp32_storage_step_in_large_tiles(nx, ny):
    _check(*_step(nx, ny, "rough", "mixed", F.FDLBM_FP32_STORE, FP32_LARGE))
