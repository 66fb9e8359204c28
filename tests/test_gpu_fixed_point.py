"""One step of the kernels that form f_eq (with FP64 storage, moments and stencils too) in fixed point, against the oracle from the same f, at the edges of
their tiles and of their number range; and every launch shape against the others, bit for bit.

Tolerance. FP32 storage rounds each value of f_eq's pair, the pair and the products of Eq. 17 (at most nine,
weights of sum below 4) to 2^-24 relative: 16 x 2^-24 of the largest value that the result is formed from.
FP64 storage: each side evaluates F_k's polynomial and a bracket with up to 16 roundings of its largest term, and
takes them from moments that carry 2^-53 kappa, kappa = sum|f| / n; Eq. 17 multiplies by weights. So 32 x 2^-53 W
(kappa max|f| + C), W a bound of the sum of a stencil's |weights|, C the largest sum of the terms' magnitudes.
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
    "smooth": (1.0, (1.0, 1.001), 0.1, 2.0, 1.0, 0.01),
    "hypersonic": (1.0, (60.0, 80.0), 19.0, 2.0, 1.0, 0.01),
    "stiff": (1.0, (0.4, 3.0), 1.0, 600.0, 1.0, 0.01),       # FP64 storage: nu above what the integer weights allow
    "coarse": (1.0, (0.9, 1.1), 0.3, 2.0, 1.0, 1.0),         # ... weights whose sum leaves them no room
    "huge": (1e250, (0.9, 1.1), 0.3, 2.0, 1.0, 0.01),        # ... exponents beyond the classes
    "tiny": (1e-250, (0.9, 1.1), 0.3, 2.0, 1.0, 0.01),
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
    if prec == F.FDLBM_FP32_STORE:
        return f0, out, o.get_f(), 16 * 2.0**-24 * np.abs(f0).max()
    n, T, uu = m[0], m[3], np.hypot(m[1], m[2])
    b, p, c = uu**2 / (2 * T), uu / T, 4.49 * k
    v2 = np.array([1.0, 1.92, 2.99, 4.49]) ** 2
    sums = np.zeros((5, ny, nx))
    for i in range(4):
        x, y, z = (v2[(i + j) % 4] for j in (1, 2, 3))
        Fk = (48 * T**4 + 6 * (x + y + z) * T**3 + (x * y + y * z + z * x) * T**2 + x * y * z / 4 * T) / abs(
            v2[i] * (v2[i] - x) * (v2[i] - y) * (v2[i] - z))
        q = np.sqrt(v2[i]) * p
        sums[i] = n * Fk * (1 + b + b * b / 2 + (1 + b) * (q + q * q / 2) + q**3 / 6 + q**4 / 24)
        sums[4] += 8 * n * Fk * (1 + b + b * b / 2)
    W = abs(1 - 1 / tau) + 2 * (c + c * c + c * abs(1 - c * c) / 3) + 8 * lam / 2 * u * k
    kappa = (np.abs(f0).sum(0) / f0.sum(0)).max()
    return f0, out, o.get_f(), 32 * 2.0**-53 * max(W, 1.0) * (kappa * np.abs(f0).max() + sums.max() + n.max())


def _check(f0, out, ref, tol):
    for g in out[1:]:
        assert np.array_equal(out[0], g)
    assert np.abs(out[0] - ref).max() <= tol


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


FP64_SMALL, FP64_LARGE = (9, 8, 0, 13, 14, 15), (0, 1, 2, 3, 9)


@pytest.mark.parametrize("bc", sorted(BCS))
@pytest.mark.parametrize("nx,ny,state", [
    (2, 2, "rough"), (4, 4, "hypersonic"), (5, 3, "rough"), (8, 4, "viscous"), (9, 5, "stiff"), (17, 9, "huge"),
    (33, 9, "rough"), (31, 7, "tiny"), (65, 13, "relaxed"), (40, 21, "coarse"), (64, 4, "smooth"),
])
def test_fp64_storage_step_in_small_tiles(nx, ny, state, bc):
    _check(*_step(nx, ny, state, bc, F.FDLBM_FP64, FP64_SMALL))


# above the size that the small tiles take: 32 x 4 and 32 x 8 against 8 x 4 and 4 x 4
@pytest.mark.parametrize("nx,ny,state,bc", [
    (321, 129, "rough", "mixed"), (127, 323, "rough", "periodic"), (10243, 4, "smooth", "periodic"),
    (13700, 3, "rough", "mixed"), (205, 201, "hypersonic", "mixed"), (205, 201, "stiff", "periodic"),
    (205, 201, "coarse", "mixed"), (161, 257, "huge", "periodic"), (161, 257, "relaxed", "mixed"),
])
def test_fp64_storage_step_in_large_tiles(nx, ny, state, bc):
    _check(*_step(nx, ny, state, bc, F.FDLBM_FP64, FP64_LARGE))
