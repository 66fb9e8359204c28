"""FP64 storage where the density spans many orders of magnitude within a tile, or from one node to the next: every value
of f_new against the oracle, relative to that node's own numbers, and all tile shapes against each other, bit for bit.

Tolerance, per value. Both sides evaluate r f_eq with up to 16 roundings of its terms' magnitudes C, from moments of the
node's own values (kappa = sum|f| / n), and Eq. 17 with up to 16 roundings of the sum S of its products' magnitudes:
32 x 2^-53 (S + kappa C) for the two. A sum of integers is taken where it has 2^45 units or more, or the node's density n
2^49; its nine products and r f_eq carry up to 2 units each: 20 x (2^-45 of the result + 2^-49 n).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fdlbm as O  # noqa: E402
from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402

PER, OUT = F.FDLBM_BC_PERIODIC, F.FDLBM_BC_OUTFLOW
SPEED = np.array([1.0, 1.92, 2.99, 4.49])
K, LAM = 0.01, 2.0


def _density(kind, nx, ny):
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    r2 = (x - 0.4 * nx) ** 2 + (y - 0.5 * ny) ** 2
    if kind == "blob":  # 2^73 from the middle of a tile to its edge
        return 1e-22 + np.exp(-r2 / 25.0)
    if kind == "cliff":  # 2^40 from one node to the next
        return np.where(x < nx // 2, 1.0, 2.0**-40) * (1 + 0 * y)
    if kind == "abyss":  # 2^70
        return np.where((x // 5 + y // 3) % 2 == 0, 1.0, 2.0**-70)
    rng = np.random.default_rng(nx)  # every node its own scale
    return 2.0 ** rng.uniform(-80, 0, (ny, nx))


def _near(a, dx, dy):
    return np.abs(a[:, 2 + dy:a.shape[1] - 2 + dy, 2 + dx:a.shape[2] - 2 + dx])


@pytest.mark.parametrize("nx,ny,variants", [(97, 13, (9, 8, 0, 13, 15)), (64, 4, (9, 0, 13)), (331, 129, (0, 1, 2, 3, 9, 14)),
                                            (10301, 4, (2, 0, 1, 8, 9))])
@pytest.mark.parametrize("flags", [0, F.FDLBM_NO_DISP])
@pytest.mark.parametrize("kind,tau", [("blob", 4.0), ("cliff", 1.0), ("abyss", 2.0), ("noise", 1.0)])
def test_each_node_keeps_its_own_precision(kind, tau, flags, nx, ny, variants):
    n = _density(kind, nx, ny)
    rng = np.random.default_rng(ny)
    u, v = rng.uniform(-0.3, 0.3, (2, ny, nx))
    T = rng.uniform(0.9, 1.1, (ny, nx))
    bc = [OUT, OUT, PER, PER]
    out = []
    for var in variants:
        s = F.Solver(nx, ny, 1e-3, 1e-3, K * 1e-3, tau * K * 1e-3, LAM, bc, F.FDLBM_FP64, flags)
        s.set_variant(var)
        s.set_macro(n, u, v, T)
        f0 = s.get_f()
        s.step(1)
        assert s.sync() == F.FDLBM_OK
        out.append(s.get_f())
        s.close()
    o = O.Sim(nx, ny, 1e-3, 1e-3, K * 1e-3, tau * K * 1e-3, LAM, bc, flags=flags)
    o.set_f(f0)
    pad = o.get_f_padded()
    assert o.step(1) == 0
    ref = o.get_f()
    for g in out[1:]:
        assert np.array_equal(out[0], g)

    vx, vy = O.velocities()
    b, p = (u * u + v * v) / (2 * T), np.hypot(u, v) / T
    C = np.zeros((33, ny, nx))
    v2 = SPEED**2
    for i in range(4):
        x, y, z = (v2[(i + j) % 4] for j in (1, 2, 3))
        Fk = (48 * T**4 + 6 * (x + y + z) * T**3 + (x * y + y * z + z * x) * T**2 + x * y * z / 4 * T) / abs(
            v2[i] * (v2[i] - x) * (v2[i] - y) * (v2[i] - z))
        q = SPEED[i] * p
        C[1 + 8 * i:9 + 8 * i] = n * Fk * (1 + b + b * b / 2 + (1 + b) * (q + q * q / 2) + q**3 / 6 + q**4 / 24)
        C[0] += 8 * n * Fk * (1 + b + b * b / 2)
    C[0] += n * (1 + b + b * b / 2)
    kappa = np.abs(f0).sum(0) / f0.sum(0)
    S = np.abs(f0) * (abs(1 - 1 / tau) + 4 * K**2 * v2[3] + 2 * LAM * 0.3 * K)
    nu = LAM / 2 * 0.3 * K
    for axis, vel in ((0, vx), (1, vy)):
        c = np.abs(vel)[:, None, None] * K
        d = 0 if flags & F.FDLBM_NO_DISP else c / 12
        for m in (-1, 1):
            S += (c / 2 + c * c / 2 + 2 * d + nu) * _near(pad, *((m, 0) if axis == 0 else (0, m)))
            S += d * _near(pad, *((2 * m, 0) if axis == 0 else (0, 2 * m)))
    tol = 32 * 2.0**-53 * (S + kappa * C) + 20 * (2.0**-45 * np.abs(ref) + 2.0**-49 * n)
    assert np.all(np.abs(out[0] - ref) <= tol), (np.abs(out[0] - ref) / tol).max()
