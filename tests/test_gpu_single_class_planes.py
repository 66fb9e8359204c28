"""FP64 storage: a plane of one exponent class beside a plane of several, in the same ring and tile. Results of the first
are tiny beside its values (2^-17), and they stay sums of integers whatever the other plane holds: a shape whose tile holds
a value of another class, and one whose tile does not, give the same bits. A value of another class stands at one node of
each 32 x 8 tile, so that nearly all 4 x 4 tiles hold none; the moments are the same at every node."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402

SPEEDS = (1.0, 1.92, 2.99, 4.49)


def _velocities():
    a = np.arange(8) * np.pi / 4 + np.pi / 4  # direction i of a ring: 45 degrees first, then counter-clockwise
    v = [np.zeros(2)] + [s * np.array([np.cos(t), np.sin(t)]) for s in SPEEDS for t in a]
    return np.array(v)


def _state(nx, ny, ring):
    s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, (0, 0, 0, 0), F.FDLBM_FP64)
    y, x = np.mgrid[0:ny, 0:nx]
    s.set_macro(1 + 0.1 * np.sin(2 * np.pi * x / nx), 0.1 * np.cos(2 * np.pi * y / ny), np.full((ny, nx), 0.05),
                np.full((ny, nx), 0.9))
    f = s.get_f()
    s.close()
    big, first = 2.0 ** 14 * 1.5, 1 + 8 * ring
    f[first:first + 8] += big * np.array([1, -1] * 4)[:, None, None]  # no density, momentum or energy
    # at one node of a 32 x 8 tile, direction 2 of the ring becomes small; the other rings make up for its moments
    v = _velocities()
    rows = np.stack([np.ones(33), v[:, 0], v[:, 1], (v ** 2).sum(1)])
    rest = [q for q in range(33) if not first <= q < first + 8]
    fill = np.linalg.lstsq(rows[:, rest], rows[:, first + 2] * big, rcond=None)[0]
    f[first + 2, 5::8, 17::32] -= big
    f[rest, 5::8, 17::32] += fill[:, None, None]
    return f


def _step(f, ny, nx, variant):
    s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, (0, 0, 0, 0), F.FDLBM_FP64)
    s.set_variant(variant)
    s.set_f(f)
    s.step(1)
    assert s.sync() == F.FDLBM_OK
    out = s.get_f()
    s.close()
    return out


@pytest.mark.parametrize("ring", [0, 2])
def test_planes_of_one_class_do_not_depend_on_the_tile(ring):
    ny, nx = 203, 301
    f = _state(nx, ny, ring)
    small = _step(f, ny, nx, 9)
    plane = 1 + 8 * ring + 5
    assert np.abs(f[plane]).min() > 2.0 ** 14 and np.median(np.abs(small[plane])) < 1  # what the test is about
    for variant in (8, 0, 1, 2):
        out = _step(f, ny, nx, variant)
        assert np.array_equal(out, small), (variant, int((out != small).sum()))
