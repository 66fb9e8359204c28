"""Tiles that hold a y-periodic grid's whole height: they take the ghost rows' macros from the interior rows they copy, and
the 32 x 4 tile of FP64 storage converts a 4-row grid's rows once. The reference without either is the same state stacked
in y until it is taller than any tile: a periodic grid of several equal copies, in which every copy must step to the same
bits as the grid alone. FP64 storage runs its large tiles above 40960 sites only, so the long grids here lie above."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402

OUT, PER = F.FDLBM_BC_OUTFLOW, F.FDLBM_BC_PERIODIC


def _step(fields, prec, variant, steps):
    ny, nx = fields[0].shape
    s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, [OUT, OUT, PER, PER], prec)
    s.set_variant(variant)
    s.set_macro(*fields)
    s.step(steps)
    assert s.sync() == F.FDLBM_OK
    f = s.get_f()
    s.close()
    return f


def _check(nx, ny, prec, variants, tallest, steps=3):
    rng = np.random.default_rng(nx + ny)
    fields = [rng.uniform(0.8, 1.2, (ny, nx)), rng.uniform(-0.5, 0.5, (ny, nx)), rng.uniform(-0.5, 0.5, (ny, nx)),
              rng.uniform(0.5, 2.0, (ny, nx))]
    reps = tallest // ny + 1
    for v in variants:
        one = _step(fields, prec, v, steps)
        many = _step([np.tile(a, (reps, 1)) for a in fields], prec, v, steps)
        for r in range(reps):
            assert np.array_equal(one, many[:, r * ny:(r + 1) * ny, :]), (v, r)


@pytest.mark.parametrize("nx,ny", [(41003, 1), (20507, 2), (13667, 3), (10273, 4), (8231, 5), (5153, 8)])
def test_fp64_large_tiles(nx, ny):
    _check(nx, ny, F.FDLBM_FP64, (0, 1, 2), 8)


@pytest.mark.parametrize("nx,ny", [(61, 1), (70, 2), (133, 3), (90, 4)])
def test_fp64_small_tiles(nx, ny):
    _check(nx, ny, F.FDLBM_FP64, (9, 8, 13, 14), 4)


@pytest.mark.parametrize("nx,ny", [(70, 3), (133, 4), (90, 8), (64, 16), (33, 29)])
def test_fp32_storage_tiles(nx, ny):
    _check(nx, ny, F.FDLBM_FP32_STORE, (0, 1, 2, 3, 5, 6), 32)
