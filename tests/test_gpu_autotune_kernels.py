"""FP64 storage runs several variants with one kernel: the autotuner times each kernel once and keeps the first of its
variants, where timed apart the order of equals was noise."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402


def _solver(nx, ny, **kw):
    s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, (0, 0, 0, 0), F.FDLBM_FP64, **kw)
    s.set_macro(*[np.full((ny, nx), a) for a in (1.0, 0.2, -0.1, 0.8)])
    return s


@pytest.mark.parametrize("nx,ny,groups", [
    (160, 100, [(0, 1, 2, 3, 4, 5, 6, 7, 8, 12), (9,), (13,), (14,), (15,)]),
    (211, 197, [(0,), (1, 12), (2, 4, 5, 6, 7), (3, 8), (9,), (13,), (14,), (15,)]),  # no split variants up to 65536 sites
    (311, 307, [(0,), (1, 12), (2, 4, 5, 6, 7, 10, 11), (3, 8), (9,), (13,), (14,), (15,)])])
def test_each_kernel_of_a_solve_is_timed_once(nx, ny, groups):
    s = _solver(nx, ny)
    times = s.autotune(2)
    best = F.fdlbm_get_variant(s.h)
    s.close()
    for g in groups:
        assert times[g[0]] > 0 and len({times[v] for v in g}) == 1
    assert best == min((times[g[0]], g[0]) for g in groups)[1]


def test_each_kernel_of_a_batch_is_timed_once():
    members = [_solver(nx, 4) for nx in (700, 901)]
    b = F.fdlbm_batch_create()
    for s in members:
        F.fdlbm_batch_add(b, s.h)
    times = F.fdlbm_batch_autotune(b, 2)
    F.fdlbm_batch_destroy(b)
    for s in members:
        s.close()
    assert times[0] > 0 and times[1] > 0 and len(set(times[1:8])) == 1
