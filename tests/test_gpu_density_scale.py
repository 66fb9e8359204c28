"""The step is linear in f, so with f times a power of 16 every result is the same number times that power, bit for
bit, as long as a node is computed in one and the same arithmetic at both scales. A state whose density leaves the
range that the fixed-point form takes is computed in the FP64 form instead, seven times slower, and its rounding differs.
Number densities (1e25 and more) and a tenuous gas are ordinary input."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0801_4169_gb300 import fdlbm as F  # noqa: E402

PER, OUT, WALL = F.FDLBM_BC_PERIODIC, F.FDLBM_BC_OUTFLOW, F.FDLBM_BC_WALL


def _state(nx, ny, seed):
    """Smooth waves with a jump of density and pressure in the middle."""
    rng = np.random.default_rng(seed)
    x, y = np.arange(nx)[None, :] / nx, np.arange(ny)[:, None] / ny
    w = [sum(a * np.sin(2 * np.pi * (k * x + m * y) + p) for k, m, a, p in
             zip(rng.integers(1, 4, 3), rng.integers(0, 3, 3), rng.uniform(0.01, 0.05, 3), rng.uniform(0, 6, 3)))
         for _ in range(4)]
    left = x < 0.5
    return [np.where(left, 1.0, 0.3) * (1 + w[0]), 0.2 + w[1], w[2], np.where(left, 1.1, 0.8) * (1 + w[3])]


def _run(nx, ny, bc, prec, variant, power, steps):
    s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, bc, prec)
    s.set_variant(variant)
    s.set_macro(*_state(nx, ny, nx + ny))
    s.set_f(np.ldexp(s.get_f(), power))
    s.step(steps)
    assert s.sync() == F.FDLBM_OK
    f = s.get_f()
    s.close()
    return np.ldexp(f, -power)


@pytest.mark.parametrize("power", [84, -84, 104])
@pytest.mark.parametrize("nx,ny,bc,variant", [(61, 9, [OUT, OUT, WALL, WALL], 9), (130, 4, [OUT, OUT, PER, PER], 0),
                                              (259, 171, [PER] * 4, 0), (11003, 4, [OUT, OUT, PER, PER], 2)])
def test_fp64_step_at_any_density(nx, ny, bc, variant, power):
    assert np.array_equal(_run(nx, ny, bc, F.FDLBM_FP64, variant, power, 3),
                          _run(nx, ny, bc, F.FDLBM_FP64, variant, 0, 3))


@pytest.mark.parametrize("power", [84, -72])
@pytest.mark.parametrize("nx,ny,bc,variant", [(61, 9, [OUT, OUT, WALL, WALL], 9), (131, 77, [PER] * 4, 6),
                                              (259, 171, [OUT] * 4, 12), (130, 4, [OUT, OUT, PER, PER], 2)])
def test_fp32_storage_step_at_any_density(nx, ny, bc, variant, power):
    assert np.array_equal(_run(nx, ny, bc, F.FDLBM_FP32_STORE, variant, power, 3),
                          _run(nx, ny, bc, F.FDLBM_FP32_STORE, variant, 0, 3))


@pytest.mark.parametrize("prec", [F.FDLBM_FP64, F.FDLBM_FP32_STORE])
def test_a_step_takes_as_long_at_any_density(prec):
    """FP32 storage rounds most of the forms' differences away, so its form shows in the time: 1.5 times the step at
    n ~ 1 was what all steps took in FP64 arithmetic, 2.4 the FP64 form out of line."""
    nx, ny, steps = 1024, 768, 10
    best = {}
    for power in (0, 84, -84):
        s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, [OUT] * 4, prec)
        m = _state(nx, ny, 5)
        s.set_macro(m[0] * 2.0**power, *m[1:])
        s.step(3)
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        for _ in range(5):
            a.record()
            s.step(steps)
            b.record()
            torch.cuda.synchronize()
            best[power] = min(best.get(power, np.inf), a.elapsed_time(b))
        s.close()
    assert max(best[84], best[-84]) <= 1.5 * best[0]


@pytest.mark.parametrize("power", [1004, 1008, 1012, -960])
@pytest.mark.parametrize("nx,ny,bc,variant", [(61, 9, [OUT, OUT, WALL, WALL], 9), (259, 171, [PER] * 4, 0)])
def test_fp64_step_near_the_ends_of_the_exponent_range(nx, ny, bc, variant, power):
    """The moments' integer sums carry 10^4 n and 10^4 sum |v|^2 f, which pass 2^1024 where n and its sums do not. There
    the step computes in FP64: three steps from sum|f| / n below 10 agree to 1000 x 2^-53 of the largest value each."""
    f = _run(nx, ny, bc, F.FDLBM_FP64, variant, 0, 3)
    g = _run(nx, ny, bc, F.FDLBM_FP64, variant, power, 3)
    assert np.abs(f - g).max() <= 3 * 1000 * 2.0**-53 * np.abs(f).max()
