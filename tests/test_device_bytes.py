"""What a solve reserves: the split step's moment buffer only where a kernel reads it."""
import pytest

from paper_0801_4169_gb300 import fdlbm as F


def _bytes(nx, ny, prec):
    return F.fdlbm_device_bytes(F.make_config(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, (1, 1, 0, 0), prec))


def _base(nx, ny, size):
    plane = (nx + 4 + 31) // 32 * 32 * (ny + 4)
    up = lambda n: (n + 255) // 256 * 256  # noqa: E731
    return 2 * up(33 * plane * size) + 256 + up(4 * nx * ny * 8), up(plane * (32 + size))


@pytest.mark.parametrize("nx,ny", [(256, 256), (1000, 700), (16385, 4)])
def test_fp64_storage_holds_no_moment_buffer(nx, ny):
    assert _bytes(nx, ny, F.FDLBM_FP64) == _base(nx, ny, 8)[0]
    assert _bytes(nx, ny, F.FDLBM_FP64_STRICT) == sum(_base(nx, ny, 8))
    base, mom = _base(nx, ny, 4)
    assert _bytes(nx, ny, F.FDLBM_FP32_STORE) == base + (mom if nx * ny > 65536 else 0)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [F.FDLBM_FP64, F.FDLBM_FP32_STORE, F.FDLBM_FP64_STRICT])
def test_the_split_variants_are_taken_and_refused_as_before(prec):
    for nx, taken in ((256, prec == F.FDLBM_FP64_STRICT), (257, True)):
        s = F.Solver(nx, 256, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, (0, 0, 0, 0), prec)
        for v in (10, 11):
            if taken:
                s.set_variant(v)
            else:
                with pytest.raises(F.FdlbmError) as e:
                    s.set_variant(v)
                assert e.value.code == F.FDLBM_E_ARG
        s.close()
