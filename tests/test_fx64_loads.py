"""The loads of the FP64-storage step (csrc/fdlbm_fx64.cuh). Its launches are programmatically dependent: a step's
blocks are resident while the step before writes the values they will read, and the read-only path (__ldg) is
defined only for data that nobody writes while a kernel runs. So every load of f goes through ldf."""
import os
import re

import numpy as np
import pytest

from paper_0801_4169_gb300 import fdlbm as F

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_0801_4169_gb300", "csrc")


def test_no_read_only_load_is_named_in_the_dependent_step():
    with open(os.path.join(CSRC, "fdlbm_fx64.cuh")) as fh:
        code = re.sub(r"//[^\n]*", "", fh.read())
    # the loads of fdlbm_kernels.cuh that may take the read-only path, and what is built on them
    found = re.findall(r"\b(__ldg|ldc|ld|node_moments|node_macro|quad_macro|moment_slot|stencil_dir)\s*[<(]", code)
    assert found == []


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [9, 0, 2])
@pytest.mark.parametrize("bad", [np.inf, np.nan, -np.inf])
def test_a_non_finite_value_is_reported_by_the_step_that_reads_it(variant, bad):
    nx, ny = 257, 161
    s = F.Solver(nx, ny, 1e-3, 1e-3, 1e-5, 1e-5, 2.0, (0, 0, 0, 0), F.FDLBM_FP64)
    s.set_variant(variant)
    s.set_macro(*[np.full((ny, nx), a) for a in (1.0, 0.2, -0.1, 0.8)])
    s.step(6)  # dependent launches in flight before the value appears
    assert s.sync() == F.FDLBM_OK
    f = s.get_f()
    f[11, 77, 130] = bad
    s.set_f(f)
    s.step(1)
    assert F.fdlbm_health(s.h) & F.FDLBM_HEALTH_NUMERIC
    with pytest.raises(F.FdlbmError) as e:
        s.sync()
    assert e.value.code == F.FDLBM_E_NUMERIC
    s.close()
