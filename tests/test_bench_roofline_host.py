"""The roofline that bench.py reports belongs to the kernel that runs: FP64 storage has small tiles on grids of up to
40960 sites, whatever the variant (no GPU)."""
import pytest

import bench


@pytest.mark.parametrize("variant", [2, 4, 5, 6, 7, 10, 11])
def test_fp64_instruction_count_is_the_large_tiles_alone(variant):
    assert bench.issue_roofline("fp64", variant, 40960, 1e9, 2070.0) is None
    assert bench.issue_roofline("fp64", variant, 40961, 1e9, 2070.0)["frac"] > 0


def test_kernel_names():
    for prec, variant, sites, name in (
            ("fp64", 2, 40960, "k_step_fx_small"), ("fp64", 2, 40961, "k_step_fx "), ("fp64", 9, 1 << 20, "k_step_fx_small"),
            ("fp64", 8, 1 << 20, "k_step_fx_small"), ("fp64", 11, 1 << 20, "k_step_fx "), ("fp64", 13, 1600, "k_persist"),
            ("fp64", 15, 1600, "small-grid steps"), ("fp64", 12, 1 << 20, "k_step_fx "), ("fp32", 12, 1 << 20, "k_step_tma"),
            ("fp32", 11, 1 << 20, "k_moments + k_update"), ("fp32", 2, 1600, "k_step "), ("fp32dw", 12, 1600, "k_step_tma"),
            ("fp32dw", 13, 1600, "k_step "), ("fneq32", 1, 1600, "k_step_fneq")):
        assert bench.step_kernel(prec, variant, sites).startswith(name), (prec, variant, sites)
