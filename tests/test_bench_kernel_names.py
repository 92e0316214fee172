"""Names of the kernels that a built plan's stages launch, as the benchmark reports
them: the rules of the library on its geometry."""
import pytest

import bench

PLAN = dict(n_pad=2048, kernel_width=7, tile=64, records=1, double_float=0)


@pytest.mark.parametrize("change,want", [
    (dict(), "spread_fixed_kernel<7, true, 2, 256>"),
    (dict(tile=32), "spread_fixed_kernel<7, true, 2, 256>"),
    (dict(kernel_width=13), "spread_fixed_kernel<16, false, 2, 256>"),
    (dict(tile=16), "spread_fixed_kernel<7, true, 2, 128>, spread_fixed_kernel<7, true, 2, 256> or "
                    "spread_private_kernel<float, 7, true>"),
])
def test_fp32_spreading(change, want):
    assert bench.kernel_of_stage("spread", dict(PLAN, **change), False) == want


@pytest.mark.parametrize("n_pad,tol,want", [(128, 1e-12, "dfc"), (128, 1e-6, "dfc"), (256, 9e-13, "double2"),
                                            (512, 1e-14, "dfc")])
def test_fp64_passes(n_pad, tol, want):
    info = dict(PLAN, n_pad=n_pad, kernel_width=13, tol=tol)
    lognp = n_pad.bit_length() - 1
    assert bench.kernel_of_stage("row_t1", info, True) == f"row_t1_kernel<{want}, {lognp}>"
    assert bench.kernel_of_stage("col_inv", info, True) == f"col_kernel<{want}, {lognp}, 1>"


def test_columns_of_the_largest_planes():
    info = dict(PLAN, n_pad=8192)
    for stage, mode in (("col_fwd_fold", 0), ("col_inv", 1), ("col_fwd", 2), ("col_inv_fold", 3)):
        assert bench.kernel_of_stage(stage, info, False) == f"col2_kernel<13, {mode}>"
