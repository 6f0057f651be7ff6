"""Fewer than 32 trajectories on the sliced-ELL stream are staged as float32: the
roofline names that kernel and counts its bytes."""
import pytest

import bench
import mqo_inputs as mi


@pytest.mark.parametrize("x_dtype,batch,f32", [("bf16", 8, True), ("f16", 16, True), ("f32", 32, True),
                                               ("f32", 4, True), ("bf16", 32, False), ("f16", 128, False)])
def test_float32_stream(x_dtype, batch, f32):
    plan = {"step_kernel": "smem_wide", "ell": True}
    assert bench.step_kernel_name(plan, x_dtype, batch) == ("mqo::k_step_f" if f32 else "mqo::k_step_s")
    assert bench.step_kernel_name(dict(plan, ell=False), x_dtype, batch) == "mqo::k_step_s"
    g = mi.erdos_renyi(100, 0.1, 1)
    size = 4 if x_dtype == "f32" else 2
    roof = bench.step_roofline(g, batch, size, size, 0.1, plan, "none", x_dtype, 6000.0, "measured", {"sm_mhz": 2000},
                               152, {})
    assert roof["algorithmic_bytes_per_launch"] == g.nnz * batch * (4 if f32 else size)
    assert roof["hbm"]["algorithmic_bytes_per_launch"] == bench.algorithmic_bytes_per_step(
        g, batch, size, size, 2 if f32 else 4)
