"""bench.py counts the operations of the sweep kernel that runs, under its name."""
import types

import bench


def test_roofline_of_both_sweeps():
    p = types.SimpleNamespace(cells=1000, n_angles=10, nf=1)
    st = [{"sweep_ms": 2.0, "sweep_launches": 2}]
    rates = {"fp32_fma_flops": 1e12, "fp32x2_fma_flops": 2e12, "mufu_ex2_per_s": 1e12, "mufu_rcp_per_s": 5e11}
    upd = 1e4 / 1e-3
    s = bench.sweep_roofline(st, p, rates, True)
    # S-, I- bilinear (4 multiplies, 3 adds each), two differences, two fused products, J
    assert abs(s["achieved"] - (2 * 7 + 2 + 4 + 2) * upd / 1e12) < 1e-12
    assert abs(s["frac"] - s["achieved"] / 2) < 1e-12
    assert abs(s["weights_gbs"] - 8 * upd / 1e9) < 1e-9 and "mufu_frac" not in s
    q = bench.sweep_roofline(st, p, rates, False)
    assert abs(q["achieved"] - 34 * upd / 1e12) < 1e-12
    assert abs(q["mufu_frac"] - 2 * upd / 5e11) < 1e-12 and "weights_gbs" not in q
    plan = {"variant": 3}
    assert bench.sweep_kernel_name(plan, True) == "sc_sweep_stream_kernel<float>"
    assert bench.sweep_kernel_name(plan, False) == "sc_sweep_pipe_kernel<float>"
