"""The bench's rooflines of the fixed-point and orbital kernels at the times measured for them: against
the pipe that binds each, a fraction that a pipe can have, and the one that ncu shows it busy."""
import types

import bench


def test_fixed_point_kernels_against_the_pipe_that_binds_them():
    plan = types.SimpleNamespace(sizes=lambda: {"lsteps": 6.63e9}, nalm=525825)
    r = bench.kernel_roofs({"lcontract_fx": (1, 28.1), "interp_fx": (1, 18.0)}, plan, "fp64", 1024, 16, 1024, 2048, 3, 10 ** 8,
                           {"fp64": None, "fp32": None})
    r.update(bench.adjoint_roofs({"interp_adj_fx": (1, 27.0), "lcontract_adj_fx": (1, 26.1)}, plan, 16, 10 ** 8, {}))
    busy = {"lcontract_fx": 0.66, "interp_fx": 0.46, "interp_adj_fx": 0.54, "lcontract_adj_fx": 0.66}   # ncu, profiles/
    for name, b in busy.items():
        assert r[name]["bound"] == "alu" and abs(r[name]["frac"] - b) <= 0.06, (name, r[name])


def test_orbital_kernels():
    # 1e8 samples, s = 20: 5,000,436 nodes in 0.357 ms, the samples in 0.681 ms
    assert 0.3 < bench.ORB_NODE_FLOPS * 5000436 / 0.357e-3 / 1e12 / bench.PEAK_FP64_TFLOPS < 0.9
    assert 0.5 < bench.ORB_SAMPLE_FLOPS * 1e8 / 0.681e-3 / 1e12 / bench.PEAK_FP64_TFLOPS < 0.9
    import numpy as np
    assert bench.orbital_bytes(np.array([0, 41, 61]), 61, 20)[0] == 8 * 61 + 32 * 4 + 24 * 19


def test_sweep_fractions():
    # lmax 4096, kmax 10: 2.5e11 steps; the FP64 plans' 1.0 s would be 2.2 of the FP64 peak, which their sums do not use
    assert bench.sweep_fraction("fp64", 2.5e11, 1009.0) is None and bench.sweep_fraction("df64", 2.5e11, 746.0) is None
    assert 0.0 < bench.sweep_fraction("fp32", 2.5e11, 69.2) < 0.79
