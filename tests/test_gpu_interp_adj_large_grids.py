"""Which kernel sums the transpose of the interpolation on grids of a million cells and more: the
samples per occupied cell from which the fixed-point form is the faster one lie lower there.  The one that
does not run returns at once; both give the same cube to rounding (FP64: both within 2^-44 of the sum of |y| at
a node's scale; the cube's norm here)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,N,K,per_cell,fixed,prec", [
    (724, 1500, 8, 4, False, "fp64"), (724, 1500, 4, 6, True, "fp64"), (724, 1500, 2, 6, False, "fp64"), (724, 1500, 2, 8, True, "fp64"),
    (1024, 2048, 16, 6, True, "fp64"), (1024, 2048, 1, 9, False, "fp64"), (724, 1500, 8, 9, False, "df64"),
    (724, 1500, 8, 14, True, "df64"), (724, 1500, 2, 20, False, "df64")])
def test_the_faster_kernel_runs(R, N, K, per_cell, fixed, prec):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    plan = sl.sidelobe_plan_create(max(K, 4), K, W.equiangular_ring_theta(R), N, precision=prec)
    n = per_cell * (R + 1) * N
    g = torch.Generator(device="cuda").manual_seed(1)
    u = torch.rand(4, n, dtype=torch.float64, device="cuda", generator=g)
    t = [torch.acos(1 - 2 * u[0]), 2 * np.pi * u[1], 2 * np.pi * u[2]]
    y = u[3] - 0.5
    plan.enable_timing(True)
    plan.kernel_stats(reset=True)
    whole = sl.adjoint_interp(plan, *t, y)
    plan.sync()
    ms = {"fx": 0.0, "tiled": 0.0}
    for k, (_, v) in plan.kernel_stats(reset=True).items():
        if k.startswith("interp_adj"):
            ms["fx" if k == "interp_adj_fx" else "tiled"] += v
    assert (ms["fx"] > ms["tiled"]) == fixed, ms
    # in small calls, which take other routes
    parts = torch.zeros_like(whole)
    for a in range(0, n, n // 2 + 1):
        b = min(n, a + n // 2 + 1)
        parts += sl.adjoint_interp(plan, *(v[a:b].contiguous() for v in t), y[a:b].contiguous())
    tol = 2.0 ** -44 if prec == "fp64" else 1e-11
    assert float(torch.linalg.norm(whole - parts)) <= tol * float(torch.linalg.norm(whole))
