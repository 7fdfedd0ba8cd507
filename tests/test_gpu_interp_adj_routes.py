"""Which kernel sums the transpose of the interpolation: on mid-sized grids and beyond four orders
the samples per occupied cell decide, in small and in large calls.  The one that does not run
returns at once."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,N,K,n,scan,fixed,prec", [
    (199, 200, 8, 159000, False, False, "fp64"),        # 4.5 per occupied cell
    (199, 200, 4, 318000, False, False, "fp64"),
    (199, 200, 16, 159000, True, True, "fp64"),         # a scan: hundreds
    (127, 128, 16, 65000, False, False, "fp64"),
    (127, 128, 8, 195000, False, True, "fp64"),
    (250, 256, 8, 100000, False, False, "fp64"),
    (300, 600, 24, 2160000, False, False, "fp64"),      # 12.4
    (300, 600, 8, 2520000, False, True, "fp64"),        # 14.4
    (199, 200, 16, 1050000, False, False, "df64"),      # 27
    (199, 200, 4, 318000, False, False, "df64"),
    (300, 600, 16, 5000000, False, True, "df64")])
def test_the_faster_kernel_runs(R, N, K, n, scan, fixed, prec):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    plan = sl.sidelobe_plan_create(max(K, 4), K, W.equiangular_ring_theta(R), N, precision=prec)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (W.pointings_scan(n, t0=3e6) if scan else W.pointings_uniform(n, seed=1))]
    y = torch.from_numpy(np.random.default_rng(2).standard_normal(n)).cuda()
    sl.adjoint_interp(plan, *t, y)
    plan.enable_timing(True)
    plan.kernel_stats(reset=True)
    for _ in range(5):
        sl.adjoint_interp(plan, *t, y)
    plan.sync()
    ms = {"fx": 0.0, "tiled": 0.0}
    for k, (_, v) in plan.kernel_stats(reset=True).items():
        if k.startswith("interp_adj"):
            ms["fx" if k == "interp_adj_fx" else "tiled"] += v
    assert (ms["fx"] > ms["tiled"]) == fixed, ms
