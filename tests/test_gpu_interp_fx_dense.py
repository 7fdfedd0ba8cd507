"""The tensor-core interpolation in the instances that only dense calls reach: few orders at p = 4, the
p = 2 and 6 stencils with one block of orders and with several; and that it is the kernel that runs.

Bound per sample: every product term carries at most 2 x 2^-54 of operand rounding and 2^-51.7 of
dropped digit products, relative to the cell's largest |F| = m, and e^{ik psi} a relative error of
k 2^-53 from psi in both: |err| <= 2 sum|w| m 2 K (2^-51 + 2 K 2^-53) plus the direct sum's own
rounding, below 16 (K + 1)^2 2^-53 sum|w| m, with sum|w| <= 3.2 (p = 6)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R, N = 31, 48


@pytest.mark.parametrize("p,K", [(4, 1), (4, 2), (4, 3), (2, 3), (2, 9), (2, 17), (6, 4), (6, 5), (6, 16), (6, 17), (4, 18)])
def test_dense_calls_match_the_direct_sum(p, K):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    from paper_2201_03478_gb300 import _lib
    from paper_2201_03478_gb300.binding import _ptr
    n, m = 100 * (R + 1) * N, 40000
    plan = sl.sidelobe_plan_create(max(K, 4), K, W.healpix_ring_theta(8), N, interp_order=p)
    rng = np.random.default_rng(K)
    cube = rng.standard_normal((R, N, K + 1)) + 1j * rng.standard_normal((R, N, K + 1))
    th, ph, ps = W.pointings_uniform(n, seed=p)
    maps, t = torch.from_numpy(cube).cuda(), [torch.from_numpy(a).cuda() for a in (th, ph, ps)]
    plan.enable_timing(True)
    got = sl.interp_tod(plan, maps, *t)
    plan.sync()
    st = plan.kernel_stats(reset=True)
    assert "interp_fx" in st and "interp_f64" not in st
    s, out = [a[:m].contiguous() for a in t], torch.empty(m, dtype=torch.float64, device="cuda")
    _lib.check(_lib.load().interp_tod_noalloc(plan.ptr, _ptr(maps), *(_ptr(a) for a in s), m, _ptr(out)))
    plan.sync()
    bound = 16.0 * (K + 1) ** 2 * 2.0 ** -53 * 3.2 * np.abs(np.concatenate([cube.real.ravel(), cube.imag.ravel()])).max()
    assert float((got[:m] - out).abs().max()) <= bound
