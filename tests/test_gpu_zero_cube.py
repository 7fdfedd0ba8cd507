"""A cube of zeros (the first step of a fit that starts from a zero sky) is interpolated at the
speed of any other, gives zeros, and zero cells next to others leave these as they are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _kernel_ms(plan, f, reps=8):
    f()
    plan.enable_timing(True)
    plan.kernel_stats(reset=True)
    for _ in range(reps):
        f()
    plan.sync()
    st = plan.kernel_stats(reset=True)
    plan.enable_timing(False)
    return sum(ms for k, (_, ms) in st.items() if k.startswith("interp")) / reps


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("K,p,n", [(16, 4, 3000000), (16, 4, 300000), (24, 4, 3000000), (8, 6, 3000000)])
def test_zero_cube_takes_no_longer(K, p, n, prec):
    """Twice the time where zero cells were summed directly; the same where they are not."""
    import paper_2201_03478_gb300 as sl
    import workloads as W
    R, N = 100, 200
    plan = sl.sidelobe_plan_create(K, K, W.equiangular_ring_theta(R), N, precision=prec, interp_order=p)
    g = torch.Generator(device="cuda").manual_seed(1)
    maps = torch.view_as_complex(torch.randn(R, N, K + 1, 2, dtype=torch.float64, device="cuda", generator=g))
    t = [torch.from_numpy(a).cuda() for a in W.pointings_uniform(n, seed=2)]
    full = _kernel_ms(plan, lambda: sl.interp_tod(plan, maps, *t))
    zero = torch.zeros_like(maps)
    out = sl.interp_tod(plan, zero, *t)
    assert not out.any()
    assert _kernel_ms(plan, lambda: sl.interp_tod(plan, zero, *t)) <= 1.4 * full


@pytest.mark.parametrize("n", [300, 60000, 400000])
def test_zero_region(n):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    K, R, N = 5, 40, 80
    plan = sl.sidelobe_plan_create(8, K, W.equiangular_ring_theta(R), N)
    g = torch.Generator(device="cuda").manual_seed(1)
    maps = torch.view_as_complex(torch.randn(R, N, K + 1, 2, dtype=torch.float64, device="cuda", generator=g))
    maps[:20] = 0
    maps[:10] *= -1.0                       # zeros of either sign
    t = [torch.from_numpy(a).cuda() for a in W.pointings_uniform(n, seed=2)]
    out = sl.interp_tod(plan, maps, *t).cpu().numpy()
    row = np.floor(t[0].cpu().numpy() * R / np.pi - 0.5)
    assert not out[(row >= 1) & (row <= 17)].any() and out[row >= 20].all()
