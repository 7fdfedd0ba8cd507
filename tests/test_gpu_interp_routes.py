"""Which kernel sums a call of a double-precision cube: the sort's count of occupied cells decides
between the fixed-point sums and the others where the call's size alone does not tell.  The
kernels' values differ in their last bits, which shows the one that ran."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _plan(K, R, N, prec):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    return sl, sl.sidelobe_plan_create(max(K, 4), K, W.equiangular_ring_theta(R), N, precision=prec)


def _cube(K, R, N):
    g = torch.Generator(device="cuda").manual_seed(1)
    return torch.view_as_complex(torch.randn(R, N, K + 1, 2, dtype=torch.float64, device="cuda", generator=g))


def _points(n, ncells, seed=3):
    """n samples, uniform (ncells = 0) or around ncells points."""
    import workloads as W
    th, ph, ps = W.pointings_uniform(n, seed=seed)
    if ncells:
        rng = np.random.default_rng(seed)
        c = rng.integers(0, ncells, n)
        th, ph = th[:ncells][c] + 1e-9 * rng.random(n), ph[:ncells][c]
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (np.clip(th, 0, np.pi), ph, ps)]


@pytest.mark.parametrize("K,n,ncells,fixed", [(13, 40000, 0, False), (16, 40000, 0, False), (13, 40000, 200, True), (16, 40000, 200, True),
                                              (16, 130000, 0, True), (16, 20000, 0, False), (12, 400000, 0, False)])
def test_df64_by_samples_per_occupied_cell(K, n, ncells, fixed):
    """3280 cells.  Fixed point gives the bits of an FP64 plan's; the double-float sums do not."""
    sl, plan = _plan(K, 40, 80, "df64")
    ref = sl.sidelobe_plan_create(max(K, 4), K, plan.ring_theta, 80)
    maps, t = _cube(K, 40, 80), _points(n, ncells)
    got, want = sl.interp_tod(plan, maps, *t), sl.interp_tod(ref, maps, *t)
    assert torch.equal(got, want) == fixed
    assert float((got - want).abs().max()) <= 1e-11 * float(want.abs().max())


@pytest.mark.parametrize("K,n", [(4, 20480), (8, 20480)])
def test_values_across_the_switch_by_size(K, n):
    """One sample more takes another kernel: same values to rounding (both forms' bound of the direct
    comparison, 16 (K + 1)^2 2^-53 of the largest |F| at sum |w| <= 2); on the same side, same bits."""
    sl, plan = _plan(K, 200, 400, "fp64")
    maps, t = _cube(K, 200, 400), _points(n + 1, 0)
    more = sl.interp_tod(plan, maps, *t)
    few = sl.interp_tod(plan, maps, *(a[:n].contiguous() for a in t))
    less = sl.interp_tod(plan, maps, *(a[:n - 7000].contiguous() for a in t))
    top = float(torch.view_as_real(maps).abs().max())
    assert not torch.equal(more[:n], few)
    assert float((more[:n] - few).abs().max()) <= 16.0 * (K + 1) ** 2 * 2.0 ** -53 * 2.0 * top
    assert torch.equal(few[:n - 7000], less)


@pytest.mark.parametrize("n", [300, 30000, 400000])
def test_eleven_to_sixteen_orders_have_one_value(n):
    """FP64, four-point stencil: the same bits in calls of any size."""
    sl, plan = _plan(12, 200, 400, "fp64")
    maps, t = _cube(12, 200, 400), _points(500000, 0)
    whole = sl.interp_tod(plan, maps, *t)
    assert torch.equal(sl.interp_tod(plan, maps, *(a[:n].contiguous() for a in t)), whole[:n])
