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
