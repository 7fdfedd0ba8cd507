"""The fixed-point contraction of FP64 plans against the oracle at the edges of its 64-l
batches, 8-l steps, 16- and 32-pair groups, and for the inputs that take the plain FP64 loop.

Bound.  The cube's error is that of the recurrence: a' and b' rounded to 2^-53 each step, which
a polar ring integrates twice over at most L steps: relative L2 below L^2 2^-52 (3.8e-12 at
L = 130)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(L, K, R, ncomp=1, seed=0):
    import workloads as W
    rng = np.random.default_rng(seed)
    rt = W.equiangular_ring_theta(R)
    sky = W.sky_gaussian(L, [np.ones(L + 1)] * ncomp, seed=seed)
    beam = rng.standard_normal((ncomp, K + 1, L + 1)) + 1j * rng.standard_normal((ncomp, K + 1, L + 1))
    beam[:, 0] = beam[:, 0].real
    for k in range(K + 1):
        beam[:, k, :k] = 0
    nphi = 8
    while nphi < 2 * L + 2:
        nphi *= 2
    return rt, sky, beam, nphi


def _cube(L, K, rt, nphi, sky, beam):
    import paper_2201_03478_gb300 as sl
    plan = sl.sidelobe_plan_create(L, K, rt, nphi, ncomp=sky.shape[0])
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = sl.synth_spin_maps(plan, d(sky), d(beam))
    plan.sync()
    return out.cpu().numpy()


@pytest.mark.parametrize("L,K,R,ncomp", [(1, 1, 4, 1), (7, 2, 8, 3), (8, 0, 9, 1), (63, 3, 31, 1), (64, 5, 33, 1),
                                         (65, 5, 64, 3), (130, 2, 67, 1), (40, 40, 20, 1)])
def test_cube_matches_the_oracle(L, K, R, ncomp):
    import oracle
    rt, sky, beam, nphi = _case(L, K, R, ncomp)
    ref = oracle.cube(sky, beam, rt, nphi)
    got = _cube(L, K, rt, nphi, sky, beam)
    assert np.linalg.norm(got - ref) <= L * L * 2.0 ** -52 * np.linalg.norm(ref) + 4e-16 * np.linalg.norm(ref)


def test_powers_of_two_scale_exactly_and_extremes_agree():
    """Scaling the sky by 2^n only shifts the digits' scale; beyond its range (V below 2^-959)
    the plain loop takes over."""
    rt, sky, beam, nphi = _case(70, 3, 40)
    one = _cube(70, 3, rt, nphi, sky, beam)
    for n in (-200, 300):
        assert np.array_equal(_cube(70, 3, rt, nphi, sky * 2.0 ** n, beam), one * 2.0 ** n)
    tiny = _cube(70, 3, rt, nphi, sky * 2.0 ** -980, beam) * 2.0 ** 980
    assert np.linalg.norm(tiny - one) <= 70 * 70 * 2.0 ** -52 * np.linalg.norm(one)


def test_non_finite_sky_reaches_its_own_order_only():
    """A NaN at (l, m) = (30, 5): every map value sums over all m, so every ring whose recurrence
    reaches l = 30 is NaN, and the FP64 oracle-side count of finite values is none."""
    rt, sky, beam, nphi = _case(40, 1, 20)
    sky[0, 5 * (2 * 40 + 1 - 5) // 2 + 30] = np.nan
    got = _cube(40, 1, rt, nphi, sky, beam)
    assert not np.isfinite(got).any()
