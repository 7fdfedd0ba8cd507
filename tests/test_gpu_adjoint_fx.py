"""The fixed-point contraction transpose at the edges of its 16-l steps, 64-l batches and
16- and 32-pair groups, by the adjoint identity against the forward contraction, and for
adjoint cubes that take the plain FP64 loop.

Bound.  <A x, y> and <x, A^T y> are sums of N products whose terms carry the recurrence's
L^2 2^-52 (as the forward test): |difference| <= 4 L^2 2^-52 |A x| |y| (L >= 8; both sides)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(L, K, R, prec, seed=0):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    nphi = 8
    while nphi < 2 * L + 2:
        nphi *= 2
    plan = sl.sidelobe_plan_create(L, K, W.equiangular_ring_theta(R), nphi, precision=prec)
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = lambda *s: torch.view_as_complex(torch.randn(*s, 2, dtype=torch.float64, device="cuda", generator=g))
    sky = torch.from_numpy(W.sky_gaussian(L, [np.ones(L + 1)], seed=seed)).cuda()
    beam = c(1, K + 1, L + 1)
    beam[:, 0] = beam[:, 0].real + 0j
    for k in range(K + 1):
        beam[:, k, :k] = 0
    return sl, plan, sky, beam, c(R, nphi, K + 1)


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("L,K,R", [(8, 2, 8), (15, 0, 9), (16, 3, 31), (63, 3, 32), (64, 5, 33), (65, 5, 64), (130, 2, 67), (40, 40, 20)])
def test_adjoint_identity(L, K, R, prec):
    sl, plan, sky, beam, mb = _setup(L, K, R, prec)
    fwd = sl.sidelobe_plan_create(L, K, plan.ring_theta, plan.nphi) if prec != "fp64" else plan
    maps = sl.synth_spin_maps(fwd, sky, beam)
    gs, gb = sl.adjoint_synth(plan, mb, sky, beam)
    lhs = float((maps.conj() * mb).sum().real)
    scale = float(torch.linalg.norm(maps)) * float(torch.linalg.norm(mb))
    assert abs(float((gs.conj() * sky).sum().real) - lhs) <= 4 * L * L * 2.0 ** -52 * scale
    assert abs(float((gb.conj() * beam).sum().real) - lhs) <= 4 * L * L * 2.0 ** -52 * scale


def test_scales_and_extremes():
    """A power of two only shifts the digits' scale (up to the order of the atomic additions);
    below 2^-959 the plain loop takes over; a NaN reaches the gradient; zeros give zeros."""
    sl, plan, sky, beam, mb = _setup(70, 3, 40, "fp64")
    one = sl.adjoint_synth(plan, mb, sky, beam)
    for n, tol in ((200, 1e-14), (-990, 4 * 70 * 70 * 2.0 ** -52)):
        got = sl.adjoint_synth(plan, mb * 2.0 ** n, sky, beam)
        for g, o in zip(got, one):
            assert float(torch.linalg.norm(g * 2.0 ** -n - o)) <= tol * float(torch.linalg.norm(o))
    assert all(float(g.abs().max()) == 0 for g in sl.adjoint_synth(plan, mb * 0, sky, beam))
    mb[3, 5, 1] = float("nan")
    assert torch.isnan(sl.adjoint_synth(plan, mb, sky, beam)[0].real).any()
