"""The fixed-point contraction and its transpose in the form that takes 32 ring pairs a warp (two
groups of 16, from 9728 units on): ragged numbers of pairs, the second group full, partly filled and
empty.  The contraction against the oracle, the transpose by the adjoint identity.

Bounds.  Contraction: a' and b' rounded to 2^-53 each step, which a polar ring integrates twice over at
most L steps, relative L2 below L^2 2^-52.  Identity: both sides are sums of products whose terms
carry that, |difference| <= 4 L^2 2^-52 |A x| |y|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SLOTS = 152 * 4 * 4          # warps of one wave: SMs x CTAs x warps


def _units(L, K, R):
    return (L + 1) * (K + 1) * (((R + 1) // 2 + 31) // 32)


CASES = [(130, 40, 67), (130, 40, 97), (130, 40, 127), (120, 80, 32), (120, 80, 33), (99, 99, 24)]


def _setup(L, K, R, prec="fp64"):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    assert _units(L, K, R) >= 4 * SLOTS
    nphi = 8
    while nphi < 2 * L + 2:
        nphi *= 2
    plan = sl.sidelobe_plan_create(L, K, W.equiangular_ring_theta(R), nphi, precision=prec)
    sky = W.sky_gaussian(L, [np.ones(L + 1)], seed=1)
    rng = np.random.default_rng(2)
    beam = rng.standard_normal((1, K + 1, L + 1)) + 1j * rng.standard_normal((1, K + 1, L + 1))
    beam[:, 0] = beam[:, 0].real
    for k in range(K + 1):
        beam[:, k, :k] = 0
    return sl, plan, sky, beam, nphi


@pytest.mark.parametrize("L,K,R", CASES)
def test_contraction_matches_the_oracle(L, K, R):
    import oracle
    sl, plan, sky, beam, nphi = _setup(L, K, R)
    got = sl.synth_spin_maps(plan, torch.from_numpy(sky).cuda(), torch.from_numpy(beam).cuda()).cpu().numpy()
    ref = oracle.cube(sky, beam, plan.ring_theta, nphi)
    assert np.linalg.norm(got - ref) <= L * L * 2.0 ** -52 * np.linalg.norm(ref)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("L,K,R", CASES)
def test_adjoint_identity(L, K, R, prec):
    sl, plan, sky, beam, nphi = _setup(L, K, R, prec)
    fwd = plan if prec == "fp64" else sl.sidelobe_plan_create(L, K, plan.ring_theta, nphi)
    sky, beam = torch.from_numpy(sky).cuda(), torch.from_numpy(beam).cuda()
    g = torch.Generator(device="cuda").manual_seed(3)
    mb = torch.view_as_complex(torch.randn(R, nphi, K + 1, 2, dtype=torch.float64, device="cuda", generator=g))
    maps = sl.synth_spin_maps(fwd, sky, beam)
    gs, gb = sl.adjoint_synth(plan, mb, sky, beam)
    lhs = float((maps.conj() * mb).sum().real)
    tol = 4 * L * L * 2.0 ** -52 * float(torch.linalg.norm(maps)) * float(torch.linalg.norm(mb))
    assert abs(float((gs.conj() * sky).sum().real) - lhs) <= tol
    assert abs(float((gb.conj() * beam).sum().real) - lhs) <= tol
