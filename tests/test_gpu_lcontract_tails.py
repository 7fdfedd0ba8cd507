"""The fixed-point contraction where sky x beam leaves the normal range: the tail of a Gaussian beam,
which passes through the smallest doubles to zero, and products that are all below 2^-959.  They
stay on the tensor cores (the plain FP64 loop, which such a tail had sent whole units to, took five times as
long), so a tail too small to count changes no bit.

Bound of the scaled sums: the recurrence's, L^2 2^-52 (test_gpu_lcontract_fx.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(L, K, R, seed=5):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    nphi = 8
    while nphi < 2 * L + 2:
        nphi *= 2
    plan = sl.sidelobe_plan_create(L, K, W.equiangular_ring_theta(R), nphi)
    rng = np.random.default_rng(seed)
    beam = rng.standard_normal((1, K + 1, L + 1)) + 1j * rng.standard_normal((1, K + 1, L + 1))
    beam[:, 0] = beam[:, 0].real
    for k in range(K + 1):
        beam[:, k, :k] = 0
    sky = W.sky_gaussian(L, [np.ones(L + 1)], seed=seed)
    return lambda b: sl.synth_spin_maps(plan, torch.from_numpy(sky).cuda(), torch.from_numpy(b).cuda()), beam


@pytest.mark.parametrize("L,K,R,sigma", [(130, 4, 40, 3.0), (200, 8, 67, 4.0), (130, 40, 97, 3.0)])
def test_a_tail_too_small_to_count_changes_no_bit(L, K, R, sigma):
    cube, beam = _setup(L, K, R)
    beam = beam * np.exp(-0.5 * (np.arange(L + 1) / sigma) ** 2)
    cut = np.where(np.abs(beam) < 1e-250, 0, beam)
    assert np.any((beam != cut) & (np.abs(beam) < 2.0 ** -1000)) and np.any(beam[..., -1] == 0)
    a, b = torch.view_as_real(cube(beam)), torch.view_as_real(cube(cut))
    sees = b.abs() > 1e-200
    assert float(sees.double().mean()) > 0.5
    assert torch.equal(a[sees], b[sees])


@pytest.mark.parametrize("L,K,R", [(63, 3, 24), (130, 40, 97)])
@pytest.mark.parametrize("e", [-962, -980, -1000])
def test_products_below_the_scales(L, K, R, e):
    cube, beam = _setup(L, K, R)
    want = cube(beam)
    got = torch.view_as_complex(torch.view_as_real(cube(beam * 2.0 ** e)) * 2.0 ** 500 * 2.0 ** (-e - 500))
    # results below 2^-1022 are rounded to 2^-1074: (e + 1074) bits after the point
    floor = 2.0 ** (-1074 - e) * np.sqrt(want.numel()) * 4 * L
    assert float(torch.linalg.norm(got - want)) <= L * L * 2.0 ** -52 * float(torch.linalg.norm(want)) + floor


@pytest.mark.parametrize("L,K,R", [(130, 3, 40), (130, 40, 97)])
def test_a_tail_behind_large_sums(L, K, R):
    """From 2^460 to zero within a unit: sums that 2^600 would carry past the largest double."""
    cube, beam = _setup(L, K, R)
    beam = beam * np.exp2(np.maximum(460.0 - 16.0 * np.arange(L + 1), -1100.0))
    a, b = (torch.view_as_real(cube(v)) for v in (beam, np.where(np.abs(beam) < 1e-250, 0, beam)))
    assert bool(torch.isfinite(a).all())
    a, b = a * 2.0 ** -400, b * 2.0 ** -400
    assert float(torch.linalg.norm(a - b)) <= L * L * 2.0 ** -52 * float(torch.linalg.norm(b))
