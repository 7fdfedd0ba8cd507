"""The fixed-point tensor-core interpolation of double-precision cubes against the
direct FP64 sum over the same stencil records (interp_tod_noalloc of an FP64 plan, whose
parity with the oracle test_zz_no_alloc and test_gpu_parity hold): edges of its 8-sample groups, 32-sample batches, 16-order blocks and 16-node
row tiles, and the cells and samples that take the direct sum.

Bound per sample.  Every product term carries at most 2 x 2^-54 of operand rounding
and 2^-51.7 of dropped digit products, relative to the cell's largest |F| = m, and
e^{ik psi} a relative error of k 2^-53 from psi in both:
|err| <= 2 sum|w| m 2 K (2^-51 + 2 K 2^-53) plus the direct sum's own rounding, below
16 (K + 1)^2 2^-53 sum|w| m, with sum|w| <= 2 at these grids.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R, NPHI = 31, 48


def _setup(K, p, prec, seed=0, scale=1.0):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    rt = W.healpix_ring_theta(8)
    plan = sl.sidelobe_plan_create(max(K, 4), K, rt, NPHI, precision=prec, interp_order=p)
    rng = np.random.default_rng(seed)
    cube = (rng.standard_normal((R, NPHI, K + 1)) + 1j * rng.standard_normal((R, NPHI, K + 1))) * scale
    return sl, plan, rt, cube, rng


def _run(sl, plan, cube, th, ph, ps):
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = sl.interp_tod(plan, d(cube), d(th), d(ph), d(ps))
    plan.sync()
    return out.cpu().numpy()


def _direct(sl, rt, cube, p, th, ph, ps):
    """The direct FP64 sum, in calls of at most 2^18 samples."""
    K = cube.shape[2] - 1
    plan = sl.sidelobe_plan_create(max(K, 4), K, rt, NPHI, precision="fp64", interp_order=p)
    from paper_2201_03478_gb300 import _lib
    from paper_2201_03478_gb300.binding import _ptr
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    maps, t = d(cube), [d(a) for a in (th, ph, ps)]
    tod = torch.full((len(th),), float("nan"), dtype=torch.float64, device="cuda")
    _lib.check(_lib.load().interp_tod_noalloc(plan.ptr, _ptr(maps), *(_ptr(a) for a in t), len(th), _ptr(tod)))
    plan.sync()
    return tod.cpu().numpy()


def _points(rng, n, ncells):
    """n samples in ncells cells (poles and the phi seam among them)."""
    t0 = np.concatenate([[1e-3, np.pi - 1e-3], np.arccos(rng.uniform(-1, 1, max(0, ncells - 2)))])[:ncells]
    p0 = np.concatenate([[0.0, 2 * np.pi - 1e-9], rng.uniform(0, 2 * np.pi, max(0, ncells - 2))])[:ncells]
    c = rng.integers(0, ncells, n)
    return (np.clip(t0[c] + 1e-4 * rng.standard_normal(n), 0, np.pi), np.mod(p0[c] + 1e-4 * rng.standard_normal(n), 2 * np.pi),
            rng.uniform(-20.0, 20.0, n))


def _bound(K, cube):
    return 16.0 * (K + 1) ** 2 * 2.0 ** -53 * 2.0 * np.abs(np.concatenate([cube.real.ravel(), cube.imag.ravel()])).max()


@pytest.mark.parametrize("K", [0, 1, 4, 7, 8, 9, 16])
@pytest.mark.parametrize("n,ncells", [(1, 1), (9, 1), (33, 2), (5000, 40), (12000, 11000), (50000, 30)])
def test_matches_the_direct_sum(K, n, ncells):
    """p = 4 and K <= 16: every call; groups, batches and both kernels (few, many samples per cell)."""
    sl, plan, rt, cube, rng = _setup(K, 4, "fp64")
    th, ph, ps = _points(rng, n, ncells)
    err = np.abs(_run(sl, plan, cube, th, ph, ps) - _direct(sl, rt, cube, 4, th, ph, ps))
    assert err.max() <= _bound(K, cube)


@pytest.mark.parametrize("p,K,prec,n", [(4, 17, "fp64", 80000), (4, 33, "fp64", 80000), (4, 128, "fp64", 80000),
                                        (2, 16, "fp64", 80000), (2, 20, "fp64", 80000), (6, 5, "fp64", 80000),
                                        (6, 20, "fp64", 80000), (4, 16, "df64", 20000)])
def test_dense_calls_match_the_direct_sum(p, K, prec, n):
    """Blocks of orders, row tiles and DF64 plans: from 48 (8) samples per grid cell on."""
    sl, plan, rt, cube, rng = _setup(K, p, prec)
    th, ph, ps = _points(rng, n, 300)
    err = np.abs(_run(sl, plan, cube, th, ph, ps) - _direct(sl, rt, cube, p, th, ph, ps))
    assert err.max() <= _bound(K, cube)


def test_values_do_not_depend_on_the_other_samples():
    """The few-samples and the many-samples kernel give the same bits: a sample's value is the
    same alone, among few and among many."""
    sl, plan, rt, cube, rng = _setup(16, 4, "fp64")
    th, ph, ps = _points(rng, 60000, 20000)
    whole = _run(sl, plan, cube, th, ph, ps)
    for m in (1, 2000, 11000):
        assert np.array_equal(_run(sl, plan, cube, th[:m], ph[:m], ps[:m]), whole[:m])
    rep = np.repeat(np.arange(3000), 20)
    assert np.array_equal(_run(sl, plan, cube, th[rep], ph[rep], ps[rep]), whole[rep])


@pytest.mark.parametrize("scale", [1e-300, 1e-200, 1e200])
def test_extreme_scales(scale):
    sl, plan, rt, cube, rng = _setup(5, 4, "fp64", scale=scale)
    th, ph, ps = _points(rng, 500, 9)
    err = np.abs(_run(sl, plan, cube, th, ph, ps) - _direct(sl, rt, cube, 4, th, ph, ps))
    assert err.max() <= _bound(5, cube)


def test_non_finite_values_stay_where_they_are():
    """An infinite or NaN node, a zero cube region and a NaN psi reach the same samples as the direct sum."""
    sl, plan, rt, cube, rng = _setup(6, 4, "fp64")
    cube[10, 7, 3] = np.nan
    cube[20, 30, 0] = np.inf
    cube[:6] = 0.0
    th, ph, ps = rng.uniform(0, np.pi, 20000), rng.uniform(0, 2 * np.pi, 20000), rng.uniform(0, 6, 20000)
    ps[::97] = np.nan
    got, ref = _run(sl, plan, cube, th, ph, ps), _direct(sl, rt, cube, 4, th, ph, ps)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    ok = np.isfinite(ref)
    assert np.abs(got[ok] - ref[ok]).max() <= _bound(6, cube[np.isfinite(cube)].reshape(-1))
