"""The spline of the orbital dipole at the edges of its rounds of 2048 rows, its threads' 8 rows
and the 8-thread scan (numbers of nodes around 1, 9, 65, 257, 2049 and 4097), and angles that the
fixed-point sine does not take, against the oracle.

Bound: every value is a sum of a few FP64 products of at most 4 max |y|, and the sweeps damp
their rounding by 0.268 a row: |difference| <= 64 x 2^-53 max |y|, both sides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s", [2, 5])
def test_rounds(s):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    from oracle import orbital as orb
    cfg = W.config_small(n=10)
    plan = sl.sidelobe_plan_create(cfg["lmax"], cfg["kmax"], cfg["ring_theta"], cfg["nphi"])
    lens = [s * (m - 1) + 1 + r for m in (1, 2, 3, 4, 9, 10, 11, 65, 66, 257, 258, 2049, 2050, 2051, 4097, 4098) for r in (0, s - 1)]
    n = int(sum(lens))
    th, ph, ps = W.pointings_scan(n, t0=99.0)
    ph, ps = ph.copy(), ps.copy()
    ph[::3] += 2 * np.pi * 100          # beyond 2^9
    ps[::5] -= 2 * np.pi * 7
    starts = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    beta = np.random.default_rng(1).standard_normal((len(lens), 3)) * 1e-4
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = sl.orbital_dipole_tod(plan, d(cfg["beam"]), 2.7, 1.4, d(th), d(ph), d(ps), starts, beta, subsample=s).cpu().numpy()
    want = orb.dipole_subsampled(orb.moments(cfg["beam"][0]), 2.7, 1.4, th, ph, ps, starts, beta, s)
    assert np.abs(got - want).max() <= 128 * 2.0 ** -53 * np.abs(want).max()
