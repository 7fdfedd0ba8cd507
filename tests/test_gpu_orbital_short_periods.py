"""The orbital dipole in short pointing periods, alone and beside long ones: numbers of nodes around
1, 8 (a thread's rows), 64 (the scan's) and 256 (where eight warps take a period instead of one),
against the oracle.

Bound: every value is a sum of a few FP64 products of at most 4 max |y|, and the sweeps damp
their rounding by 0.268 a row: |difference| <= 64 x 2^-53 max |y|, both sides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHORT = (1, 2, 3, 4, 8, 9, 10, 11, 63, 64, 65, 66, 67, 254, 255, 256)


@pytest.mark.parametrize("nodes", [SHORT, SHORT + (257, 258, 259, 3000), (0, 0, 1), (5,) * 400, (257, 5000)])
@pytest.mark.parametrize("s", [2, 20])
def test_short_periods(nodes, s):
    import paper_2201_03478_gb300 as sl
    import workloads as W
    from oracle import orbital as orb
    cfg = W.config_small(n=10)
    plan = sl.sidelobe_plan_create(cfg["lmax"], cfg["kmax"], cfg["ring_theta"], cfg["nphi"])
    lens = [max(0, s * (m - 1) + 1 + r) if m else 0 for m in nodes for r in (0, s - 1)]
    n = int(sum(lens))
    th, ph, ps = W.pointings_scan(n, t0=99.0)
    starts = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    beta = np.random.default_rng(1).standard_normal((len(lens), 3)) * 1e-4
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = sl.orbital_dipole_tod(plan, d(cfg["beam"]), 2.7, 1.4, d(th), d(ph), d(ps), starts, beta, subsample=s).cpu().numpy()
    want = orb.dipole_subsampled(orb.moments(cfg["beam"][0]), 2.7, 1.4, th, ph, ps, starts, beta, s)
    assert np.abs(got - want).max() <= 128 * 2.0 ** -53 * np.abs(want).max()
