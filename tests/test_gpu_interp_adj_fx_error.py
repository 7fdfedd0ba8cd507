"""Error of the fixed-point transpose of the interpolation against extended precision (numpy's
longdouble, at least 64 significant bits), on dense and sparse calls.

Bound, relative L2 of the adjoint cube.  A term y w_theta w_phi e^{ik psi} of the FP64 form carries
at most ten roundings of 2^-54 (four in each weight, the phase, the product), k 2^-53 from psi's
recurrence; terms of random sign keep the ratio in their sum; the FP64 additions of a node's some
20 partial sums add sqrt(20) 2^-54: 6 x 2^-53 + K 2^-53."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R, N = 31, 48


def _reference(K, rt, th, ph, ps, y):
    q = np.longdouble
    pi = np.arccos(q(-1))
    ext = np.concatenate([-rt[1::-1].astype(q), rt.astype(q), 2 * pi - rt[:-3:-1].astype(q)])    # rows -2 .. R + 1
    i = np.searchsorted(rt, th, side="right") - 1
    u = ph.astype(q) * N / (2 * pi)
    j = np.floor(u).astype(int)
    f, t = u - j, th.astype(q)
    wt, wp = [q(1)] * 4, [q(1)] * 4
    for a in range(4):
        for b in range(4):
            if b != a:
                na, nb = ext[i + 1 + a], ext[i + 1 + b]                # row i - 1 + a, at index + 2
                wt[a] = wt[a] * (t - nb) / (na - nb)
                wp[a] = wp[a] * (f - (b - 1)) / q(a - b)
    out = np.zeros((R * N, K + 1, 2), dtype=q)
    for k in range(K + 1):
        e = [(2 if k else 1) * y.astype(q) * g(k * ps.astype(q)) for g in (np.cos, np.sin)]
        for a in range(4):
            row = i - 1 + a
            ghost = (row < 0) | (row >= R)
            ring = np.where(row < 0, -1 - row, np.where(row >= R, 2 * R - 1 - row, row))
            for b in range(4):
                node = ring * N + (j - 1 + b + ghost * (N // 2)) % N
                w = wt[a] * wp[b] * np.where(ghost & (k % 2 == 1), -1, 1)
                np.add.at(out[:, k, 0], node, w * e[0])
                np.add.at(out[:, k, 1], node, -w * e[1])
    return out.reshape(R, N, K + 1, 2)


@pytest.mark.parametrize("K,n", [(0, 40000), (4, 40000), (7, 9000), (16, 3000)])
def test_error_is_that_of_fp64(K, n):
    import paper_2201_03478_gb300 as sl
    rng = np.random.default_rng(K)
    rt = np.pi * (np.arange(R) + 0.5) / R
    th, ph, ps = np.arccos(rng.uniform(-1, 1, n)), rng.uniform(0, 2 * np.pi, n), rng.uniform(0, 2 * np.pi, n)
    y = 1e-3 * rng.standard_normal(n)
    plan = sl.sidelobe_plan_create(max(K, 4), K, rt, N)
    plan.enable_timing(True)
    got = sl.adjoint_interp(plan, *(torch.from_numpy(a).cuda() for a in (th, ph, ps, y)))
    plan.sync()
    assert "interp_adj_fx" in plan.kernel_stats()
    ref = _reference(K, rt, th, ph, ps, y)
    err = np.stack([got.cpu().numpy().real, got.cpu().numpy().imag], -1).astype(np.longdouble) - ref
    rel = float(np.sqrt((err ** 2).sum() / (ref ** 2).sum()))
    assert rel <= (6 + K) * 2.0 ** -53, rel


def test_zero_weights_and_samples_add_nothing():
    """Samples on the nodes and samples of amplitude zero leave their neighbours at exactly zero."""
    import paper_2201_03478_gb300 as sl
    rt = np.pi * (np.arange(R) + 0.5) / R
    plan = sl.sidelobe_plan_create(8, 3, rt, N)
    y = np.tile([1.0, 0.0, -3.0], 40)
    th, ps = np.full(y.size, rt[10]), np.linspace(0, 6, y.size)
    got = sl.adjoint_interp(plan, *(torch.from_numpy(a).cuda() for a in (th, np.zeros(y.size), ps, y)))
    got = got.cpu().numpy()
    assert got[10, 0].any()
    got[10, 0] = 0
    assert not got.any()
