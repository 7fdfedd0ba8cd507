"""The fixed-point interpolation is no further from extended precision (numpy's longdouble) than
the direct FP64 sum over the same stencil records (interp_tod_noalloc of an FP64 plan).

Both errors are relative L2 over the same samples; both are sums of some thousand independent
roundings of the same terms, so the comparison is allowed 5%."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L, R, N = 40, 40, 80


def _reference(p, rt, cube, th, ph, ps):
    q, h = np.longdouble, p // 2
    pi = np.arccos(q(-1))
    ext = np.concatenate([-rt[:h][::-1].astype(q), rt.astype(q), 2 * pi - rt[-h:][::-1].astype(q)])    # rows -h .. R + h - 1
    i = np.searchsorted(rt, th, side="right") - 1
    u = ph.astype(q) * N / (2 * pi)
    j = np.floor(u).astype(int)
    f, t = u - j, th.astype(q)
    wt, wp = [q(1)] * p, [q(1)] * p
    for a in range(p):
        for b in range(p):
            if b != a:
                na, nb = ext[i + 1 + a], ext[i + 1 + b]                # row i - h + 1 + a, at index + h
                wt[a] = wt[a] * (t - nb) / (na - nb)
                wp[a] = wp[a] * (f - (b - h + 1)) / q(a - b)
    out = np.zeros(th.size, dtype=q)
    for k in range(cube.shape[2]):
        re, im = np.zeros(th.size, dtype=q), np.zeros(th.size, dtype=q)
        for a in range(p):
            row = i - h + 1 + a
            ghost = (row < 0) | (row >= R)
            ring = np.where(row < 0, -1 - row, np.where(row >= R, 2 * R - 1 - row, row))
            for b in range(p):
                v = cube[ring, (j - h + 1 + b + ghost * (N // 2)) % N, k]
                w = wt[a] * wp[b] * np.where(ghost & (k % 2 == 1), -1, 1)
                re, im = re + w * v.real.astype(q), im + w * v.imag.astype(q)
        a = k * ps.astype(q)
        out += (2 * (np.cos(a) * re - np.sin(a) * im)) if k else re
    return out


@pytest.mark.parametrize("p,K", [(4, 5), (4, 16), (4, 32), (2, 8), (6, 8), (6, 20)])
def test_no_further_from_extended_precision_than_the_direct_sum(p, K):
    """The LFI-like sky and far-sidelobe beam on a small grid; dense calls.  Pooled over four of
    them: the fixed point's unit follows the power of two above the largest |F|, one to two times it."""
    import paper_2201_03478_gb300 as sl
    import workloads as W
    from paper_2201_03478_gb300 import _lib
    from paper_2201_03478_gb300.binding import _ptr
    rt, n, m = W.equiangular_ring_theta(R), 100 * R * N, 2000
    plan = sl.sidelobe_plan_create(L, K, rt, N, ncomp=3, interp_order=p)
    plan.enable_timing(True)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    e2 = np.zeros(2)
    for seed in range(4):
        th, ph, ps = W.pointings_uniform(n, seed=seed)
        maps, t = sl.synth_spin_maps(plan, d(W.sky_polarised(L, seed)), d(W.beam_far_sidelobe(L, K, seed + 1))), [d(a) for a in (th, ph, ps)]
        got = sl.interp_tod(plan, maps, *t).cpu().numpy()[:m]
        direct = torch.full((m,), float("nan"), dtype=torch.float64, device="cuda")
        s = [a[:m].contiguous() for a in t]
        _lib.check(_lib.load().interp_tod_noalloc(plan.ptr, _ptr(maps), *(_ptr(a) for a in s), m, _ptr(direct)))
        plan.sync()
        ref = _reference(p, rt, maps.cpu().numpy(), th[:m], ph[:m], ps[:m])
        e2 += [float(((x.astype(np.longdouble) - ref) ** 2).sum() / (ref ** 2).sum()) for x in (got, direct.cpu().numpy())]
    assert "interp_fx" in plan.kernel_stats()
    assert e2[0] <= 1.05 ** 2 * e2[1], np.sqrt(e2 / 4)


@pytest.mark.parametrize("p,K,n", [(4, 16, 300), (4, 16, 40000), (4, 24, 180000), (6, 8, 180000)])
@pytest.mark.parametrize("top", [1 - 2.0 ** -53, 1 - 2.0 ** -8, 1 - 2.0 ** -9, 1 - 2.0 ** -9 - 2.0 ** -30, 1 - 2.0 ** -12, 1.0, 1 + 2.0 ** -52])
def test_values_at_the_ends_of_the_digit_range(p, K, n, top):
    """Every |Re F| and |Im F| at the largest value, in phase with the sample: the sums reach their
    limits.  Bound: the fixed point's and the direct sum's terms, as in the comparison with it elsewhere:
    16 (K + 1)^2 2^-53 of the largest |F| at sum |w| <= 2."""
    import paper_2201_03478_gb300 as sl
    import workloads as W
    from paper_2201_03478_gb300 import _lib
    from paper_2201_03478_gb300.binding import _ptr
    rt = W.equiangular_ring_theta(R)
    plan = sl.sidelobe_plan_create(L, K, rt, N, interp_order=p)
    th, ph, ps = W.pointings_uniform(n, seed=3)
    ps = np.repeat(np.array([0.0, np.pi / 4, np.pi, -np.pi / 2]), (n + 3) // 4)[:n]
    k = np.arange(K + 1)
    a = 2 * np.pi * 7 * k / 64
    cube = np.where(np.cos(a + 0.1) >= 0, top, -top) + 1j * np.where(np.sin(a + 0.1) >= 0, -top, top)
    maps = torch.from_numpy(np.ascontiguousarray(np.broadcast_to(cube, (R, N, K + 1)))).cuda()
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (th, ph, np.where(np.arange(n) % 2, ps, a[1]))]
    got = sl.interp_tod(plan, maps, *t)
    for i in range(0, n, 1 << 18):
        s, out = [x[i:i + (1 << 18)].contiguous() for x in t], torch.empty(min(n - i, 1 << 18), dtype=torch.float64, device="cuda")
        _lib.check(_lib.load().interp_tod_noalloc(plan.ptr, _ptr(maps), *(_ptr(x) for x in s), out.numel(), _ptr(out)))
        plan.sync()
        assert float((got[i:i + out.numel()] - out).abs().max()) <= 16.0 * (K + 1) ** 2 * 2.0 ** -53 * 2.0 * top
