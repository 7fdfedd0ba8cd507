"""The work that a user of this library has it do, as measurable cases.

Each case is one call (or one training step) through the package's public entry
points with the inputs, plan or batch that a program keeps beside it:

    forward    convolve_tod: cube and TOD of one detector
    interp     interp_tod: the TOD of a stretch of pointings on a kept cube
    adjoint    adjoint_tod: gradients of <tod, c> with respect to sky and beam
    gradient   sidelobe_tod and its backward pass (autograd), one least-squares step
    multisky   synth_spin_maps_multi: one cube per sky of a posterior sample set
    batch      sl_batch_run: the forward operator of several detectors, one graph
    orbital    orbital_dipole_tod: orbital dipole and quadrupole, 4 pi beam

Inputs are seeded and made on the GPU: Gaussian skies with C_l = (l+1)^-2 (EE and
BB at 5% and 1% of TT), beams falling as (l+1)^-1.5 ("sidelobe") or as a Gaussian
in l and 0.5^k ("taper"), pointings of a 1 rpm satellite scan at 32.5 Hz or uniform
on the rotation group.  ``exact`` evaluates the same operator in plain 64-bit torch.
"""
import math

import numpy as np
import torch

import paper_2201_03478_gb300 as sl

TWO_PI = 2.0 * math.pi


# ------------------------------------------------------------------ the cases
def _case(name, kind, precision, lmax, kmax, ncomp, nrings, nphi, n, beam="sidelobe", grid="equiangular",
          pointing="scan", order=4, count=0):
    c = dict(kind=kind, precision=precision, lmax=lmax, kmax=kmax, ncomp=ncomp, nrings=nrings, nphi=nphi, n=n,
             beam=beam, grid=grid, pointing=pointing, order=order, count=count)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a unit-test sized call: launches and latency are all there is
        _case("small_1k_fp64", "forward", "fp64", 64, 4, 1, 127, 128, 1000, "taper", "healpix", "uniform"),
        # a coarse model on rings of 2 3 5^3 points, an odd number of rings, six-point interpolation
        _case("ragged_p6_fp32", "forward", "fp32", 300, 7, 1, 301, 750, 333331, "sidelobe", "equiangular", "uniform", 6),
        # one pointing period (55 minutes at 32.5 Hz) on a kept cube
        _case("period_interp_fp64", "interp", "fp64", 1024, 16, 3, 1024, 2048, 107251),
        # the headline workload in each accuracy class
        _case("lfi_forward_fp64", "forward", "fp64", 1024, 16, 3, 1024, 2048, 100000000),
        _case("lfi_forward_fp32", "forward", "fp32", 1024, 16, 3, 1024, 2048, 100000000),
        _case("lfi_forward_df64", "forward", "df64", 1024, 16, 3, 1024, 2048, 20000000),
        # the differentiation workload: many uniform pointings on the small grid
        _case("small_adjoint_fp64", "adjoint", "fp64", 64, 4, 1, 127, 128, 10000000, "taper", "healpix", "uniform"),
        # one step of a fit of sky and beam to a day or two of data
        _case("lfi_gradient_fp64", "gradient", "fp64", 1024, 16, 3, 1024, 2048, 5000000),
        # the high-resolution variant
        _case("highres_forward_fp32", "forward", "fp32", 2048, 32, 1, 2048, 4096, 20000000, "taper", "equiangular",
              "uniform"),
        # one beam over the skies of a posterior sample set
        _case("multisky_16_fp32", "multisky", "fp32", 512, 16, 3, 512, 1024, 0, count=16),
        # a focal plane of uneven detectors in one graph (count detectors; lmax and kmax are the largest)
        _case("detectors_6_fp32", "batch", "fp32", 1500, 24, 3, 1500, 3000, 2000000, count=6),
        # the orbital dipole of two weeks of data, rotation at every 20th sample
        _case("orbital_40m", "orbital", "fp64", 1024, 16, 3, 1024, 2048, 40000000),
    ]


def _smooth_even(x):
    """The smallest even 2^a 3^b 5^c >= x."""
    q = max(8, int(x) + (int(x) & 1))
    while True:
        r = q
        for f in (2, 3, 5):
            while r % f == 0:
                r //= f
        if r == 1:
            return q
        q += 2


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward"] * 5 + ["interp"] * 2 + ["adjoint", "gradient", "multisky", "batch", "orbital"])
    prec = rng.choice(["fp64", "fp64", "fp32", "fp32", "df64"])
    if kind in ("multisky", "batch"):
        prec = "fp32"
    if kind == "orbital":
        return _case("", kind, "fp64", _log_int(rng, 48, 300), 2 + rng.randrange(8), rng.choice([1, 3]), 128, 256,
                     _log_int(rng, 1000, 60000000))
    if kind == "multisky":
        lmax, kmax = _log_int(rng, 48, 512), rng.randrange(0, 13)
        return _case("", kind, prec, lmax, kmax, rng.choice([1, 3]), lmax + rng.randrange(0, 9), _smooth_even(2 * lmax + 2),
                     0, count=rng.randrange(2, 21))
    if kind == "batch":
        return _case("", kind, prec, rng.choice([300, 500, 768]), rng.choice([5, 8, 12]), rng.choice([1, 3]), 512, 1024,
                     _log_int(rng, 20000, 2000000), count=rng.randrange(2, 8))
    lmax = _log_int(rng, 48, 2048 if prec == "fp32" and kind in ("forward", "interp") else 800)
    kmax = min(lmax, rng.choice([0, 1, 2, 4, 5, 8, 11, 16, 16, 23, 32]))
    if lmax > 1024:
        kmax = min(kmax, 16)
    order = rng.choice([4, 4, 4, 2, 6])
    grid = rng.choice(["equiangular", "equiangular", "healpix"])
    nrings = lmax + rng.randrange(0, 17)
    if grid == "healpix":
        nrings = 4 * max(2, (lmax + 3) // 2 // 2) - 1
    hi = 30000000 if kind in ("forward", "interp") else 6000000
    return _case("", kind, prec, lmax, kmax, rng.choice([1, 3]), nrings, _smooth_even(2 * lmax + rng.randrange(0, 40)),
                 _log_int(rng, 1000, hi), rng.choice(["sidelobe", "taper"]), grid, rng.choice(["scan", "uniform"]), order)


# ------------------------------------------------------------------ inputs
def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + salt)


def _ring_theta(case):
    nr = case["nrings"]
    if case["grid"] == "healpix":      # the 4 Nside - 1 HEALPix ring colatitudes
        ns = (nr + 1) // 4
        i = np.arange(1, 2 * ns, dtype=np.float64)
        north = np.arccos(np.where(i < ns, 1.0 - i * i / (3.0 * ns * ns), 4.0 / 3.0 - 2.0 * i / (3.0 * ns)))
    else:
        north = math.pi * (np.arange(nr // 2, dtype=np.float64) + 0.5) / nr
    th = np.empty(nr, dtype=np.float64)
    h = nr // 2
    th[:h] = north[:h]
    if nr % 2:
        th[h] = 0.5 * math.pi
    th[nr - h:] = (math.pi - north[:h])[::-1]
    return th


def _lm(lmax):
    """l and m of the m-major packing idx(l, m) = m (2 lmax + 1 - m) / 2 + l."""
    m = torch.arange(lmax + 1, device="cuda").repeat_interleave(torch.arange(lmax + 1, 0, -1, device="cuda"))
    first = m * (2 * lmax + 1 - m) // 2
    return torch.arange(m.numel(), device="cuda") - first, m


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _sky(g, lmax, ncomp, nsky=None):
    l, m = _lm(lmax)
    ell = l.to(torch.float64)
    amp = (ell + 1.0) ** -1.0 * torch.where(m == 0, 1.0, math.sqrt(0.5))
    shape = (ncomp, l.numel()) if nsky is None else (nsky, ncomp, l.numel())
    z = torch.complex(_normal(g, *shape), _normal(g, *shape) * (m > 0))
    comp = torch.ones(ncomp, 1, dtype=torch.float64, device="cuda")
    if ncomp == 3:
        comp = torch.tensor([[1.0], [math.sqrt(0.05)], [0.1]], dtype=torch.float64, device="cuda")
        comp = comp * torch.where((l >= 2)[None, :] | (torch.arange(3, device="cuda") == 0)[:, None], 1.0, 0.0)
    return (z * (comp * amp)).contiguous()


def _beam(g, lmax, kmax, ncomp, kind):
    ell = torch.arange(lmax + 1, dtype=torch.float64, device="cuda")
    k = torch.arange(kmax + 1, dtype=torch.float64, device="cuda")[:, None]
    if kind == "taper":
        amp = torch.exp(-ell * ell / (2.0 * 20.0 ** 2)) * 0.5 ** k
    else:
        amp = (ell + 1.0) ** -1.5 * torch.ones_like(k)
    amp = amp * (ell >= k)
    z = torch.complex(_normal(g, ncomp, kmax + 1, lmax + 1), _normal(g, ncomp, kmax + 1, lmax + 1) * (k > 0))
    if ncomp == 3:
        z = z * (torch.tensor([1.0, 0.1, 0.1], dtype=torch.float64, device="cuda")[:, None, None]
                 * ((ell >= 2) | (torch.arange(3, device="cuda") == 0)[:, None])[:, None, :])
    return (z * amp).contiguous()


def _pointing(g, n, kind):
    if kind == "uniform":
        u = torch.rand(3, n, generator=g, dtype=torch.float64, device="cuda")
        return torch.arccos(2.0 * u[0] - 1.0), TWO_PI * u[1], TWO_PI * u[2]
    # spin axis in the ecliptic at longitude 2 pi t / 1 yr, boresight 85 degrees from it, 1 rpm, 32.5 Hz
    r = torch.rand(2, generator=g, dtype=torch.float64, device="cuda").tolist()
    year, ca, sa = 365.25 * 86400.0, math.cos(math.radians(85.0)), math.sin(math.radians(85.0))
    th, ph, ps = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3))
    for a in range(0, n, 1 << 25):
        e = min(n, a + (1 << 25))
        t = r[0] * year + torch.arange(a, e, dtype=torch.float64, device="cuda") / 32.5
        lam, w = t * (TWO_PI / year), t * (TWO_PI / 60.0)
        cl, sn, cw, sw = torch.cos(lam), torch.sin(lam), torch.cos(w), torch.sin(w)
        nx, ny, nz = ca * cl - sa * sw * sn, ca * sn + sa * sw * cl, sa * cw
        yz = nx * (cw * cl) + ny * (cw * sn)            # z component of boresight x scan direction
        th[a:e] = torch.arccos(nz.clamp(-1.0, 1.0))
        ph[a:e] = torch.atan2(ny, nx).remainder(TWO_PI)
        ps[a:e] = (torch.atan2(yz, sw) + TWO_PI * r[1]).remainder(TWO_PI)
    return th, ph, ps


def _plan(case):
    return sl.sidelobe_plan_create(case["lmax"], case["kmax"], _ring_theta(case), case["nphi"], ncomp=case["ncomp"],
                                   precision=case["precision"], interp_order=case["order"])


def _detectors(case):
    """The detectors of a batch: band limits in the proportions of a real focal plane."""
    out = []
    for d in range(case["count"]):
        lmax = max(32, int(case["lmax"] * (1.0, 0.1707, 0.5, 0.6827, 0.3413)[d % 5]))
        kmax = max(2, int(case["kmax"] * (1.0, 0.1667, 0.6667, 0.3334, 0.5)[(3 * d) % 5]))
        n = max(1, int(case["n"] * (1.0, 0.31, 0.062, 0.6, 0.14)[(2 * d) % 5]))
        out.append(dict(case, lmax=lmax, kmax=kmax, nrings=lmax, nphi=_smooth_even(2 * lmax), n=n))
    return out


def _orbital_periods(n, seed):
    """Offsets of 40-70 minute pointing periods at 32.5 Hz and the velocity / c of each."""
    rng = np.random.default_rng(int(seed) + 77)
    starts = [0]
    while starts[-1] < n:
        starts.append(min(n, starts[-1] + int(rng.integers(78000, 136501))))
    starts = np.asarray(starts, dtype=np.int64)
    lam = TWO_PI * 0.5 * (starts[:-1] + starts[1:]) / 32.5 / (365.25 * 86400.0)
    v = 29.78e3 * np.stack([-np.sin(lam), np.cos(lam), np.zeros_like(lam)], -1)
    return starts, (v + 0.3e3 * rng.standard_normal(v.shape)) / 299792458.0


def _inputs(case, seed):
    """Everything random of a case: device tensors (and the orbital periods on the host)."""
    g, kind = _gen(seed), case["kind"]
    L, K, nc, n = case["lmax"], case["kmax"], case["ncomp"], case["n"]
    if kind == "batch":
        sky = _sky(g, L, nc)
        l, _ = _lm(L)
        dets = []
        for d, c in enumerate(_detectors(case)):
            gd = _gen(seed, 1 + d)
            th, ph, ps = _pointing(gd, c["n"], c["pointing"])
            dets.append(dict(case=c, sky=sky[:, l <= c["lmax"]].contiguous(),
                             beam=_beam(gd, c["lmax"], c["kmax"], nc, c["beam"]), theta=th, phi=ph, psi=ps))
        return dict(dets=dets)
    x = dict(beam=_beam(g, L, K, nc, case["beam"]))
    if kind == "multisky":
        x["sky"] = _sky(g, L, nc, case["count"])
        return x
    x["theta"], x["phi"], x["psi"] = _pointing(g, n, case["pointing"])
    if kind == "orbital":
        x["starts"], x["beta"] = _orbital_periods(n, seed)
        return x
    x["sky"] = _sky(g, L, nc)
    if kind in ("adjoint", "gradient"):
        x["y"] = 1e-3 * _normal(g, n)      # a residual, or data of noise alone
    return x


def prepare(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "batch":
        items = []
        for d in x["dets"]:
            plan = _plan(d["case"])
            maps = torch.empty(plan.maps_shape(), dtype=plan.maps_dtype, device="cuda")
            items.append(dict(plan=plan, sky=d["sky"], beam=d["beam"], maps=maps, theta=d["theta"], phi=d["phi"],
                              psi=d["psi"], tod=torch.empty(d["theta"].numel(), dtype=torch.float64, device="cuda")))
        torch.cuda.current_stream().synchronize()
        return dict(kind=kind, items=items, batch=sl.sl_batch_create(items))
    s = dict(x, kind=kind, plan=_plan(case))
    if kind == "interp":
        s["maps"] = sl.synth_spin_maps(s["plan"], s["sky"], s["beam"])
    if kind == "gradient":
        s["sky"].requires_grad_(True)
        s["beam"].requires_grad_(True)
    if kind == "orbital":
        s["q"] = sl.quad_factor(70e9, 2.7255)
    return s


def run(s):
    kind = s["kind"]
    if kind == "forward":
        return sl.convolve_tod(s["plan"], s["sky"], s["beam"], s["theta"], s["phi"], s["psi"])
    if kind == "interp":
        return sl.interp_tod(s["plan"], s["maps"], s["theta"], s["phi"], s["psi"])
    if kind == "adjoint":
        return sl.adjoint_tod(s["plan"], s["theta"], s["phi"], s["psi"], s["y"], s["sky"], s["beam"])
    if kind == "gradient":
        tod = sl.sidelobe_tod(s["plan"], s["sky"], s["beam"], s["theta"], s["phi"], s["psi"])
        gs, gb = torch.autograd.grad(tod, (s["sky"], s["beam"]), tod.detach() - s["y"])
        return tod.detach(), gs, gb
    if kind == "multisky":
        return sl.synth_spin_maps_multi(s["plan"], s["sky"], s["beam"])
    if kind == "batch":
        sl.sl_batch_run(s["batch"])
        return [(it["maps"], it["tod"]) for it in s["items"]]
    return sl.orbital_dipole_tod(s["plan"], s["beam"], 2.7255, s["q"], s["theta"], s["phi"], s["psi"], s["starts"],
                                 s["beta"], 20)


def work(case):
    """Bytes read and written once, and the operations of the two-step algorithm as it is
    stated: complex x real products and three-term recurrences over every (ring, m, l),
    N log2 N transforms, p x p node sums per order and sample."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work(dict(c, kind="forward")) for c in _detectors(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    L, K1, R, nphi, n, p = case["lmax"], case["kmax"] + 1, case["nrings"], case["nphi"], case["n"], case["order"]
    if kind == "orbital":
        return {"bytes": 32.0 * n, "flops": n / 20 * 152.0 + 7.0 * n}
    coef = case["ncomp"] * 16.0 * ((L + 1) * (L + 2) / 2 + K1 * (L + 1))
    cube_bytes = R * nphi * K1 * (8.0 if case["precision"] == "fp32" else 16.0)
    cube = K1 * (4.0 * R * (L + 1) ** 2 + 1.5 * R * (L + 1) * (L + 2) + 5.0 * R * nphi * math.log2(nphi))
    tod = n * (4.0 * p * p * K1 + 10.0)
    if kind == "multisky":
        ns = case["count"]
        return {"bytes": ns * (coef + cube_bytes),
                "flops": K1 * (ns * (4.0 * R * (L + 1) ** 2 + 5.0 * R * nphi * math.log2(nphi))
                               + 1.5 * R * (L + 1) * (L + 2))}
    if kind == "forward":
        return {"bytes": coef + cube_bytes + 32.0 * n, "flops": cube + tod}
    if kind == "interp":
        return {"bytes": cube_bytes + 32.0 * n, "flops": tod}
    if kind == "adjoint":
        return {"bytes": 2.0 * coef + 32.0 * n, "flops": cube + tod}
    return {"bytes": 3.0 * coef + 72.0 * n, "flops": 2.0 * (cube + tod)}


# ------------------------------------------------------------------ the operator in plain 64-bit torch
def _wigner_rows(lmax, kmax, theta, each, block=16):
    """d^l_{mk}(theta_r) for k = 0..kmax, m = -l..l by the three-term recurrence in l from
    the single-term values at l = max(|m|, k); calls each(l0, D) with D [block, K+1, 2M+1, R]
    (M = the block's last l; zero where l < max(|m|, k)).  A stored value is v 2^(512 e)."""
    dev, f8 = theta.device, torch.float64
    R = theta.numel()
    x, c, s = torch.cos(theta), torch.cos(0.5 * theta), torch.sin(0.5 * theta)
    W = 2 * lmax + 1
    v = torch.zeros(kmax + 1, W, R, dtype=f8, device=dev)       # current l
    u = torch.zeros_like(v)                                     # l - 1
    e = torch.zeros(kmax + 1, W, R, dtype=torch.int16, device=dev)
    edge = [None] * (kmax + 1)      # values at m = +l and m = -l with their exponents, per k
    ks = torch.arange(kmax + 1, dtype=f8, device=dev)[:, None]
    for l0 in range(0, lmax + 1, block):
        M = min(lmax, l0 + block - 1)
        D = torch.zeros(M - l0 + 1, kmax + 1, 2 * M + 1, R, dtype=f8, device=dev)
        for l in range(l0, M + 1):
            if l > 0:
                lo, hi = lmax - (l - 1), lmax + l
                ms = torch.arange(-(l - 1), l, dtype=f8, device=dev)[None, :]
                kk = ks[:l] if kmax >= l else ks            # orders with k <= l - 1
                q = l - 1.0
                nk = kk.shape[0]
                vv, uu = v[:nk, lo:hi], u[:nk, lo:hi]
                if l == 1:
                    nxt = vv * x
                else:
                    den = q * torch.sqrt((l * l - ms * ms) * (l * l - kk * kk))
                    al, be = (2 * q + 1) * q * l / den, (2 * q + 1) * ms * kk / den
                    ga = l * torch.sqrt((q * q - ms * ms).clamp_min(0.0) * (q * q - kk * kk).clamp_min(0.0)) / den
                    nxt = torch.addcmul(-be[..., None], al[..., None], x)
                    nxt.mul_(vv)
                    nxt.addcmul_(ga[..., None], uu, value=-1.0)
                uu.copy_(vv)
                vv.copy_(nxt)
                if l % 8 == 0:
                    big = vv.abs() > 2.0 ** 256
                    vv[big] *= 2.0 ** -512
                    uu[big] *= 2.0 ** -512
                    e[:nk, lo:hi][big] += 1
            for k in range(min(l, kmax) + 1):
                if k == l:      # the whole row |m| <= k starts here
                    for m in range(-k, k + 1):
                        v[k, lmax + m] = math.sqrt(math.comb(2 * k, k + m)) * c ** (k + m) * s ** (k - m)
                    edge[k] = [v[k, lmax + k].clone(), v[k, lmax - k].clone(), torch.zeros(R, dtype=torch.int16, device=dev),
                               torch.zeros(R, dtype=torch.int16, device=dev)]
            if l > 0:           # m = +-l of the orders k < l
                nk = min(l, kmax + 1)
                ratio = torch.sqrt(2.0 * l * (2.0 * l - 1.0) / ((l + ks[:nk]) * (l - ks[:nk])))
                P, N, pe, ne = (torch.stack([edge[k][i] for k in range(nk)]) for i in range(4))
                P, N = -P * ratio * (c * s), N * ratio * (c * s)
                for val, ex in ((P, pe), (N, ne)):
                    small = (val.abs() < 2.0 ** -256) & (val != 0)
                    val[small] *= 2.0 ** 512
                    ex[small] -= 1
                for k in range(nk):
                    edge[k] = [P[k], N[k], pe[k], ne[k]]
                v[:nk, lmax + l], v[:nk, lmax - l] = P, N
                e[:nk, lmax + l], e[:nk, lmax - l] = pe, ne
                u[:nk, lmax + l] = u[:nk, lmax - l] = 0.0
            nk = min(l, kmax) + 1
            D[l - l0, :nk, M - l:M + l + 1] = v[:nk, lmax - l:lmax + l + 1] * (e[:nk, lmax - l:lmax + l + 1] == 0)
        each(l0, D)


def _full_sky(sky, lmax):
    """s_{l,m} as [ncomp, L+1 (l), 2L+1 (m + L)]."""
    l, m = _lm(lmax)
    out = torch.zeros(sky.shape[0], lmax + 1, 2 * lmax + 1, dtype=torch.complex128, device=sky.device)
    out[:, l, lmax + m] = sky
    pos = m > 0
    out[:, l[pos], lmax - m[pos]] = sky[:, pos].conj() * (1.0 - 2.0 * (m[pos] % 2))
    return out


def _exact_cube(case, skies, beam):
    """F [nsky][R, nphi, K+1] complex128."""
    L, K, nphi = case["lmax"], case["kmax"], case["nphi"]
    theta = torch.from_numpy(_ring_theta(case)).cuda()
    R, ns = theta.numel(), len(skies)
    full = [_full_sky(s, L) for s in skies]
    G = torch.zeros(K + 1, 2 * L + 1, R, 2 * ns, dtype=torch.float64, device="cuda")

    def add(l0, D):
        M = (D.shape[2] - 1) // 2
        nb = D.shape[0]
        cols = []
        for f in full:
            A = torch.einsum("xlm,xkl->kmlx", f[:, l0:l0 + nb, L - M:L + M + 1], beam[:, :, l0:l0 + nb].conj()).sum(-1)
            cols += [A.real, A.imag]
        A = torch.stack(cols, -1)                                   # [K+1, 2M+1, nb, 2 ns]
        for k in range(K + 1):
            G[k, L - M:L + M + 1] += torch.matmul(D[:, k].permute(1, 2, 0), A[k])
    _wigner_rows(L, K, theta, add)
    cubes = []
    q = torch.arange(-L, L + 1, device="cuda") % nphi
    for i in range(ns):
        H = torch.zeros(K + 1, nphi, R, dtype=torch.complex128, device="cuda")
        H.index_add_(1, q, torch.complex(G[..., 2 * i], G[..., 2 * i + 1]))
        cubes.append((torch.fft.ifft(H, dim=1) * nphi).permute(2, 1, 0).contiguous())
    return cubes


def _stencil(case, theta, phi):
    """Node indices and Lagrange weights of the p x p stencil: rows [n, p], columns [n, p], sign flags."""
    p, nphi = case["order"], case["nphi"]
    rt = torch.from_numpy(_ring_theta(case)).cuda()
    R, h = rt.numel(), p // 2
    ext = torch.cat([-rt[:h].flip(0), rt, TWO_PI - rt[-h:].flip(0)])
    i = torch.searchsorted(rt, theta, right=True) - 1
    rows = i[:, None] - h + 1 + torch.arange(p, device="cuda")
    nodes = ext[rows + h]
    wt = torch.ones_like(nodes)
    for a in range(p):
        for b in range(p):
            if a != b:
                wt[:, a] *= (theta - nodes[:, b]) / (nodes[:, a] - nodes[:, b])
    t = phi * (nphi / TWO_PI)
    j = torch.floor(t)
    f = t - j
    cols = j.long()[:, None] - h + 1 + torch.arange(p, device="cuda")
    wp = torch.ones_like(nodes)
    for a in range(p):
        for b in range(p):
            if a != b:
                wp[:, a] *= (f - (b - h + 1)) / (a - b)
    ghost = (rows < 0) | (rows >= R)
    ring = torch.where(rows < 0, -1 - rows, torch.where(rows >= R, 2 * R - 1 - rows, rows))
    return ring, cols, ghost, wt, wp


def _chunks(case, x, each):
    """each(slice, node index [m, p p], weight [m, p p], ghost [m, p p], psi) over chunks of the pointings."""
    n = x["theta"].numel()
    step = max(1, int(4e7) // (case["order"] ** 2 * (case["kmax"] + 1)))
    for a in range(0, n, step):
        sl_ = slice(a, min(n, a + step))
        ring, cols, ghost, wt, wp = _stencil(case, x["theta"][sl_], x["phi"][sl_])
        col = (cols[:, None, :] + ghost[:, :, None] * (case["nphi"] // 2)) % case["nphi"]
        node = (ring[:, :, None] * case["nphi"] + col).flatten(1)
        w = (wt[:, :, None] * wp[:, None, :]).flatten(1)
        each(sl_, node, w, ghost[:, :, None].expand_as(col).flatten(1), x["psi"][sl_])


def _exact_tod(case, cube, x):
    K = case["kmax"]
    F = cube.reshape(-1, K + 1)
    tod = torch.empty_like(x["theta"])
    sgn = 1.0 - 2.0 * (torch.arange(K + 1, device="cuda") % 2)
    eps = torch.full((K + 1,), 2.0, dtype=torch.float64, device="cuda")
    eps[0] = 1.0

    def add(sl_, node, w, ghost, psi):
        v = F[node]                                                  # [m, pp, K+1]
        ws = torch.where(ghost[:, :, None], sgn, torch.ones_like(sgn)) * w[:, :, None]
        ang = psi[:, None] * torch.arange(K + 1, device="cuda")
        S = torch.complex((v.real * ws).sum(1), (v.imag * ws).sum(1))
        tod[sl_] = ((S.real * torch.cos(ang) - S.imag * torch.sin(ang)) * eps).sum(1)
    _chunks(case, x, add)
    return tod


def _exact_adjoint(case, x, y):
    """Gradients of sum_i y_i c_i with respect to the packed sky and beam."""
    L, K, nphi = case["lmax"], case["kmax"], case["nphi"]
    theta = torch.from_numpy(_ring_theta(case)).cuda()
    R = theta.numel()
    bar = torch.zeros(R * nphi, K + 1, 2, dtype=torch.float64, device="cuda")
    sgn = 1.0 - 2.0 * (torch.arange(K + 1, device="cuda") % 2)
    eps = torch.full((K + 1,), 2.0, dtype=torch.float64, device="cuda")
    eps[0] = 1.0

    def add(sl_, node, w, ghost, psi):
        ang = psi[:, None] * torch.arange(K + 1, device="cuda")
        ph = torch.stack([torch.cos(ang), -torch.sin(ang)], -1) * (eps[:, None] * y[sl_][:, None, None])
        ws = torch.where(ghost[:, :, None], sgn, torch.ones_like(sgn)) * w[:, :, None]
        bar.index_add_(0, node.flatten(), (ws[..., None] * ph[:, None]).flatten(0, 1))
    _chunks(case, x, add)
    X = torch.fft.fft(torch.complex(bar[..., 0], bar[..., 1]).view(R, nphi, K + 1), dim=1)
    q = torch.arange(-L, L + 1, device="cuda") % nphi
    Gh = torch.view_as_real(X[:, q].permute(2, 1, 0).contiguous())  # [K+1, 2L+1, R, 2]
    Ab = torch.zeros(K + 1, 2 * L + 1, L + 1, 2, dtype=torch.float64, device="cuda")

    def back(l0, D):
        M = (D.shape[2] - 1) // 2
        for k in range(K + 1):
            Ab[k, L - M:L + M + 1, l0:l0 + D.shape[0]] = torch.matmul(D[:, k].permute(1, 0, 2), Gh[k, L - M:L + M + 1])
    _wigner_rows(L, K, theta, back)
    Ab = torch.view_as_complex(Ab)                                  # [K+1, 2L+1, L+1]
    beam, full = x["beam"].detach(), _full_sky(x["sky"].detach(), L)
    l, m = _lm(L)
    Ap, An = Ab[:, L + m, l], Ab[:, L - m, l]                       # [K+1, nalm]
    gs = torch.zeros_like(x["sky"].detach())
    par = 1.0 - 2.0 * (m % 2)
    for X_ in range(beam.shape[0]):
        b = beam[X_][:, l]
        g = (b * Ap + par * b.conj() * An.conj()).sum(0)
        gs[X_] = torch.where(m > 0, g, torch.complex((b * Ap).sum(0).real, torch.zeros_like(g.real)))
    gb = torch.einsum("xlm,kml->xkl", full, Ab.conj())
    gb[:, 0] = torch.complex(gb[:, 0].real, torch.zeros_like(gb[:, 0].real))
    ell = torch.arange(L + 1, device="cuda")
    return gs, gb * (ell >= torch.arange(K + 1, device="cuda")[:, None])


def _beam_moments(beam):
    """int v B dOmega of the temperature beam's l <= 2 part, by quadrature."""
    b = beam[0].cpu().numpy()
    z, wz = np.polynomial.legendre.leggauss(8)
    ph = TWO_PI * np.arange(16) / 16
    Z, P = np.meshgrid(z, ph, indexing="ij")
    S = np.sqrt(1.0 - Z * Z)
    pi = math.pi
    Y = {(0, 0): math.sqrt(1 / (4 * pi)) + 0 * Z, (1, 0): math.sqrt(3 / (4 * pi)) * Z,
         (1, 1): -math.sqrt(3 / (8 * pi)) * S, (2, 0): math.sqrt(5 / (16 * pi)) * (3 * Z * Z - 1),
         (2, 1): -math.sqrt(15 / (8 * pi)) * S * Z, (2, 2): math.sqrt(15 / (32 * pi)) * S * S}
    B = np.zeros_like(Z)
    for (l, k), y in Y.items():
        if k < b.shape[0] and l < b.shape[1]:
            B += (1 if k == 0 else 2) * (b[k, l] * y * np.exp(1j * k * P)).real
    w = wz[:, None] * (TWO_PI / 16) * B
    v = [S * np.cos(P), S * np.sin(P), Z]
    return [float((w * f).sum()) for f in (v[0], v[1], v[2], v[0] * v[0], v[1] * v[1], v[2] * v[2], v[0] * v[1],
                                           v[0] * v[2], v[1] * v[2])]


def _dipole(S, T0, q, th, ph, ps, beta):
    ct, st, cp, sp, cs, ss = torch.cos(th), torch.sin(th), torch.cos(ph), torch.sin(ph), torch.cos(ps), torch.sin(ps)
    bx, by, bz = beta.unbind(-1)
    e1 = cp * bx + sp * by
    e2 = cp * by - sp * bx
    a = ct * e1 - st * bz
    x, y, z = cs * a + ss * e2, cs * e2 - ss * a, st * e1 + ct * bz
    return T0 * (S[0] * x + S[1] * y + S[2] * z + q * (S[3] * x * x + S[4] * y * y + S[5] * z * z
                                                      + 2 * (S[6] * x * y + S[7] * x * z + S[8] * y * z)))


def _exact_orbital(x, s=20, T0=2.7255, nu=70e9):
    a = 6.62607015e-34 * nu / (1.380649e-23 * T0)
    q = 0.5 * a * (math.exp(a) + 1.0) / (math.exp(a) - 1.0)
    S = _beam_moments(x["beam"])
    beta = torch.from_numpy(x["beta"]).cuda()
    starts = torch.from_numpy(x["starts"]).cuda()
    n = x["theta"].numel()
    i = torch.arange(n, device="cuda")
    per = torch.searchsorted(starts, i, right=True) - 1
    loc, length = i - starts[per], (starts[1:] - starts[:-1])
    nodes = (length - 1) // s + 1
    out = _dipole(S, T0, q, x["theta"], x["phi"], x["psi"], beta[per])
    # second derivatives of each period's natural spline, all periods side by side
    M = int(nodes.max())
    idx = (starts[:-1, None] + s * torch.arange(M, device="cuda")).clamp_max(n - 1)
    y = out[idx].cpu().numpy()
    nn = nodes.cpu().numpy()
    cp, dp, m2 = np.zeros_like(y), np.zeros_like(y), np.zeros((y.shape[0], M + 1))
    for j in range(1, M - 1):
        den = 4.0 - cp[:, j - 1]
        cp[:, j] = 1.0 / den
        dp[:, j] = (6.0 * (y[:, j + 1] - 2.0 * y[:, j] + y[:, j - 1]) / (s * s) - dp[:, j - 1]) / den
    for j in range(M - 2, 0, -1):
        m2[:, j] = np.where(j <= nn - 2, dp[:, j] - cp[:, j] * m2[:, j + 1], 0.0)
    m2 = torch.from_numpy(m2).cuda()
    yt = torch.from_numpy(y).cuda()
    j = torch.minimum(loc // s, (nodes[per] - 2).clamp_min(0))
    B = (loc - j * s).to(torch.float64) / s
    A = 1.0 - B
    sp = A * yt[per, j] + B * yt[per, (j + 1).clamp_max(M - 1)] + ((A ** 3 - A) * m2[per, j] + (B ** 3 - B) * m2[per, j + 1]) * (s * s / 6.0)
    inside = (loc <= s * (nodes[per] - 1)) & (nodes[per] > 1)
    return torch.where(inside, sp, out)


def exact(case, seed):
    """What ``run`` returns, from plain 64-bit torch."""
    x, kind = _inputs(case, seed), case["kind"]
    with torch.no_grad():
        if kind == "batch":
            out = []
            for d in x["dets"]:
                F, = _exact_cube(d["case"], [d["sky"]], d["beam"])
                out.append((F, _exact_tod(d["case"], F, d)))
            return out
        if kind == "orbital":
            return _exact_orbital(x)
        if kind == "multisky":
            return torch.stack(_exact_cube(case, list(x["sky"]), x["beam"]))
        if kind == "adjoint":
            return _exact_adjoint(case, x, x["y"])
        F, = _exact_cube(case, [x["sky"]], x["beam"])
        tod = _exact_tod(case, F, x)
        if kind == "forward":
            return F, tod
        if kind == "interp":
            return tod
        del F
        gs, gb = _exact_adjoint(case, x, tod - x["y"])
        return tod, gs, gb
