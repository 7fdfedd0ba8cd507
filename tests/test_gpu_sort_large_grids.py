"""The pointing sort on grids beyond the lines where its scans take another form (160,000 tiles,
2.7e8 cells): every sample's value against the two-point formula written out, which needs the
right cell, tile and work item of every sample; two tile widths give the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,N,prec,widths", [(4608, 6144, "fp32", (32, 16)), (4608, 6144, "df64", (32, 8)), (16384, 16384, "fp32", (32,))])
def test_values_on_a_large_grid(R, N, prec, widths):
    import paper_2201_03478_gb300 as sl
    rt = np.pi * (np.arange(R) + 0.5) / R
    rt[R // 2:] = np.pi - rt[:R // 2][::-1]
    plan = sl.sidelobe_plan_create(2, 0, rt, N, precision=prec, interp_order=2)
    g = torch.Generator(device="cuda").manual_seed(1)
    maps = torch.zeros(plan.maps_shape(), dtype=plan.maps_dtype, device="cuda")
    torch.view_as_real(maps)[..., 0] = torch.rand(R, N, 1, generator=g, device="cuda")
    n = 300000
    u = torch.rand(3, n, generator=g, dtype=torch.float64, device="cuda")
    u[:, :5000] = 0.3 + 1e-4 * u[:, :5000]                       # and a crowd in a few cells
    th, ph, ps = 0.01 + 3.12 * u[0], 2 * np.pi * u[1], 2 * np.pi * u[2]
    i = torch.searchsorted(torch.from_numpy(rt).cuda(), th, right=True) - 1
    t0, t1 = torch.from_numpy(rt).cuda()[i], torch.from_numpy(rt).cuda()[i + 1]
    x = ph * (N / (2 * np.pi))
    j = torch.floor(x).long()
    a, b = (th - t0) / (t1 - t0), x - j
    F = maps[..., 0].real
    f = lambda r, c: F[r, c % N].double()
    want = (1 - a) * ((1 - b) * f(i, j) + b * f(i, j + 1)) + a * ((1 - b) * f(i + 1, j) + b * f(i + 1, j + 1))
    first = None
    for tc in widths:
        plan.set_tile_cols(tc)
        got = sl.interp_tod(plan, maps, th, ph, ps)
        plan.sync()
        # FP32: offsets and weights of 2^-24 each, of values below 1
        assert float((got - want).abs().max()) <= (2e-6 if prec == "fp32" else 1e-10)
        first = got if first is None else first
        assert torch.equal(got, first)
