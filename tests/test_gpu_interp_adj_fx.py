"""The fixed-point transpose of the interpolation against the tiled FP64 kernel: a plan with more
than 32 orders takes the latter, and its first orders are the same sums.  Edges of the
32-sample batches, blocks of four orders and runs of cells, both sides of the choice by occupied
cells, poles, phi seam, amplitudes 2^40 apart, and samples that take the plain loop.

Bound per node.  With B the sum of |y| over the samples that touch it (|w| eps_k < 3.2), each
side carries k 2^-53 from psi and the recurrences' growth (below 8 K 2^-53), the fixed point
at most 64 x 2^-53 of the run's largest |y|, the FP64 sums n_node 2^-53: |err| <= 4 B (8 K + 64 +
n_node) 2^-53."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _adjoint(K, R, N, prec, th, ph, ps, y):
    import paper_2201_03478_gb300 as sl
    rt = np.pi * (np.arange(R) + 0.5) / R
    plan = sl.sidelobe_plan_create(max(K, 4), K, rt, N, precision=prec)
    out = sl.adjoint_interp(plan, *(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (th, ph, ps, y)))
    plan.sync()
    return out.cpu().numpy()


def _touching(R, N, th, ph, y):
    """Per node: sum of |y| and number of the samples that may touch it (stencils one node wider)."""
    i, j = np.floor(th * R / np.pi - 0.5).astype(int), np.floor(ph * N / (2 * np.pi)).astype(int)
    b, cnt = np.zeros((R, N)), np.zeros((R, N))
    for a in range(-2, 4):
        for c in range(-2, 4):
            row, col = i + a, j + c
            over = (row < 0) | (row >= R)
            row = np.where(row < 0, -1 - row, np.where(row >= R, 2 * R - 1 - row, row))
            col = (col + np.where(over, N // 2, 0)) % N
            np.add.at(b, (row, col), np.abs(y))
            np.add.at(cnt, (row, col), 1)
    return b, cnt


def _check(K, R, N, prec, th, ph, ps, y):
    got, ref = _adjoint(K, R, N, prec, th, ph, ps, y), _adjoint(33, R, N, "fp64", th, ph, ps, y)[..., :K + 1]
    b, cnt = _touching(R, N, th, ph, y)
    assert (np.abs(got - ref) <= (4 * b * (8 * K + 64 + cnt) * 2.0 ** -53)[..., None]).all()
    return got


def _points(n, ncells, seed=0):
    rng = np.random.default_rng(seed)
    t0 = np.concatenate([[1e-3, np.pi - 1e-3], np.arccos(rng.uniform(-1, 1, ncells))])[:ncells]
    p0 = np.concatenate([[0.0, 2 * np.pi - 1e-9], rng.uniform(0, 2 * np.pi, ncells)])[:ncells]
    c = rng.integers(0, ncells, n)
    return (np.clip(t0[c] + 1e-2 * rng.standard_normal(n), 0, np.pi), np.mod(p0[c] + 0.1 * rng.standard_normal(n), 2 * np.pi),
            rng.uniform(-20.0, 20.0, n), rng.standard_normal(n) * 2.0 ** (-40 * (c % 2)))


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("K,n,ncells", [(0, 33, 3), (1, 1, 1), (3, 31, 40), (4, 32, 2), (5, 5000, 7), (8, 4000, 900),
                                        (13, 20000, 4), (16, 3001, 60), (32, 2000, 30)])
def test_against_tiled_kernel(K, n, ncells, prec):
    _check(K, 31, 48, prec, *_points(n, ncells))


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("ncells", [20, 100000])
def test_choice_by_occupied_cells(ncells, prec):
    _check(2, 200, 256, prec, *_points(100000, ncells, seed=1))


def test_scales_and_extremes():
    """Zeros give zeros; amplitudes beyond the fixed point and phases beyond its table agree;
    a NaN or an infinity reaches the nodes that it reaches in the tiled kernel."""
    th, ph, ps, y = _points(3000, 10, seed=2)
    assert not _check(6, 31, 48, "fp64", th, ph, ps, y * 0).any()
    for s in (2.0 ** 600, 2.0 ** 975, 2.0 ** -700, 2.0 ** -980):
        with np.errstate(over="ignore"):
            _check(6, 31, 48, "fp64", th, ph, ps, np.sign(y) * s)
    ps[::7] *= 1e4
    _check(6, 31, 48, "fp64", th, ph, ps, y)
    for k, bad in ((5, np.nan), (9, np.inf)):
        v = y.copy()
        v[k] = bad
        got, ref = _adjoint(6, 31, 48, "fp64", th, ph, ps, v), _adjoint(33, 31, 48, "fp64", th, ph, ps, v)[..., :7]
        assert (np.isfinite(got) == np.isfinite(ref)).all() and not np.isfinite(got).all()
