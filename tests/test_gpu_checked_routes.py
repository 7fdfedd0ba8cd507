"""The bounds-checked library variant (-DSL_CHECKED) on every route of the interpolation and of its
transpose: few and many samples per cell, every stencil, several blocks of orders, the kernels that
the count of occupied cells decides between.  No guard may fire, the results match the oracle, and
the kernels named are the ones launched, so that a change of the routes cannot drop one silently.  In
a child process: a process loads one library variant."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
from paper_2201_03478_gb300 import _lib
_lib.use_checked_build()
import paper_2201_03478_gb300 as sl
import oracle
oracle.build()
import workloads as W
lib = _lib.load()
assert lib._name.endswith("libsidelobe_checked.so"), lib._name
dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
def points(n, cells, seed=1):
    """poles, phi = 0 and 2 pi among n samples, uniform or around `cells` points"""
    th, ph, ps = W.pointings_uniform(n, seed=seed)
    if cells:
        c = np.random.default_rng(seed).integers(0, cells, n)
        th, ph = th[c], ph[c]
    k = min(n, 6)
    th[:k], ph[:k] = [0.0, 1e-9, np.pi, np.pi - 1e-9, 0.02, 3.12][:k], [0.0, 2 * np.pi - 1e-12, 1.0, 0.0, 6.28, 3.0][:k]
    return th, ph, ps
def run(name, got, ref, tol, plan, kernels):
    plan.sync()
    st, ks = lib.sl_debug_check_status(), plan.kernel_stats(reset=True)
    assert st == 0, (name, hex(st))
    for k in kernels:
        assert k in ks, (name, k, sorted(ks))
    err = np.linalg.norm(np.ravel(got.cpu().numpy() - ref)) / np.linalg.norm(np.ravel(ref))
    assert err < tol, (name, err)
    print("%s: %.1e, %s" % (name, err, ",".join(kernels)))
#        name                precision  R    N    K  p  n       cells  kernels
forward = [("few",           "fp64", 31,  48,  4, 4, 3000,   0,   ["interp_fx"]),
           ("short",         "fp64", 60, 120, 16, 4, 15000,  0,   ["interp_fx", "interp_fx_short"]),
           ("dense",         "fp64", 31,  48, 16, 4, 60000,  0,   ["interp_fx"]),
           ("direct",        "fp64", 60, 120,  5, 4, 25000,  0,   ["interp_f64"]),
           ("p2",            "fp64", 31,  48,  5, 2, 150000, 0,   ["interp_fx"]),
           ("p2 blocks",     "fp64", 31,  48, 18, 2, 80000,  0,   ["interp_fx"]),
           ("p6",            "fp64", 31,  48,  9, 6, 80000,  0,   ["interp_fx"]),
           ("p6 blocks",     "fp64", 31,  48, 18, 6, 80000,  0,   ["interp_fx"]),
           ("blocks",        "fp64", 31,  48, 20, 4, 80000,  0,   ["interp_fx"]),
           ("df64 both",     "df64", 31,  48, 16, 4, 20000,  0,   ["interp_fx", "interp_df"]),
           ("df64 few cells", "df64", 31, 48, 16, 4, 20000,  30,  ["interp_fx", "interp_df"]),
           ("df64 dense",    "df64", 31,  48, 16, 4, 100000, 0,   ["interp_fx"])]
for name, prec, R, N, K, p, n, cells, kernels in forward:
    rt = W.equiangular_ring_theta(R)
    plan = sl.sidelobe_plan_create(max(K, 4), K, rt, N, precision=prec, interp_order=p)
    rng = np.random.default_rng(K)
    cube = rng.standard_normal((R, N, K + 1)) + 1j * rng.standard_normal((R, N, K + 1))
    th, ph, ps = points(n, cells)
    plan.enable_timing(True)
    got = sl.interp_tod(plan, dev(cube), dev(th), dev(ph), dev(ps))
    run(name, got, oracle.interp(cube, rt, th, ph, ps, p=p), 1e-10, plan, kernels)
adjoint = [("few",           "fp64", 31,  48,  4, 4, 3000,   0,   ["interp_adj_fx"]),
           ("both",          "fp64", 127, 128, 16, 4, 30000, 0,   ["interp_adj_fx", "interp_adj"]),
           ("both, few cells", "fp64", 127, 128, 16, 4, 30000, 50, ["interp_adj_fx", "interp_adj"]),
           ("dense",         "fp64", 31,  48, 32, 4, 60000,  0,   ["interp_adj_fx"]),
           ("p2",            "fp64", 31,  48,  5, 2, 20000,  0,   ["interp_adj"]),
           ("p6",            "fp64", 31,  48,  5, 6, 20000,  0,   ["interp_adj"]),
           ("33 orders",     "fp64", 31,  48, 33, 4, 20000,  0,   ["interp_adj"]),
           ("df64 both",     "df64", 127, 128, 8, 4, 30000,  0,   ["interp_adj_fx", "interp_adj_df"]),
           ("df64 p6",       "df64", 31,  48,  5, 6, 20000,  0,   ["interp_adj_df"])]
for name, prec, R, N, K, p, n, cells, kernels in adjoint:
    rt = W.equiangular_ring_theta(R)
    plan = sl.sidelobe_plan_create(max(K, 4), K, rt, N, precision=prec, interp_order=p)
    th, ph, ps = points(n, cells)
    y = np.random.default_rng(3).standard_normal(n)
    plan.enable_timing(True)
    got = sl.adjoint_interp(plan, dev(th), dev(ph), dev(ps), dev(y))
    run("adjoint " + name, got, oracle.interp_adjoint(y, rt, N, K, th, ph, ps, p=p), 1e-10, plan, kernels)
'''


def test_no_guard_fires_on_any_route():
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=1200)
    print(r.stdout[-4000:])
    assert r.returncode == 0, r.stderr[-4000:]
