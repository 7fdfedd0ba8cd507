"""The fixed-point kernels' 64-bit integer arithmetic (csrc/fxint.cuh), compiled for the host with
checks for undefined behaviour that end the program, against exact integers: the limits of its
ranges (psi = 0, where a step's product is 2^63, among them) and random values."""
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2201_03478_gb300", "csrc")
ONE = 1 << 62

MAIN = r"""
#include <stdio.h>
#include "fxint.cuh"
int main() {
    long long op, a, b, c;
    while (scanf("%lld %lld %lld %lld", &op, &a, &b, &c) == 4)
        printf("%lld\n", op == 0 ? sl::fx_mulhi(a, b) : op == 1 ? sl::fx_mul(a, b) : op == 2 ? sl::fx_mulhi_rn(a, b)
               : op == 3 ? sl::fx_mul_rn(a, b) : op == 4 ? sl::fx_cheb(a, b, c) : sl::fx_shift_even(a, (int)b));
}
"""


def _signed64(x):
    return (x + (1 << 63)) % (1 << 64) - (1 << 63)


def test_no_undefined_behaviour_and_stated_errors(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    subprocess.run([gxx, "-O1", "-std=c++17", "-x", "c++", "-fsanitize=undefined", "-fsanitize-undefined-trap-on-error",
                    "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rng = random.Random(1)
    q62 = [0, 1, -1, ONE, -ONE, ONE - 1, ONE // 2, (1 << 31) - 1, 1 << 31, -(1 << 31), (1 << 32) + (1 << 31)]
    q62 += [rng.randrange(-ONE, ONE + 1) for _ in range(300)]
    wide = [23 << 58, -(23 << 58)] + [rng.randrange(-(23 << 58), 23 << 58) for _ in range(100)]
    weights = [3 << 61, -(3 << 61), 0] + [rng.randrange(-(3 << 61), 3 << 61) for _ in range(20)]
    cases, bound = [], []
    for a in q62:
        for b in q62[::7]:
            # floor of the middle products and the low product left out (a quarter): 1 + 1/4 units
            cases += [(0, a, b, 0), (1, a, b, 0), (3, a, b, 0)]
            bound += [(a * b, 64, 1.25), (a * b, 62, 5.0), (a * b, 62, 1.5)]
    for a in wide:
        for b in weights:
            cases.append((2, a, b, 0))
            bound.append((a * b, 64, 0.75))
    for a, b, c in [(ONE, ONE, ONE), (-ONE, ONE, -ONE), (ONE, -ONE, -ONE), (-ONE, -ONE, ONE)]:
        cases.append((4, a, b, c))                       # X = 1 or -1 again: the product wraps, the step does not
        bound.append((2 * a * b - (c << 62), 62, 0.0))
    for a in q62[:60]:
        for n in (0, 1, 3, 13, 40, 61):
            cases.append((5, a, n, 0))
            bound.append((a, n, 0.5))
    text = "".join("%d %d %d %d\n" % c for c in cases)
    r = subprocess.run([str(exe)], input=text, capture_output=True, text=True)
    assert r.returncode == 0, "undefined behaviour (status %d)" % r.returncode
    got = [int(x) for x in r.stdout.split()]
    assert len(got) == len(cases)
    for c, g, (exact, n, units) in zip(cases, got, bound):
        d = (g << n) - exact
        assert g == _signed64(g) and abs(d) <= int(units * 4) << max(n - 2, 0) if n >= 2 else abs(d) <= units * (1 << n), (c, g)
    odd = [c for c in cases if c[0] == 5 and c[2] == 1 and c[1] % 2]
    for c in odd:                                        # ties go to even
        assert got[cases.index(c)] % 2 == 0
