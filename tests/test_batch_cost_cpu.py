"""The estimate that orders a batch's detectors (csrc/batchcost.cuh), compiled for the host: within
a fifth of the measured steps of every precision at LFI size, so that detectors of unlike
precisions are ordered by their times."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include <stdio.h>
#include "batchcost.cuh"
int main() {
    const int modes[4] = {SL_FP32, SL_TF32X3, SL_FP64, SL_DF64};
    for (int m : modes) printf("%.6g\n", sl::batch_cost_ms(m, 6.63e9, 17e8));
}
"""


def test_the_estimate_is_the_measured_step(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-x", "c++", "-I", os.path.join(ROOT, "paper_2201_03478_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    got = [float(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]
    for ms, measured in zip(got, (7.95, 14.3, 51.0, 44.7)):
        assert 0.8 * measured <= ms <= 1.2 * measured, (got, measured)
