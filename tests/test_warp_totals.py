"""The sum of the warps' totals of a target (sum_totals of msp_hostdev.cuh)
against exact sums: up to four totals in order, more with the lost parts
collected.  Bounds: N - 1 roundings in order; with the lost parts two, plus
terms of second order (N^2 2^-48 of the sum of magnitudes)."""
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include "msp_hostdev.cuh"
int main() {
    float v[TOTALS];
    while (std::fread(v, 4, TOTALS, stdin) == TOTALS) {
        const float s = msp::sum_totals<TOTALS>([&](int k) { return v[k]; });
        std::fwrite(&s, 4, 1, stdout);
    }
    return 0;
}
"""


@pytest.mark.parametrize("n", [4, 8, 16])
def test_sum_of_the_warps_totals(tmp_path, n):
    src, exe = tmp_path / "sum.cpp", tmp_path / "sum"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O2", f"-DTOTALS={n}", "-x", "c++", "-I",
                           os.path.join(ROOT, "paper_2301_10570_gb300", "csrc"), str(src), "-o",
                           str(exe)])
    rng = np.random.default_rng(n)
    v = np.concatenate([
        rng.uniform(0, 1, (4000, n)), np.exp(rng.uniform(-20, 5, (4000, n))),
        np.where(np.arange(n) == 0, 2.0 ** 24, 1.0)[None].repeat(2, 0),   # ones lost in order
        np.zeros((1, n))]).astype(np.float32)
    got = np.frombuffer(subprocess.run([str(exe)], input=v.tobytes(), capture_output=True,
                                       check=True).stdout, np.float32)
    assert got.shape == (len(v),)
    for row, s in zip(v.astype(np.float64), got):
        exact, mag = math.fsum(row), float(np.abs(row).sum())
        bound = (3 if n == 4 else 2) * 2.0 ** -24 * abs(exact) + n * n * 2.0 ** -48 * mag
        assert abs(float(s) - exact) <= bound
