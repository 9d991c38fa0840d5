"""The per-atmosphere adjoint's path-length sums (csrc/sum3.h, compiled for the host): no less
accurate than FP64 additions of the same FP32 terms, for alternating terms, a wide range and sums
that cancel; and where a partial sum leaves FP32's range, what FP64 additions give."""
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1912_07759_gb300", "csrc")
PROBE = r'''
#include <cstdio>
#include <vector>
#include "sum3.h"
int main() {
  int n;
  while (std::scanf("%d", &n) == 1) {
    std::vector<float> v(n);
    for (float& x : v) std::scanf("%a", &x);
    std::printf("%a\n", tr::sum_fp32_terms([&](auto add) {
      for (int i = 0; i < n; i += 2) add(v[i], i + 1 < n ? v[i + 1] : 0.f);
    }));
  }
}
'''


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    d = tmp_path_factory.mktemp("sum3")
    (d / "p.cpp").write_text(PROBE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + CSRC, "-o", str(d / "p"), str(d / "p.cpp")],
                   check=True)

    def run(rows):
        text = "\n".join(f"{len(r)} " + " ".join(float(x).hex() for x in r) for r in rows)
        out = subprocess.run([str(d / "p")], input=text, capture_output=True, text=True, check=True)
        return [float.fromhex(x) for x in out.stdout.split()]
    return run


def test_sums_are_as_accurate_as_fp64_additions(sums):
    rng = np.random.default_rng(4)
    rows = []
    for n in (1, 2, 17, 100, 180):
        v = rng.normal(size=(40, n))
        rows += list(v) + list(v * 10.0 ** rng.uniform(-9, 9, v.shape)) + list(np.cumsum(v, 1) * 1e7)
    rows = [r.astype(np.float32) for r in rows]
    rows += [np.concatenate([r, rng.permutation(-r)]) for r in rows]     # sums that cancel
    for r, s in zip(rows, sums(rows)):
        exact, peak = math.fsum(map(float, r)), float(np.abs(r.astype(np.float64)).sum())
        # rounding to FP64, and n^2 2^-72 of the partial sums (n <= 360)
        assert abs(s - exact) <= 2.0 ** -53 * abs(exact) + 2.0 ** -55 * peak


def test_sums_beyond_the_range_of_fp32(sums):
    big = np.float32(3e38)
    rows = [[big, big, -big, 1.0], [big] * 8, [-big, -big, big, big, 2.5], [np.inf, 1.0, big],
            [np.inf, -np.inf], [1.0, np.nan]]
    for r, s in zip(rows, sums(rows)):
        ref = 0.0
        for x in r:
            ref += float(np.float32(x))
        assert s == ref or (math.isnan(s) and math.isnan(ref)), (r, s, ref)
