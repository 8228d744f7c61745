"""The stopping test's sums of squares (csrc/hz_norm_acc.cuh) compiled on their own for the host, against exact rational
sums.  The bound for both sums of n entries is that of FP64 sums, a relative error of 2^-53 for the result alone, and
for the differences an underflow below 2^-140 of the largest entry's square.  No GPU is involved."""

import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from conftest import ROOT

SRC = r"""
#include <cstdio>
#include <vector>
#include "hz_norm_acc.cuh"

int main() {
  int n;
  while (std::scanf("%d", &n) == 1) {
    std::vector<float> now(n), before(n);
    float big = 0.f;
    for (int k = 0; k < n; ++k) {
      unsigned a, b;
      if (std::scanf("%x %x", &a, &b) != 2) return 1;
      now[k] = hz::norm_acc::from_bits(a);
      before[k] = hz::norm_acc::from_bits(b);
      big = std::fmax(std::fmax(big, std::fabs(now[k])), std::fabs(before[k]));
    }
    hz::NormAcc acc;
    acc.start(big);
    now.push_back(0.f);  // an odd one's mate
    before.push_back(0.f);
    for (int k = 0; k < n; k += 2) acc.add(make_float2(now[k], now[k + 1]), make_float2(before[k], before[k + 1]));
    double dn, un;
    acc.finish(dn, un);
    std::printf("%a %a\n", dn, un);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("norm_acc")
    (d / "t.cu").write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2606_21695_gb300", "csrc")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-I", csrc, "-o", str(d / "t"),
                    str(d / "t.cu")], check=True)

    def run(cases):
        text = "".join(f"{len(a)}\n" + "".join(f"{x:x} {y:x}\n" for x, y in zip(a.view(np.uint32), b.view(np.uint32)))
                       for a, b in cases)
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(float.fromhex(v) for v in line.split()) for line in out.splitlines()]

    return run


def _cases():
    rng = np.random.default_rng(5)
    f = np.float32
    out = []
    for n in (1, 2, 34, 50, 128):
        for scale in (1.0, 1e-30, 1e-44, 3e37):
            a = (rng.standard_normal(n) * scale).astype(f)
            for rel in (1.0, 1e-3, 3e-7, 1e-12):  # from one iterate to the next
                out.append((a, (a * (1 + rel * rng.standard_normal(n))).astype(f)))
            out.append((np.nextafter(a, f(np.inf)), a))                                   # one unit in the last place
        wide = (rng.standard_normal(n) * 10.0 ** rng.uniform(-20, 20, n)).astype(f)       # wide range in a thread
        out.append((wide, (wide * (1 + 1e-5 * rng.standard_normal(n))).astype(f)))
        out.append((np.zeros(n, f), a))                                                   # new iterate zero
        out.append((a, np.zeros(n, f)))
        out.append((np.zeros(n, f), np.zeros(n, f)))
        out.append(((1e-25 * rng.standard_normal(n)).astype(f), (1e5 * rng.standard_normal(n)).astype(f)))  # > 2^64 apart
        out.append((np.full(n, np.finfo(f).max), np.full(n, -np.finfo(f).max)))           # the largest difference
        out.append((np.full(n, np.finfo(f).smallest_subnormal), np.zeros(n, f)))
    return out


def test_sums_of_squares_are_as_good_as_fp64(sums):
    cases = _cases()
    for (now, before), (dn, un) in zip(cases, sums(cases)):
        a, b = ([Fraction(float(v)) for v in x] for x in (now, before))
        d, u = sum((x - y) ** 2 for x, y in zip(a, b)), sum(x * x for x in a)
        tiny = Fraction(2) ** -140 * max(x * x for x in a + b) * len(a)
        eps = Fraction(2) ** -53 * (1 + Fraction(2) ** -10)
        assert np.isfinite(dn) and np.isfinite(un)
        assert abs(Fraction(dn) - d) <= eps * d + tiny, (now, before)
        assert abs(Fraction(un) - u) <= eps * u + tiny, (now, before)


def test_non_finite_entries_never_pass_for_converged(sums):
    f = np.float32
    one = np.ones(4, f)
    cases = []
    for bad in (np.nan, np.inf, -np.inf):
        for both in (False, True):
            a = one.copy()
            a[2] = bad
            cases.append((a, a.copy() if both else one))
    for dn, un in sums(cases):
        assert not dn <= 1e-8 * un
