"""Constants of the FP64 collision (csrc/olb_fold.h): in exact arithmetic on the rounded
constants a step must leave mass and momentum unchanged, or every step would multiply
them by the same factor beside 1 and the error would grow with the number of steps.

The header is compiled with the host compiler; the sums are evaluated as fractions."""
import os
import shutil
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2307_11752_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "olb_fold.h"
int main() {
  int dim;
  double omega, odd;
  while (std::scanf("%d %la %la", &dim, &omega, &odd) == 3) {
    const olb::Fold64 r = olb::fold64_rates(dim, omega, odd);
    std::printf("%a %a %a %a %a %a %a %a\n", r.keep, 2.0 * r.odd, r.ow[0], r.ow[1], r.ow[2], r.t[1], r.t[2], 2.0 * r.even);
  }
}
"""


def _rates():
    taus = [0.5 + 2.0 ** -k for k in range(1, 30)]
    taus += [0.5001, 0.52, 0.54725, 0.55, 0.6, 0.62, 0.7, 0.75, 0.8, 0.9, 1.0, 1.1, 1.25, 1.3, 1.5, 1.7, 1.99, 2.0]
    taus += [2.01, 3.0, 5.5, 10.0, 64.0, 1000.0, 1e6]
    taus += [0.5 + 0.0137 * k for k in range(1, 400)]
    for tau in taus:
        omega = 1.0 / tau
        yield omega, omega
        for magic in (1e-4, 3.0 / 16.0, 0.25, 7.0):
            yield omega, 1.0 / (magic / (tau - 0.5) + 0.5)


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
@pytest.mark.parametrize("dim", [2, 3])
def test_a_step_keeps_mass_and_momentum_exactly(tmp_path, dim):
    src, exe = tmp_path / "drv.cpp", tmp_path / "drv"
    src.write_text(DRIVER)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    rates = list(_rates())
    text = "".join(f"{dim} {a.hex()} {b.hex()}\n" for a, b in rates)
    r = subprocess.run([str(exe)], input=text, capture_output=True, text=True)
    lines = r.stdout.splitlines()
    assert r.returncode == 0 and len(lines) == len(rates)
    n1, n2, m = (4, 4, 4) if dim == 2 else (6, 12, 8)
    w = (4 / 9, 1 / 9, 1 / 36) if dim == 2 else (1 / 3, 1 / 18, 1 / 36)
    for (omega, odd), line in zip(rates, lines):
        keep, keep_odd, ow0, ow1, ow2, t1, t2, keep_even = map(float.fromhex, line.split())
        assert keep == keep_even == 1.0 - omega and keep_odd == 1.0 - odd
        F = Fraction
        assert F(keep) + F(ow0) + n1 * F(ow1) + n2 * F(ow2) == 1, (omega, odd)
        assert F(keep_odd) + 2 * F(t1) + m * F(t2) == 1, (omega, odd)
        # and each constant is the product it stands for: the small ones to 4 units in the
        # last place, the remainders to what 1 - omega's own rounding leaves of them
        for got, want, slack in ((ow1, omega * w[1], 0.0), (ow2, omega * w[2], 0.0), (t2, 3 * odd * w[2], 0.0),
                                 (ow0, omega * w[0], 2.0 ** -53), (t1, 3 * odd * w[1], 2.0 ** -53)):
            assert abs(got - want) <= 2.0 ** -50 * want + slack, (omega, odd)
