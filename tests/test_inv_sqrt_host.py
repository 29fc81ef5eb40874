"""The scale 1 / |w| of an FP32 Krylov vector from the squared norm held as an FP32 pair (csrc/dd.h, compiled on
the host with contraction disabled): 1 / sqrt(hi + lo) rounded once.

The host's estimate is within 2^-23 relatively, so the Newton step leaves 3/8 (2^-22)^2 < 2^-45 and its own
rounding about as much: 2^-44 together, 2^-19 of the half unit that the final rounding allows.  The error stays
below 0.5 + 2^-19 units in the last place (of the result's binade)."""
import shutil
import subprocess
import textwrap
from decimal import Decimal, getcontext
from fractions import Fraction

import numpy as np
import pytest

from tests.test_dd_host import CSRC

PROG = textwrap.dedent(r"""
    #include <cstdio>
    #include "dd.h"
    int main() {
      float h, l;
      while (std::scanf("%a %a", &h, &l) == 2) std::printf("%a\n", lfx::inv_sqrt_once(h, l));
      return 0;
    }
    """)


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("inv_sqrt")
    (d / "p.cpp").write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I" + CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)
    return str(d / "p")


def run(exe, pairs):
    inp = "\n".join(f"{float(h).hex()} {float(l).hex()}" for h, l in pairs) + "\n"
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout.split()
    return [float.fromhex(x) if "0x" in x else float(x) for x in out]


def exact(h, l):
    getcontext().prec = 60
    x = Fraction(float(h)) + Fraction(float(l))
    return Fraction(1 / (Decimal(x.numerator) / Decimal(x.denominator)).sqrt())


@pytest.mark.parametrize("lo_exp,hi_exp", [(-20, 20), (-79, -75), (75, 79), (-148, -110), (100, 127)])
def test_rounded_once(exe, lo_exp, hi_exp):
    rng = np.random.default_rng(hi_exp + 200)
    n = 400
    h = (rng.uniform(1.0, 2.0, n) * np.exp2(rng.integers(lo_exp, hi_exp, n))).astype(np.float32)
    l = (rng.uniform(-0.5, 0.5, n) * np.spacing(h).astype(np.float64)).astype(np.float32)
    keep = h > 0
    for (a, b), y in zip(zip(h[keep], l[keep]), run(exe, zip(h[keep], l[keep]))):
        want = exact(a, b)
        ulp = Fraction(float(np.spacing(np.float32(y))))
        assert abs(Fraction(y) - want) <= (Fraction(1, 2) + Fraction(1, 2 ** 19)) * ulp, (a, b, y)


def test_limits(exe):
    assert run(exe, [(0.0, 0.0), (float("nan"), 0.0), (float("inf"), 0.0), (1.0, 0.0), (4.0, 0.0)]) == [0.0, 0.0, 0.0, 1.0, 0.5]
