"""The minimiser's division (quick_div in fit_dev.cuh), restated with exact rational arithmetic: the FP32
reciprocal of the rounded denominator, two Newton steps for the reciprocal and one correction of the
quotient by its residual, each fused step rounded once. The FP32 reciprocal is within 1.2e-7, a Newton
step squares that (1.5e-14, then below the rounding of a double), and the correction leaves the
quotient within one unit in the last place of the exact one."""
import os
import re
from fractions import Fraction

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))   # (one rounding, to nearest even)


def _quick_div(num, den):
    d = np.float32(den)
    r = float(np.float32(1.0 / float(d)))   # 1 / d in double, then FP32: within an ulp of the rounded reciprocal
    r = _fma(r, _fma(-den, r, 1.0), r)
    r = _fma(r, _fma(-den, r, 1.0), r)
    q = num * r
    return _fma(r, _fma(-den, q, num), q)


def test_within_a_unit_in_the_last_place():
    rng = np.random.default_rng(1)
    dens = np.exp(rng.uniform(np.log(1e-29), np.log(1e29), 4000)) * rng.choice([-1.0, 1.0], 4000)
    nums = np.exp(rng.uniform(np.log(1e-30), np.log(1e30), 4000))
    nums[:500], dens[500:1000] = 1.0, 1.0 + rng.uniform(0, 1, 500)
    for num, den in zip(nums.tolist(), dens.tolist()):
        exact = Fraction(num) / Fraction(den)
        assert abs(Fraction(_quick_div(num, den)) - exact) <= Fraction(float(np.spacing(abs(float(exact)))))


def test_steps_are_those_of_the_kernel():
    src = open(os.path.join(ROOT, "paper_2502_15253_gb300", "csrc", "fit_dev.cuh")).read()
    body = src[src.index("double quick_div(double num, double den)"):]
    body = re.sub(r"\s+", " ", body[:body.index("\n}\n")])
    assert "if (!(fabsf(d) > 1e-30f && fabsf(d) < 1e30f)) return num / den;" in body
    assert body.count("r = fma(r, fma(-den, r, 1.0), r);") == 2
    assert body.endswith("const double q = num * r; return fma(r, fma(-den, q, num), q);")
