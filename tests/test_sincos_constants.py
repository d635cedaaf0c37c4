"""sin and cos of pi r as the evaluation kernels form them, read from the source."""
import os
import re

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sincos_polynomials():
    """FP32 Horner with fused multiply-adds over |r| <= 1/2: two roundings of values below 1 and the fit's
    5e-9, so both within 2 * 2^-24 + 1e-8; the packed form carries the same constants."""
    src = open(os.path.join(ROOT, "paper_2502_15253_gb300", "csrc", "dev_model.cuh")).read()
    one = src[src.index("void sincos_half(float r"):]
    one = one[:one.index("\n}\n")]
    two = src[src.index("void sincos_half2(f32x2 r"):]
    two = two[:two.index("\n}\n")]
    num = r"-?\d+\.\d+(?:e-?\d+)?f"
    k = [x for x in re.findall(num, one)]
    assert k == re.findall(num, two)
    t = [np.float32(x[:-1]) for x in k if x != "3.14159274f" and x != "1.f"]
    fma = lambda a, b, c: (a.astype(np.float64) * b + np.float64(c)).astype(np.float32)
    r = np.linspace(-0.5, 0.5, 1_000_001).astype(np.float32)
    u = (r * r).astype(np.float32)
    p, q = np.full_like(u, t[0]), np.full_like(u, t[5])
    for c in t[1:5]:
        p = fma(p, u, c)
    for c in t[6:] + [np.float32(1)]:
        q = fma(q, u, c)
    pi = np.float32(np.pi)
    s = ((r * p).astype(np.float32).astype(np.float64) + r.astype(np.float64) * pi).astype(np.float32)
    bar = 2 * 2.0 ** -24 + 1e-8
    R = np.pi * r.astype(np.float64)
    assert np.abs(s - np.sin(R)).max() < bar
    assert np.abs(q - np.cos(R)).max() < bar
