"""The training kernel's GELU and slope (gelu_tail2 and gelu_and_grad2 in
csrc/mlp.cu), restated step by step in FP32 with the source's own constants, are
within the errors the kernel states of x Phi(x) and Phi(x) + x phi(x).  Every
operation is rounded once (products and sums in FP64, then to FP32, as the fused
multiply-adds round); 2^x is rounded from FP64, and shifted by the two ulps the
instruction may be off."""
import math
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_18401_gb300", "csrc", "mlp.cu")
f32, f64 = np.float32, np.float64


def constants():
    text = open(SRC).read()
    c = re.search(r"constexpr float c\[8\] = \{([^}]*)\}", text).group(1)
    return [f32(v.strip().rstrip("f")) for v in c.split(",")]


def fma(a, b, c):
    return (f64(a) * f64(b) + f64(c)).astype(f32)


def ex2(x, ulps):
    y = np.exp2(f64(x)).astype(f32)
    y = np.where(y < f32(2.0 ** -126), f32(0.0), y)  # flushes subnormal results
    return (y.view(np.int32) + np.where(y > 0, ulps, 0).astype(np.int32)).view(f32)


def gelu_and_slope(x, ulps):
    c = constants()
    h = f32(-0.5) * np.abs(x)
    s = np.full_like(x, c[7])
    for k in range(6, -1, -1):
        s = fma(s, h, np.full_like(x, c[k]))
    e = ex2((f64(s) * f64(h)).astype(f32), ulps)
    g = fma(h, e, np.maximum(x, f32(0)))
    hh = (f64(h) * f64(h)).astype(f32)
    d = ex2((f64(hh) * f64(f32(-2.8853900817779268))).astype(f32), ulps)
    p = np.where(x >= 0, fma(e, np.full_like(e, f32(-0.5)), np.ones_like(e)), f32(0.5) * e)
    xs = (f64(x) * f64(f32(0.39894228040143268))).astype(f32)
    return g, fma(xs, d, p)


def points():
    rng = np.random.default_rng(4)
    return np.concatenate([rng.uniform(-6, 6, 200_000), rng.normal(0, 1, 100_000), rng.uniform(-40, 40, 50_000),
                           10.0 ** rng.uniform(-30, 30, 20_000) * rng.choice([-1, 1], 20_000),
                           [0.0, -0.0, 5.8, -5.8, 1e20, -1e20, 3e38, -3e38]]).astype(f32)


@pytest.mark.parametrize("ulps", [-2, 0, 2])
def test_within_the_stated_errors(ulps):
    x = points()
    with np.errstate(over="ignore", invalid="ignore", under="ignore"):
        g, dg = gelu_and_slope(x, ulps)
    X = x.astype(f64)
    cdf = np.array([0.5 * math.erfc(-v / math.sqrt(2.0)) for v in X])
    with np.errstate(over="ignore", under="ignore"):
        pdf = np.exp(-0.5 * X * X) / math.sqrt(2.0 * math.pi)
    slack = 1.2e-7 * (ulps != 0)  # two ulps of 2^x <= 1 reach the result halved
    assert np.max(np.abs(g - X * cdf) / np.maximum(1.0, np.abs(X))) <= 8.5e-8 + slack
    assert np.max(np.abs(dg - (cdf + np.where(np.isinf(X * X), 0.0, X * pdf)))) <= 1.35e-7 + slack
