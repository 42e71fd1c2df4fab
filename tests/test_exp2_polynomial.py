"""The polynomial that takes a share of the attention kernel's exponentials: its coefficients, read from the source, in the
kernel's order of fp32 operations, against 2^x in 64 bits."""

import os
import re

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_01805_b200", "csrc", "attn_tc.cu")


def _exp2_poly(x):
    body = open(SRC).read().split("void exp2_poly2")[1].split("\n}\n")[0]
    floor = np.float32(re.search(r"max_nan\(x0, (-[0-9.]+)f\)", body).group(1))
    coef = [np.float32(re.search(r"uint64_t y = pack_f32x2\(([0-9.]+)f", body).group(1))]
    coef += [np.float32(c) for c in re.findall(r"fma_f32x2\(y, f, pack_f32x2\(([0-9.]+)f", body)]
    assert len(coef) == 6
    magic = np.float32(12582912.0)
    x = np.maximum(x.astype(np.float32), floor)
    t = x + magic
    n = t - magic
    f = (x.astype(np.float64) - n).astype(np.float32)
    y = np.full_like(x, coef[0])
    for c in coef[1:]:   # fused: the product of two fp32 is exact in 64 bits, one rounding at the end
        y = (y.astype(np.float64) * f + c).astype(np.float32)
    scale = ((t.view(np.uint32) << np.uint32(23)) + np.uint32(0x3F800000)).view(np.float32)
    return y * scale


def test_relative_error_over_the_normal_range():
    x = np.concatenate([np.linspace(-126, 100, 2_000_001), np.arange(-126, 101), np.arange(-126, 100) + 0.5]).astype(np.float32)
    ref = np.exp2(x.astype(np.float64))
    assert np.abs(_exp2_poly(x) / ref - 1).max() <= 1.7e-7


def test_zero_where_the_weight_is_nothing():
    x = np.array([-127.0, -127.5, -200.0, -1e30, -np.inf], np.float32)
    assert (_exp2_poly(x) == 0).all()
    # between: no more than the smallest normal number, as ex2.approx.ftz gives it to within that number
    x = np.linspace(-127, -126, 1001).astype(np.float32)
    got = _exp2_poly(x).astype(np.float64)
    assert (got >= 0).all() and (np.abs(got - np.exp2(x.astype(np.float64))) <= 2.0 ** -126).all()
