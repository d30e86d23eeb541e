"""The exponential that the scoring kernels evaluate on the FMA pipe, its fp32 steps repeated in numpy (no GPU)."""
import os
import re

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_19906_b200", "csrc", "exp2.cuh")
f32 = np.float32


def coefficients():
    text = re.search(r"kExp2Poly\[7\] = \{(.*?)\};", open(SRC).read(), re.S).group(1)
    return [f32(c.strip().rstrip("f")) for c in text.split(",")]


def fma(a, b, c):
    """fp32 fused multiply-add: the product is exact in fp64, the sum is rounded twice (to fp64, then to fp32)."""
    return (a.astype(np.float64) * b.astype(np.float64) + np.float64(c)).astype(f32)


def exp2_factors(x, k=f32(12582912.0)):
    x = np.clip(x, f32(-127), f32(128))             # (NaN stays NaN)
    t = x + k
    f = x - (t - k)
    c = coefficients()
    p = np.full_like(f, c[-1])
    for a in c[-2::-1]:
        p = fma(p, f, a)
    pow2 = ((t.view(np.uint32) << np.uint32(23)) + np.uint32(0x3F800000)).view(f32)
    with np.errstate(all="ignore"):
        r = p * pow2
    return np.where(np.abs(r) < f32(2.0 ** -126), f32(0), r)      # .ftz


def test_error_is_below_that_of_the_special_function_unit():
    """Measured for ex2.approx.ftz on [-30, 0]: 1.42e-7 at the most, mean -5.1e-8, rms 5.9e-8."""
    for lo, hi in ((-1, 0), (-30, 0), (-125.9, 0), (0, 127.4)):
        x = np.linspace(lo, hi, 2000001).astype(f32)
        e = exp2_factors(x).astype(np.float64) / np.exp2(x.astype(np.float64)) - 1
        assert np.abs(e).max() < 7e-8 and abs(e.mean()) < 1e-9 and np.sqrt((e ** 2).mean()) < 3e-8


def test_ends_of_the_range():
    x = np.array([-np.inf, -1e30, -200, -127, -126.6, -126.4, 128, 129, 1e30, np.inf], dtype=f32)
    np.testing.assert_array_equal(exp2_factors(x), [0, 0, 0, 0, 0, 0, np.inf, np.inf, np.inf, np.inf])
    assert exp2_factors(np.array([-126, 0, 127], dtype=f32)).tolist() == [2.0 ** -126, 1.0, 2.0 ** 127]
    assert np.isnan(exp2_factors(np.array([np.nan], dtype=f32)))[0]
