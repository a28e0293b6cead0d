"""The projection on a level set, whose quotient comes from a reciprocal and two corrections: bit for bit what the correctly
rounded single-precision division gives, at half levels and their neighbours, for spacings of every kind of mantissa and
where the quotient is tiny, overflows or is not a number."""

import numpy as np
import pytest

from paper_2105_09837_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [2, 16, 256, 2048, 65536])
@pytest.mark.parametrize("scale", [1.0, 1.9999999, 1.0000001, 0.1, 0.011764706, 3.3333333e-5, 7.7e18, 9.99e-20, 1e-20, 9.9e-21,
                                   1e-30, 3e25])
def test_codes_are_those_of_the_rounded_division(m, scale):
    f = np.float32
    scale = f(scale)
    lo = f(-3) * scale
    rng = np.random.default_rng(m)
    with np.errstate(all="ignore"):
        half = lo + (rng.integers(-2, m + 2, 200000).astype(f) + f(0.5)) * scale
        x = np.concatenate([half, np.nextafter(half, f(np.inf)), np.nextafter(half, f(-np.inf)),
                            (rng.uniform(-2, m + 2, 200000) * scale).astype(f), rng.standard_normal(1000).astype(f) * f(1e-38),
                            np.array([0.0, -0.0, 3e38, -3e38, np.inf, -np.inf, np.nan, 1e-45], dtype=f)]).astype(f)
        v = np.floor((x - lo) / scale + f(0.5))
        want = np.where(np.isnan(v), f(0), np.clip(v, f(0), f(m - 1)))
    codes, p = B.quantize(x, float(scale), m, lo=float(lo))
    assert np.array_equal(codes, want.astype(codes.dtype))
    assert np.array_equal(p, lo + want * scale)
