"""The FP64 reciprocal of the tau = 0 kernels (csrc/gks_rcp.cuh) restated in exact arithmetic: within one
ulp of 1/x over the range the launch rules allow, for any FP32 seed within 1 ulp."""
from fractions import Fraction

import numpy as np
import pytest


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))     # one rounding


@pytest.mark.parametrize("seed_ulp", [-1, 0, 1])
def test_fp64_reciprocal_is_within_an_ulp(seed_ulp):
    rng = np.random.default_rng(5 + seed_ulp)
    xs = list(rng.uniform(1.0, 2.0, 1500) * 2.0 ** rng.integers(-110, 111, 1500))
    xs += [1.0, 2.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0), 3.0, 2.0 ** -100, 2.0 ** 101]
    for x in xs:
        u = int(np.float64(x).view(np.uint64))
        hi, lo = u >> 32, u & 0xffffffff
        f = np.uint32((((hi - (896 << 20)) << 3) | (lo >> 29)) & 0xffffffff).view(np.float32)
        assert 0 <= x - float(f) < x * 2.0 ** -23
        b = int((np.float32(1.0) / f).view(np.int32)) + seed_ulp
        r = float(np.uint64((((b >> 3) + (896 << 20)) << 32) | ((b << 29) & 0xffffffff)).view(np.float64))
        assert r == float(np.int32(b).view(np.float32))
        e = _fma(-x, r, 1.0)
        q = _fma(r, _fma(e, e, e), r)
        err = abs(Fraction(q) * Fraction(float(x)) - 1) / Fraction(2) ** -52
        assert err <= 1, (x, float(err))
