"""Host-side check of the claims the GPTQ kernel's short rounding step rests on (csrc/gptq.cu): with d of 24 bits and
1 / d = yh + yl by three Newton steps from any 22-bit approximation, fma(x, yh, x yl) is the correctly rounded quotient x / d; and
the upper word of the distance to a code tells every quotient that could round the other way."""
import math
from fractions import Fraction

import numpy as np


def _rn(q: Fraction) -> float:
    return float(q)  # CPython rounds a rational to the nearest double, ties to even


def _fma(a: float, b: float, c: float) -> float:
    return _rn(Fraction(a) * Fraction(b) + Fraction(c))


def _reciprocal_pair(d: float, y0: float):
    y1 = _fma(y0, _fma(-d, y0, 1.0), y0)
    yh = _fma(y1, _fma(-d, y1, 1.0), y1)
    return yh, _rn(Fraction(yh) * Fraction(_fma(-d, yh, 1.0)))


def test_two_part_reciprocal_divides_correctly():
    rng = np.random.default_rng(11)
    for trial in range(400):
        d = float(np.float32(np.ldexp(rng.uniform(1, 2), int(rng.integers(-90, 90)))) * (1 if trial % 3 else -1))
        if trial % 5 == 0:
            d = float(np.nextafter(np.float32(abs(d)), np.float32(np.inf)))  # odd significands
        approx = float(np.float32(1.0 / d)) * (1 + rng.uniform(-1, 1) * 2.0 ** -22)
        yh, yl = _reciprocal_pair(d, float(np.float32(approx)))
        assert abs(Fraction(yh) + Fraction(yl) - 1 / Fraction(d)) <= abs(1 / Fraction(d)) / 2 ** 99
        for _ in range(20):
            x = float(np.ldexp(rng.uniform(-1, 1), int(rng.integers(-200, 200))))
            # next to the midpoint of two doubles, where a quotient by a 24-bit number comes as near as it can
            if rng.random() < 0.5:
                m = Fraction(2 * int(rng.integers(2 ** 52, 2 ** 53)) + 1, 2 ** 53)
                x = _rn(m * Fraction(d))
            want = _rn(Fraction(x) / Fraction(d))
            assert _fma(x, yh, _rn(Fraction(x) * Fraction(yl))) == want
        assert _fma(0.0, yh, 0.0 * yl) == 0.0


def test_codes_are_refused_wherever_the_product_could_round_apart():
    rng = np.random.default_rng(12)
    refused = 0
    for _ in range(3000):
        s = float(np.float32(np.exp(rng.uniform(-12, 2))))
        s_inv = _rn(1 / Fraction(s))
        k = int(rng.integers(-300, 300))
        w = _rn(Fraction(s) * (Fraction(k) + Fraction(1, 2))) * (1 + float(rng.choice([0, 1, -1, 3, 1e4])) * 2.0 ** -52)
        if rng.random() < 0.5:
            w = float(rng.uniform(-300, 300)) * s
        for hi in (127, 7):
            t = Fraction(w) * Fraction(s_inv)
            fast = min(max(round(t), -hi - 1), hi)
            want = min(max(round(Fraction(_rn(Fraction(w) / Fraction(s)))), -hi - 1), hi)  # rint of the rounded quotient, clipped
            frac = np.float64(abs(_fma(w, s_inv, -float(fast))))
            upper = int(frac.view(np.uint64) >> np.uint64(32))
            if upper in (0x3FDFFFFF, 0x3FE00000) or upper >= 0x40780000:
                refused += 1
            else:
                assert fast == want, (w, s)
    assert refused > 500 and math.isfinite(refused)
