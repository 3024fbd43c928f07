"""The anchor index difference of a separation is wrapped to its nearest
periodic image in FP32 (k - n rint(k / n), 1 / n rounded down, the rounding by
one FMA onto 1.5 2^23): the same index as the integer rule, for every lattice
size and at every k where the rule changes."""
from fractions import Fraction

import numpy as np


def _wrapped(k, n, inv):
    # the FMA's exact value rounds to a whole number (one unit in the last
    # place of 1.5 2^23 is 1), ties to even
    return k - n * round(Fraction(k) * inv)


def test_float_wrap_equals_the_integer_rule():
    for n in list(range(1, 2100)) + list(range(2100, 65536, 37)) + [65535]:
        r = np.float32(1.0 / n)
        inv = Fraction(float(np.nextafter(r, np.float32(0.0), dtype=np.float32)))
        assert inv < Fraction(1, n)
        half = n // 2
        for k in {0, 1, half - 1, half, half + 1, n - 1}:
            for q in (k, -k):
                if abs(q) >= n:
                    continue
                want = q - n if 2 * q > n else q + n if 2 * q < -n else q
                assert _wrapped(q, n, inv) == want, (n, q)
