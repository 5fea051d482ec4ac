"""FP32 from both words of a double in seven integer operations, as the kernels
convert (a funnel shift, one addition that rounds and rebiases, the flush),
modelled operation for operation and checked without a GPU: against the
definition (round half away from zero to 23 mantissa bits, magnitudes below
2^-126 to signed zero) and, bit for bit, against the longer sequence of
test_convert_model, over FP32's whole range and both sides of its edges."""
from fractions import Fraction

import numpy as np

from test_convert_model import _bits64, _doubles, _f32_of_bits, _round_away
from test_convert_model import f32_from_f64_bits as long_form

M32 = 0xFFFFFFFF


def f32_from_f64_bits(lo, hi):
    funnel = ((hi << 4) | (lo >> 28)) & M32
    v = ((funnel + 0x80000001) & M32) >> 1
    return (hi & 0x80000000) | (v if ((hi << 1) & M32) >= 0x70200000 else 0)


def _edges():
    rng = np.random.default_rng(12)
    x = [2.0 ** -126, np.nextafter(2.0 ** -126, 0), np.nextafter(2.0 ** -126, 1), 2.0 ** -127, 5e-324, 0.0,
         np.float64(np.finfo(np.float32).max), 2.0 ** 127, (2 - 2.0 ** -23) * 2.0 ** 126,
         (2 - 2.0 ** -24) * 2.0 ** 126, 1.0, np.nextafter(1.0, 0), np.nextafter(2.0, 0)]
    for e in range(-126, 128):                       # every exponent, with mantissas at the rounding's edges
        for m in (0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (3 << 28) - 1, 3 << 28, (1 << 52) - (1 << 28) - 1):
            x.append(float(np.ldexp(1.0 + m * 2.0 ** -52, e)))
    x += list(np.ldexp(rng.uniform(1, 2, 4000), rng.integers(-126, 127, 4000)))
    x = np.array(x)
    return np.concatenate([x, -x, _doubles(2000, seed=3)])


def test_seven_operations_convert_to_fp32():
    for x in _edges():
        b = _bits64(x)
        bits = f32_from_f64_bits(b & M32, b >> 32)
        f = _f32_of_bits(bits)
        assert (bits >> 31) == (b >> 63)
        if abs(x) < 2.0 ** -126:
            assert f == 0.0
        else:
            assert Fraction(f) == _round_away(x, 24), x
        assert f == long_form(b & M32, b >> 32)
