"""The compensated-FP32 form's 8-operation accumulation step (the kernel that
keeps the inner sums in scratch, two rows per packed operation), modelled on
the host with every FP32 rounding reproduced and checked against exact
rational arithmetic without a GPU.

acc += x y with h = x y rounded: s = hi + h, z = s - hi, and TwoSum's two
error terms, a = hi - (s - z) and, in place of (h - z) plus the product's
residual x y - h, b = fma(x, y, -z): the same exact quantity in one rounding
instead of two (h - z is exact, so the 10-operation step rounds the residual's
sum where this one rounds b).  The inner sum's pair enters the outer sum as
one step on its high word and one FMA on its low word.

The bound is Dot2's (test_fp32c_dot2_model): one rounding of the result plus
c n^2 2^-48 sum |w u e| with c n^2 = 2^8.  Also on sums that cancel: each
second term the negative of the one before it but for its last bits."""
from fractions import Fraction

import numpy as np
import pytest

from fp32_model import F32, Q, add, f32, fma, mul, sub
from test_fp32c_dot2_model import dot2_step


def packed_step(acc, x, y):
    h = mul(x, y)
    s = add(acc[0], h)
    z = sub(s, acc[0])
    a = sub(acc[0], sub(s, z))
    b = fma(x, y, -z)
    return (s, add(acc[1], add(a, b)))


def contracted_step(acc, x, y):
    """The step with its product contracted into the addition that follows."""
    s = fma(x, y, acc[0])
    z = sub(s, acc[0])
    a = sub(acc[0], sub(s, z))
    b = fma(x, y, -z)
    return (s, add(acc[1], add(a, b)))


def h_value(CX, CY, E, step):
    acc = (F32(0), F32(0))
    for p0 in range(E.shape[0]):
        F = (F32(0), F32(0))
        for p2 in range(E.shape[1]):
            F = step(F, CY[p2], E[p0, p2])
        acc = step(acc, CX[p0], F[0])
        acc = (acc[0], fma(CX[p0], F[1], acc[1]))
    return add(acc[0], acc[1])


def _cases(cancel):
    rng = np.random.default_rng(9)
    for _ in range(12):
        E = rng.standard_normal((32, 32)) * 10.0 ** rng.uniform(-6, 0, (32, 32))
        E = np.array([[f32(Q(v)) for v in row] for row in E], dtype=np.float32)
        CX = rng.standard_normal(32).astype(np.float32)
        CY = rng.standard_normal(32).astype(np.float32)
        if cancel:
            CY[1::2] = CY[::2]
            E[:, 1::2] = -E[:, ::2] * (1 + rng.integers(-8, 9, (32, 16)) * 2.0 ** -22).astype(np.float32)
        yield CX, CY, E


def _worst(step, cancel):
    """Largest (|H - exact| - 2^-24 |exact|) / (2^-40 sum |w u e|) over the cases."""
    worst = Fraction(0)
    for CX, CY, E in _cases(cancel):
        terms = [Q(CX[p]) * Q(CY[q]) * Q(E[p, q]) for p in range(32) for q in range(32)]
        exact, mag = sum(terms), sum(abs(t) for t in terms)
        err = abs(Q(h_value(CX, CY, E, step)) - exact)
        worst = max(worst, (err - abs(exact) / 2 ** 24) * 2 ** 40 / mag)
    return float(worst)


@pytest.mark.parametrize("cancel", [False, True])
def test_packed_step_reaches_the_bound(cancel):
    w, w10 = _worst(packed_step, cancel), _worst(dot2_step, cancel)
    print(f"share of the bound's second term: 8 operations {w:.4f}, 10 operations {w10:.4f}")
    assert w <= 1.0 and w10 <= 1.0


def test_step_is_error_free_where_the_sum_is():
    """hi + lo after one step from (hi, 0): hi + x y but for the roundings of b
    (a half ulp of an error term, 2^-48 of the larger operand) and of a + b."""
    rng = np.random.default_rng(2)
    for _ in range(2000):
        x, y = (F32(v) for v in rng.standard_normal(2))
        hi = F32(-float(x) * float(y) * (1 + 2.0 ** -rng.integers(10, 24))) if rng.integers(2) else F32(rng.standard_normal())
        s, lo = packed_step((hi, F32(0)), x, y)
        exact = Q(hi) + Q(x) * Q(y)
        assert abs(Q(s) + Q(lo) - exact) <= (abs(Q(hi)) + abs(Q(x) * Q(y))) / 2 ** 46


def test_contracted_product_is_not():
    """The reason the product is two scalar multiplications."""
    rng = np.random.default_rng(2)
    worst = 0.0
    for _ in range(2000):
        x, y, hi = (F32(v) for v in rng.standard_normal(3))
        s, lo = contracted_step((hi, F32(0)), x, y)
        exact = Q(hi) + Q(x) * Q(y)
        worst = max(worst, float(abs(Q(s) + Q(lo) - exact) / (abs(Q(hi)) + abs(Q(x) * Q(y)))))
    print(f"contracted: 2^{np.log2(worst):.1f}")
    assert worst > 2.0 ** -40
