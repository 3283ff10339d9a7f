"""The integer digits of the float64 tensor-core products, restated in exact integers: what they hold and drop.

Nine-bit form (gradient): f = round(v 2^(1083 - e)) as seven digits of at most 256, digit products of weight
d = s + t <= 6 kept.  Eight-bit form (Grams): f = round(v 2^(1084 - e)) as eight digits of at most 128, d <= 7 kept.
Bounds per term, in units of the power of two of either vector's largest magnitude: what is dropped and half a unit
of either f times the other.
"""
import math
import random
from fractions import Fraction

import pytest

FORMS = {"nine": (9, 7, 60, Fraction(720, 100) / 2 ** 59), "eight": (8, 8, 61, Fraction(804, 100) / 2 ** 60)}


def fixed(v, e, top):
    """round(v 2^(1023 + top - e)) as the device rounds it (ties away from zero)."""
    f = Fraction(v) * Fraction(2) ** (1023 + top - e)
    return int(math.copysign(1, v)) * int(abs(f) + Fraction(1, 2))


def digits(f, bits, count):
    q = []
    for s in range(count - 1, -1, -1):
        half = 1 << (bits - 1)
        lo = ((f + half) % (1 << bits)) - half if s > 0 else f
        f = (f - lo) >> bits
        q.insert(0, lo)
    return q


def exponent(vec):
    return max(math.frexp(v)[1] + 1022 for v in vec if v)


def product(a, b, form):
    """(kept digit products, bound in the same unit, exact) of sum a_k b_k, as fractions."""
    bits, count, top, _ = FORMS[form]
    ea, eb = exponent(a), exponent(b)
    acc = [0] * count
    for x, y in zip(a, b):
        qa, qb = digits(fixed(x, ea, top), bits, count), digits(fixed(y, eb, top), bits, count)
        assert all(abs(q) <= 1 << (bits - 1) for q in qa + qb)
        assert abs(qa[0]) <= (1 << (top + 1 - bits * (count - 1))) + 1
        for d in range(count):
            acc[d] += sum(qa[s] * qb[d - s] for s in range(d + 1))
    unit = Fraction(2) ** (ea + eb - 2 * (1023 + top))
    kept = sum(v << (bits * (2 * (count - 1) - d)) for d, v in enumerate(acc)) * unit
    ref = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
    return kept, Fraction(2) ** (ea + eb - 2046) * len(a), ref, acc


def extreme(form, rng):
    """A value near a power of two whose lower digits are all the most negative."""
    bits, count, top, _ = FORMS[form]
    f = (1 << top) + (1 << (bits * (count - 1)))
    for s in range(1, count):
        f -= 1 << (bits * (count - 1 - s) + bits - 1)
    f -= f % (1 << (top - 52))
    return math.ldexp(float(f), -top)


def vectors(form, kind, n, seed):
    rng = random.Random(seed)
    if kind == "extreme":
        return [extreme(form, rng)] * n, [extreme(form, rng)] * n
    if kind == "small":                           # one large value, the rest far below it
        return ([1.0] + [math.ldexp(rng.uniform(1, 2), -rng.randint(5, 70)) for _ in range(n - 1)],
                [math.ldexp(rng.uniform(1, 2), -rng.randint(5, 70)) for _ in range(n - 1)] + [1.5])
    return [rng.uniform(-2, 2) for _ in range(n)], [rng.uniform(-2, 2) for _ in range(n)]


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("kind", ["extreme", "small", "random"])
@pytest.mark.parametrize("n", [1, 16, 42, 43, 48, 64])
def test_what_the_digits_drop(form, kind, n):
    for seed in range(5):
        kept, unit, ref, _ = product(*vectors(form, kind, n, seed), form)
        assert abs(kept - ref) <= FORMS[form][3] * unit


def test_the_nine_bit_bound_is_nearly_reached():
    kept, unit, ref, _ = product(*vectors("nine", "extreme", 48, 0), "nine")
    assert abs(kept - ref) > unit / 2 ** 57


def test_accumulators_stay_whole_in_float32():
    """Below 2^24 every partial sum is exact; the nine-bit form's lowest one passes it from 43 terms on, where the
    few units a rounding may take (two per product and term, say) weigh 2^54: the 0.19 2^61 per term that the
    bound of 7.2 2^61 leaves over what the digits drop holds them."""
    for k in range(1, 49):
        most = [k * sum(256 * 256 if 0 < s < d else 128 * 256 for s in range(d + 1)) for d in range(7)]
        assert max(most[:6]) < 2 ** 24
        assert (most[6] < 2 ** 24) == (k <= 42)
        assert 2 ** 54 * 2 * 7 * k <= 0.19 * 2 ** 61 * k
    most = [64 * sum(128 * 128 if 0 < s < d else 65 * 128 for s in range(d + 1)) for d in range(8)]
    assert max(most) < 2 ** 23
