"""The balanced base-2^8 digit split behind the byte-digit tensor-core product, on the host.

X = rint(x 2^(8 ND - e)), |X| <= 2^(8 ND - 1), is cut into ND digits (7; 5 for corrections) with
one addition: byte k of Y = X + sum_k 128 2^(8k) (the ND - 1 low bytes), minus 128, is the digit of
weight 2^(8k) and Y >> 8 (ND - 1) the top one.  The digits must reproduce X and stay within 128,
so that they are exact in FP16, and an accumulator's sum must stay exact in FP32.
"""
import random

import pytest


def _digits(X, nd):
    Y = X + sum(128 << (8 * k) for k in range(nd - 1))
    return [((Y >> (8 * k)) & 255) - 128 for k in range(nd - 1)] + [Y >> (8 * (nd - 1))]


@pytest.mark.parametrize("nd", [5, 7])
def test_digits_reproduce_the_value(nd):
    rng = random.Random(nd)
    top = 8 * nd - 1
    xs = [0, 1, -1, 127, 128, -128, -129, 1 << top, -(1 << top), (1 << top) - 1]
    xs += [sum(127 << (8 * k) for k in range(nd)), -sum(128 << (8 * k) for k in range(nd - 1))]
    xs += [rng.randrange(-(1 << top), (1 << top) + 1) for _ in range(20000)]
    xs += [rng.randrange(-(1 << b), 1 << b) for b in range(1, top) for _ in range(50)]
    for X in xs:
        d = _digits(X, nd)
        assert sum(v << (8 * k) for k, v in enumerate(d)) == X
        assert all(-128 <= v <= 127 for v in d[:-1]) and -128 <= d[-1] <= 128


def test_accumulators_stay_exact():
    """Pass of 128 complex terms (256 real): one slice product's sum is at most 2^22, so four fit
    in an FP32 accumulator; the seven-digit split gives group 4's fifth product a spare one, and
    the combination of the group sums stays below 2^63."""
    one = 256 * 128 * 128
    assert 4 * one <= 1 << 24
    groups = [g + 1 for g in range(7)]
    assert [g for g, m in enumerate(groups) if m * one > 1 << 24] == [4, 5, 6]
    total = sum(m * one << (8 * (6 - g)) for g, m in enumerate(groups)) >> 8
    assert total < 1 << 63
    assert (one << 8) + 2 * one < 1 << 31     # the two top groups in 32 bits
