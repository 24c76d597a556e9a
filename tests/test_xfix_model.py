"""The two-limb integer arithmetic of the FP64-accurate hop (xfix.cuh) in
Python integers: conversion, limb ranges, the bounds that keep the 64-bit
sums exact, and the error of a colour product against exact rationals."""
from fractions import Fraction

import numpy as np
import pytest

SPINOR_BITS, LINK_BITS, LIMB = 57, 59, 30


def exponent(values):
    """e with |v| < 2^e for every v (frexp's exponent of the largest)."""
    return int(np.frexp(np.max(np.abs(values)))[1])


def to_int(v, e, bits):
    """v 2^(bits - e) rounded to nearest, halves away from zero."""
    f = Fraction(float(v)) * Fraction(2) ** (bits - e)
    n = (2 * abs(f.numerator) + f.denominator) // (2 * f.denominator)
    return -n if v < 0 else n


def split(n):
    lo = ((n + (1 << (LIMB - 1))) & ((1 << LIMB) - 1)) - (1 << (LIMB - 1))
    return (n - lo) >> LIMB, lo


@pytest.mark.parametrize("spread", [0.0, 3.0, 12.0])
def test_conversion_and_limbs(spread):
    rng = np.random.default_rng(7)
    for bits in (SPINOR_BITS, LINK_BITS):
        v = rng.standard_normal(500) * np.exp(spread * rng.standard_normal(500))
        e = exponent(v)
        for x in v:
            n = to_int(x, e, bits)
            assert abs(n) <= 1 << bits
            hi, lo = split(n)
            assert hi * (1 << LIMB) + lo == n
            assert abs(hi) <= 1 << (bits - LIMB) and -(1 << 29) <= lo < 1 << 29
            # half a unit of the common exponent, far below FP64's ulp of the largest entry
            assert abs(Fraction(float(x)) - Fraction(n) * Fraction(2) ** (e - bits)) <= Fraction(2) ** (e - bits - 1)


def test_sums_stay_in_64_bits():
    """Worst case of every operand: hops, colours and complex parts all add up."""
    u_hi, u_lo = 1 << 29, 1 << 29
    h_hi, h_lo = 2 * (1 << 27), 2 * (1 << 29)
    assert h_lo <= (1 << 31) - 1 and h_hi <= (1 << 31) - 1
    hh = 6 * u_hi * h_hi
    cross = 6 * (u_hi * h_lo + u_lo * h_hi) + (1 << 29)
    assert hh < 1 << 63 and cross < 1 << 63
    one_hop = hh + (cross >> LIMB) + 1
    assert 8 * one_hop < 1 << 63


def test_colour_product_error():
    """Sum of six limb products against the exact value: within 2^-55 of the
    largest link and spinor entry (the FP64 sum has an error near 2^-53 of
    the summed terms)."""
    rng = np.random.default_rng(3)
    worst = 0.0
    for _ in range(200):
        u, h = rng.standard_normal(6), rng.standard_normal(6)
        eu, eh = exponent(u), exponent(h)
        hh = cross = 0
        for a, b in zip(u, h):
            ah, al = split(to_int(a, eu, LINK_BITS))
            bh, bl = split(to_int(b, eh, SPINOR_BITS))
            hh += ah * bh
            cross += ah * bl + al * bh
        got = Fraction(hh + ((cross + (1 << 29)) >> LIMB)) * Fraction(2) ** (eu + eh - 56)
        exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(u, h))
        worst = max(worst, float(abs(got - exact) / Fraction(2) ** (eu + eh)))
    assert worst < 2.0 ** -55
    assert worst > 0.0


@pytest.mark.parametrize("kind", ["worst", "random"])
def test_hop_error_with_projected_operands(kind):
    """One colour sum of a hop with h = upper +- lower limb by limb, in units of
    2^-56 of the largest product of entries: 3 for the six products of low
    limbs, 1 for the two roundings, 3.75 for the rounding of the inputs.
    worst: every low limb -2^29, so that the dropped products add up."""
    rng = np.random.default_rng(11)
    worst = 0
    for _ in range(200):
        hh = cross = 0
        exact = Fraction(0)
        u, up, lo = rng.uniform(-1, 1, 6), rng.uniform(-1, 1, 6), rng.uniform(-1, 1, 6)
        u[0] = up[0] = 1 - 2.0 ** -53  # exponent 0 for all
        for a, p, l in zip(u, up, lo):
            na, np_, nl = to_int(a, 0, LINK_BITS), to_int(p, 0, SPINOR_BITS), to_int(l, 0, SPINOR_BITS)
            if kind == "worst":
                na, np_, nl = ((n >> LIMB << LIMB) - (1 << (LIMB - 1)) for n in (na, np_, nl))
                exact += Fraction(na * (np_ + nl)) / 2 ** (LINK_BITS + SPINOR_BITS)
            else:
                exact += Fraction(float(a)) * (Fraction(float(p)) + Fraction(float(l)))
            (ah, al), (ph, pl), (lh, ll) = split(na), split(np_), split(nl)
            hh += ah * (ph + lh)
            cross += ah * (pl + ll) + al * (ph + lh)
        units = abs(Fraction(hh + ((cross + (1 << 29)) >> LIMB)) - exact * 2 ** 56)
        worst = max(worst, units)
        assert units <= (4 if kind == "worst" else 7.75)
    if kind == "worst":
        assert worst > 2.5  # the dropped products are there
