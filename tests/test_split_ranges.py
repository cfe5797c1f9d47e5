"""The split products' lazy ranges (mul_split, fold_s, fold_u of common.cuh and the engine
that uses them), in exact integers and fractions: every intermediate fits its register, every
value stays in the range the next step needs, for every prime length and the largest c the
library takes (split_prime)."""
import random
from fractions import Fraction as Fr

import pytest

from oracle.params import BfvParams
from tests import rules_lib

BITS = list(range(41, 61))


def _largest_c(b):
    return (1 << 24) - 1 if b >= 59 else (1 << (b - 33)) - 1


def _error(b, a):
    """max |hi32(H)| c / 2^b for |y| <= a 2^b."""
    return (Fr(2) ** 30 + a * Fr(2) ** (b - 33) + 1) * _largest_c(b) / Fr(2) ** b


def _product(b, lo, hi):
    """Range of mul_split(0, y, w), y in [lo, hi] (units of 2^b)."""
    a = max(-lo, hi)
    e = _error(b, a)
    return (-(Fr(1, 2) + max(-lo, 0) * Fr(2) ** (b - 64) + e), Fr(3, 2) + max(hi, 0) * Fr(2) ** (b - 64) + e)


@pytest.mark.parametrize("b", BITS)
def test_forward_ranges(b):
    """Four Cooley-Tukey stages from a folded value stay inside (-7, 8) (units of 2^b), where
    the product's inputs have to be and 64 bits end for b = 60; with 8 q (two stages: 4 q)
    added they are positive and below 2^64."""
    tiny = Fr(1, 1 << 20)   # what a fold leaves outside [0, 1]
    lo, hi = -tiny, 1 + tiny
    for stage in range(4):   # (the last one ends below 7.97, the products' largest operand)
        plo, phi = _product(b, lo, hi)
        lo, hi = lo - max(-plo, phi), hi + max(-plo, phi)
        assert -8 < lo and hi < 8
        q = 1 - Fr(_largest_c(b), 1 << b)
        if stage == 1:
            assert lo > Fr(-333, 100) and hi < Fr(433, 100) and lo + 4 * q > 0
    assert lo > -7 and hi < Fr(797, 100) and lo + 8 * q > 0 and (hi + 8) * Fr(2) ** b < Fr(2) ** 64
    assert 8 * _largest_c(b) < Fr(2) ** b * tiny and (1 << (64 - b)) * _largest_c(b) < (1 << b) - 2 * _largest_c(b)


@pytest.mark.parametrize("b", BITS)
def test_inverse_ranges(b):
    """Two Gentleman-Sande stages, the second one's sums folded, keep [-0.87, 1.87]; every sum
    stays below 8; the scaled last stage's products, from 2 q, are in (0.9 q, 4.1 q)."""
    lo, hi = Fr(-87, 100), Fr(187, 100)
    for start in ((Fr(0), Fr(1)), _product(b, Fr(0), Fr(1)), (lo, hi)):
        slo, shi = start
        assert lo <= slo and shi <= hi
        p1 = _product(b, slo - shi, shi - slo)
        r1 = min(2 * slo, p1[0]), max(2 * shi, p1[1])
        assert -8 < 2 * r1[0] and 2 * r1[1] < 8 and r1[1] - r1[0] < 8
        p2 = _product(b, r1[0] - r1[1], r1[1] - r1[0])
        assert lo <= p2[0] and p2[1] <= hi
        for plo, phi in (_product(b, 2 * r1[0], 2 * r1[1]), _product(b, r1[0] - r1[1], r1[1] - r1[0]),
                         _product(b, 2 * slo, 2 * shi)):
            q = 1 - Fr(_largest_c(b), 1 << b)
            assert plo + 2 * q > Fr(9, 10) and phi + 2 * q < Fr(41, 10) * q


def _signed(v, bits):
    assert -(1 << (bits - 1)) <= v < 1 << (bits - 1), (v, bits)
    return v


def _mul_split(base, y, words, b, c):
    """mul_split with every intermediate checked against its register."""
    (w0, w1), (v0, v1) = words
    y0 = (y + (1 << 31)) % (1 << 32) - (1 << 31)
    y1 = _signed((y - y0) >> 32, 32)
    h = _signed(_signed(y0 * w1, 64) + y1 * v1, 64)
    low = _signed(_signed(base + y0 * w0, 64) + y1 * v0, 64)
    low = _signed(low + (h >> 32) * c, 64)
    return _signed(low + ((h % (1 << 32)) << (b - 32)), 64)


@pytest.mark.parametrize("ring", [(12, 2, 54), (13, 3, 60), (14, 4, 60), (13, 4, 59), (12, 1, 50), (12, 2, 57)])
def test_products_of_extreme_operands(ring):
    r = random.Random(ring[2])
    for q in BfvParams(log_n=ring[0], num_primes=ring[1], prime_bits=ring[2]).primes:
        if not rules_lib.split_prime(q):
            continue
        b = q.bit_length()
        c, one = (1 << b) - q, 1 << b
        ws = [0, 1, 2, q // 2, q // 2 + 1, q - 1, (1 << (b - 1)) - 1, 1 << 31, (1 << 32) - 1] + \
            [r.randrange(q) for _ in range(40)]
        ys = [0, 1, -1, one, one - 1, -7 * one + 1, 797 * one // 100, (1 << 31) - 1, 1 << 31, -(1 << 31), -(1 << 31) - 1] + \
            [r.randrange(-7 * one, 797 * one // 100) for _ in range(40)]
        for w in ws:
            words = rules_lib.split_words(w % q, q)
            for y in ys:
                for base in (0, 2 * q) if b == 60 else (0, 2 * q, -one):
                    if base and not -4 * one < y < one * 15 // 2:
                        continue
                    v = _mul_split(base, y, words, b, c)
                    assert (v - base - y * w) % q == 0
                    lo, hi = _product(b, Fr(min(y, 0), one), Fr(max(y, 0), one))
                    assert lo <= Fr(v - base, one) <= hi


def test_shorter_primes_pass_the_60_bit_bound():
    """The error term for b <= 58 is up to 1/8, four times that of 60-bit primes: a bound
    stated for those alone would not hold for 54-bit ones."""
    assert _error(60, 8) <= Fr(1, 32) + Fr(1, 1 << 30)
    assert all(Fr(1, 9) < _error(b, 1) <= Fr(1, 6) for b in range(44, 59))
