"""Launch rules (csrc/rules.h) on the host."""
import ctypes
import random

import pytest

from oracle.params import BfvParams
from tests import rules_lib

# words that fit a 284 208 MiB device beside nothing else
MOST_WORDS = 284208 * (1 << 20) // 8


@pytest.mark.parametrize("k", [1, 16, 17, 784, 6272, (1 << 31) + 5, (1 << 34) - 1, 1 << 34, (1 << 34) + 1, 1 << 35,
                               MOST_WORDS])
@pytest.mark.parametrize("tiles", [1, 3, 100, 457, 100000])
def test_ring_parts_cover_every_reduction_that_fits_the_device(k, tiles):
    """Every reduction whose operand fits the device is taken, in launches of at most
    ring_launch_k elements: a launch's parts cover its chunks once, none is empty, and no
    chunk number (the kernel looks three ahead) leaves 32 bits."""
    most, start = rules_lib.ring_launch_k(), 0
    assert most % 16 == 0
    while start < k:
        part = min(k - start, most)
        chunks, per, parts = rules_lib.ring_split(part, tiles)
        assert chunks == -(-part // 16) and chunks + 3 < 1 << 31
        assert (parts - 1) * per < chunks <= parts * per
        assert 1 <= parts <= 65535 and (parts == 1 or per >= 4)
        start += part


# (B, Ci, Co, H, kernel, pad), role, t_bits -> form, where the measured times of the forms
# are at least 1.2 apart (us: integer form / tensor cores)
RING_FORMS = [
    ((1, 256, 100, 1, 1, 0), 2, 41, "tile"),          # 4.8 / 9.5
    ((1, 2048, 1001, 1, 1, 0), 2, 41, "tile"),        # 13.0 / 18.9
    ((64, 2048, 1, 1, 1, 0), 1, 41, "tile"),          # 5.0 / 9.5
    ((1000, 3, 8, 1, 1, 0), 0, 59, "tile"),           # 6.9 / 7.4 and less
    ((64, 3, 64, 56, 1, 0), 0, 41, "tile"),           # 59.8 / 94.9
    ((64, 3, 3, 56, 3, 1), 0, 41, "tile"),            # 20.9 / 36.9
    ((64, 64, 3, 56, 3, 1), 0, 59, "tile"),           # 381 / 468
    ((1, 1, 1, 28, 5, 2), 2, 41, "offsets"),          # 8.8 / 15.0
    ((1, 16, 8, 28, 3, 1), 2, 59, "offsets"),         # 4.2 / 17.1
    ((1, 16, 64, 28, 1, 0), 2, 41, "offsets"),        # 5.2 / 15.8
    ((64, 2048, 2, 1, 1, 0), 0, 59, "digits"),        # 1240 / 13.4
    ((64, 2048, 2, 1, 1, 0), 0, 41, "digits"),
    ((1000, 10, 3, 1, 1, 0), 2, 59, "digits"),        # 535 / 15
    ((8, 64, 3, 14, 3, 1), 0, 59, "digits"),          # 285 / 16
    ((64, 16, 16, 32, 3, 1), 0, 41, "digits"),        # 104 / 48
    ((64, 16, 16, 32, 3, 1), 2, 59, "digits"),        # 190 / 70
    ((64, 2048, 1001, 1, 1, 0), 2, 41, "digits"),     # 97 / 38
    ((128, 128, 128, 16, 3, 1), 2, 41, "digits"),
]


@pytest.mark.parametrize("layer,role,t_bits,form", RING_FORMS)
def test_ring_form_is_the_faster_one(layer, role, t_bits, form):
    assert rules_lib.ring_form(layer, role, t_bits) == form


def test_a_small_bias_gradient_is_no_cluster_launch():
    parts = rules_lib.load().bias_parts_
    assert [parts(ctypes.c_longlong(n)) for n in (1, 4096, 4097, 1 << 40)] == [1, 1, 8, 8]


def test_small_linear_combinations_take_one_element_a_thread():
    assert not rules_lib.lincomb_pairs(100000) and rules_lib.lincomb_pairs(1 << 17)


# (log2 N, primes, bits): every ring the repository's tests and benchmark use, and the
# shortest and longest primes a context takes
PRIMES = [q for ring in ((12, 2, 54), (12, 2, 60), (13, 3, 60), (14, 4, 60), (13, 4, 59), (12, 2, 48))
          for q in BfvParams(log_n=ring[0], num_primes=ring[1], prime_bits=ring[2]).primes]


@pytest.mark.parametrize("q", sorted(set(PRIMES)))
def test_split_words_are_the_centred_residues(q):
    """(compiled with undefined behaviour trapped: no shift leaves its type)"""
    if not rules_lib.split_prime(q):
        pytest.skip("not of the split products' form")
    sh, r = q.bit_length() - 32, random.Random(q)
    for w in [0, 1, 2, q // 2, q // 2 + 1, q - 2, q - 1] + [r.randrange(q) for _ in range(200)]:
        for (low, rest), v in zip(rules_lib.split_words(w, q), (w, (w << 32) % q)):
            x = (rest << sh) + low
            assert x % q == v and -q // 2 <= x <= q // 2
            assert 0 <= low < 1 << sh and -(1 << 31) <= rest < 1 << 31


def test_short_primes_take_no_split_products():
    for bits in (30, 31, 32, 36, 39):
        for q in BfvParams(log_n=12, num_primes=2, prime_bits=bits).primes:
            assert not rules_lib.split_prime(q)
    assert not rules_lib.split_prime((1 << 61) - 1)


def test_multiply_accumulate_forms():
    """Alg. 1 with few input blocks streams; digit products where a tile's 4 x 16 (weight
    gradients 8 x 16) outputs mostly exist; the knobs and the primes decide the rest."""
    form = rules_lib.mac_form
    assert form(10, 6, 16) == "short" and form(10, 16, 16) == "digits" and form(64, 32, 43, dual=True) == "digits"
    assert form(2, 16, 64) == "bulk" and form(5, 9, 7) == "bulk" and form(3, 2, 5, dual=True) == "bulk"
    assert form(10, 16, 16, staging=0) == "ring" and form(10, 16, 16, columns=0) == "smem"
    assert form(10, 2, 16, split=False) == "digits" and form(10, 16, 16, split=False, columns=0) == "generic"


def test_mask_polynomials_skip_where_many_warps_are_empty():
    skips = rules_lib.mask_skips
    assert skips(2752, 8192, 18) and skips(2048, 8192, 51)
    assert not skips(2048, 8192, 52) and not skips(1920, 8192, 64)   # nearly full
    assert not skips(2, 8192, 4) and not skips(37, 8192, 4) and skips(38, 8192, 4)   # one wave


def test_compact_form_skips_where_half_of_the_groups_are_empty():
    skips = rules_lib.load().compact_skips_
    assert [bool(skips(8192, f)) for f in (1, 128, 129, 256)] == [True, True, False, False]
