"""Bounds of the two-word ladders that let residues grow past 2 m (Python integers, word for
word what the device keeps): the half-reduced ladder of moduli up to 1.02e12, with the exponent
bookkeeping of a term (R 2^w0 start) and of a prime (2^t start), and the three-word squaring
of 47-bit moduli.  Every dropped word is asserted to be zero and every power to be right."""

import random

import pytest

HALF = 1_020_000_000_000
R = 1 << 64


def redc(T, m, words):
    for _ in range(words):
        u = (T * pow(-m, -1, 1 << 32)) % (1 << 32)
        T = (T + u * m) >> 32
    return T


def half(x, m):
    assert x < 1 << 48 and x * x < 1 << 96
    y = redc(x * x, m, 1)
    assert y < 1 << 64          # two words
    return y


def full(x, m, s):
    assert x >> 32 < 1 << 16 and x * x < 1 << 96
    t = redc(x * x, m, 1)
    assert t < 1 << 64          # two words, then shifted into three
    y = redc(t << s, m, 1)
    assert y < 2 * m
    return y


def general(x, m, s):
    assert x < 1 << 61
    y = redc((x * x) << s, m, 2)
    assert y < 2 * m
    return y


MODULI = [HALF - 1, HALF - 7, 2**39 + 1, 2**39 - 1, 2**31 + 11, 10**12 - 11, 2**36 - 5, 2**32 + 15]


@pytest.mark.parametrize("m", MODULI)
def test_half_reduced_ladder_of_terms(m):
    rng = random.Random(m)
    first_max = (63 - m.bit_length()) // 2
    exponents = [64, 96, 127, 128, 320, 1312, 2**40 - 1, 10**12, 10**13] + [64 * 4**k // 3 + d for k in (5, 17, 18) for d in (-1, 0, 1, 2)]
    exponents += [rng.randrange(64, 2**44) for _ in range(60)]
    for e_min in exponents:
        for E in (e_min, e_min + rng.randrange(0, min(e_min // 64 + 1, 65536))):   # lanes of a warp
            e_max = e_min + min(e_min // 64, 65535)
            k = (((3 * e_min - 128) >> 6).bit_length() - 1) // 2
            off = 128 * (4**k - 1) // 3
            c = 1
            while (((e_max + off) >> (2 * k)) - 64) >> c > first_max:
                c += 1
            u = E + off
            f1 = (u >> (2 * k)) - 64
            assert f1 >= 0 and f1 >> c <= first_max
            x = (R % m) << (f1 >> c)
            bits = (f1 & ((1 << c) - 1)) << (2 * k) | u & (4**k - 1)
            p = 2 * k + c - 1
            x = general(x, m, bits >> p & 1)
            while p > 2 * k:
                p -= 1
                x = full(x, m, bits >> p & 1)
            x -= m if x >= m else 0
            while p > 0:
                p -= 2
                x = full(half(x, m), m, bits >> p & 3)
            assert x < 2 * m and x % m == pow(2, E, m)


@pytest.mark.parametrize("p", [1019999999989, 2**32 + 15, 2**36 - 5, 2**39 - 7, 549755813881, 10**12 - 11, 2147483659])
def test_half_reduced_ladder_of_primes(p):
    assert pow(2, p - 1, p) == 1
    rng = random.Random(p)
    l = p.bit_length()
    j = l - 5
    off = (32 << j if j & 1 else 0) + 128 * (4 ** (j // 2) - 1) // 3
    for e in [10**6, p - 2, p - 1, p, 7 * p + 3] + [rng.randrange(20 * p) for _ in range(40)]:
        u = (e + off - l * 2**j) % (p - 1) + l * 2**j - (p - 1)
        assert 0 <= u < l << j
        x, b = 1 << (u >> j), j
        assert x < 2 * p
        if b & 1:
            b -= 1
            x = full(x, p, u >> b & 1)
        while b > 0:
            b -= 2
            x = full(half(x, p), p, u >> b & 3)
        assert x < 2 * p and x % p == pow(2, e, p)


@pytest.mark.parametrize("m", [2**47 - 1, 2**47 - 115, 2**46 + 1, 10**14 + 7])
def test_three_word_square_of_47_bit_moduli(m):
    rng = random.Random(m)
    for _ in range(40):
        x = (R % m) << rng.choice([7, 8])
        f = 64 + (x // (R % m)).bit_length() - 1
        s = rng.choice([0, 1])
        x, f = general(x, m, s), 2 * f - 64 + s
        x -= m if x >= m else 0
        for i in range(24):
            s = rng.choice([0, 0, 0, 15, rng.randrange(16)])
            x, f = full(x, m, s), 2 * f - 64 + s
            assert x < m + (1 << 47) - (1 << 45)
            if f < 10**7:
                assert x % m == pow(2, f, m)
