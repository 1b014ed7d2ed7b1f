"""Word-level bounds of the prime form's ladders that take every reduction step: the two-word
one of primes past 1.02e12 (up to 2.18e13, Eq. 1's largest modulus) and the one-word ones,
with their exponent bookkeeping, for a warp whose largest prime has more bits.  The
half-reduced ladder is in test_half_ladder_bounds.py."""

import random

import pytest

from test_half_ladder_bounds import full


def is_prime(p):
    return all(pow(a, p - 1, p) == 1 and p % a for a in (2, 3, 5, 7, 11, 13, 17, 19, 23))


def primes_from(v, count):
    v |= 1
    while count:
        if is_prime(v):
            yield v
            count -= 1
        v += 2


def reduced_exponent(e, off, p, l, j):
    """As the device forms it, in 64-bit words with a single-precision quotient off by at most one."""
    a = e + off - l * 2**j
    assert 0 <= a < 1 << 63
    assert a // (p - 1) < 1 << 20        # single precision is far within one
    u = a % (p - 1) + l * 2**j - (p - 1)
    assert 0 <= u < l << j
    return u


@pytest.mark.parametrize("above", [1_020_000_000_000, 2**40, 3 * 10**12, 2**42, 2**43 - 300, 10_900_000_000_000,
                                   2**44 - 500, 21_800_000_000_000])
def test_two_word_ladder(above):
    rng = random.Random(above)
    for p in primes_from(above, 3):
        assert p < 1 << 45
        l, n = p.bit_length(), p // 2 + 1
        j = l - 5
        for e in [n + 64, n + 1279, 2 * n, p - 2, p - 1, p] + [rng.randrange(p // 2, 23 * p) for _ in range(25)]:
            u = reduced_exponent(e, 64 * (2**j - 1), p, l, j)
            x, rem, b = 1 << (u >> j), u & (2**j - 1), j
            assert x < 2 * p
            length = (b - 1 & 3) + 1
            while b > 0:
                b -= length
                shift = rem >> b & 15 if length == 4 else rem >> b
                assert shift < 1 << length
                for _ in range(length - 1):
                    x = full(x, p, 0)
                x = full(x, p, shift)      # asserts the words and x < 2 p
                length = 4
            assert x % p == pow(2, e, p)


# path 0: lazy residues below 2 p, p < 2^29; path 3: reduced ones, p < 2^31
@pytest.mark.parametrize("path,above", [(0, 700_000), (0, 2**23 - 40), (0, 13_000_000), (0, 2**24 + 1), (0, 23_400_000), (0, 2**28 + 1), (0, 2**29 - 100),
                                        (3, 2**29 + 1), (3, 2**30 - 70), (3, 2**31 - 90)])
def test_one_word_ladder(path, above):
    rng = random.Random(above)
    for p in primes_from(above, 3):
        if p >> (29 if path == 0 else 31):
            continue
        # the list's primes reach from A / 23 to A
        for l in range(p.bit_length(), min(p.bit_length() + 5, 29) + 1) if path == 0 else (p.bit_length(), 31):
            j = l - 4
            inv = pow(p, -1, 1 << 32)
            for e in [p, 2 * p + 64, 20 * p + 3] + [rng.randrange(p, 23 * p) for _ in range(30)]:
                u = reduced_exponent(e, 32 * (2**j - 1), p, l, j)
                x = 1 << (u >> j)
                for b in range(j - 1, -1, -1):
                    y = 2 * x if u >> b & 1 else x
                    assert x < 1 << 32 and y < 1 << 32
                    T = x * y
                    h = (T % 2**32 * inv % 2**32) * p >> 32
                    if path == 3:
                        r = (T >> 32) - h
                        assert -p < r < p
                        x = r if r >= 0 else r + p
                    else:
                        x = (T >> 32) + p - h
                        assert 0 < x < 1 << 32
                assert x < 2 * p and x % p == pow(2, e, p)
