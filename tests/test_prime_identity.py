"""The identity behind queries summed by primes, in exact fractions: the head terms of both
formulas up to the prime form's limits equal, mod 1, the sum over prime powers q of
(residue) / q with the residues the kernels form -- closed sums over c with their signs,
exponents and limits, and for long sums one period times a geometric sum."""

from fractions import Fraction

import pytest

from oracle import bbp_oracle as o1


def primes_upto(n):
    return [p for p in range(3, n + 1, 2) if all(p % q for q in range(3, int(p**0.5) + 1, 2))]


def limits(formula, d):
    odd = lambda v: v - 1 + v % 2
    if formula == 0:
        A = odd(d + 1)
        return A, odd(A // 5), odd(1 + 2 * (d - 1) // 5)
    return 2 * d + 5, odd(d + 2), odd((d + 1) // 2)


def head_terms(formula, d):
    """Sum mod 1 of the head terms that the prime form covers."""
    f = o1.FORMULAS[formula]
    lim, total = limits(formula, d), Fraction(0)
    for s in f.series:
        top = 2 * d + 6 if formula else lim[0] if s.a == 10 else lim[2]
        k = 0
        while s.a * k + s.b <= top and d + s.c - f.step * k >= 0:
            m = s.a * k + s.b
            sign = s.sign * (-1) ** (k * f.alternating)
            total += sign * Fraction(pow(2, d + s.c - f.step * k, m), m)
            k += 1
    return total % 1


def sums(formula, q, d):
    """(c0, stride, sign of i, log2 of the ratio per i over q, exponent and sign at i = 0, period)"""
    r = q % 4
    alternate, twos, none = (lambda i: (-1) ** i), (lambda i: -1 if i & 2 else 1), (lambda i: 1)
    chi, psi = (1 if r == 1 else -1), (1 if q % 8 in (1, 3) else -1)
    if formula == 0:
        return [(1, 2, alternate, 2, d + 3 - q, chi, q), (1, 2, alternate, 10, d + 1 - 5 * q, -chi, q),
                (1, 2, twos, 5, d - 1 - 5 * (q - 1) // 2, -psi, 4 * q)]
    return [(r, 4, alternate, 2, d + 2 - (q * r - 1) // 2, 1 if q * r % 8 == 1 else -1, q),
            (4 - r, 4, none, 4, d + 2 - (4 - r) * q, -1, q), (1, 2, none, 4, d + 1 - 2 * q, -1, q)]


def residue(formula, p, q, d):
    total = 0
    for (c0, stride, sign, ratio, start, minus, period), top in zip(sums(formula, q, d), limits(formula, d)):
        n = (top // q - c0) // stride + 1 if top // q >= c0 else 0
        step = sign(period) * pow(2, -ratio * q * period, q)
        for i in range(min(n, period)):
            c = stride * i + c0
            if c % p:
                times = (n - i + period - 1) // period
                geometric = sum(pow(step, v, q) for v in range(times))
                total += minus * sign(i) * pow(2, start - ratio * q * i, q) * pow(c, -1, q) * geometric
    return total % q


@pytest.mark.parametrize("formula", [0, 1])
def test_prime_powers_give_the_head_terms(formula):
    for d in list(range(1, 34)) + [77, 100, 257, 500]:
        total = Fraction(0)
        for p in primes_upto(limits(formula, d)[0]):
            q = p
            while q <= limits(formula, d)[0]:
                total += Fraction(residue(formula, p, q, d), q)
                q *= p
        assert total % 1 == head_terms(formula, d), d
