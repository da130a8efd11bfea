"""Bounds of the two-step Montgomery reduction (R = 2^60) on 30-bit-split partial sums, with exact integers: no partial
value leaves 64 bits, the result is V 2^-60 mod p and below V / 2^60 + p, for the numbers of terms and primes
the kernels use it with."""
import random

import pytest

M30, M64 = (1 << 30) - 1, (1 << 64) - 1
PRIMES = {20: (1 << 20) - 3, 40: (1 << 40) - 87, 50: (1 << 50) - 27, 56: (1 << 56) - 5, 60: (1 << 60) - 93}


def mont60(s00, s01, s11, p, norm):
    """As the kernel computes it; every 64-bit value is checked."""
    def fits(x):
        assert 0 <= x <= M64, "a partial sum leaves 64 bits"
        return x

    p0, p1, np_ = p & M30, p >> 30, -pow(p, -1, 1 << 30) & M30
    fits(s00), fits(s01), fits(s11)
    if norm:
        s11 = fits(s11 + (s01 >> 30))
        s01 &= M30
    m0 = (s00 & 0xFFFFFFFF) * np_ & M30
    s01 = fits(m0 * p1 + fits(s01 + (fits(m0 * p0 + s00) >> 30)))
    m1 = (s01 & 0xFFFFFFFF) * np_ & M30
    return fits(m1 * p1 + fits(s11 + (fits(m1 * p0 + s01) >> 30)))


# (terms, factor bound in bits or None for the prime itself, prime bits, NORM): basis conversion sums up to 4 terms
# without and up to 8 with the normalisation, the key inner product up to 4 / 8 of any prime and 12 below 2^56
@pytest.mark.parametrize("terms,ybits,pbits,norm", [
    (1, 60, 60, False), (4, 60, 60, False), (4, 60, 20, False), (4, 60, 40, False), (8, 60, 60, True), (8, 60, 50, True),
    (4, None, 60, False), (8, None, 60, True), (8, None, 40, True), (12, None, 56, True), (12, None, 50, True)])
def test_mont60(terms, ybits, pbits, norm):
    p = PRIMES[pbits]
    top = (1 << ybits) - 1 if ybits else p - 1
    rng = random.Random(terms * 1000 + pbits)
    cases = [([top] * terms, [p - 1] * terms), ([0] * terms, [p - 1] * terms), ([M30 & top] * terms, [min(M30, p - 1)] * terms)]
    cases += [([rng.randint(0, top) for _ in range(terms)], [rng.randrange(p) for _ in range(terms)]) for _ in range(300)]
    for ys, cs in cases:
        s00 = sum((y & M30) * (c & M30) for y, c in zip(ys, cs))
        s11 = sum((y >> 30) * (c >> 30) for y, c in zip(ys, cs))
        sm = sum(((y & M30) + (y >> 30)) * ((c & M30) + (c >> 30)) for y, c in zip(ys, cs)) & M64
        s01 = (sm - s00 - s11) & M64  # the Karatsuba middle sum, exact modulo 2^64
        v = sum(y * c for y, c in zip(ys, cs))
        assert s01 == sum((y & M30) * (c >> 30) + (y >> 30) * (c & M30) for y, c in zip(ys, cs))
        r = mont60(s00, s01, s11, p, norm)
        assert r * (1 << 60) % p == v % p and r <= (v >> 60) + p
        if ybits is None:
            assert r < (2 * p if pbits <= 56 else 9 * p)
        else:
            assert r < (terms + 1) * p
