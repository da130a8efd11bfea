"""Ranges around a basis conversion, with exact integers: its outputs lie in [0, 5t), and every consumer takes them.
The forward transform's uncorrected butterflies (primes below 2^57) grow by less than 4q a stage, below 69q after the
16 stages of N = 2^16, which the final reduction by a 32-bit quotient estimate handles; the corrected ones (up to
2^60) take anything below 8q."""
import random

import pytest

RNG = random.Random(20261205)
INPUT, STAGES = 5, 16
BOUND = INPUT + 4 * STAGES  # in units of q


@pytest.mark.parametrize("sources", range(1, 9))
def test_conversion_outputs(sources):
    """The reduction leaves a sum of `sources` products below (sources + 1) t; more than four take 4t off where it
    fits."""
    t = (1 << 60) - 93
    top = (sources + 1) * t - 1
    for x in [0, 4 * t - 1, 4 * t, INPUT * t - 1, top] + [RNG.randrange(top + 1) for _ in range(200)]:
        if x > top:
            continue
        assert x < 1 << 64
        y = x - 4 * t if sources > 4 and x >= 4 * t else x
        assert 0 <= y < INPUT * t and y % t == x % t


def test_uncorrected_growth():
    """X + WY and X - WY + 4q with WY in [0, 4q) stay below the next bound and within 64 bits."""
    q = (1 << 57) - 1
    bound = INPUT
    for _ in range(STAGES):
        assert (bound * q - 1) + (4 * q - 1) < (bound + 4) * q  # the sum
        assert 0 < 0 - (4 * q - 1) + 4 * q and (bound * q - 1) + 4 * q < (bound + 4) * q  # the difference
        bound += 4
    assert bound == BOUND == 69 and bound * q < 2 ** 63.2 < 1 << 64


def test_corrected_range():
    """A corrected butterfly reduces X below 4q first (X < 8q), so its outputs are below 8q again, for 60-bit primes."""
    q = (1 << 60) - 93
    for x in [0, 4 * q - 1, 4 * q, INPUT * q - 1, 8 * q - 1]:
        assert x < 1 << 64
        x = x - 4 * q if x >= 4 * q else x
        for wy in (0, 4 * q - 1):
            assert 0 <= x + wy < 8 * q and 0 <= x - wy + 4 * q < 8 * q


def reduce_below69(x, q):
    s = q.bit_length() - 1
    mu = (1 << (64 + s)) // q
    r, xh = mu >> 32, x >> (s - 24)
    assert r < 1 << 32 and xh < 1 << 32
    est = ((xh * r) >> 32) >> 24
    v = x - est * q
    assert 0 <= v < 2 * q, (x / q, est)
    return v - q if v >= q else v


@pytest.mark.parametrize("bits", [25, 26, 30, 40, 50, 56, 57])
def test_reduction(bits):
    primes = [RNG.randrange(1 << (bits - 1), 1 << bits) | 1 for _ in range(300)]
    primes += [(1 << (bits - 1)) + 1, (1 << bits) - 1]
    for q in primes:
        edges = [k * q + d for k in range(BOUND) for d in (0, q - 1)] + [BOUND * q - 1]
        for x in edges + [RNG.randrange(BOUND * q) for _ in range(20)]:
            assert reduce_below69(x, q) == x % q
