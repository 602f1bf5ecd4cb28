"""The wide product-accumulate (rns.cuh mac and settle, moduli below 2^60),
restated with explicit words: the low and high products as one carry chain, the
middle ones in a word of their own that kMidBudget = 8 products never wrap."""
import random

import pytest

from paper_2609_35352_gb300 import workloads as W

M32, M64, M128 = (1 << 32) - 1, (1 << 64) - 1, (1 << 128) - 1


@pytest.mark.parametrize("fill", ["max", "random"])
@pytest.mark.parametrize("bits", [52, 54, 60])
def test_settled_sum(bits, fill):
    rng = random.Random(bits)
    q = W.ntt_primes(1024, bits, 1)[0]
    acc = mid = want = 0
    for n in range(256):  # the least number of products a 128-bit accumulator takes
        a, b = (q - 1, q - 1) if fill == "max" else (rng.randrange(q), rng.randrange(q))
        acc += (a & M32) * (b & M32) + ((a >> 32) * (b >> 32) << 64)
        mid += (a & M32) * (b >> 32) + (a >> 32) * (b & M32)
        assert mid <= M64 and acc <= M128
        if n % 8 == 7:
            acc += mid << 32
            mid = 0
            assert acc <= M128
        want += a * b
    assert acc == want
