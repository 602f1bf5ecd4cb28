"""The twiddle product of the transforms mod q (ntt.cuh mul_twiddle), restated
in Python integers with explicit 32- and 64-bit words: for a table entry w,
v = w 2^32 mod q, om = floor(2^32 w / 2q), ov = floor(2^32 v / 2q) and any
64-bit x, the result is congruent to x w and lies in [0, 6q); and the bounds
of the butterflies built on it (forward with and without the conditional
subtraction, inverse) hold at the widest moduli each takes."""
import random

import pytest

from paper_2609_35352_gb300 import workloads as W

M32, M64 = (1 << 32) - 1, (1 << 64) - 1


def entry(w, q):
    qw, v = divmod(w << 32, q)
    om, ov = qw // 2, (v << 31) // q
    assert om == (w << 32) // (2 * q) and ov == (v << 32) // (2 * q)
    assert om < 1 << 31 and ov < 1 << 31
    return w, v, om, ov


def mul_twiddle(x, e, q):
    w, v, om, ov = e
    xl, xh = x & M32, x >> 32
    m = xl * om + xh * ov
    assert m <= M64  # the 64-bit sum does not wrap
    k = m >> 32
    n = (1 << 64) - 2 * q
    p = (xl * (w & M32) + xh * (v & M32)) & M64
    hi = ((p >> 32) + xl * (w >> 32) + xh * (v >> 32) + k * (n >> 32)) & M32
    return (((hi << 32) | (p & M32)) + k * (n & M32)) & M64


@pytest.mark.parametrize("bits", [20, 31, 40, 50, 55, 56, 60])
def test_product_range(bits):
    rng = random.Random(bits)
    for q in W.ntt_primes(1024, bits, 2):
        for w in [0, 1, 2, q - 1, q - 2, q // 2, q // 2 + 1] + [rng.randrange(q) for _ in range(200)]:
            e = entry(w, q)
            xs = [0, 1, q - 1, M32, M32 + 1, M64, M64 - 1, M64 - M32, (6 * q - 1) & M64, (12 * q - 1) & M64]
            for x in xs + [rng.randrange(1 << 64) for _ in range(20)]:
                r = mul_twiddle(x, e, q)
                assert r < 6 * q and (r - x * w) % q == 0, (q, w, x)


def test_butterfly_bounds():
    q = (1 << 56) - 1  # FAST: every q below 2^56, inputs below 8q, 17 stages
    bound = 8 * q
    for _ in range(17):
        bound += 6 * q  # x + t and x - t + 6q, t below 6q
    assert bound < 1 << 63 and bound <= 128 * q  # 128q - t in the rescale's last step is positive
    assert q - 1 + 128 * q < 1 << 64
    q = (1 << 60) - 1  # general: x below 12q, brought below 6q
    assert 6 * q + 6 * q <= 1 << 64 and q - 1 + 12 * q < 1 << 64
    # inverse: sums of two values below 6q, and x - y + 6q below 12q
    assert 12 * q < 1 << 64
