"""The matrix kernel's arithmetic (gemm.h, kernel_gemm.cu), restated in Python
integers: balanced digits, the accumulators' bounds, the biased recombination
and the final reduction with explicit words, at the extreme residues."""
import random

import pytest

from paper_2609_35352_gb300 import workloads as W

M32, M64, M128 = (1 << 32) - 1, (1 << 64) - 1, (1 << 128) - 1
OFFSET = 0x8080808080 + (512 << 40)
MAGIC = 0x4B400000


def digits(c):
    """Digits of a centred residue: bytes of c + OFFSET minus 128, the rest minus 512."""
    u = c + OFFSET
    assert 0 <= u < 1 << 51
    d = [((u >> (8 * i)) & 255) - 128 for i in range(5)] + [(u >> 40) - 512]
    assert sum(v << (8 * i) for i, v in enumerate(d)) == c
    assert all(-128 <= v <= 127 for v in d[:5]) and -512 <= d[5] <= 512
    return d


def test_class_bounds():
    """64 raw terms: every class sum is an integer of at most 2^24, classes 0 to
    3 and the signed sums at most 2^22 (the conversion by a magic addend)."""
    top = [128] * 5 + [512]
    for s in range(11):
        worst = 64 * sum(top[a] * top[s - a] for a in range(6) if 0 <= s - a < 6)
        assert worst <= (1 << 22 if s < 4 else 1 << 24), s
    assert 96 * 512 <= 1 << 22


def magic_sum(n):
    return sum(MAGIC << (8 * s) for s in range(n))


def finish(l0, l1, l2, s, g, q):
    k = q.bit_length()
    mk, shift = (1 << (k + 63)) // q // 2, k - 34
    assert 0 <= l0 <= M64 and 0 <= l1 <= M64 and s < 1 << 58 and g < 1 << 50
    x = (l0 + (l1 << 32) + ((l2 & M64) << 64) + s * g) & M128
    assert x < 1 << (2 * k + 9)
    mid = (s >> 32) * (g & M32) + (s & M32) * (g >> 32)
    assert mid <= M64
    A = x >> (k - 2)
    assert A < 1 << 61 and mk < 1 << 63 and shift >= 0
    a0, a1, m0, m1 = A & M32, A >> 32, mk & M32, mk >> 32
    m = a0 * m1 + a1 * m0
    assert m <= M64
    h = a1 * m1 + (m >> 32)
    r = ((x & M64) - h * q) & M64
    assert r < 4 * q
    r = r - 2 * q if r >= 2 * q else r
    return r - q if r >= q else r


@pytest.mark.parametrize("bits", [34, 40, 49, 50])
def test_output(bits):
    rng = random.Random(bits)
    for q in W.ntt_primes(1024, bits, 2):
        half, k = q // 2, q.bit_length()
        edge = [0, 1, q - 1, half, half + 1, half - 1]
        for trial in range(60):
            n = 64 if trial < 20 else rng.randint(0, 64)
            pick = (lambda: rng.choice(edge)) if trial % 2 else (lambda: rng.randrange(q))
            fixed = trial < 6
            X = [edge[trial] if fixed else pick() for _ in range(96)]
            G = [edge[-1 - trial] if fixed else pick() for _ in range(n)]
            w = [1 if fixed else rng.choice((-1, 0, 1)) for _ in range(96)]
            g = q - 1 if trial % 3 == 0 else rng.randrange(q)
            xd = [digits(x - half) for x in X]
            gd = [digits(v - q if v > half else v) for v in G]
            e = [sum(xd[i][a] * gd[i][s - a] for i in range(n) for a in range(6) if 0 <= s - a < 6) for s in range(11)]
            f = [sum(w[i] * xd[i][a] for i in range(96)) for a in range(6)]
            rs = sum(v - q if v > half else v for v in G)
            t = q * (1 << (k + 6)) + half * rs % q - magic_sum(4)
            b0, b1, b2 = t & M32, ((t >> 32) & M32) + (1 << 50), (t >> 64) - (1 << 18)
            l0 = b0 + sum((MAGIC + e[s]) << (8 * s) for s in range(4))
            l1 = b1 + sum(e[4 + s] << (8 * s) for s in range(4))
            l2 = b2 + sum(e[8 + s] << (8 * s) for s in range(3))
            ws = sum(w)
            sc = abs(ws) * half % q
            sb = ((q - sc) if ws < 0 else sc) + 128 * q
            lo = sum((MAGIC + f[s]) << (8 * s) for s in range(4))
            hi = sum((MAGIC + f[4 + s]) << (8 * s) for s in range(2))
            s = (lo + (hi << 32) + sb - magic_sum(4) - (magic_sum(2) << 32)) & M64
            want = (sum(a * b for a, b in zip(G, X)) + g * sum(a * b for a, b in zip(w, X))) % q
            assert finish(l0, l1, l2, s, g, q) == want
