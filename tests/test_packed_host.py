"""Bounds of the carry-free sums (modarith.cuh) and the run split of the
automorphism that the diagonal kernel uses, restated with exact integers."""
import random

import pytest

from paper_2605_17222_gb300 import synth

M32, M64 = (1 << 32) - 1, (1 << 64) - 1


def primes40():
    return [synth.ntt_primes(40, 1, 1 << 17)[0], synth.ntt_primes(34, 1, 1 << 13)[0], (1 << 32) + 15]


def words(rng, q, n):
    """Extreme and random residues."""
    return [rng.choice([0, 1, q - 1, q - 2, rng.randrange(q)]) for _ in range(n)]


def sum40(d, k, add, q):
    mu32 = (1 << 64) // q
    assert mu32 <= M32
    L = sum((x & 0xFFFFF) * (y & M32) for x, y in zip(d, k))
    M = sum((x >> 20) * (y & M32) for x, y in zip(d, k))
    P = sum((x & 0xFFFFF) * (y >> 32) for x, y in zip(d, k))
    Q = sum((x >> 20) * (y >> 32) for x, y in zip(d, k))
    assert max(L, M) <= M64 and max(P, Q) <= M32
    m = M + (P << 12) + (Q << 32)
    assert m <= M64
    m -= ((m >> 32) * mu32 >> 32) * q
    assert 0 <= m < 3 * q
    y = L + add + (m << 20)
    assert y <= M64
    return y - ((y >> 32) * mu32 >> 32) * q


def reduce_top(x, q):
    b = q.bit_length()
    assert x >> (63 + b) == 0
    x1, mu = x >> (b - 1), (1 << (63 + b)) // q
    assert x1 <= M64 and mu <= M64
    qe = (x1 >> 32) * (mu >> 32) + ((x1 & M32) * (mu >> 32) >> 32) + ((x1 >> 32) * (mu & M32) >> 32)
    return x - qe * q


@pytest.mark.parametrize("q", primes40())
def test_sum40(q):
    rng = random.Random(1)
    for _ in range(300):
        n = rng.randint(1, 8)
        d, k, add = words(rng, q, n), words(rng, q, n), rng.choice([0, 4 * q, q - 1])
        v = sum40(d, k, add, q)
        assert 0 <= v < 3 * q and (v - add - sum(x * y for x, y in zip(d, k))) % q == 0


@pytest.mark.parametrize("bits", [18, 31, 32, 33, 41, 54, 55, 56, 60])
def test_sum60_reduces_below_5q(bits):
    q = synth.ntt_primes(bits, 1, 1 << 13)[0]
    rng = random.Random(bits)
    lo = (1 << 30) - 1
    for _ in range(300):
        n = rng.randint(1, 8)
        d, k, add = words(rng, q, n), words(rng, q, n), rng.choice([0, 6 * q - 1])
        L = sum((x & lo) * (y & lo) for x, y in zip(d, k)) + add
        M = sum((x & lo) * (y >> 30) + (x >> 30) * (y & lo) for x, y in zip(d, k))
        H = sum((x >> 30) * (y >> 30) for x, y in zip(d, k))
        assert max(L, M, H) <= M64
        x = L + (M << 30) + (H << 60)
        v = reduce_top(x, q)
        assert 0 <= v < 5 * q and (v - x) % q == 0


def test_outer_sums_fit():
    """The outer sums' halves: v f = v0 f0 + 2^32 (v0 f1 + v1 f0) + 2^64 v1 f1, L's carries added to H."""
    def fits(v, f, terms, h_max):
        v1, f1 = v >> 32, f >> 32
        return terms * (M32 * f1 + v1 * M32) <= M64 and terms * (v1 * f1 + 1) <= h_max

    assert fits(3 * (1 << 40) - 1, (1 << 40) - 1, 16384, M32)  # packed: v < 3q
    assert fits(5 * (1 << 55) - 1, (1 << 55) - 1, 64, M64)     # up to 55 bits: v < 5q
    assert 32 * (5 * (1 << 60) - 1) * ((1 << 60) - 1) + (1 << 60) < 1 << 128  # 128-bit sums


@pytest.mark.parametrize("q", primes40())
def test_packed_outer_value(q):
    """The reduction of L + 2^32 M + 2^64 H in the steps of the kernel."""
    mu32, rng = (1 << 64) // q, random.Random(3)
    red = lambda x: x - ((x >> 32) * mu32 >> 32) * q
    for _ in range(200):
        L, M, H = rng.choice([0, M64, rng.getrandbits(64)]), rng.randrange(1 << 58), rng.randrange(3 << 30)
        assert M + (H << 32) <= M64
        u = (L >> 32) + red(M + (H << 32))
        assert u < 1 << 43
        r = red(u << 20 | (L & M32) >> 12)
        y = r << 12 | (L & 0xFFF)
        assert r < 3 * q and y <= M64
        assert 0 <= red(y) < 3 * q and (red(y) - (L + (M << 32) + (H << 64))) % q == 0


@pytest.mark.parametrize("log_n", [12, 13, 15, 16])
def test_gather_splits_at_the_run(log_n):
    """Word l of run `run` reads word brv_7(C + g brv_7(l) mod 128) of run srun (Eq. 7)."""
    brv = lambda x, n: int(format(x, f"0{n}b")[::-1], 2)
    N, lr, rng = 1 << log_n, log_n - 7, random.Random(log_n)
    for _ in range(40):
        g, run = pow(5, rng.randrange(N // 2), 2 * N), rng.randrange(N // 128)
        E = ((g * (2 * brv(run, lr) + 1) - 1) >> 1) % N
        srun, C = brv(E % (1 << lr), lr), E >> lr
        for l in [0, 1, 127, rng.randrange(128)]:
            e = g * (2 * brv(run * 128 + l, log_n) + 1) % (2 * N)
            want = brv((e - 1) // 2, log_n)
            assert srun * 128 + brv((C + g * brv(l, 7)) % 128, 7) == want
