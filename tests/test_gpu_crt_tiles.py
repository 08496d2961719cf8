"""The tiled CRT digit kernel (CUDA cores) with CUDA-core limbs
(crt_form = 1) and, where the shape rule takes it, with tensor-core limbs
(crt_form = 0): prime counts at the edges of its sub-blocks (4), half blocks
(32) and digit blocks (64), coefficient counts at the edges of its tiles (16
and 32) and of the limb kernel's (128), against the exact oracle; many pairs
of few primes through the one-thread-per-coefficient kernel."""
import random

import pytest

from oracle import exact
from tests.helpers import check_sampled_31, rand_bipoly

pytestmark = pytest.mark.gpu


def pair_with_primes(rng, dx, K):
    """A pair of y-degree 1 and x-degree dx whose resultant takes K primes."""
    from paper_1010_1386_gb300 import rs
    lo, hi = 8, 4000
    while True:
        bits = (lo + hi) // 2
        f, g = rand_bipoly(rng, dx, 1, bits), rand_bipoly(rng, dx, 1, bits)
        k = rs.result_bound(f, g)["primes"]
        if k == K or hi - lo <= 1:
            return f, g, k
        lo, hi = (bits, hi) if k < K else (lo, bits)


@pytest.mark.parametrize("form", [1, 0])
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 8, 9, 23, 24, 31, 32, 33, 60, 63, 64, 65, 68, 95, 96, 97, 127, 128, 129,
                               160, 193])
def test_prime_counts(form, K):
    from paper_1010_1386_gb300 import rs
    rng = random.Random(100 * K + form)
    pairs, ks = [], set()
    for dx in (3, 8):  # 7 and 17 coefficients
        f, g, k = pair_with_primes(rng, dx, K)
        pairs.append((f, g))
        ks.add(k)
    assert min(abs(k - K) for k in ks) <= 1
    with rs.Context(crt_form=form) as ctx:
        assert ctx.resultant_batch(pairs) == [exact.resultant_y(f, g) for f, g in pairs]


@pytest.mark.parametrize("form", [1, 0])
@pytest.mark.parametrize("n", [15, 16, 17, 31, 32, 33, 127, 128, 129, 257])
def test_coefficient_counts(form, n):
    from paper_1010_1386_gb300 import rs
    rng = random.Random(n + form)
    f, g = rand_bipoly(rng, (n - 1 + 1) // 2, 1, 900), rand_bipoly(rng, (n - 1) // 2, 1, 900)
    with rs.Context(crt_form=form) as ctx:
        R = ctx.resultant_y(f, g)
    assert len(R) == n
    assert R == exact.resultant_y(f, g)


@pytest.mark.parametrize("form", [1, 0])
def test_tiles_of_32(form):
    """Enough coefficients for 32 a tile: 120 pairs of 113 coefficients, 100 to
    200 primes, each equal to the pair alone (16 a tile)."""
    from paper_1010_1386_gb300 import rs
    rng = random.Random(5)
    pairs = []
    for i in range(120):
        b = 380 + 3 * i
        pairs.append((rand_bipoly(rng, 14, 4, b), rand_bipoly(rng, 14, 4, b)))
    with rs.Context(crt_form=form) as ctx:
        got = ctx.resultant_batch(pairs)
        for i in (0, 1, 59, 60, 118, 119):
            assert got[i] == ctx.resultant_y(*pairs[i])
            check_sampled_31(*pairs[i], got[i], rng, samples=1)


def test_one_thread_per_coefficient_with_few_primes():
    from paper_1010_1386_gb300 import rs
    rng = random.Random(6)
    pairs = [(rand_bipoly(rng, 4 + i % 3, 3, 14), rand_bipoly(rng, 5, 2 + i % 2, 14)) for i in range(900)]
    with rs.Context() as ctx:
        got = ctx.resultant_batch(pairs)
    for i in range(0, 900, 29):
        assert got[i] == exact.resultant_y(*pairs[i])


@pytest.mark.parametrize("n,bits", [(40, 900), (1500, 900), (1500, 2300)])  # limbs on the tensor cores, then on the CUDA cores twice
def test_one_long_pair(n, bits):
    """One pair of about 120 or 300 primes with many of a few."""
    from paper_1010_1386_gb300 import rs
    rng = random.Random(n + bits)
    pairs = [(rand_bipoly(rng, 2, 2, 20), rand_bipoly(rng, 2, 2, 20)) for _ in range(n)]
    pairs.insert(n // 2, (rand_bipoly(rng, 6, 2, bits), rand_bipoly(rng, 6, 2, bits)))
    with rs.Context() as ctx:
        got = ctx.resultant_batch(pairs)
    for i in [n // 2] + list(range(0, n, 97)):
        assert got[i] == exact.resultant_y(*pairs[i])
    with rs.Context(crt_form=1) as ctx:
        assert ctx.resultant_batch(pairs) == got
