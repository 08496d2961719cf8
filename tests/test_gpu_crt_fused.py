"""The Chinese remaindering in one kernel (few primes): every prime count to 16
and, with the many coefficients that take them there, counts around the groups
of four digits, the chunks of 16 limbs and the largest (80); coefficient counts
around its blocks of 128; against the exact oracle and the separate kernels."""
import random

import pytest

from oracle import exact
from tests.helpers import rand_bipoly

pytestmark = pytest.mark.gpu


def pair_with_primes(rng, dx, K):
    """A pair of y-degree 1 whose resultant takes about K primes."""
    from paper_1010_1386_gb300 import rs
    lo, hi = 1, 4000
    while True:
        bits = (lo + hi) // 2
        f, g = rand_bipoly(rng, dx, 1, bits), rand_bipoly(rng, dx, 1, bits)
        k = rs.result_bound(f, g)["primes"]
        if k == K or hi - lo <= 1:
            return f, g, bits
        lo, hi = (bits, hi) if k < K else (lo, bits)


def run(pairs, form=0):
    """Results, and the number of kernels a pass launches."""
    from paper_1010_1386_gb300 import rs
    with rs.Context(crt_form=form) as ctx:
        b = ctx.batch(pairs)
        b.run()
        b.sync()
        out, launches = b.results(), b.info()["kernel_launches"]
        b.close()
        return out, launches


@pytest.mark.parametrize("K", list(range(1, 17)))
def test_few_primes(K):
    rng = random.Random(K)
    pairs = [pair_with_primes(rng, dx, K)[:2] for dx in (0, 3, 63, 64, 80)]  # 1, 7, 127, 129 and 161 coefficients
    got, launches = run(pairs)
    assert got == [exact.resultant_y(f, g) for f, g in pairs]
    assert launches < run(pairs, form=1)[1]


@pytest.mark.parametrize("K", [17, 18, 32, 33, 34, 63, 66, 79, 80])
def test_more_primes(K):
    from paper_1010_1386_gb300 import rs
    rng = random.Random(K)
    _, _, bits = pair_with_primes(rng, 12, K)
    pairs = []
    while len(pairs) < 1000:  # 25,000 coefficients
        f, g = rand_bipoly(rng, 12, 1, bits), rand_bipoly(rng, 12, 1, bits)
        if rs.result_bound(f, g)["primes"] <= K:  # some ask for one prime more than the probe's
            pairs.append((f, g))
    assert max(rs.result_bound(f, g)["primes"] for f, g in pairs) == K
    got, launches = run(pairs)
    tiles, more = run(pairs, form=1)
    assert got == tiles
    assert launches < more
    for i in range(0, len(pairs), 97):
        assert got[i] == exact.resultant_y(*pairs[i])
