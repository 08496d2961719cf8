"""The direct interpolation form (g2_form = 1): point-pair counts around its
output blocks of 7, with the pairs alone (few blocks: many segments, the even
and odd part in a block each) and among many (few segments, small blocks),
against the exact oracle; the largest count of its range against the oracle
modulo a prime it does not use itself, and mixed sizes in one batch against
the transform form."""
import random

import pytest

from oracle import exact
from tests.helpers import check_sampled_31, rand_bipoly

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def direct():
    from paper_1010_1386_gb300 import rs
    with rs.Context(g2_form=1) as ctx:
        yield ctx


# y-degree 1 and x-degree M - 1 give 2 M - 1 coefficients, M point pairs
@pytest.mark.parametrize("M", [1, 2, 6, 7, 8, 13, 14, 15, 21, 22, 27, 28, 29, 35, 36, 63, 64, 65, 112, 113, 127, 128])
@pytest.mark.parametrize("n", [1, 40])
def test_point_counts(direct, M, n):
    rng = random.Random(100 * M + n)
    pairs = [(rand_bipoly(rng, M - 1, 1, 40), rand_bipoly(rng, M - 1, 1, 40)) for _ in range(n)]
    got = direct.resultant_batch(pairs)
    assert got[:3] == [exact.resultant_y(f, g) for f, g in pairs[:3]]
    assert got[-1] == exact.resultant_y(*pairs[-1])


def test_many_tasks(direct):
    rng = random.Random(5)
    pairs = [(rand_bipoly(rng, dx, 2, 60), rand_bipoly(rng, dx, 2, 60)) for dx in (2, 4, 9, 16, 30) for _ in range(400)]
    got = direct.resultant_batch(pairs)
    for i in range(0, len(pairs), 67):
        assert got[i] == exact.resultant_y(*pairs[i])
    from paper_1010_1386_gb300 import rs
    with rs.Context(g2_form=2) as ctx:
        assert ctx.resultant_batch(pairs) == got


@pytest.mark.parametrize("dx,dy", [(2047, 1), (812, 8), (814, 8), (1023, 8)])  # up to 8,185 point pairs
def test_largest_counts(direct, dx, dy):
    rng = random.Random(dx)
    f, g = rand_bipoly(rng, dx, dy, 6), rand_bipoly(rng, dx, dy, 6)
    check_sampled_31(f, g, direct.resultant_y(f, g), rng)


@pytest.mark.parametrize("dx", [820, 812])
def test_largest_counts_with_many_primes(direct, dx):
    """More than two blocks per SM: the halves in turn (6,561 point pairs), and
    both at once at the shared-memory limit (6,497)."""
    from paper_1010_1386_gb300 import rs
    rng = random.Random(dx)
    f, g = rand_bipoly(rng, dx, 8, 650), rand_bipoly(rng, dx, 8, 650)
    assert rs.result_bound(f, g)["primes"] > 304
    R = direct.resultant_y(f, g)
    check_sampled_31(f, g, R, rng)
