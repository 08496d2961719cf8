"""Inputs of many limbs: limb counts around where the staging changes to summed
products (8) and up to the largest (128), values at the ends of their range
and of both signs, in full rows and in sparse ones (missing coefficients and
whole missing columns), against the exact oracle."""
import random

import pytest

from oracle import exact

pytestmark = pytest.mark.gpu


def value(rng, limbs):
    b = 32 * limbs - 1
    return rng.choice([2**b - 1, 1 - 2**b, 2 ** (b - 1), 1, -1, rng.getrandbits(b), -rng.getrandbits(b), rng.getrandbits(31)])


def poly(rng, dx, dy, limbs, keep):
    """[i][j]: coefficient of x^i y^j; `keep` of the coefficients, whole columns missing below the top."""
    cols = [j == dy or rng.random() < max(keep, 0.5) for j in range(dy + 1)]
    f = [[value(rng, limbs) if cols[j] and rng.random() < keep else 0 for j in range(dy + 1)] for _ in range(dx + 1)]
    f[0][dy] = 2 ** (32 * limbs - 1) - 1  # the full limb count, and the leading column
    return f


@pytest.mark.parametrize("limbs", [1, 7, 8, 9, 31, 32, 33, 127, 128])
@pytest.mark.parametrize("keep", [1.0, 0.3])
@pytest.mark.parametrize("shape", [(0, 3), (3, 2), (9, 1), (2, 7), (1, 9)])
def test_limb_counts(limbs, keep, shape):
    from paper_1010_1386_gb300 import rs
    dx, dy = shape
    rng = random.Random(limbs * 100 + dx * 10 + dy)
    pairs = [(poly(rng, dx, dy, limbs, keep), poly(rng, max(dx - 1, 0), 2, rng.choice([1, limbs]), keep))
             for _ in range(2)]
    with rs.Context() as ctx:
        assert ctx.resultant_batch(pairs) == [exact.resultant_y(f, g) for f, g in pairs]
