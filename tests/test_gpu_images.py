"""The image kernel.  The remainder sequence's double steps (two degrees of one polynomial per
pass): every image equals the oracle's determinant of the formal Sylvester
matrix, over degrees at the edges of the register capacities and phases,
equal, adjacent and far apart, on dense inputs and on sparse ones whose
sequence meets vanishing pivots; the evaluation's row groups (7 products per
fold, two parities) at their edges, with zero coefficients and inputs so large
that the evaluation takes no shared columns."""
import random

import pytest

from oracle import modp
from tests.helpers import check_sampled_31, rand_bipoly

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1010_1386_gb300 import rs
    with rs.Context() as c:
        yield c


def check(ctx, f, g, primes=2, points=6):
    ps, xs, zs = ctx.images(f, g, primes, points)
    for k in range(primes):
        for i in range(points):
            assert int(zs[k, i]) == modp.resultant_image(f, g, int(ps[k]), int(xs[k, i])), (k, i)


DEGREES = [(1, 1), (2, 1), (1, 2), (3, 1), (1, 4), (2, 2), (3, 3), (7, 7), (7, 6), (8, 8), (9, 7), (12, 12), (13, 12),
           (15, 16), (16, 16), (19, 20), (21, 20), (23, 23), (24, 23), (27, 28), (28, 28), (29, 30), (31, 32), (36, 35),
           (37, 36), (39, 39), (40, 40), (41, 20), (20, 43), (47, 47), (48, 47), (55, 54), (56, 56), (57, 29), (63, 63),
           (64, 64), (65, 3), (3, 66), (71, 71), (71, 70), (70, 71), (71, 1), (1, 71)]


@pytest.mark.parametrize("m,n", DEGREES)
def test_dense(ctx, m, n):
    rng = random.Random(1000 * m + n)
    check(ctx, rand_bipoly(rng, 2, m, 40), rand_bipoly(rng, 3, n, 40))


@pytest.mark.parametrize("m,n", [(6, 4), (9, 9), (17, 16), (29, 28), (37, 20), (41, 41), (57, 50), (71, 64)])
def test_vanishing_pivots(ctx, m, n):
    """Every third power of y, a common factor, and leading coefficients that
    vanish at the first point pair (x = 1 and x = -1)."""
    rng = random.Random(77 * m + n)
    f, g = rand_bipoly(rng, 2, m, 20), rand_bipoly(rng, 2, n, 20)
    sf = [[c if (m - j) % 3 == 0 else 0 for j, c in enumerate(row)] for row in f]
    sg = [[c if (n - j) % 3 == 0 else 0 for j, c in enumerate(row)] for row in g]
    check(ctx, sf, sg)
    check(ctx, sf, g)
    check(ctx, f, sg)
    lead = [-1, 0, 1]  # x^2 - 1
    for i in range(3):
        f[i][m] = lead[i]
    check(ctx, f, g)
    for i in range(3):
        g[i][n] = 2 * lead[i]
    check(ctx, f, g)
    h = [[3, -1, 2], [1, 0, 0], [0, 5, 0]]  # common factor: R = 0

    def times(a, b):
        out = [[0] * (len(a[0]) + len(b[0]) - 1) for _ in range(len(a) + len(b) - 1)]
        for i, r in enumerate(a):
            for j, c in enumerate(r):
                for k, s in enumerate(b):
                    for l, d in enumerate(s):
                        out[i + k][j + l] += c * d
        return out
    if m <= 69:
        ps, xs, zs = ctx.images(times(f, h), times(g, h), 2, 6)
        assert not zs.any()


@pytest.mark.parametrize("dx", [0, 1, 2, 5, 6, 11, 12, 13, 14, 15, 16, 26, 27, 28, 29, 41, 42, 43])
def test_evaluation_rows(ctx, dx):
    rng = random.Random(31 * dx + 5)
    for m, n, other in ((9, 9, 3), (17, 3, dx), (33, 10, 1)):
        f, g = rand_bipoly(rng, dx, m, 33), rand_bipoly(rng, other, n, 33)
        for j in (1, m // 2):  # zero coefficients of y^j, and one of low x-degree
            for row in f:
                row[j] = 0
        for row in g[1:]:
            row[n // 2] = 0
        check(ctx, f, g, primes=1, points=70)


def test_largest_staged_inputs(ctx):
    """deg_y = 71 with deg_x = 470 and 190: the staged coefficients leave too
    little shared memory for 128 threads' columns."""
    rng = random.Random(9)
    check(ctx, rand_bipoly(rng, 470, 71, 12), rand_bipoly(rng, 190, 1, 12), primes=1, points=4)


@pytest.mark.parametrize("cap", range(8, 80, 8))
def test_without_columns(ctx, cap):
    """About 28,100 words staged: two blocks of 128 threads fit an SM's shared
    memory without their columns (28,800 words each), one with them."""
    rng = random.Random(cap)
    dx = 27900 // (cap + 1) - 8
    check(ctx, rand_bipoly(rng, dx, cap - 1, 12), rand_bipoly(rng, 3, 1, 12), primes=1, points=70)


def test_both_forms_of_a_capacity():
    """One batch with pairs of the same register capacity in both forms."""
    from paper_1010_1386_gb300 import rs
    rng = random.Random(12)
    pairs = [(rand_bipoly(rng, dx, 39, 12), rand_bipoly(rng, 2, 2, 12)) for dx in (3, 672, 5, 672, 17)]
    with rs.Context() as c:
        for (f, g), R in zip(pairs, c.resultant_batch(pairs)):
            check_sampled_31(f, g, R, rng)
