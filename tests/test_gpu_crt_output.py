"""The carry and output kernel of the Chinese remaindering: coefficients whose
two's-complement limbs are all ones or all zeros over whole 16-limb chunks
(carries and borrows that run through several chunks), result lengths at the
edges of its steps (1, 2, 4, 5, 8, 9, 16 and 17 chunks) and coefficient counts
around 32 and 128, with limbs from both limb kernels, against exact integers."""
import random

import pytest

from oracle import exact

pytestmark = pytest.mark.gpu


def scaled_pair(coeffs, shift):
    """2^s y and y^m + d(x): their resultant in y is +-2^(s m) d, coefficient by coefficient."""
    m = max(1, -(-shift // 3900))
    f = [[0, 2 ** (shift // m)]]
    g = [[c] + [0] * m for c in coeffs]
    g[0][m] = 1
    return f, g, shift // m * m


@pytest.mark.parametrize("form", [1, 0, 2])
@pytest.mark.parametrize("chunks", [1, 2, 4, 5, 8, 9, 16, 17, 33])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 300])
def test_carries(form, chunks, n):
    from paper_1010_1386_gb300 import rs
    rng = random.Random(1000 * chunks + n)
    bits = 512 * chunks - 40
    top = min(bits, 4000)  # input coefficients have at most 128 limbs
    special = [0, 1, -1]
    for b in range(8, top, 8):
        special += [2**b, 2**b - 1, 1 - 2**b, -(2**b), -(2**b) - 1, 2**b + 1]
    cs = [2**top - 1] + [rng.choice(special) for _ in range(n - 1)]
    with rs.Context(crt_form=form) as ctx:
        for sign in (1, -1):
            f, g, s = scaled_pair([sign * x for x in cs], bits - top)
            want = exact.resultant_y(f, g)
            assert max(abs(x) for x in want) >> s == 2**top - 1
            assert ctx.resultant_y(f, g) == want


@pytest.mark.parametrize("bits", [984, 1000, 1496, 1900, 2200, 2430])
def test_carries_in_one_kernel(bits):
    """The same values in the one-kernel remaindering, 2 to 5 chunks of 16 limbs
    (up to 80 primes), which many coefficients take."""
    from paper_1010_1386_gb300 import rs
    rng = random.Random(bits)
    special = [0, 1, -1]
    for b in range(8, bits, 8):
        special += [2**b, 2**b - 1, 1 - 2**b, -(2**b), -(2**b) - 1, 2**b + 1]
    pairs, want = [], []
    for i in range(100):
        cs = [(1 - 2 * (i & 1)) * (2**bits - 1)] + [rng.choice(special) for _ in range(298)] + [1]
        f, g, _ = scaled_pair(cs, 0)
        pairs.append((f, g))
        want.append(cs)
    sign = exact.resultant_y(*pairs[0])[299]
    want = [[sign * c for c in cs] for cs in want]
    assert want[1] == exact.resultant_y(*pairs[1])
    launches = []
    for form in (0, 1):
        with rs.Context(crt_form=form) as ctx:
            b = ctx.batch(pairs)
            b.run()
            b.sync()
            assert b.results() == want
            launches.append(b.info()["kernel_launches"])
            b.close()
    assert launches[0] == launches[1] - 2
