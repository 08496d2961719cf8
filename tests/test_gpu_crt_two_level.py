"""CRT digits in two levels (groups of 256 digits from the tiled kernel, their
products with the later residues on the tensor cores): prime counts at the
edges of a digit block (64) and of a group (256), coefficient counts at the
edges of the tiles (16 and 128), pairs with fewer groups than the longest in
one batch, against the exact oracle; and the same digits as the tiled kernel
gives by itself."""
import random

import pytest

from oracle import exact
from tests.helpers import rand_bipoly

pytestmark = pytest.mark.gpu


def pair_with_primes(rng, dx, K):
    """A pair of y-degree 6 and x-degree dx whose resultant takes about K primes."""
    from paper_1010_1386_gb300 import rs
    lo, hi = 8, 4090
    while True:
        bits = (lo + hi) // 2
        f, g = rand_bipoly(rng, dx, 6, bits), rand_bipoly(rng, dx, 6, bits)
        k = rs.result_bound(f, g)["primes"]
        if k == K or hi - lo <= 1:
            return f, g, k
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


@pytest.mark.parametrize("K", [1023, 1024, 1025, 1087, 1088, 1089, 1281])
def test_prime_counts(K):
    rng = random.Random(K)
    f, g, k = pair_with_primes(rng, 1, K)
    assert abs(k - K) <= 1
    got, launches = run([(f, g)])
    assert launches == 5 + 2 * ((k - 1) // 256)  # the two-level digits were taken
    assert got == [exact.resultant_y(f, g)]


def test_uneven_batch():
    """Prime counts from 20 to 1,300 and coefficient counts from 1 to 301 in one batch."""
    rng = random.Random(77)
    pairs = []
    for dx, K in ((0, 1300), (1, 1100), (2, 1030), (4, 300), (5, 256), (5, 257), (10, 700), (25, 20)):
        f, g, _ = pair_with_primes(rng, dx, K)
        pairs.append((f, g))
    got, launches = run(pairs)
    tiles, fewer = run(pairs, form=1)
    assert launches > fewer
    assert got == tiles
    assert got[:2] == [exact.resultant_y(f, g) for f, g in pairs[:2]]


def test_repeated_and_zero():
    """A second pass over the same buffers, and a pair with a zero resultant beside a long one."""
    from paper_1010_1386_gb300 import rs
    rng = random.Random(78)
    f, g, _ = pair_with_primes(rng, 1, 1200)
    with rs.Context() as ctx:
        b = ctx.batch([(f, g), (f, f)])
        want = [exact.resultant_y(f, g), []]
        for _ in range(3):
            b.run()
            b.sync()
            got = b.results()
            assert got[0] == want[0] and not any(got[1])
        b.close()


def test_wait_runs_out_and_context_recovers():
    """The copies of the far products held back by the test hook: their waits
    give up, the context reports the timeout and is exact again afterwards."""
    from paper_1010_1386_gb300 import rs
    rng = random.Random(79)
    f, g, _ = pair_with_primes(rng, 1, 1030)
    want = exact.resultant_y(f, g)
    with rs.Context() as ctx:
        assert ctx.resultant_y(f, g) == want
        ctx.stall_tensor_cores(True)
        with pytest.raises(rs.RsError) as ei:
            ctx.resultant_y(f, g)
        assert ei.value.code == -5  # RS_ERR_TIMEOUT
        ctx.stall_tensor_cores(False)
        assert ctx.resultant_y(f, g) == want
