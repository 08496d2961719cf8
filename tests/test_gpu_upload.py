"""What a batch uploads: the rows of each accepted pair up to its true
x-degree.  A rejected pair's coefficients are not read again (its extents may
be anything), and a batch that is used again with arrays padded by zero rows
takes the same rows."""
import ctypes

import numpy as np
import pytest

from paper_1010_1386_gb300 import inputs, rs

pytestmark = pytest.mark.gpu


def padded(f, rows):
    c = f.coeffs
    return inputs.BiPoly(np.concatenate([c, np.zeros((rows,) + c.shape[1:], dtype=np.uint32)]))


def some_pairs(n, deg):
    return inputs.workload_batch(7, n=n, deg_lo=deg, deg_hi=deg)


def test_input_bytes():
    (f, g), = some_pairs(1, 5)
    too_long = inputs.BiPoly(np.ones((4, 3, 200), dtype=np.uint32))  # more limbs than the library takes
    zero = inputs.BiPoly(np.zeros((9, 3, 1), dtype=np.uint32))
    F, G = rs._Polys([f, too_long, f, zero, padded(f, 6)]), rs._Polys([g, g, too_long, g, padded(g, 1)])
    lib, h, info = rs.load(), ctypes.c_void_p(), rs.rs_batch_info()
    with rs.Context() as ctx:
        assert lib.rs_batch_create(ctx.h, 5, F.structs, G.structs, ctypes.byref(h)) == 0
        assert lib.rs_batch_info_get(h, ctypes.byref(info)) == 0
        assert info.input_bytes == 2 * 4 * (f.coeffs.size + g.coeffs.size)
        assert lib.rs_batch_destroy(h) == 0


@pytest.mark.parametrize("n", [4, 200])  # copied by the calling thread, and by several
def test_padded_arrays(n):
    pairs = some_pairs(n, 6)
    wide = [(padded(f, 40 + i % 7), padded(g, 3 * (i % 5))) for i, (f, g) in enumerate(pairs)]
    with rs.Context() as ctx:
        want = ctx.resultant_batch(pairs)
        assert ctx.resultant_batch(wide) == want  # the batch of the call before, more rows in the arrays
        assert ctx.resultant_batch(pairs) == want
        b = ctx.batch(pairs)
        b.upload(wide)
        b.run()
        b.sync()
        assert b.results() == want
        b.close()


@pytest.mark.parametrize("field,value", [("coeffs", 0), ("deg_x", -3), ("deg_x", 1 << 30), ("deg_y", -7),
                                         ("limbs", 0), ("limbs", 129), ("limbs", 1 << 30)])
def test_rejected_pairs(field, value):
    lib = rs.load()
    pairs = some_pairs(6, 5)
    with rs.Context() as ctx:
        want = ctx.resultant_batch(pairs)
        F, G = rs._Polys([p[0] for p in pairs]), rs._Polys([p[1] for p in pairs])
        F.raw[1][field] = value
        G.raw[4][field] = value
        out = rs._Outputs(pairs)
        status = (ctypes.c_int32 * len(pairs))()
        for _ in range(2):  # built, then used again
            assert lib.rs_resultant_batch(ctx.h, len(pairs), F.structs, G.structs, out.structs, status) < 0
            assert [s == 0 for s in status] == [i not in (1, 4) for i in range(6)]
            got = out.ints()
            assert [got[i] for i in (0, 2, 3, 5)] == [want[i] for i in (0, 2, 3, 5)]
