"""Results copied back in pieces (large batches): every pair equals the same
pair alone, with zero resultants, a buffer that is too small and a pair that
fails to plan among them."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_pieces():
    from paper_1010_1386_gb300 import inputs, rs
    lib = rs.load()
    base = inputs.workload_shift(5, 15, False, 2048)  # about 1.7 MB of results per pair
    zero = inputs.BiPoly(np.zeros((3, 3, 1), dtype=np.uint32))
    pairs = [(zero, base[0][1])] + (base * 3)[:14] + [(base[0][0], zero)] + (base * 3)[14:] + [(zero, zero)]
    with rs.Context() as ctx:
        want = [rs.limbs_to_ints(w, d, l) for d, l, w in (ctx.resultant_batch([p], raw=True)[0] for p in base)]
        F, G = rs._Polys([p[0] for p in pairs]), rs._Polys([p[1] for p in pairs])
        F.raw[4]["limbs"] = 500  # above the limit
        out = rs._Outputs(pairs)
        out.structs[9].capacity_words = 10
        status = (ctypes.c_int32 * len(pairs))()
        for _ in range(2):
            rc = lib.rs_resultant_batch(ctx.h, len(pairs), F.structs, G.structs, out.structs, status)
            assert rc == status[4] != 0
            assert status[9] == -2 and (out.structs[9].deg + 1) * out.structs[9].limbs > 10
            assert not out.bufs[9].any()
            order = (list(range(10)) * 3)
            k = 0
            for i, (f, g) in enumerate(pairs):
                if f is zero or g is zero:
                    assert status[i] == 0 and out.structs[i].deg == -1
                    continue
                j = order[k]
                k += 1
                if i in (4, 9):
                    continue
                assert status[i] == 0
                assert rs.limbs_to_ints(out.bufs[i], out.structs[i].deg, out.structs[i].limbs) == want[j], i
