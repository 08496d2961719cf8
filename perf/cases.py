"""Timed cases: exact resultants through the library's C ABI, host buffers in
and host buffers out, over the range of work a program gives it.

A pass uploads the inputs, runs the batch and copies the trimmed results back
(or makes one call that does all three).  Results are integers: per pair a
degree, a limb count and the coefficients' two's-complement limbs.
"""
import ctypes
import math

import numpy as np

from paper_1010_1386_gb300 import inputs, rs
from paper_1010_1386_gb300.inputs import BiPoly

_UPOLY = np.dtype([("deg", "<i4"), ("limbs", "<i4"), ("capacity_words", "<i8"), ("coeffs", "<u8")])
_CTX = {}  # the program's handles: one context for calls and batches, one that serves


def _ctx(what="calls"):
    if what not in _CTX:
        _CTX[what] = rs.Context()
        if what == "server":
            _CTX["served"] = rs.Server(_CTX[what])
    return _CTX[what]


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # one call on one small pair of curves: two plane curves of degree 6 as a
        # geometry program meets them, planning, launches and copies included
        {"name": "one_call_deg6", "kind": "dense", "call": "once", "n": 1, "deg": 6, "bits": 11},
        # a batch of many small systems (curve arrangements: conics to octics)
        {"name": "small_1024", "kind": "uneven", "call": "batch", "n": 1024, "lo": 2, "hi": 8, "bits": "16,32"},
        # a single ordinary pair of dense curves
        {"name": "single_deg30", "kind": "dense", "call": "batch", "n": 1, "deg": 30, "bits": 32},
        # a single large pair: the largest request of the serving mix
        {"name": "single_deg64_128", "kind": "dense", "call": "batch", "n": 1, "deg": 64, "bits": 128},
        # a ragged handful of pairs of uneven degrees
        {"name": "uneven_17", "kind": "uneven", "call": "batch", "n": 17, "lo": 8, "hi": 40, "bits": "16,32,64"},
        # the large batch of uneven pairs
        {"name": "uneven_512", "kind": "uneven", "call": "batch", "n": 512, "lo": 8, "hi": 40, "bits": "16,32,64"},
        # topology computation: f = p q^2 against the derivative of p q or, where no one took the square-free
        # part, of f itself (that resultant vanishes and every image degenerates)
        {"name": "critical_32", "kind": "critical", "call": "batch", "n": 32, "p": 24, "q": 12, "bits": 64,
         "zeros": 16},
        # long coefficients (shifted curves), both projections: about 500, 1,200 and
        # 2,000 primes
        {"name": "shift15_k512", "kind": "shift", "call": "batch", "deg": 15, "k": 512, "sparse": False},
        {"name": "shift15_k2048", "kind": "shift", "call": "batch", "deg": 15, "k": 2048, "sparse": False},
        {"name": "shift9_sparse_k2048", "kind": "shift", "call": "batch", "deg": 9, "k": 2048, "sparse": True},
        # requests of mixed degrees and sizes submitted at once to the continuous-batching server
        {"name": "serve_96", "kind": "mixed", "call": "serve", "n": 96, "lo": 8, "hi": 64, "bits_lo": 16,
         "bits_hi": 128},
        # square-free factorisation of the resultants of such curves
        {"name": "squarefree_16", "kind": "critical", "call": "squarefree", "n": 16, "p": 24, "q": 12, "bits": 64,
         "zeros": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "uneven", "uneven", "critical", "shift", "mixed", "squarefree"])
    if kind == "dense":
        deg, bits = _log_int(rng, 3, 64), rng.randint(8, 128)
        # K (D + 1) images of about 2 deg^2 products each: at most the 512-pair batch's
        cost = 2.0 * deg * bits / 31 * deg ** 2 * 2 * deg ** 2
        return {"kind": "dense", "call": rng.choice(["once", "batch"]),
                "n": _log_int(rng, 1, max(1, min(512, int(2e10 / cost)))), "deg": deg, "bits": bits}
    if kind == "uneven":
        lo = rng.randint(2, 20)
        return {"kind": "uneven", "call": "batch", "n": _log_int(rng, 1, 400), "lo": lo, "hi": lo + rng.randint(1, 18),
                "bits": rng.choice(["16", "32", "16,32", "16,32,64"])}
    if kind in ("critical", "squarefree"):
        n = _log_int(rng, 1, 24 if kind == "critical" else 12)
        return {"kind": "critical", "call": "batch" if kind == "critical" else "squarefree", "n": n,
                "p": rng.randint(4, 24), "q": rng.randint(2, 12), "bits": rng.randint(16, 64),
                "zeros": rng.choice([0, n // 2]) if kind == "critical" else 0}
    if kind == "shift":
        return {"kind": "shift", "call": "batch", "deg": rng.randint(4, 15), "k": _log_int(rng, 32, 2048),
                "sparse": rng.random() < 0.5}
    lo = rng.randint(4, 16)
    return {"kind": "mixed", "call": "serve", "n": _log_int(rng, 4, 96), "lo": lo, "hi": rng.randint(lo + 4, 64),
            "bits_lo": rng.randint(8, 32), "bits_hi": rng.randint(33, 128)}


# ----------------------------------------------------------------- the inputs


def _kronecker(poly, width, ny):
    """The polynomial's values as one integer: coefficient (i, j) at digit
    i ny + j of 32 width bits (negative coefficients borrow)."""
    c = poly.coeffs
    nx, nyp, L = c.shape
    neg = (c[..., -1] >> 31).astype(bool)
    mag = c.astype(np.uint64)
    carry = neg.astype(np.uint64)
    for l in range(L):  # two's complement magnitude
        v = np.where(neg, mag[..., l] ^ np.uint64(0xFFFFFFFF), mag[..., l]) + carry
        mag[..., l] = v & np.uint64(0xFFFFFFFF)
        carry = v >> np.uint64(32)
    out = 0
    for sel, sign in ((~neg, 1), (neg, -1)):
        w = np.zeros((nx, ny, width), dtype="<u4")
        w[:, :nyp, :L] = np.where(sel[..., None], mag, 0)
        out += sign * int.from_bytes(w.tobytes(), "little")
    return out


def _from_kronecker(value, nx, ny, width):
    half = int.from_bytes(np.tile(np.array([0] * (width - 1) + [1 << 31], dtype="<u4"), nx * ny).tobytes(), "little")
    raw = (value + half).to_bytes(4 * (nx * ny * width + 1), "little", signed=True)
    w = np.frombuffer(raw, dtype="<u4")[: nx * ny * width].reshape(nx, ny, width).copy()
    w[..., -1] ^= np.uint32(1 << 31)
    return BiPoly(w.astype(np.uint32))


def _derivative_y(poly):
    c = poly.coeffs[:, 1:, :].astype(np.uint64) * np.arange(1, poly.deg_y + 1, dtype=np.uint64)[None, :, None]
    for l in range(c.shape[2]):
        if l + 1 < c.shape[2]:
            c[..., l + 1] += c[..., l] >> np.uint64(32)
        c[..., l] &= np.uint64(0xFFFFFFFF)
    return BiPoly(np.ascontiguousarray(c.astype(np.uint32)))


def _critical(rng, dp, dq, bits, coprime):
    """f = p q^2 and its y-derivative, or that of p q: curves with a repeated
    component, as a curve's topology is computed from them."""
    p, q = (inputs.dense_total_degree(rng, d, bits) for d in (dp, dq))
    terms = (dq + 1) * (dq + 2) // 2
    width = -(-(3 * bits + 2 * terms.bit_length() + (dp + 2 * dq).bit_length() + 2) // 32)
    n = dp + 2 * dq + 1
    P, Q = _kronecker(p, width, n), _kronecker(q, width, n)
    f = _from_kronecker(P * Q * Q, n, n, width)
    if not coprime:
        return f, _derivative_y(f)
    m = dp + dq + 1
    pq = _from_kronecker(P * Q, m, n, width)
    return f, _derivative_y(BiPoly(np.ascontiguousarray(pq.coeffs[:, :m, :])))


def _shapes(case):
    """Per pair the shapes of f and g: (x-degree, y-degree, total degree, bound
    on log2 of a coefficient's size, monomials).  They belong to the case; the
    seed draws the coefficients."""
    rng = np.random.Generator(np.random.PCG64(81))

    def total(d, bits):
        return d, d, d, bits, (d + 1) * (d + 2) // 2

    kind, out = case["kind"], []
    if kind == "dense":
        out = [(total(case["deg"], case["bits"]),) * 2] * case["n"]
    elif kind == "uneven":  # one bidegree and one coefficient size per pair
        for _ in range(case["n"]):
            dx, dy = (int(rng.integers(case["lo"], case["hi"] + 1)) for _ in range(2))
            out.append(((dx, dy, dx + dy, int(rng.choice([int(b) for b in case["bits"].split(",")])),
                         (dx + 1) * (dy + 1)),) * 2)
    elif kind == "critical":
        dp, dq, b = case["p"], case["q"], case["bits"]
        terms = (dq + 1) * (dq + 2) // 2
        d, bits = dp + 2 * dq, 3 * b + 2 * terms.bit_length()
        for i in range(case["n"]):
            dg, bg = (d, bits) if i < case["zeros"] else (dp + dq, 2 * b + terms.bit_length())
            out.append((total(d, bits), (dg - 1, dg - 1, dg - 1, bg + dg.bit_length(), dg * (dg + 1) // 2)))
    elif kind == "shift":  # both projections of the ten pairs of five curves
        d, _, _, bits, terms = total(case["deg"], 16 + case["k"])
        out = [((d, d, d, bits, terms // (4 if case["sparse"] else 1)),) * 2] * 20
    else:  # requests: independent total degrees, one coefficient size
        for _ in range(case["n"]):
            df, dg = (int(rng.integers(case["lo"], case["hi"] + 1)) for _ in range(2))
            b = int(rng.integers(case["bits_lo"], case["bits_hi"] + 1))
            out.append((total(df, b), total(dg, b)))
    return out


def _pairs(case, seed):
    rng = np.random.Generator(np.random.PCG64([int(seed), 77]))
    kind = case["kind"]
    if kind == "critical":
        return [_critical(rng, case["p"], case["q"], case["bits"], i >= case["zeros"]) for i in range(case["n"])]
    if kind == "shift":
        base = inputs.workload_shift([int(seed), 79], case["deg"], case["sparse"], case["k"])
        return base + [(inputs.swap_xy(f), inputs.swap_xy(g)) for f, g in base]
    if kind == "uneven":
        return [tuple(inputs.dense_bidegree(rng, s[0], s[1], s[3]) for s in pair) for pair in _shapes(case)]
    return [tuple(inputs.dense_total_degree(rng, s[0], s[3]) for s in pair) for pair in _shapes(case)]


# ------------------------------------------------------- sizes of the results


def _bounds(case):
    """Per pair (degree bound, bit bound) of Res_y from the shapes: Sylvester
    degrees, Hadamard's bound on the rows."""
    out = []
    for a, b in _shapes(case):
        rows = [s[3] + math.log2(s[0] + 1) + 0.5 * math.log2(s[1] + 1) for s in (a, b)]
        out.append((min(a[0] * b[1] + b[0] * a[1], a[2] * b[2]), int(math.ceil(b[1] * rows[0] + a[1] * rows[1])) + 2))
    return out


class _Results:
    """rs_upoly structs whose coefficients lie in one buffer."""

    def __init__(self, words):
        self.raw = np.zeros(max(1, len(words)), dtype=_UPOLY)
        self.buf = np.zeros(max(1, sum(words)), dtype=np.uint32)
        at = np.concatenate([[0], np.cumsum(words)[:-1]]).astype(np.uint64)
        self.raw["capacity_words"] = words
        self.raw["coeffs"] = np.uint64(self.buf.ctypes.data) + np.uint64(4) * at
        self.structs = (rs.rs_upoly * len(self.raw)).from_buffer(self.raw)

    def outputs(self):
        return {"deg": self.raw["deg"].copy(), "limbs": self.raw["limbs"].copy(), "coeffs": self.buf.view(np.int32)}


def _polys(pairs):
    out = []
    for side in range(2):
        a = (rs.rs_bipoly * len(pairs))()
        for s, p in zip(a, (pair[side] for pair in pairs)):
            c = p.coeffs
            s.deg_x, s.deg_y, s.limbs = c.shape[0] - 1, c.shape[1] - 1, c.shape[2]
            s.coeffs = c.ctypes.data_as(ctypes.POINTER(ctypes.c_uint32))
        out.append(a)
    return out


class _State:
    batch = None

    def __del__(self):
        if self.batch is not None:
            self.batch.close()


def _words(case):
    return [(d + 1) * (b // 32 + 1) for d, b in _bounds(case)]


_MULT = 4  # multiplicities a square-free call reports here (p q^2 gives 1, 2, 3)


def prepare(case, seed):
    s = _State()
    s.call, s.pairs = case["call"], _pairs(case, seed)
    s.f, s.g = _polys(s.pairs)
    s.ctx = _ctx("server" if s.call == "serve" else "calls")
    if s.call == "squarefree":
        bounds = _bounds(case)
        s.content = _Results([b // 32 + 1 for _, b in bounds])
        s.factors = _Results([(d // m + 1) * ((b + 2 * d + 64) // 32 + 1) for d, b in bounds
                              for m in range(1, _MULT + 1)])
        s.nmult = np.zeros(len(s.pairs), dtype=np.int32)
        return s
    s.out = _Results(_words(case))
    if s.call == "batch":
        s.batch = s.ctx.batch(s.pairs)
    elif s.call == "serve":
        s.ctx.autotune(s.pairs)  # the server itself never tunes
    return s


def _ok(rc, ctx):
    if rc < 0:
        raise rs.RsError(rc, (rs.load().rs_last_error(ctx.h) or b"").decode())


def run(state):
    s, lib = state, rs.load()
    n = len(s.pairs)
    if s.call == "batch":
        s.batch.upload()
        s.batch.run()
        _ok(lib.rs_batch_results(s.batch.h, s.out.structs, None), s.ctx)
    elif s.call == "once":
        _ok(lib.rs_resultant_batch(s.ctx.h, n, s.f, s.g, s.out.structs, None), s.ctx)
    elif s.call == "serve":
        tickets = [ctypes.c_uint64() for _ in range(n)]
        for i, t in enumerate(tickets):
            _ok(lib.rs_server_submit(s.ctx.h, ctypes.byref(s.f[i]), ctypes.byref(s.g[i]), ctypes.byref(t)), s.ctx)
        for i, t in enumerate(tickets):
            _ok(lib.rs_server_wait(s.ctx.h, t.value, ctypes.byref(s.out.structs[i]), None, -1), s.ctx)
    else:
        nm = s.nmult.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))
        _ok(lib.rs_squarefree_batch(s.ctx.h, n, s.f, s.g, _MULT, s.content.structs, s.factors.structs, nm, None), s.ctx)
        return {"content": s.content.outputs(), "factors": s.factors.outputs(), "nmult": s.nmult.copy()}
    return s.out.outputs()


def work(case):
    """Bytes: coefficients in, result limbs out.  Flops: two per modular
    product of the images (half of an evaluation each, one remainder sequence)
    over the primes and points that the result's size asks for."""
    nbytes = flops = 0.0
    for pair, (d, bits) in zip(_shapes(case), _bounds(case)):
        a, b = pair
        images = (bits / 31.0 + 1) * (d + 1)
        nbytes += sum(4 * (s[0] + 1) * (s[1] + 1) * -(-s[3] // 32) for s in pair) + 4 * (d + 1) * (bits // 32 + 1)
        flops += 2 * images * ((a[4] + b[4]) / 2 + a[1] * b[1])
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------- exact values


def _determinant(m):
    """Fraction-free elimination over the integers."""
    m, sign, prev = [r[:] for r in m], 1, 1
    for k in range(len(m) - 1):
        if m[k][k] == 0:
            swap = next((r for r in range(k + 1, len(m)) if m[r][k]), None)
            if swap is None:
                return 0
            m[k], m[swap], sign = m[swap], m[k], -sign
        for r in range(k + 1, len(m)):
            for c in range(k + 1, len(m)):
                m[r][c] = (m[r][c] * m[k][k] - m[r][k] * m[k][c]) // prev
        prev = m[k][k]
    return sign * m[-1][-1]


def _integers(poly):
    c = poly.coeffs.astype("<u4")
    return [[int.from_bytes(v.tobytes(), "little", signed=True) for v in row] for row in c]


def _resultant(f, g, D):
    """Coefficients of Res_y(f, g): Sylvester determinants at 0..D, Newton's
    divided differences on them, expanded."""
    F, G, m, n = _integers(f), _integers(g), f.deg_y, g.deg_y
    values = []
    for x in range(D + 1):
        fx = [sum(F[i][j] * x ** i for i in range(len(F))) for j in range(m, -1, -1)]
        gx = [sum(G[i][j] * x ** i for i in range(len(G))) for j in range(n, -1, -1)]
        values.append(_determinant([[0] * r + fx + [0] * (n - 1 - r) for r in range(n)] +
                                   [[0] * r + gx + [0] * (m - 1 - r) for r in range(m)]))
    diffs, out, basis, fact = values, [0] * (D + 1), [1], 1
    num, common = [], math.factorial(D)
    for k in range(D + 1):  # k-th forward difference over k!
        num.append(diffs[0] * (common // fact))
        diffs = [b - a for a, b in zip(diffs, diffs[1:])]
        fact *= k + 1
    for k in range(D + 1):
        for i, c in enumerate(basis):
            out[i] += num[k] * c
        basis = [(basis[i - 1] if i else 0) - (k * basis[i] if i < len(basis) else 0) for i in range(len(basis) + 1)]
    out = [c // common for c in out]
    while out and out[-1] == 0:
        out.pop()
    return out


def exact(case, seed):
    if case["call"] == "squarefree" or case["kind"] != "dense" or case["n"] * case["deg"] ** 5 > 80000:
        return None
    pairs = _pairs(case, seed)
    out = _Results(_words(case))
    at = 0
    for i, ((f, g), (D, _)) in enumerate(zip(pairs, _bounds(case))):
        r = _resultant(f, g, D)
        limbs = max([1] + [-(-(max(c, ~c).bit_length() + 1) // 32) for c in r])
        raw = b"".join(c.to_bytes(4 * limbs, "little", signed=True) for c in r)
        out.buf[at: at + len(r) * limbs] = np.frombuffer(raw, dtype="<u4")
        out.raw["deg"][i], out.raw["limbs"][i] = len(r) - 1, limbs
        at += int(out.raw["capacity_words"][i])
    return out.outputs()
