"""The launch shape of the direct interpolation (rs_g2_shape, called in the
library): over point-pair counts and task counts, its shared memory holds the
inputs, b and the partial sums the kernel lays out there and stays within the
kernel's limit, and the shapes that only few sizes take are the ones the GPU
tests of those sizes mean."""
import ctypes
import os

import pytest

from paper_1010_1386_gb300 import rs

PAD, MAX_BYTES, SMS = 8, 4 * (8192 + 16) * 4, 152


class Shape(ctypes.Structure):
    _fields_ = [("threads", ctypes.c_int), ("seg", ctypes.c_int), ("halves", ctypes.c_int), ("split", ctypes.c_int),
                ("smem", ctypes.c_size_t)]


@pytest.fixture(scope="module")
def shape():
    if not os.path.exists(rs.LIB_PATH):
        from paper_1010_1386_gb300 import build
        build.build()
    fn = getattr(rs.load(), "_Z11rs_g2_shapeiliPK9RsG2Shape")
    fn.restype, fn.argtypes = Shape, [ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.POINTER(Shape)]
    return fn


def check(s, M):
    assert s.threads % 32 == 0 and 32 <= s.threads <= 512
    assert s.split in (0, 1) and s.halves in ((1,) if s.split else (1, 2)) and s.seg >= 1
    inputs = 1 if s.split else 2  # halves a block holds; s.halves of them are convolved at once
    words = (inputs + 1) * (M + 2 * PAD) + max(s.seg * s.halves, 1) * M  # the inverses take the sums' first M words
    assert words * 4 <= s.smem <= MAX_BYTES


MS = sorted(set(range(1, 130)) | {int(1.09 ** k) for k in range(57, 105)} | set(range(6480, 6600)) | set(range(8000, 8193)))


@pytest.mark.parametrize("tasks", [1, 69, 152, 304, 305, 341, 4000, 100000])
def test_shared_memory(shape, tasks):
    for M in MS:
        if M > 8192:
            continue
        s = shape(M, tasks, SMS, None)
        check(s, M)
        for m in (M, (M + 3) // 2, M // 2 + 1):  # smaller counts of the octave in the same launch
            t = shape(m, tasks, SMS, ctypes.byref(s))
            if t.halves == s.halves:
                assert (t.threads, t.split) == (s.threads, s.split)
                check(t, m)


def test_shapes_of_few_sizes(shape):
    """The halves in turn, above 6,556 pairs with more than two tasks per SM;
    both at once at the shared-memory limit; few tasks in clusters."""
    for M in (6557, 6561, 8192):
        s = shape(M, 341, SMS, None)
        assert (s.halves, s.split, s.seg) == (1, 0, 1)
    s = shape(6497, 341, SMS, None)
    assert (s.halves, s.split, s.seg) == (2, 0, 1) and s.smem > MAX_BYTES - 4096
    for M in (6497, 8192):
        assert shape(M, 20, SMS, None).split == 1
