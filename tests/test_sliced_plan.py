"""The plan of a sliced FP64 product (host code; sizes only, no GPU)."""
import ctypes

import pytest

from paper_2407_18947_gb300 import _lib


class Plan(ctypes.Structure):
    _fields_ = [("swap", ctypes.c_bool), ("nt", ctypes.c_int), ("seg", ctypes.c_int),
                ("nseg", ctypes.c_int), ("spc", ctypes.c_int), ("nsplit", ctypes.c_int),
                ("cost", ctypes.c_double)]


def _plan(M, N, K):
    f = _lib.load()._ZN5rtcc37oz_planExxx  # rtcc3::oz_plan(long long, long long, long long)
    f.restype, f.argtypes = Plan, [ctypes.c_longlong] * 3
    return f(M, N, K)


# the triples' products over (o, v): build, back-contractions, densities, cotangents
SHAPES = [(o, v) for o, v in ((3, 8), (5, 19), (7, 23), (9, 31), (10, 38), (11, 41), (15, 57), (20, 76),
                              (2, 97), (25, 12))]


@pytest.mark.parametrize("o,v", SHAPES)
def test_scratch_is_one_sum_per_output_or_304_tiles(o, v):
    """Not one per segment of 128 terms: that was v / 128 of a triples tensor."""
    for M, N, K in ((o * o * v, o * v * v, o + v), (v, v, o**3 * v * v), (o, o, o * o * v**3),
                    (o * o * v, v, o * v * v), (o * v * v, o, o * o * v), (o * o * v * v, 1, o * v),
                    (o * v * v, v, o * o * v), (o, o * o * v**3, o), (v, o**3 * v * v, v),
                    ((o + v)**2, (o + v)**2, 3 * (o + v))):
        p = _plan(M, N, K)
        assert p.nt in (16, 32, 48, 64) and 0 < p.seg <= 128 and p.seg % 8 == 0
        assert (p.nseg - 1) * p.seg < K <= p.nseg * p.seg
        assert (p.nsplit - 1) * p.spc < p.nseg <= p.nsplit * p.spc  # every CTA has a segment
        assert p.nsplit * M * N <= max(M * N, 304 * 128 * p.nt // 2)
        if p.nsplit > 1:
            rows = N if p.swap else M
            assert (rows + 127) // 128 <= 65535  # the grid's y axis
