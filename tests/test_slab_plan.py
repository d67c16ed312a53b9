"""The slabs of a digit product that does not fit its scratch whole
(csrc/oz_gemm.cu), worked out on the host: no GPU.

A product needs room for one tile of 128 lane rows and one of 80 column rows
(an embedded operand counts two rows for each of its own), and must run with
that and with anything above it."""
import itertools

import pytest

from paper_2304_05505_gb300 import thc

SHAPES = [
    # M, N, K, batch, real
    (163, 112, 432, 1, 0),
    (400, 1080, 110592, 1, 0),      # the sum over a 48^3 grid of the orbital gradient
    (170, 1080, 115200, 1, 0),
    (200, 540, 114000, 1, 0),
    (1200, 60, 1200, 64, 0),
    (60, 1200, 300, 7, 0),
    (41, 4000, 97, 3, 0),
    (129, 81, 33, 2, 0),
    (1, 1, 1, 1, 0),
    (3, 500, 20, 5, 0),
    (600, 4096, 600, 1, 1),
    (81, 129, 1000, 1, 1),
    (79, 127, 5, 1, 1),
]


def _least(shape):
    """The smallest scratch (to a byte) that the product runs with."""
    lo, hi = 0, 1 << 40
    assert thc.thc_debug_slab_plan(*shape, hi) is not None
    while lo + 1 < hi:
        mid = (lo + hi) // 2
        if thc.thc_debug_slab_plan(*shape, mid) is None:
            lo = mid
        else:
            hi = mid
    return hi


@pytest.mark.parametrize("shape", SHAPES)
def test_more_scratch_never_fails(shape):
    """From the least scratch upward every amount has a plan; its slabs are
    whole tiles or the whole operand, and they grow with the scratch."""
    M, N, K, batch, real = shape
    least = _least(shape)
    whole = 1 << 40
    # one tile of each side in eight digits, magnitudes and exponents, with some room for bookkeeping
    kr = K if real else 2 * K
    tile = (128 + 80) * (18 * (kr + 8) + 8)
    assert least <= tile + 16384
    before = 0
    for f in itertools.chain((1.0 + i / 40 for i in range(160)), (1.3 ** i for i in range(6, 60))):
        bytes_ = min(whole, int(least * f))
        p = thc.thc_debug_slab_plan(*shape, bytes_)
        assert p is not None, (shape, f)
        bs, rows, cols = p
        assert 1 <= bs <= batch and 1 <= rows <= M and 1 <= cols <= N
        assert rows == M or rows % 40 == 0 or rows % 64 == 0
        assert cols == N or cols % 40 == 0 or cols % 64 == 0
        assert bs == 1 or (rows == M and cols == N)
        before = max(before, bs * rows * cols)
    assert before == batch * M * N      # at the end the whole product in one slab


def test_scratch_below_one_tile_is_refused():
    assert thc.thc_debug_slab_plan(300, 300, 100, 1, 0, 2048) is None
