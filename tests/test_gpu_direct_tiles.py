"""The tiled direct kernel against the oracle, bit for bit: channel counts around its tiles, ragged pixel tiles,
borders, strides, and a weight that is not finite beside the padding."""
import numpy as np
import pytest

from oracle import oracle as O
from tests import cases as K

pytestmark = pytest.mark.gpu

SHAPES = [
    (O.Shape(2, 8, 8, 16, 16, groups=4), "one block of 16 channels"),
    (O.Shape(1, 3, 5, 16, 12, groups=2), "c_out = 12"),
    (O.Shape(3, 9, 7, 32, 32, groups=4), "32 channels"),
    (O.Shape(2, 6, 6, 48, 40, groups=4), "c_out = 40"),
    (O.Shape(1, 5, 4, 64, 100, groups=4), "two channel blocks, the second ragged"),
    (O.Shape(16, 20, 21, 16, 16, groups=4), "100 thousand outputs"),
    (O.Shape(40, 20, 21, 16, 16, groups=4), "two pixels per thread, 16 channels"),
    (O.Shape(40, 15, 16, 16, 32, groups=4), "two pixels per thread, 32 channels"),
    (O.Shape(64, 20, 16, 8, 24, groups=2), "two pixels per thread, 24 channels"),
    (O.Shape(100, 20, 16, 8, 24, groups=2), "four pixels per thread, 32 channels"),
    (O.Shape(40, 16, 15, 8, 64, groups=2), "two pixels per thread, 64 channels"),
    (O.Shape(70, 18, 16, 8, 64, groups=2), "four pixels per thread, 64 channels"),
    (O.Shape(2, 11, 9, 16, 16, 5, 5, 2, 2, groups=4), "5x5, stride 2"),
    (O.Shape(2, 7, 7, 16, 16, 1, 1, 1, 0, groups=1), "1x1, no conditional path"),
    (O.Shape(3, 1, 1, 16, 40, groups=4), "one pixel: one tap of nine"),
    (O.Shape(2, 1, 4, 64, 16, groups=2), "one row: three taps of nine"),
    (O.Shape(2, 2, 3, 16, 16, 7, 7, 1, 3, groups=4), "15 taps of 49"),
    (O.Shape(1, 3, 1, 16, 16, 5, 5, 2, 2, groups=2), "stride 2, taps from the first on"),
    (O.Shape(1, 2, 9, 16, 16, 3, 3, 4, 2, groups=2), "stride 4, padding 2"),
    (O.Shape(2, 1, 1, 16, 16, 3, 3, 20, 5, groups=2), "padding only"),
    (O.Shape(1500, 1, 4, 8, 64, groups=2), "one row, two pixels per thread"),
    (O.Shape(4000, 4, 1, 8, 64, groups=2), "one column, four pixels per thread"),
]


@pytest.mark.parametrize("s,why", SHAPES, ids=[w for _, w in SHAPES])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_bit_exact(s, why, dtype):
    import torch
    from paper_1805_12549_b200 import binding as B
    c = K.make_float_case("tile", s, dtype, density=0.4, residual=s.n % 2 == 0, smooth=False)
    ref = K.run_oracle(c)
    g = K.GpuCase(c, algo=1)
    y, mask, st = g.run()
    K.compare(c, ref, y, mask, st, exact=True)
    p = torch.empty((s.m, s.c_out), dtype=torch.float32, device="cuda")
    B.cg_conv_partial_sums(g.conv.handle, g.x, g.wb, p)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(p.cpu().numpy().reshape(ref.p.shape), ref.p)
    g.close()


def test_taps_in_the_padding_are_left_out():
    """An infinite weight times the zero padding would be NaN: only outputs that really use the tap see it."""
    s = O.Shape(1, 6, 6, 16, 16, groups=4)
    c = K.make_float_case("tileinf", s, "f32", density=0.5, smooth=False)
    c.wb = c.wb.copy()
    c.wb[3, 0, 0, 1] = np.inf                    # the upper left tap: outputs of the first row and column do not use it
    ref = K.run_oracle(c)
    assert np.isfinite(ref.p[0, 0, :, 3]).all() and not np.isfinite(ref.p[0, 1:, 1:, 3]).any()
    g = K.GpuCase(c, algo=1)
    y, mask, _ = g.run()
    np.testing.assert_array_equal(mask, ref.mask)
    np.testing.assert_array_equal(np.isfinite(y), np.isfinite(ref.y))
    g.close()


SIZES_OF_PRODUCTS = [(O.Shape(2, 8, 8, 16, 16, groups=2), "one channel per thread"),
                     (O.Shape(40, 15, 16, 16, 32, groups=2), "two pixels per thread"),
                     (O.Shape(64, 20, 16, 8, 64, groups=2), "four pixels per thread")]


@pytest.mark.parametrize("s,why", SIZES_OF_PRODUCTS, ids=[w for _, w in SIZES_OF_PRODUCTS])
def test_bf16_products_outside_the_normal_range_are_rounded_by_themselves(s, why):
    """Products below 2^-126 round to multiples of 2^-149 and products from 2^128 on are infinite before they are added:
    a fused multiply-add would keep what the separate multiplication of the definition loses."""
    c = K.make_float_case("tiny", s, "bf16", density=0.5, smooth=False)
    c.x, c.wb, c.wc = (np.ldexp(a, -68).astype(np.float32) for a in (c.x, c.wb, c.wc))
    c.x[0, 0, 0, :2] = np.float32(2.0) ** 64     # P = -2^127 + 2^128: infinite by itself
    c.wb[5] = 0.0
    c.wb[5, 1, 1, :2] = -np.float32(2.0) ** 63, np.float32(2.0) ** 64
    ref = K.run_oracle(c)
    assert np.isinf(ref.p[0, 0, 0, 5])
    g = K.GpuCase(c, algo=1)
    y, mask, st = g.run()
    K.compare(c, ref, y, mask, st, exact=True)
    import torch
    from paper_1805_12549_b200 import binding as B
    p = torch.empty((s.m, s.c_out), dtype=torch.float32, device="cuda")
    B.cg_conv_partial_sums(g.conv.handle, g.x, g.wb, p)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(p.cpu().numpy().reshape(ref.p.shape), ref.p)
    g.close()
