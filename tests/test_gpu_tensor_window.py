"""The window kernel (CG_ALGO_AUTO, tc4_conv.cu) against the oracle: tile edges, ragged last tiles, every
weight layout, the K loop shared by a cluster, int8, stride 2, residual, the two-sided gate."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1805_12549_b200 import binding as B
from tests import cases as K

pytestmark = pytest.mark.gpu
WINDOW = 4


def _run(c, **kw):
    ref = K.run_oracle(c)
    g = K.GpuCase(c, algo=0, **kw)
    assert g.conv.kernel_id == WINDOW, g.conv.plan
    print(g.conv.plan)
    y, mask, st = g.run()
    exempt = K.compare(c, ref, y, mask, st)
    assert st.tiles_skipped == 0 and st.rows_total == c.s.m * c.s.words
    g.close()
    return ref, st, exempt


SHAPES = [
    (O.Shape(1, 7, 7, 512, 512, groups=4), "one image: K loop over eight CTAs"),
    (O.Shape(1, 14, 14, 256, 256, groups=4), "K loop over a cluster, two pixel tiles"),
    (O.Shape(1, 28, 28, 128, 128, groups=4), "c_p = 32, K loop over a cluster"),
    (O.Shape(1, 1, 1, 128, 64, groups=4), "a single pixel"),
    (O.Shape(2, 3, 5, 64, 96, groups=2), "half-empty channel tile"),
    (O.Shape(3, 56, 56, 64, 64, groups=4), "c_p = 16"),
    (O.Shape(40, 28, 28, 128, 128, groups=4), "several jobs per pair, streamed weights"),
    (O.Shape(40, 56, 56, 64, 64, groups=4), "several jobs per pair, resident weights"),
    (O.Shape(150, 8, 8, 256, 256, groups=4), "images share padding rows"),
    (O.Shape(256, 4, 4, 512, 512, groups=4), "a third of the rows is padding"),
    (O.Shape(21, 13, 19, 256, 192, groups=2), "odd extents, c_out = 192"),
    (O.Shape(2, 9, 127, 64, 64, groups=4), "a patch of two loads"),
    (O.Shape(2, 4, 250, 64, 64, groups=4), "rows too wide for a patch: one patch per tap"),
    (O.Shape(5, 56, 56, 64, 128, stride=2, groups=4), "stride 2, c_p = 16"),
    (O.Shape(20, 28, 28, 128, 256, stride=2, groups=4), "stride 2, c_p = 32, pairs"),
    (O.Shape(3, 15, 9, 64, 64, stride=2, groups=4), "stride 2, odd extents"),
    (O.Shape(1, 14, 14, 256, 512, stride=2, groups=4), "stride 2, K loop over a cluster"),
    (O.Shape(4, 1, 9, 64, 64, stride=2, groups=2), "stride 2, one row"),
    (O.Shape(2, 17, 23, 128, 64, stride=3, groups=4), "stride 3"),
    (O.Shape(5, 7, 1, 64, 128, groups=1), "one column, ungated"),
    (O.Shape(33, 12, 12, 512, 256, groups=2), "four base chunks, pairs"),
    (O.Shape(9, 10, 11, 320, 128, 1, 1, 1, 0, groups=1), "1x1, ungated, five chunks"),
    (O.Shape(70, 10, 11, 64, 256, 1, 1, 1, 0, groups=1), "1x1, one chunk, pairs"),
    (O.Shape(128, 1, 1, 512, 1024, 1, 1, 1, 0, groups=1), "a classifier"),
    (O.Shape(3, 9, 9, 64, 96, 1, 1, 1, 0, groups=1), "1x1, one chunk, two jobs"),
    (O.Shape(1, 7, 5, 192, 64, 1, 1, 1, 0, groups=1), "1x1, three chunks, part of a job"),
    (O.Shape(1, 17, 16, 256, 64, 1, 1, 1, 0, groups=1), "1x1, four chunks, K loop over a cluster"),
    (O.Shape(3, 10, 10, 512, 64, groups=8), "G = 8"),
    (O.Shape(70, 14, 14, 64, 128, 1, 1, 2, 0, groups=1), "1x1, stride 2, pairs"),
    (O.Shape(1, 13, 9, 256, 64, 1, 1, 2, 0, groups=1), "1x1, stride 2, odd extents, K loop over a cluster"),
    (O.Shape(40, 10, 11, 128, 96, 1, 1, 3, 0, groups=1), "1x1, stride 3"),
]


@pytest.mark.parametrize("s,why", SHAPES, ids=[w for _, w in SHAPES])
def test_parity(s, why):
    # (a single pixel's own statistics would put every gate on its threshold)
    c = K.make_float_case("win", s, "bf16", density=0.3, delta=0.0 if s.m == 1 else None)
    ref, st, exempt = _run(c)
    assert abs(st.density - ref.density) < 2e-3 + 2.0 / st.outputs
    assert st.executed_macs >= st.dense_macs


@pytest.mark.parametrize("s", [SHAPES[0][0], SHAPES[10][0]], ids=["cluster", "pairs"])
@pytest.mark.parametrize("how", ["residual", "band", "open", "shut"])
def test_options(s, how):
    c = K.make_float_case("winopt", s, "bf16", density=0.4, residual=how == "residual",
                          delta={"open": -K.INF, "shut": K.INF}.get(how))
    if how == "band":
        c.delta_high = (c.delta + np.float32(0.8)).astype(np.float32)
    _run(c)


@pytest.mark.parametrize("n", [1, 40], ids=["cluster", "pairs"])
def test_a_nan_stays_where_it_is_used(n):
    c = K.make_float_case("winnan", O.Shape(n, 12, 11, 128, 128, groups=4), "bf16", density=0.3)
    c.x[0, 5, 10, 3] = np.nan          # beside the right edge: the next row's left padding shares the position
    c.x[n - 1, 11, 0, 100] = np.nan    # the last row: the next image's upper padding
    _run(c)


INT8 = [
    (O.Shape(3, 28, 28, 128, 128, groups=4), "one K slice of base channels"),
    (O.Shape(40, 14, 14, 256, 256, groups=4), "two base slices, several jobs per pair"),
    (O.Shape(1, 7, 7, 512, 512, groups=4), "a whole base chunk, K loop over a cluster"),
    (O.Shape(4, 13, 6, 128, 64, groups=2), "c_out = 64"),
    (O.Shape(5, 28, 28, 128, 256, stride=2, groups=4), "stride 2"),
    (O.Shape(2, 9, 7, 256, 64, 1, 1, 1, 0, groups=1), "1x1, two chunks"),
]


@pytest.mark.parametrize("s,why", INT8, ids=[w for _, w in INT8])
def test_int8_is_exact(s, why):
    _run(K.make_int8_case("wini8", s, density=0.3))


@pytest.mark.parametrize("n", [2, 30], ids=["cluster", "pairs"])
def test_outputs_that_are_only_16_byte_aligned(n):
    import torch
    c = K.make_float_case("winal", O.Shape(n, 12, 12, 128, 128, groups=4), "bf16", density=0.3)
    g = K.GpuCase(c, algo=0)
    g.run()
    buf = torch.zeros(g.y.numel() + 64, dtype=torch.bfloat16, device="cuda")
    off = (-buf.data_ptr() % 32 + 16) // 2
    y1 = buf[off:off + g.y.numel()].view(g.y.shape)
    g.conv.forward(g.x, g.wb, g.wc, g.bn, g.delta, y1, g.mask, None)
    torch.cuda.synchronize()
    assert torch.equal(y1, g.y) and float(buf[:off].abs().sum()) == 0 and float(buf[off + g.y.numel():].abs().sum()) == 0
    g.close()


SHUT = [
    (O.Shape(40, 56, 56, 64, 64, groups=4), "one base slice, resident weights"),
    (O.Shape(40, 28, 28, 128, 128, groups=4), "two base slices"),
    (O.Shape(256, 4, 4, 512, 512, groups=4), "base chunks"),
    (O.Shape(70, 28, 28, 64, 128, stride=2, groups=4), "stride 2, one base slice"),
    (O.Shape(60, 28, 28, 128, 256, stride=2, groups=4), "stride 2, two base slices"),
    (O.Shape(21, 13, 19, 256, 192, groups=2), "half-empty channel tile"),
    (O.Shape(48, 7, 7, 512, 512, groups=8), "one job per pair"),
]


@pytest.mark.parametrize("s,why", SHUT, ids=[w for _, w in SHUT])
@pytest.mark.parametrize("how", ["all", "some", "residual", "band", "dense"])
def test_column_tiles_whose_gates_cannot_fire(s, why, how):
    c = K.make_float_case("winshut", s, "bf16", density=0.3, residual=how == "residual")
    if how == "some":
        c.delta[:(s.c_out + 1) // 2] = K.INF
        c.delta[-1] = np.nan                     # (fires nowhere either)
    else:
        c.delta[:] = K.INF
    if how == "band":
        c.delta_high = np.full(s.c_out, 2.0, np.float32)
    ref, st, _ = _run(c, cond_mode=1 if how == "dense" else 0)
    if how != "some":
        skips = how != "dense"
        assert st.active == 0 and (st.executed_macs < st.dense_macs) == skips and (st.tiles_total == 0) == skips


@pytest.mark.parametrize("s", [O.Shape(40, 28, 28, 128, 128, groups=4), O.Shape(60, 14, 14, 256, 256, groups=4),
                               O.Shape(40, 28, 28, 256, 128, stride=2, groups=4)],
                         ids=["one chunk", "two chunks", "stride 2"])
def test_int8_thresholds_beyond_every_sum(s):
    c = K.make_int8_case("winshut8", s, density=0.3)
    top = 9 * s.c_p * 128 * 128                  # (the largest sum there is)
    for thr, skips in ((top, False), (top + 1, True)):
        c.bn["q_gate_thr"] = np.full(s.c_out, thr, np.int32)
        _, st, _ = _run(c)
        assert (st.executed_macs < st.dense_macs) == skips


@pytest.mark.parametrize("s,residual", [(O.Shape(40, 20, 20, 128, 128, groups=4), False),
                                        (O.Shape(40, 20, 20, 128, 128, groups=4), True),
                                        (O.Shape(40, 20, 20, 128, 192, groups=2), False),
                                        (O.Shape(40, 20, 20, 128, 256, stride=2, groups=4), True)],
                         ids=["128 channels", "residual", "64 channels per tile", "stride 2"])
def test_an_infinite_sum_meets_an_infinite_threshold(s, residual):
    """A tie fires, at +inf too: those outputs are the full sum under its batch norm."""
    c = K.make_float_case("winshutinf", s, "bf16", density=0.3, residual=residual)
    c.delta[:] = K.INF
    c.x[1, 7, 19, 3] = np.inf                    # P = +-inf around it
    c.x[39, 19, 0, 5] = np.inf
    c.x[39, 18, 1, 77] = -np.inf                 # R = +-inf there: P + R is infinite or not a number
    c.x[2, 3, 4, 6] = np.nan
    ref = K.run_oracle(c)
    assert ref.active > 0 and np.isnan(ref.p).any()
    g = K.GpuCase(c, algo=0)
    assert g.conv.kernel_id == WINDOW
    for with_mask in (True, False):
        y, mask, st = g.run(with_mask=with_mask)
        if with_mask:
            np.testing.assert_array_equal(mask, ref.mask)
        assert st.executed_macs < st.dense_macs and st.active == ref.active
        fin = np.isfinite(ref.y)
        np.testing.assert_array_equal(y[~fin], ref.y[~fin])
        assert (np.abs(y[fin] - ref.y[fin]) <= K.BF16_ATOL + K.BF16_RTOL * np.abs(ref.y[fin])).all()
    g.close()


# K loops of pairs: packed weights and stride-2 windows, with the plan that the shape has to take.
K_LOOPS = [
    (O.Shape(40, 28, 28, 128, 128, groups=8), "one patch for all taps", "packed", "G = 8: one base slice"),
    (O.Shape(60, 13, 15, 128, 256, groups=4), "one patch for all taps", "packed", "odd extents, two column tiles"),
    (O.Shape(70, 28, 28, 64, 128, stride=2, groups=2), "four patches", "packed", "one chunk, two base slices"),
    (O.Shape(30, 28, 28, 128, 256, stride=2, groups=8), "four patches", "packed", "two chunks, one base slice"),
    (O.Shape(70, 30, 26, 64, 64, stride=2, groups=4), "four patches", "packed", "64 columns to a job"),
    (O.Shape(40, 14, 14, 256, 512, stride=2, groups=4), "four patches", "streamed", "a base chunk, streamed"),
    (O.Shape(150, 28, 28, 128, 64, stride=2, groups=2), "four patches", "resident", "a base chunk, resident"),
    (O.Shape(40, 28, 28, 128, 128, stride=2, groups=1), "four patches", "streamed", "ungated"),
    (O.Shape(600, 4, 4, 128, 256, stride=2, groups=4), "four patches", "packed", "four output pixels per image"),
    (O.Shape(3000, 2, 2, 128, 256, stride=2, groups=4), "one patch per tap", "streamed", "too much padding for a window"),
    (O.Shape(80, 13, 15, 128, 256, stride=2, groups=4), "one patch per tap", "streamed", "odd extents"),
    (O.Shape(60, 28, 28, 256, 256, stride=2, groups=8), "one patch per tap", "streamed", "too many chunks to pack"),
    (O.Shape(28, 28, 28, 128, 128, groups=4), "halves", "packed", "18 jobs in halves, packed"),
    (O.Shape(60, 14, 14, 128, 320, groups=4), "halves", "packed", "halves of a half-empty column tile"),
    (O.Shape(256, 4, 4, 512, 512, groups=4), "halves", "streamed", "7 jobs in halves, streamed"),
    (O.Shape(96, 14, 14, 256, 512, stride=2, groups=4), "halves", "streamed", "halves, stride 2"),
    (O.Shape(60, 28, 28, 128, 256, stride=2, groups=4), "halves", "packed", "halves, stride 2, packed"),
    (O.Shape(50, 14, 14, 256, 256, groups=8), "halves", "streamed", "halves, two base slices"),
    (O.Shape(110, 14, 14, 128, 128, 1, 1, 1, 0, groups=1), "halves", "", "halves, 1x1"),
]


@pytest.mark.parametrize("s,patch,weights,why", K_LOOPS, ids=[k[3] for k in K_LOOPS])
@pytest.mark.parametrize("how", ["density", "some shut", "all shut"])
def test_k_loops_of_pairs(s, patch, weights, why, how):
    c = K.make_float_case("winkloop", s, "bf16", density=0.3, calib_images=4)
    if how != "density":
        c.delta[:s.c_out if how == "all shut" else (s.c_out + 1) // 2] = K.INF
    ref, st, _ = _run(c)
    g = K.GpuCase(c, algo=0)
    plan = g.conv.plan
    g.close()
    assert patch in plan and (weights in plan or s.groups == 1), plan
    assert how != "all shut" or s.c_r == 0 or (st.active == 0 and st.executed_macs < st.dense_macs)


@pytest.mark.parametrize("s", [O.Shape(60, 28, 28, 128, 256, stride=2, groups=4), O.Shape(40, 28, 28, 256, 128, stride=2, groups=4),
                               O.Shape(40, 28, 28, 256, 128, stride=2, groups=8), O.Shape(40, 28, 28, 256, 128, stride=2, groups=2)],
                         ids=["one chunk", "two base slices", "one base slice", "a base chunk"])
def test_int8_stride_2_windows(s):
    _run(K.make_int8_case("wini8s2", s, density=0.3))


def test_new_inputs_and_new_weights_of_one_handle():
    """More pointers than a handle keeps tensor maps of, in an order in which the input, the weights or both are new."""
    import torch
    c = K.make_float_case("winmaps", O.Shape(28, 28, 28, 128, 128, groups=4), "bf16", density=0.3, calib_images=1)
    g = K.GpuCase(c, algo=0)
    assert "halves" in g.conv.plan
    xs = [g.x.roll(i, 0) for i in range(6)]
    weights = [(g.wb, g.wc), (g.wb.flip(0), g.wc.flip(0)), (g.wb, g.wc.flip(0))]
    order = [(i, j) for j in (0, 1, 2, 0) for i in range(6)] + [(i % 6, i % 3) for i in range(12)]
    first = {}
    for i, j in order:
        g.conv.forward(xs[i], *weights[j], g.bn, g.delta, g.y, g.mask)
        if (i, j) not in first:
            fresh = K.GpuCase(c, algo=0)
            fresh.conv.forward(xs[i], *weights[j], g.bn, g.delta, fresh.y, fresh.mask)
            first[i, j] = fresh.y.clone(), fresh.mask.clone()
            fresh.close()
        assert torch.equal(g.y, first[i, j][0]) and torch.equal(g.mask, first[i, j][1]), (i, j)
    g.close()


STRIDE_2 = [k for k in K_LOOPS if k[0].stride == 2 and k[0].h > 4]


@pytest.mark.parametrize("s", [k[0] for k in STRIDE_2], ids=[k[3] for k in STRIDE_2])
def test_a_stride_2_layer_sums_as_every_other_pixel_of_the_dense_one(s):
    """The same taps in the same order, whatever copies bring the pixels: bit for bit, gates included."""
    import torch
    c = K.make_float_case("winorder", s, "bf16", density=0.3, calib_images=4)
    g = K.GpuCase(c, algo=0)
    y2, mask2, _ = g.run()
    dense = B.GatedConv(s.n, s.h, s.w, s.c_in, s.c_out, groups=s.groups, dtype=B.CG_BF16)
    assert dense.kernel_id == WINDOW and "over 1 CTA(s)" in dense.plan and "over 1 CTA(s)" in g.conv.plan
    y1, mask1 = dense.alloc_outputs()
    dense.forward(g.x, g.wb, g.wc, g.bn, g.delta, y1, mask1)
    torch.cuda.synchronize()
    y1 = y1[:, ::2, ::2].float().cpu().numpy()
    mask1 = mask1.view(s.n, s.h, s.w, s.words)[:, ::2, ::2].cpu().numpy().view(np.uint32)
    np.testing.assert_array_equal(mask2, mask1.reshape(-1, s.words))
    np.testing.assert_array_equal(y2, y1)
    dense.close()
    g.close()


# int8 jobs of 128 columns, with gates that fire: what the plan says of patches, weights and the last round.
INT8_K_LOOPS = [
    (O.Shape(60, 14, 14, 256, 256, groups=4), "one patch for all taps", "packed", True, "two base slices"),
    (O.Shape(48, 14, 14, 256, 256, groups=8), "one patch for all taps", "packed", True, "one base slice"),
    (O.Shape(60, 14, 14, 256, 256, groups=2), "one patch for all taps", "resident", True, "a base chunk"),
    (O.Shape(64, 7, 7, 512, 512, groups=4), "one patch for all taps", "streamed", False, "a base chunk, streamed"),
    (O.Shape(96, 14, 14, 256, 512, stride=2, groups=4), "four patches", "packed", True, "stride 2, two base slices"),
    (O.Shape(96, 14, 14, 256, 512, stride=2, groups=8), "four patches", "packed", True, "stride 2, one base slice"),
    (O.Shape(96, 14, 14, 256, 512, stride=2, groups=2), "four patches", "streamed", True, "stride 2, a base chunk"),
    (O.Shape(40, 28, 28, 256, 512, stride=2, groups=4), "four patches", "packed", False, "stride 2, whole rounds"),
    (O.Shape(96, 14, 14, 512, 512, stride=2, groups=4), "four patches", "streamed", True, "stride 2, streamed"),
]


@pytest.mark.parametrize("s,patch,weights,halves,why", INT8_K_LOOPS, ids=[k[4] for k in INT8_K_LOOPS])
def test_int8_jobs_of_128_columns(s, patch, weights, halves, why):
    c = K.make_int8_case("wini8k", s, density=0.3)
    g = K.GpuCase(c, algo=0)
    plan = g.conv.plan
    g.close()
    assert "channel tiles of 128" in plan and patch in plan and weights in plan and ("halves" in plan) == halves, plan
    _, st, _ = _run(c)
    assert 0.2 < st.active / st.outputs < 0.4


# Layers of few jobs, on either side of each line between K loops shared by a cluster and CTA pairs.
FEW_JOBS = [
    (O.Shape(2, 5, 5, 64, 64, groups=4), False, 4, "36 MMAs, one job"),
    (O.Shape(1, 14, 14, 64, 64, groups=4), False, 1, "36 MMAs, two pixel tiles"),
    (O.Shape(1, 28, 28, 64, 64, groups=4), True, 4, "36 MMAs, residual, 7 jobs"),
    (O.Shape(1, 56, 56, 64, 64, groups=4), True, 1, "36 MMAs, residual, 28 jobs"),
    (O.Shape(3, 14, 14, 128, 128, groups=4), False, 8, "72 MMAs, 12 jobs"),
    (O.Shape(1, 28, 28, 128, 128, groups=4), False, 1, "72 MMAs, 16 jobs"),
    (O.Shape(1, 28, 28, 128, 128, groups=4), True, 4, "72 MMAs, residual, 14 jobs"),
    (O.Shape(2, 28, 28, 128, 128, groups=4), True, 1, "72 MMAs, residual, 28 jobs"),
    (O.Shape(1, 28, 28, 128, 256, stride=2, groups=4), False, 1, "72 MMAs, stride 2"),
    (O.Shape(3, 14, 14, 256, 256, groups=4), False, 4, "144 MMAs, room for four CTAs a job"),
    (O.Shape(5, 14, 14, 256, 256, groups=4), False, 1, "144 MMAs, room for two"),
    (O.Shape(128, 1, 1, 512, 1024, 1, 1, 1, 0, groups=1), False, 2, "a classifier: 32 MMAs, one pixel tile, 16 jobs"),
    (O.Shape(1, 10, 10, 64, 1024, groups=4), False, 4, "36 MMAs, one pixel tile, 16 jobs"),
]


@pytest.mark.parametrize("s,residual,ctas,why", FEW_JOBS, ids=[f[3] for f in FEW_JOBS])
def test_layers_of_few_jobs(s, residual, ctas, why):
    c = K.make_float_case("winfew", s, "bf16", density=0.3, residual=residual)
    _run(c)
    g = K.GpuCase(c, algo=0)
    plan = g.conv.plan
    g.close()
    assert f"over {ctas} CTA(s)" in plan, plan
