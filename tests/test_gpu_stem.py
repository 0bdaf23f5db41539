"""The fused stem (cg_stem_forward) against the oracle's 7x7 stride-2 convolution of the image."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1805_12549_b200 import synth
from tests import cases as K

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (2, 5, 5), (1, 7, 10), (3, 33, 29), (1, 12, 300), (2, 224, 224), (40, 30, 34)]


def _stem(n, h, w, x, wt, bn, delta):
    import torch
    from paper_1805_12549_b200 import binding as B
    dev = lambda a: torch.from_numpy(synth.bf16_bits(np.ascontiguousarray(a, np.float32)).view(np.int16)).cuda().view(torch.bfloat16)  # noqa: E731
    ho, wo = (h - 1) // 2 + 1, (w - 1) // 2 + 1
    conv = B.GatedConv(n, ho, wo, 192, 64, k=1, pad=0, groups=1)
    wp = np.zeros((64, 192), np.float32)
    wp[:, :147] = wt.reshape(64, -1)
    params = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in bn.items() if v is not None}
    guard = torch.full((n * ho * wo * 64 + 4096,), 7.0, dtype=torch.bfloat16, device="cuda")
    y = guard[2048:-2048].view(n, ho, wo, 64)
    ws = torch.empty(B.cg_stem_workspace_bytes(), dtype=torch.uint8, device="cuda")
    xd, wd, dd = dev(x), dev(wp), torch.from_numpy(delta).cuda()
    B.cg_stem_forward(conv.handle, xd, wd, B.make_bn(params), dd, y, ws)
    st = conv.stats()
    assert bool((guard[:2048] == 7).all()) and bool((guard[-2048:] == 7).all())
    out = y.float().cpu().numpy()
    conv.close()
    return out, st


@pytest.mark.parametrize("n,h,w", SIZES)
@pytest.mark.parametrize("dv", [K.INF, 0.0])
def test_stem_matches_the_convolution(n, h, w, dv):
    key = ("stem", n, h, w)
    x = synth.bf16_round(synth.rng(key, "x").standard_normal((n, h, w, 3), dtype=np.float32))
    wt, _ = synth.kaiming_weights(key, 64, 7, 7, 3, 1)
    wt = synth.bf16_round(wt)
    bn = synth.bn_params(key, 64)
    delta = np.full(64, dv, np.float32)
    s = O.Shape(n, h, w, 3, 64, 7, 7, 2, 3, 1, 1e-5, 1)
    ref = O.gated_conv(s, x, wt, np.zeros((64, 7, 7, 0), np.float32), bn, delta, None, out_bf16=True)
    y, st = _stem(n, h, w, x, wt, bn, delta)
    c = K.Case("stem", s, "bf16", x, wt, None, bn, delta)
    near = np.abs((ref.p.reshape(-1, 64) - bn["mean_base"]) / np.sqrt(bn["var_base"] + 1e-5) - delta) < K.NEAR_TIE
    err = np.abs(y.astype(np.float64) - ref.y) - K.BF16_ATOL - K.BF16_RTOL * np.abs(ref.y)
    assert (err[~near.reshape(ref.y.shape)] <= 0).all()
    assert st.calls == 1 and st.device_status == 0 and abs(st.active - ref.active) <= near.sum()
    assert c.s.m * 64 == st.outputs
    # blocks of a pixel and 32 channels, as the 1x1 layer over the patch matrix counts them
    words = ref.mask.reshape(-1, 2)
    assert st.rows_total == words.size and abs(st.rows_active - np.count_nonzero(words)) <= near.sum()


def test_pixels_that_are_not_finite_stay_where_they_are_used():
    n, h, w = 1, 20, 22
    key = ("steminf",)
    x = synth.bf16_round(synth.rng(key, "x").standard_normal((n, h, w, 3), dtype=np.float32))
    x[0, 9, 11, 1] = np.inf
    wt, _ = synth.kaiming_weights(key, 64, 7, 7, 3, 1)
    wt = synth.bf16_round(wt)
    bn, delta = synth.bn_params(key, 64), np.full(64, K.INF, np.float32)
    s = O.Shape(n, h, w, 3, 64, 7, 7, 2, 3, 1, 1e-5, 1)
    ref = O.gated_conv(s, x, wt, np.zeros((64, 7, 7, 0), np.float32), bn, delta, None, out_bf16=True)
    y, _ = _stem(n, h, w, x, wt, bn, delta)
    finite = np.isfinite(ref.p).all(-1)
    assert finite.sum() == finite.size - 16                       # rows 3-6 and columns 4-7 of the output use the pixel
    ok = np.abs(y.astype(np.float64) - ref.y) <= K.BF16_ATOL + K.BF16_RTOL * np.abs(ref.y)
    assert ok[finite].all()


@pytest.mark.parametrize("algo", [0, 1], ids=["auto", "direct"])
def test_a_pass_without_hooks_matches_the_recorded_one(algo):
    """forward() takes the fused stem where the stem layer runs on tensor cores, the patch matrix elsewhere."""
    import torch
    from paper_1805_12549_b200 import resnet18 as R
    net = R.CgResNet18(image=33, classes=20, algo=algo)
    net.set_density(1.0)                       # every gate open: two orders of summation agree
    x = R.synthetic_images("stemnet", 2, 33)
    inst = net.instance(2)
    a = inst.forward(x).float().clone()
    b = inst.forward(x, record=[]).float().clone()
    torch.cuda.synchronize()
    assert torch.isfinite(a).all() and float((a - b).norm()) <= (3e-2 if algo == 0 else 0.0) * float(b.norm())
    per, _ = inst.stats()
    assert per["stem"].calls == 2 and all(st.device_status == 0 for st in per.values())
    inst.close()


def test_a_short_batch_gives_its_own_logits_and_other_extents_are_refused():
    import torch
    from paper_1805_12549_b200 import binding as B, resnet18 as R
    net = R.CgResNet18(image=33, classes=20)
    net.set_density(1.0)
    x = R.synthetic_images("stemshort", 4, 33)
    inst = net.instance(3)
    full = inst.forward(x[:3]).clone()
    stem = inst.out["stem"].clone()
    for k in (1, 2):
        inst.out["stem"].fill_(3.0)
        assert torch.equal(inst.forward(x[:k].clone())[:k], full[:k])
        assert torch.equal(inst.out["stem"][:k], stem[:k]) and bool((inst.out["stem"][k:] == 3).all())
    for bad in (x, torch.cat([x, x], -1)[:3, ..., :4].contiguous(), x[:3, ..., :2].contiguous(), x[:3, :31].contiguous()):
        with pytest.raises(B.CgError):
            inst.forward(bad)
    inst.close()


@pytest.mark.parametrize("algo", [0, 1], ids=["auto", "direct"])
def test_events_and_records_are_those_of_a_plain_pass(algo):
    import torch
    from paper_1805_12549_b200 import resnet18 as R
    net = R.CgResNet18(image=33, classes=20, algo=algo)
    net.set_density(1.0)
    x = R.synthetic_images("stemhooks", 2, 33)
    inst = net.instance(2)
    plain = inst.forward(x).clone()
    stem = inst.out["stem"].clone()
    events, record = [], []
    assert torch.equal(inst.forward(x, events=events), plain)
    assert torch.equal(inst.forward(x, record=record), plain)
    torch.cuda.synchronize()
    names = [name for name, _, _ in events]
    assert names.count("stem") == 1 and ("stem.im2col" in names) == (algo == 1)
    # one kernel per operator, the fused stem two
    assert len(names) == inst.launches_per_forward() - (algo == 0)
    spec, patches, _, y, _ = record[0]
    assert spec.name == "stem" and patches.shape[-1] == spec.c_in and torch.equal(y, stem)
    assert len(record) == len(net.specs)
    inst.close()


POOL_SIZES = [(1, 2, 2), (3, 5, 6), (1, 7, 10), (5, 33, 30), (1, 12, 300), (2, 9, 224), (3, 18, 226), (13, 40, 112), (6, 224, 224)]


@pytest.mark.parametrize("n,h,w", POOL_SIZES)
@pytest.mark.parametrize("dv,relu", [(K.INF, True), (K.INF, False), (0.0, True)])
def test_stem_and_pooling_in_one_kernel(n, h, w, dv, relu):
    """Strips that end inside a group, a second column tile, odd output extents, several items per block: y against the
    oracle, the maxima against the pooling kernel over that y, bit by bit (with pixels that are not finite)."""
    import torch
    from paper_1805_12549_b200 import binding as B
    key = ("stempool", n, h, w)
    x = synth.bf16_round(synth.rng(key, "x").standard_normal((n, h, w, 3), dtype=np.float32))
    if dv == K.INF and h > 4:
        x[0, h // 2, w // 2, 1] = np.inf
        x[n - 1, h - 1, w - 1, 2] = np.nan
    wt, _ = synth.kaiming_weights(key, 64, 7, 7, 3, 1)
    wt = synth.bf16_round(wt)
    bn, delta = synth.bn_params(key, 64), np.full(64, dv, np.float32)
    ref = O.gated_conv(O.Shape(n, h, w, 3, 64, 7, 7, 2, 3, 1, 1e-5, int(relu)), x, wt, np.zeros((64, 7, 7, 0), np.float32), bn, delta,
                       None, out_bf16=True)
    dev = lambda a: torch.from_numpy(synth.bf16_bits(np.ascontiguousarray(a, np.float32)).view(np.int16)).cuda().view(torch.bfloat16)  # noqa: E731
    ho, wo = (h - 1) // 2 + 1, (w - 1) // 2 + 1
    hp, wp = (ho - 1) // 2 + 1, (wo - 1) // 2 + 1
    conv = B.GatedConv(n + 1, ho, wo, 192, 64, k=1, pad=0, groups=1, relu=relu)      # (a handle for more images)
    wflat = np.zeros((64, 192), np.float32)
    wflat[:, :147] = wt.reshape(64, -1)
    params = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in bn.items() if v is not None}
    guard = [torch.full((n * a * b * 64 + 4096,), 7.0, dtype=torch.bfloat16, device="cuda") for a, b in ((ho, wo), (hp, wp))]
    y, pooled = guard[0][2048:-2048].view(n, ho, wo, 64), guard[1][2048:-2048].view(n, hp, wp, 64)
    B.cg_stem_pool_forward(conv.handle, dev(x), dev(wflat), B.make_bn(params), torch.from_numpy(delta).cuda(), y, pooled)
    st = conv.stats()
    conv.close()
    assert all(bool((g[:2048] == 7).all()) and bool((g[-2048:] == 7).all()) for g in guard)
    with np.errstate(invalid="ignore"):
        near = np.abs((ref.p.reshape(-1, 64) - bn["mean_base"]) / np.sqrt(bn["var_base"] + 1e-5) - delta) < K.NEAR_TIE
    finite = np.isfinite(ref.p)
    out = y.float().cpu().numpy()
    with np.errstate(invalid="ignore"):
        err = np.abs(out.astype(np.float64) - ref.y) - K.BF16_ATOL - K.BF16_RTOL * np.abs(ref.y)
    assert (err[finite.reshape(ref.y.shape) & ~near.reshape(ref.y.shape)] <= 0).all()
    assert st.calls == 1 and st.device_status == 0 and abs(st.active - ref.active) <= near.sum()
    assert st.rows_total == (n * ho * wo) * 2 and abs(st.rows_active - np.count_nonzero(ref.mask)) <= near.sum()
    want = torch.empty_like(pooled)
    B.cg_maxpool_bf16(y.contiguous(), want, 3, 2, 1)
    assert torch.equal(pooled.view(torch.int16), want.view(torch.int16))


def test_a_network_of_a_large_batch_pools_in_the_stem():
    """The same logits and stem activations as the two kernels, with the operators and launches that a pass then has."""
    import torch
    from paper_1805_12549_b200 import binding as B, resnet18 as R
    assert B.cg_stem_pool_pays(8, 224, 224) and not B.cg_stem_pool_pays(1, 224, 224) and not B.cg_stem_pool_pays(500, 224, 223)
    net = R.CgResNet18(image=224, classes=20)
    net.set_density(1.0)
    x = R.synthetic_images("stempoolnet", 8, 224)
    inst = net.instance(8)
    assert inst.stem_pools
    a = inst.forward(x).clone()
    stem, pooled = inst.out["stem"].clone(), inst.pooled.clone()
    events, record = [], []
    assert torch.equal(inst.forward(x, events=events), a) and torch.equal(inst.forward(x, record=record), a)
    names = [name for name, _, _ in events]
    assert "maxpool" not in names and len(names) == inst.launches_per_forward()
    assert torch.equal(record[0][3], stem) and len(record) == len(net.specs)
    inst.stem_pools = False
    b = inst.forward(x)
    torch.cuda.synchronize()
    # (another order of fp32 sums: some outputs differ by a bf16 rounding)
    for u, v in ((inst.out["stem"], stem), (inst.pooled, pooled)):
        assert float((u.float() - v.float()).norm()) <= 1e-3 * float(v.float().norm())
    assert float((a.float() - b.float()).norm()) <= 3e-2 * float(b.float().norm())
    inst.close()
