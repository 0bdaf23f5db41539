"""CPU-side checks of the C-ABI library: it loads without a GPU, exports every symbol the
header declares, and rejects bad descriptions before touching CUDA."""
import ctypes as C
import os
import re

import pytest

from paper_1805_12549_b200 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols(header="cgconv.h"):
    text = open(os.path.join(ROOT, "include", header)).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(cg_[a-z0-9_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    lib = B.lib()
    names = _declared_symbols()
    assert set(B.EXPORTS) <= set(names)
    assert len(names) >= 11
    for n in names:
        assert hasattr(lib, n), n


def test_library_exports_the_network_operators():
    lib = B.lib()
    names = _declared_symbols("cgnet.h")
    assert set(names) == set(B.NET_EXPORTS)
    for n in names:
        assert hasattr(lib, n), n


def test_network_operators_reject_bad_arguments_before_any_launch():
    lib = B.lib()
    buf = (C.c_uint8 * 4096)()
    base = C.addressof(buf)
    p = C.c_void_p((base + 15) & ~15)
    odd = C.c_void_p(p.value + 2)
    INVALID, ALIGN = 1, 3
    assert lib.cg_im2col_bf16(None, p, 1, 8, 8, 3, 7, 2, 3, 152, None) == INVALID
    assert lib.cg_im2col_bf16(p, p, 1, 8, 8, 3, 7, 2, 3, 144, None) == INVALID      # k_pad < 147
    assert lib.cg_im2col_bf16(p, p, 1, 8, 8, 3, 7, 2, 3, 150, None) == INVALID      # not a multiple of 8
    assert lib.cg_im2col_bf16(p, p, 1, 2, 2, 3, 7, 2, 0, 152, None) == INVALID      # filter larger than the image
    assert lib.cg_im2col_bf16(odd, p, 1, 8, 8, 3, 7, 2, 3, 152, None) == ALIGN
    assert lib.cg_subsample_bf16(p, p, 1, 8, 8, 12, 2, None) == INVALID             # channels not a multiple of 8
    assert lib.cg_subsample_bf16(p, odd, 1, 8, 8, 16, 2, None) == ALIGN
    assert lib.cg_maxpool_bf16(p, p, 1, 8, 8, 16, 3, 2, 3, None) == INVALID         # a window of padding only
    assert lib.cg_maxpool_bf16(p, None, 1, 8, 8, 16, 3, 2, 1, None) == INVALID
    assert lib.cg_avgpool_bf16(p, p, 0, 49, 16, None) == INVALID
    assert lib.cg_avgpool_bf16(odd, p, 1, 49, 16, None) == ALIGN


def test_the_stem_is_told_the_images_and_channels_of_its_input(monkeypatch):
    """The extents come from x itself: a short batch is that many images, another channel count is refused."""
    import torch
    seen = []

    class Recorder:
        def cg_stem_forward(self, *args):
            seen.append(args)
            return 0

    monkeypatch.setattr(B, "_lib", Recorder())
    monkeypatch.setattr(B, "_stream_ptr", lambda stream: None)
    x = torch.zeros((3, 9, 11, 4), dtype=torch.bfloat16)
    B.cg_stem_forward(C.c_void_p(16), x, x, B.CgBnParams(), x, x, x)
    assert seen[0][2:6] == (3, 9, 11, 4)


def test_a_patch_matrix_that_does_not_fit_is_refused(monkeypatch):
    """A batch larger than the matrix was made for must not be written behind it."""
    import torch
    calls = []

    class Recorder:
        def cg_im2col_bf16(self, *args):
            calls.append(args)
            return 0

    monkeypatch.setattr(B, "_lib", Recorder())
    monkeypatch.setattr(B, "_stream_ptr", lambda stream: None)
    a = torch.zeros((2, 5, 6, 152), dtype=torch.bfloat16)
    x = torch.zeros((4, 9, 12, 3), dtype=torch.bfloat16)
    for n in (1, 2):
        B.cg_im2col_bf16(x[:n], a, 7, 2, 3)
    assert len(calls) == 2
    for bad in (x[:3], torch.zeros((2, 11, 12, 3), dtype=torch.bfloat16)):
        with pytest.raises(ValueError):
            B.cg_im2col_bf16(bad, a, 7, 2, 3)
    assert len(calls) == 2


def test_the_stem_rejects_bad_arguments_before_any_launch():
    lib = B.lib()
    buf = (C.c_uint8 * 4096)()
    p = C.c_void_p((C.addressof(buf) + 15) & ~15)
    bn = C.byref(B.CgBnParams())
    for h, x, n, ih, iw, c, w, y, ws in ((None, p, 1, 8, 8, 3, p, p, p), (p, None, 1, 8, 8, 3, p, p, p),
                                         (p, p, 0, 8, 8, 3, p, p, p), (p, p, 1, 0, 8, 3, p, p, p),
                                         (p, p, 1, 8, -1, 3, p, p, p), (p, p, 1, 8, 8, 4, p, p, p),
                                         (p, p, 1, 8, 8, 1, p, p, p), (p, p, 1, 8, 8, 3, None, p, p),
                                         (p, p, 1, 8, 8, 3, p, None, p), (p, p, 1, 8, 8, 3, p, p, None)):
        assert lib.cg_stem_forward(h, x, n, ih, iw, c, w, bn, None, y, ws, None) == 1   # (the handle is not looked at)


def test_status_strings():
    lib = B.lib()
    seen = {lib.cg_status_string(i) for i in range(8)}
    assert len(seen) == 8
    assert lib.cg_status_string(0) == b"ok"


def _desc(**kw):
    base = dict(n=2, h=8, w=8, c_in=16, c_out=16, kh=3, kw=3, stride=1, pad=1, groups=4,
                in_dtype=B.CG_F32, out_dtype=B.CG_F32, bn_eps=1e-5, relu=1, has_residual=0,
                requant_shift=0, algo=0, cond_mode=0, grouping=0)
    base.update(kw)
    return B.CgConvDesc(**base)


@pytest.mark.parametrize("kw", [dict(n=0), dict(c_in=15), dict(kh=3, kw=5), dict(groups=0),
                                dict(stride=0), dict(pad=-1), dict(in_dtype=7, out_dtype=7),
                                dict(out_dtype=B.CG_BF16), dict(h=1, w=1, pad=0),
                                dict(in_dtype=B.CG_I8, out_dtype=B.CG_I8, requant_shift=0),
                                dict(in_dtype=B.CG_I8, out_dtype=B.CG_I8, requant_shift=32),
                                dict(bn_eps=-1.0), dict(algo=9), dict(cond_mode=-1),
                                dict(grouping=2), dict(grouping=1, c_out=18),
                                dict(grouping=1, in_dtype=B.CG_I8, out_dtype=B.CG_I8,
                                     requant_shift=8)])
def test_create_rejects_bad_descriptions(kw):
    h = C.c_void_p()
    d = _desc(**kw)
    assert B.lib().cg_conv_create(C.byref(h), C.byref(d)) == 1      # CG_ERR_INVALID_ARG
    assert not h.value


def test_create_null_arguments():
    d = _desc()
    assert B.lib().cg_conv_create(None, C.byref(d)) == 1
    h = C.c_void_p()
    assert B.lib().cg_conv_create(C.byref(h), None) == 1


def test_tensor_algo_rejects_ineligible_layers():
    h = C.c_void_p()
    for kw in (dict(algo=B.CG_ALGO_TENSOR),                                  # fp32
               dict(algo=B.CG_ALGO_TENSOR, in_dtype=B.CG_BF16, out_dtype=B.CG_BF16, c_in=24,
                    c_out=16)):                                              # c_p = 6 channels
        d = _desc(**kw)
        assert B.lib().cg_conv_create(C.byref(h), C.byref(d)) == 2           # CG_ERR_UNSUPPORTED


def test_tap_stacked_algo_eligibility_is_decided_on_the_host():
    """CG_ALGO_TENSOR_STACKED: 3x3, stride 1, pad 1, bf16, 64 -> 64 channels, c_in/G a multiple of 16,
    width at most 128, no grouping, no channel-wise gate, no row compaction.  Layers outside report
    CG_ERR_UNSUPPORTED before any device is needed; a layer inside gets as far as the device."""
    import torch
    h = C.c_void_p()
    ok = dict(algo=B.CG_ALGO_TENSOR_STACKED, in_dtype=B.CG_BF16, out_dtype=B.CG_BF16, c_in=64, c_out=64,
              h=32, w=32, groups=4)
    for kw in (dict(w=129), dict(c_out=128), dict(c_in=128), dict(groups=8), dict(kh=1, kw=1, pad=0),
               dict(stride=2), dict(cond_mode=3), dict(channel_tau=0.5), dict(grouping=1),
               dict(in_dtype=B.CG_I8, out_dtype=B.CG_I8, requant_shift=8)):
        d = _desc(**{**ok, **kw})
        assert B.lib().cg_conv_create(C.byref(h), C.byref(d)) == 2, kw       # CG_ERR_UNSUPPORTED
    if not torch.cuda.is_available():
        for kw in (dict(), dict(w=56, h=56), dict(groups=1), dict(groups=2), dict(w=128, h=3)):
            d = _desc(**{**ok, **kw})
            assert B.lib().cg_conv_create(C.byref(h), C.byref(d)) == 5, kw   # CG_ERR_CUDA: eligible, no device


BEYOND_32_BITS = [dict(h=65536, w=65536), dict(h=65536, w=65536, stride=2), dict(h=32768, w=131072), dict(h=1, w=2 ** 30),
                  dict(h=2 ** 30, w=2), dict(h=2 ** 31 - 1, w=2), dict(h=2 ** 31 - 1, w=2 ** 31 - 1),
                  dict(n=2 ** 31 - 1, h=65536, w=65536), dict(n=2 ** 31 - 1, h=3, w=3),
                  dict(h=65536, w=65536, kh=1, kw=1, pad=0, groups=1)]


def test_extents_beyond_32_bits_return_a_status():
    """Products of extents that leave 32 bits (one is a multiple of 2^32) must not end the process: a layer that no
    tensor-core kernel can run goes to the direct kernels.  In a process of its own, without devices."""
    import subprocess
    import sys
    base = dict(n=1, h=8, w=8, c_in=128, c_out=64, kh=3, kw=3, stride=1, pad=1, groups=4, requant_shift=8)
    descs = [{**base, "in_dtype": t, "out_dtype": t, **kw} for t in (B.CG_F32, B.CG_BF16, B.CG_I8) for kw in BEYOND_32_BITS]
    code = ("import ctypes as C\nfrom paper_1805_12549_b200 import binding as B\nh = C.c_void_p()\n"
            "for d in %r:\n    print(B.lib().cg_conv_create(C.byref(h), C.byref(B.CgConvDesc(**d))), flush=True)" % (descs,))
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    got = r.stdout.split()
    assert r.returncode == 0, (r.returncode, descs[min(len(got), len(descs) - 1)], r.stderr[-500:])
    assert got == ["5"] * len(descs)                     # CG_ERR_CUDA: described, no device


def test_null_handle_calls_are_safe():
    lib = B.lib()
    assert lib.cg_conv_workspace_bytes(None) == 0
    assert lib.cg_conv_host_staging_bytes(None) == 0
    assert lib.cg_conv_launches_per_forward(None) == 0
    assert lib.cg_conv_uses_tensor_cores(None) == 0
    lib.cg_conv_destroy(None)
    st = B.CgStats()
    assert lib.cg_conv_stats(None, C.byref(st), None) == 1
    bn = B.CgBnParams()
    assert lib.cg_conv_forward(None, None, None, None, C.byref(bn), None, None, None, None, None,
                               0, None) == 1


def test_create_without_a_device_reports_cuda_error():
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present")
    h = C.c_void_p()
    d = _desc()
    assert B.lib().cg_conv_create(C.byref(h), C.byref(d)) == 5               # CG_ERR_CUDA
    with pytest.raises(B.CgError):
        B.cg_conv_create(d)
