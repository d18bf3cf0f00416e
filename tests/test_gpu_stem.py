"""Narrow stems (C < 8) whose A tiles the kernel builds from the input rows, against
the oracle: even and odd row lengths and pitches, inputs off a 16-byte boundary,
strides 1 to 3, kernels of one to seven rows, no padding, tiles that end in the next
image, one and several tiles per CTA, windows next to infinities (a zero weight column
must never meet a neighbouring element); both paths, residual, occupancy bit for bit."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2511_19457_gb300 import synth
from tests._parity import assert_close, assert_occ_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    from paper_2511_19457_gb300 import sparoa
    return sparoa


@pytest.fixture(scope="module")
def ctx(sp):
    c = sp.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("B,H,W,C,Co,k,stride,pad,res,off", [
    (2, 64, 64, 3, 64, 7, 2, 3, False, 0), (3, 65, 71, 3, 32, 7, 2, 3, True, 0), (1, 224, 224, 3, 64, 7, 2, 3, False, 0),
    (2, 30, 33, 3, 24, 3, 1, 1, False, 1), (5, 23, 17, 3, 64, 3, 2, 1, True, 3), (2, 40, 37, 1, 16, 7, 1, 3, False, 2),
    (1, 64, 50, 5, 8, 3, 3, 0, False, 5), (4, 16, 16, 4, 40, 5, 1, 2, False, 0), (2, 90, 61, 7, 64, 3, 2, 1, False, 7),
    (9, 13, 13, 2, 64, 3, 1, 1, True, 0), (2, 200, 131, 3, 64, 3, 1, 1, False, 0), (1, 129, 9, 6, 64, 2, 1, 0, False, 1)])
@pytest.mark.parametrize("force", [1, 2])
def test_stem(sp, ctx, B, H, W, C, Co, k, stride, pad, res, off, force):
    d = synth.conv_layer(seed=H + W, N=B, H=H, W=W, Cin=C, Cout=Co, k=k, stride=stride, pad=pad, bn="random")
    Ho, Wo = (H + 2 * pad - k) // stride + 1, (W + 2 * pad - k) // stride + 1
    R = B * Ho * Wo
    g = torch.Generator().manual_seed(3)
    rb = synth.to_bf16_bits(torch.randn(R, Co, generator=g)) if res else None
    buf = torch.full((off + B * H * W * C + 16,), float("inf"), dtype=torch.bfloat16, device="cuda")
    x = buf[off:off + B * H * W * C].view(B, H, W, C)  # infinities before and after
    x.copy_(sp.bits_to_device(d["x"]).view(B, H, W, C))
    y = torch.full((B, Ho, Wo, Co), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(R, Co)
    yo.buf.fill_(0x3C)
    st = sp.sparoa_conv2d(ctx, x, sp.bits_to_device(d["w"]).view(Co, k, k, C), y, stride=stride, pad=pad,
                          bn=torch.from_numpy(d["bn"]).cuda(), act=1,
                          residual=None if rb is None else sp.bits_to_device(rb).view(B, Ho, Wo, Co),
                          thr=sp.thresholds(force_path=force), y_occ=yo, host=True)
    assert st.path == force and st.nnz == orc.stats(d["x"], B * H * W, C).nnz
    ref = orc.conv2d(d["x"], B, H, W, C, d["w"], Co, k, k, stride, pad, bn=d["bn"], residual_bits=rb, act=1)
    assert_close(y.float().cpu().numpy(), ref, what="stem")
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), R, Co), "stem")


def test_infinity_stays_in_its_windows(sp, ctx):
    """an infinite pixel reaches exactly the outputs whose window holds it"""
    B, H, W, C, Co, k = 1, 40, 45, 3, 64, 7
    d = synth.conv_layer(seed=1, N=B, H=H, W=W, Cin=C, Cout=Co, k=k, stride=2, pad=3, bn="random")
    x = sp.bits_to_device(d["x"]).view(B, H, W, C).clone()
    x[0, 20, 22, 1] = float("inf")
    w = sp.bits_to_device(d["w"]).view(Co, k, k, C)
    y = torch.empty(B, 20, 23, Co, dtype=torch.bfloat16, device="cuda")
    sp.sparoa_conv2d(ctx, x, w, y, stride=2, pad=3)
    ref = torch.nn.functional.conv2d(x.float().permute(0, 3, 1, 2), w.float().permute(0, 3, 1, 2), stride=2, padding=3)
    assert torch.equal(torch.isfinite(y), torch.isfinite(ref.permute(0, 2, 3, 1)))


@pytest.mark.parametrize("B,H,W,C,Co,k,stride", [
    (2, 64, 48, 3, 64, 16, 16), (1, 70, 61, 3, 768, 14, 14),  # images that are not whole patches
    (3, 40, 45, 4, 40, 13, 15),                              # gaps between the windows
    (9, 50, 50, 3, 72, 25, 25),                              # 1875 values a window
    (2, 54, 54, 3, 64, 27, 27),                              # 2187: past the limit
    (5, 16, 16, 7, 128, 16, 16)])                            # one window an image
@pytest.mark.parametrize("force", [1, 2])
def test_patch_embedding(sp, ctx, B, H, W, C, Co, k, stride, force):
    """windows of more than 512 values that do not overlap"""
    d = synth.conv_layer(seed=H + W, N=B, H=H, W=W, Cin=C, Cout=Co, k=k, stride=stride, pad=0, bn="random")
    Ho, Wo = (H - k) // stride + 1, (W - k) // stride + 1
    R = B * Ho * Wo
    y = torch.full((B, Ho, Wo, Co), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(R, Co)
    yo.buf.fill_(0x3C)
    st = sp.sparoa_conv2d(ctx, sp.bits_to_device(d["x"]).view(B, H, W, C), sp.bits_to_device(d["w"]).view(Co, k, k, C), y,
                          stride=stride, pad=0, bn=torch.from_numpy(d["bn"]).cuda(), act=1,
                          thr=sp.thresholds(force_path=force), y_occ=yo, host=True)
    assert st.path == force and st.nnz == orc.stats(d["x"], B * H * W, C).nnz
    ref = orc.conv2d(d["x"], B, H, W, C, d["w"], Co, k, k, stride, 0, bn=d["bn"], act=1)
    assert_close(y.float().cpu().numpy(), ref, what="patches")
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), R, Co), "patches")


def test_stem_rounding(sp, ctx):
    """The 7x7 stem's sums are no less exact than those over im2col rows: 2-norm of
    the distance to the correctly rounded result over its norm, 2.66e-5 there.  One
    accumulator for its eleven k-steps leaves 2.8e-5, two that share them 2.0e-5."""
    err = ref2 = 0.0
    for seed in range(4):
        g = torch.Generator().manual_seed(seed)
        x = torch.randn(8, 224, 224, 3, generator=g).to(torch.bfloat16).cuda()
        w = (torch.randn(64, 7, 7, 3, generator=g) / 147 ** 0.5).to(torch.bfloat16).cuda()
        y = torch.empty(8, 112, 112, 64, dtype=torch.bfloat16, device="cuda")
        sp.sparoa_conv2d(ctx, x, w, y, stride=2, pad=3)
        want = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), w.double().permute(0, 3, 1, 2), stride=2,
                                          padding=3).permute(0, 2, 3, 1).to(torch.bfloat16).double()
        err += float((y.double() - want).pow(2).sum())
        ref2 += float(want.pow(2).sum())
    assert (err / ref2) ** 0.5 <= 2.4e-5
