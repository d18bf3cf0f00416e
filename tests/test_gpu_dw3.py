"""The 3x3 depthwise kernel at the edges of its work split: output widths around
a strip's 8 pixels, heights around a box's 3 rows and around a run's end, channel
counts around its 32-channel slices, one warp with several items, and input
values of every kind at the image border (the padding).  Values against the
64-bit oracle; occupancy bit for bit."""
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


def _bits(shape, seed, zero_p=0.4):
    g = torch.Generator().manual_seed(seed)
    v = torch.randn(*shape, generator=g)
    v[torch.rand(*shape, generator=g) < zero_p] = 0.0
    return synth.to_bf16_bits(v)


@pytest.mark.parametrize("s", [1, 2])
@pytest.mark.parametrize("N,H,W,C,act,res", [
    (1, 1, 1, 8, 0, False), (2, 2, 3, 24, 1, True), (1, 3, 7, 32, 2, False), (3, 4, 8, 40, 0, True),
    (1, 5, 9, 64, 1, False), (2, 6, 16, 72, 3, False), (1, 7, 17, 96, 2, True), (5, 31, 33, 136, 1, False),
    (64, 13, 12, 168, 2, False), (2, 200, 1, 16, 1, True), (1, 1, 300, 56, 0, False), (48, 61, 40, 32, 1, False),
    (1, 6, 5, 1400, 2, False)])
def test_depthwise_edges(sp, ctx, N, H, W, C, act, res, s):
    g = torch.Generator().manual_seed(N * H + W * C + s)
    xb = _bits((N, H, W, C), N + H + W + C)
    wb = synth.to_bf16_bits(torch.randn(C, 3, 3, 1, generator=g) * 0.4)
    bn = synth.random_bn(C, g)
    Ho, Wo = (H - 1) // s + 1, (W - 1) // s + 1
    rb = _bits((N, Ho, Wo, C), 3) if res else None
    y = torch.full((N, Ho, Wo, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(N * Ho * Wo, C)
    yo.buf.fill_(0x77)
    st = sp.sparoa_conv2d(ctx, sp.bits_to_device(xb).view(N, H, W, C), sp.bits_to_device(wb).view(C, 3, 3, 1), y,
                          stride=s, pad=1, groups=C, bn=torch.from_numpy(bn).cuda(), act=act,
                          residual=sp.bits_to_device(rb).view(N, Ho, Wo, C) if res else None, y_occ=yo, host=True)
    assert st.path == sp.PATH_DEPTHWISE
    what = f"dw {N}x{H}x{W}x{C} s{s}"
    assert_close(y.float().cpu().numpy().astype(np.float64),
                 orc.conv2d(xb, N, H, W, C, wb, C, 3, 3, s, 1, groups=C, bn=bn, residual_bits=rb, act=act), what=what)
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), N * Ho * Wo, C), what)


@pytest.mark.parametrize("kind", ["dw", "pointwise", "attention"])
def test_subnormal_outputs_count(sp, ctx, kind):
    """occupancy counts every bf16 pattern but +-0, subnormal values among them"""
    C, R = 64, 4 * 9 * 11
    pat = np.resize(np.array([0x0001, 0x8001, 0x0000, 0x8000, 0x007F, 0x3F80, 0x0010], dtype=np.uint16), R * C)
    yo = sp.OccupancyBuffer(R, C)
    yo.buf.fill_(0x77)
    x = sp.bits_to_device(pat)
    y = torch.full((R, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    if kind == "dw":
        w = torch.zeros(C, 3, 3, 1, dtype=torch.bfloat16, device="cuda")
        w[:, 1, 1] = 1.0
        sp.sparoa_conv2d(ctx, x.view(4, 9, 11, C), w, y.view(4, 9, 11, C), stride=1, pad=1, groups=C, y_occ=yo)
    elif kind == "pointwise":
        w = torch.eye(C, device="cuda").to(torch.bfloat16).view(C, 1, 1, C).contiguous()
        sp.sparoa_conv2d(ctx, x.view(4, 9, 11, C), w, y.view(4, 9, 11, C), stride=1, pad=0, y_occ=yo)
    else:
        qkv = torch.zeros(R, 1, 3 * C, dtype=torch.bfloat16, device="cuda")  # one token: the output is v
        qkv[:, 0, 2 * C:] = x.view(R, C)
        sp.sparoa_attention(ctx, qkv, y.view(R, 1, C), 1, y_occ=yo)
    yb = sp.device_to_bits(y).reshape(-1)
    if kind == "dw":
        assert np.array_equal(yb & 0x7FFF, pat & 0x7FFF)
    assert_occ_equal(yo.to_host(), orc.stats(yb, R, C), kind)
