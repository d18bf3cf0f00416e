"""Narrow 1x1 convolutions with many tiles per CTA (resident weights, bit-sliced
column counts flushed every seven tiles, one epilogue warp per tile and lane
quarter) against the oracle: one to six 32-column blocks, partial blocks, a last
tile with few rows, tile counts at and around the flush period, every activation,
residual, spatial (strided) tiles.  Counts and bitmaps bit for bit, values within
the path's tolerance (bf16 rounding of the output, 2^-9)."""
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


# rows = B H W; 152 CTAs x 4 warps per lane quarter x 7 tiles of 128 rows = 544,768 rows per flush period
@pytest.mark.parametrize("B,H,W,C,Co,stride,act,res", [
    (1, 700, 780, 16, 96, 1, 2, False), (1, 512, 1100, 8, 32, 1, 1, True), (1, 333, 501, 24, 144, 1, 2, False),
    (1, 257, 300, 64, 24, 1, 0, True), (1, 200, 640, 160, 64, 1, 1, False), (1, 151, 257, 32, 192, 1, 3, False),
    (3, 130, 131, 32, 40, 2, 1, False), (2, 160, 160, 64, 256, 1, 1, True)])
@pytest.mark.parametrize("force", [1, 2])
def test_pointwise(sp, ctx, B, H, W, C, Co, stride, act, res, force):
    d = synth.conv_layer(seed=H + C, N=B, H=H, W=W, Cin=C, Cout=Co, k=1, stride=stride, pad=0, bn="random")
    Ho, Wo = (H - 1) // stride + 1, (W - 1) // stride + 1
    R = B * Ho * Wo
    g = torch.Generator().manual_seed(3)
    rb = synth.to_bf16_bits(torch.randn(R, Co, generator=g)) if res else None
    y = torch.full((B, Ho, Wo, Co), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(R, Co)
    yo.buf.fill_(0x5A)
    x = sp.bits_to_device(d["x"]).view(B, H, W, C)
    sp.sparoa_conv2d(ctx, x, sp.bits_to_device(d["w"]).view(Co, 1, 1, C), y, stride=stride, pad=0,
                     bn=torch.from_numpy(d["bn"]).cuda(), act=act,
                     residual=None if rb is None else sp.bits_to_device(rb).view(B, Ho, Wo, Co),
                     thr=sp.thresholds(force_path=force), y_occ=yo)
    assert ctx.last_path() == force
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), R, Co), "occupancy")
    ref = orc.conv2d(d["x"], B, H, W, C, d["w"], Co, 1, 1, stride, 0, bn=d["bn"], residual_bits=rb, act=act)
    assert_close(y.float().cpu().numpy(), np.asarray(ref).reshape(y.shape), what="pointwise")


@pytest.mark.parametrize("M,N", [(1576, 6144), (130, 4104), (4000, 8200)])
def test_more_than_one_row_word(sp, ctx, M, N):
    """outputs of more than 4096 columns: every row has several bitmap words, and no
    tile's columns may lie in two"""
    g = torch.Generator().manual_seed(M)
    x = torch.randn(M, 64, generator=g)
    w = torch.randn(N, 64, generator=g)
    w[4032:4096] = 0.0  # the last 64 columns of the first word, and the first of the second
    w[4160:4200] = 0.0
    xb, wb = synth.to_bf16_bits(x), synth.to_bf16_bits(w)
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    xo, yo = sp.OccupancyBuffer(M, 64), sp.OccupancyBuffer(M, N)
    yo.buf.fill_(0x5A)
    xd, wd = sp.bits_to_device(xb).view(M, 64), sp.bits_to_device(wb).view(N, 64)
    sp.sparoa_op_stats(ctx, xd, (M, 64), occ=xo)
    sp.sparoa_gemm(ctx, xd, wd, y, x_occ=xo, y_occ=yo, thr=sp.thresholds(force_path=1))
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), M, N), "occupancy")
    assert_close(y.float().cpu().numpy(), (xd.double() @ wd.double().T).cpu().numpy(), what="gemm")


@pytest.mark.parametrize("M,K,N,act,res", [
    (1576, 768, 768, 0, True), (1576, 768, 3072, 3, False), (20000, 64, 96, 1, False), (20000, 144, 136, 2, True),
    (77777, 200, 72, 1, False), (1500, 1000, 760, 1, True), (40000, 96, 152, 0, False)])
@pytest.mark.parametrize("force", [1, 2])
def test_tiles_of_96_and_160_columns(sp, ctx, M, K, N, act, res, force):
    """one and several tiles per CTA, several column tiles, the last one partial"""
    g = torch.Generator().manual_seed(N)
    x = torch.randn(M, K, generator=g)
    x[(torch.rand((M + 127) // 128, (K + 31) // 32, generator=g) < 0.4)
      .repeat_interleave(128, 0)[:M].repeat_interleave(32, 1)[:, :K]] = 0.0  # whole 128 x 32 blocks
    w = torch.randn(N, K, generator=g) / K ** 0.5
    w[N // 3: N // 3 + 40] = 0.0
    b = torch.randn(N, generator=g)
    b[N // 3: N // 3 + 40] = 0.0
    r = torch.randn(M, N, generator=g) * (torch.rand(M, N, generator=g) < 0.5) if res else None
    xd = sp.bits_to_device(synth.to_bf16_bits(x)).view(M, K)
    wd = sp.bits_to_device(synth.to_bf16_bits(w)).view(N, K)
    rd = sp.bits_to_device(synth.to_bf16_bits(r)).view(M, N) if res else None
    bd = b.cuda()
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    xo, yo = sp.OccupancyBuffer(M, K), sp.OccupancyBuffer(M, N)
    yo.buf.fill_(0x5A)
    sp.sparoa_op_stats(ctx, xd, (M, K), occ=xo)
    sp.sparoa_gemm(ctx, xd, wd, y, bias=bd, act=act, x_occ=xo, y_occ=yo, residual=rd,
                   thr=sp.thresholds(force_path=force))
    assert ctx.last_path() == force
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), M, N), "occupancy")
    v = xd.double() @ wd.double().T + bd.double()
    if res:
        v = v + rd.double()
    v = {0: lambda t: t, 1: torch.relu, 2: lambda t: t.clamp(0, 6),
         3: lambda t: torch.nn.functional.gelu(t, approximate="tanh")}[act](v)
    assert_close(y.float().cpu().numpy(), v.cpu().numpy(), what="gemm")


@pytest.mark.parametrize("M,K,N,act,res", [
    (19451, 64, 96, 1, False), (19584, 128, 128, 1, True), (38912, 64, 128, 0, False), (38913, 64, 128, 2, True),
    (19500, 40, 64, 1, True), (5000, 128, 640, 1, True), (300, 64, 72, 3, False), (128, 64, 4928, 1, True),
    (1000, 96, 4160, 0, False)])
@pytest.mark.parametrize("force", [1, 2])
def test_one_and_two_tiles_a_cta(sp, ctx, M, K, N, act, res, force):
    """around one and two tiles per CTA of 152, where the epilogue warps share tiles
    and a lone tile's counts go straight out; one and two groups of K"""
    test_tiles_of_96_and_160_columns(sp, ctx, M, K, N, act, res, force)
