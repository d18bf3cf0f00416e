"""The one-tile-per-cluster GEMM / convolution kernel (fewer 64-wide output
tiles than SMs) against the oracle at the edges of its shapes: one row, partial
row and column tiles, one K block, K shares that do not divide evenly, a K tail,
clusters of 1 to 8 CTAs, 32- and 64-wide K blocks, spatial tiles with images
missing from the box, shares with no occupied K block, fp32 and bf16 outputs,
residual, every activation; output occupancy bit for bit.

Bounds: the bf16 output rounding is 2^-9 of each value, fp32 sums of K <= 4608
products add less than K * 2^-24 of the sum of magnitudes (3e-4 here): the
path's max 2e-2 / Frobenius 5e-3; fp32 outputs without that rounding 1e-4.
"""
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


def _sparse(shape, g, block=None):
    """ReLU of normals; with `block`, whole [128 rows, 32 columns] blocks zero"""
    v = torch.randn(*shape, generator=g).relu()
    if block:
        M, K = shape
        keep = torch.rand((M + 127) // 128, (K + 31) // 32, generator=g) >= block
        v = v * keep.repeat_interleave(128, 0)[:M].repeat_interleave(32, 1)[:, :K]
    return synth.to_bf16_bits(v)


@pytest.mark.parametrize("M,K,N,act,f32", [
    (1, 64, 8, 0, False), (1, 32, 64, 1, True), (37, 72, 200, 3, False), (127, 4096, 64, 2, False),
    (128, 2048, 72, 1, True), (129, 3072, 136, 1, False), (256, 648, 768, 0, False), (400, 256, 712, 3, False),
    (640, 1096, 256, 2, False), (1216, 128, 256, 1, False),
    # (bf16 outputs of few K blocks run in the persistent kernel: fp32 ones here)
    (1, 64, 8, 0, True), (37, 72, 200, 3, True), (400, 256, 712, 3, True), (1216, 128, 256, 1, True),
    # one CTA a tile and a long K; 15 and 16 tiles around the clusters of 8 that fit
    (128, 3104, 4992, 1, False), (128, 1600, 960, 1, False), (128, 1600, 1024, 3, False)])
@pytest.mark.parametrize("force", [1, 2])
def test_gemm(sp, ctx, M, K, N, act, f32, force):
    g = torch.Generator().manual_seed(M + K + N)
    xb = _sparse((M, K), g, 0.7)
    wb = synth.to_bf16_bits(torch.randn(N, K, generator=g) / np.sqrt(K))
    rb = synth.to_bf16_bits(torch.randn(M, N, generator=g))
    bn = synth.random_bn(N, g)
    y = torch.full((M, N), float("nan"), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    yo = None if f32 else sp.OccupancyBuffer(M, N)
    st = sp.sparoa_gemm(ctx, sp.bits_to_device(xb).view(M, K), sp.bits_to_device(wb).view(N, K), y,
                        bn=torch.from_numpy(bn).cuda(), act=act, residual=sp.bits_to_device(rb).view(M, N),
                        thr=sp.thresholds(force_path=force), y_occ=yo, host=True)
    assert st.path == force
    ref = orc.fc(xb, M, K, wb, N, bn=bn, residual_bits=rb, act=act)
    tol = dict(max_rel=1e-4, fro_rel=1e-4) if f32 and act != 3 else {}
    assert_close(y.float().cpu().numpy(), ref, what=f"{M}x{K}x{N}", **tol)
    if yo is not None:
        assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y), M, N), f"{M}x{K}x{N}")


@pytest.mark.parametrize("B,H,W,C,Co,k,stride,act", [
    (1, 7, 7, 512, 512, 3, 1, 1), (1, 14, 14, 256, 256, 3, 1, 1), (1, 14, 14, 256, 512, 1, 2, 0),
    (1, 9, 5, 32, 8, 3, 1, 2), (3, 11, 13, 96, 72, 3, 2, 1), (2, 1, 1, 64, 64, 3, 1, 1), (5, 3, 3, 128, 64, 3, 1, 3),
    (1, 15, 17, 64, 64, 5, 2, 1)])
@pytest.mark.parametrize("force", [1, 2])
def test_conv(sp, ctx, B, H, W, C, Co, k, stride, act, force):
    d = synth.conv_layer(seed=B + H + C, N=B, H=H, W=W, Cin=C, Cout=Co, k=k, stride=stride, pad=k // 2, bn="random")
    xb = d["x"].reshape(B, H, W, C).copy()
    xb[:, : H // 2] = 0  # whole taps of the upper tiles have nothing occupied
    Ho, Wo = (H + 2 * (k // 2) - k) // stride + 1, (W + 2 * (k // 2) - k) // stride + 1
    g = torch.Generator().manual_seed(1)
    rb = synth.to_bf16_bits(torch.randn(B, Ho, Wo, Co, generator=g))
    y = torch.full((B, Ho, Wo, Co), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(B * Ho * Wo, Co)
    st = sp.sparoa_conv2d(ctx, sp.bits_to_device(xb).view(B, H, W, C), sp.bits_to_device(d["w"]).view(Co, k, k, C), y,
                          stride=stride, pad=k // 2, bn=torch.from_numpy(d["bn"]).cuda(), act=act,
                          residual=sp.bits_to_device(rb).view(B, Ho, Wo, Co), thr=sp.thresholds(force_path=force),
                          y_occ=yo, host=True)
    assert st.path == force
    ref = orc.conv2d(xb.reshape(-1), B, H, W, C, d["w"], Co, k, k, stride, k // 2, bn=d["bn"],
                     residual_bits=rb.reshape(-1), act=act)
    assert_close(y.float().cpu().numpy(), ref, what="conv")
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), B * Ho * Wo, Co), "conv")
