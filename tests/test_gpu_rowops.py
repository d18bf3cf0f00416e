"""Layer norm, attention and global average pooling at the edges of their work
splits: runs of rows around 128-row blocks, rows of one to five register chunks,
parameters off a 16-byte boundary, query tiles around a CTA's seven and around
block seams, pooling by clusters of 1 to 8 CTAs; occupancy bit for bit.  Values:
bf16 output rounding 2^-9 (attention: the probabilities' too), fp32 sums."""
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


def _bits(shape, seed, zero_p=0.3):
    g = torch.Generator().manual_seed(seed)
    v = torch.randn(*shape, generator=g)
    v[torch.rand(*shape, generator=g) < zero_p] = 0.0
    return synth.to_bf16_bits(v)


@pytest.mark.parametrize("R,C", [(1, 8), (127, 64), (129, 256), (5000, 264), (6304, 768), (2500, 1024), (300, 1032),
                                 (20001, 200)])
@pytest.mark.parametrize("params", ["none", "aligned", "off"])
def test_layernorm(sp, ctx, R, C, params):
    xb = _bits((R, C), R + C)
    xb.reshape(R, C)[R // 2] = 0  # a constant row
    gb = None
    if params != "none":
        g = torch.Generator().manual_seed(C)
        gb = np.stack([1 + 0.1 * torch.randn(C, generator=g).numpy(), np.zeros(C)]).astype(np.float32)
        gb[:, ::3] = 0.0  # whole columns of zeros
    t = None
    if gb is not None:
        buf = torch.zeros(2 * C + 1, dtype=torch.float32, device="cuda")
        t = buf[1:] if params == "off" else buf[:-1]
        t.copy_(torch.from_numpy(gb).reshape(-1))
    y = torch.full((R, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(R, C)
    yo.buf.fill_(0x77)
    sp.sparoa_layernorm(ctx, sp.bits_to_device(xb).view(R, C), y, gamma_beta=t, y_occ=yo)
    yb = sp.device_to_bits(y)
    assert_occ_equal(yo.to_host(), orc.stats(yb.reshape(-1), R, C), f"layernorm {R}x{C}")
    assert_close(y.float().cpu().numpy(), orc.layernorm(xb, R, C, gb, 1e-6), what=f"layernorm {R}x{C}")


@pytest.mark.parametrize("N,T,heads,hd", [(1, 1, 1, 64), (3, 16, 2, 64), (2, 112, 3, 64), (5, 113, 2, 32), (2, 128, 4, 16),
                                          (3, 129, 1, 64), (2, 225, 5, 32), (1, 512, 2, 64), (2, 197, 12, 64)])
@pytest.mark.parametrize("emit", [True, False])
def test_attention(sp, ctx, N, T, heads, hd, emit):
    D = heads * hd
    qb = _bits((N, T, 3 * D), T + D, 0.0)
    q = qb.reshape(N, T, 3 * D)
    q[:, :, 2 * D: 2 * D + 3] = 0  # three zero columns of v
    y = torch.full((N, T, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(N * T, D) if emit else None
    if emit:
        yo.buf.fill_(0x11)
    sp.sparoa_attention(ctx, sp.bits_to_device(qb).view(N, T, 3 * D), y, heads, y_occ=yo)
    if emit:
        assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), N * T, D), "attention")
    assert_close(y.float().cpu().numpy(), orc.attention(qb, N, T, heads, hd), what=f"attention {N} {T} {heads} {hd}")


@pytest.mark.parametrize("T", [31, 32, 33, 63, 64, 65, 96, 257])
@pytest.mark.parametrize("hd", [16, 32, 64])
def test_attention_key_blocks(sp, ctx, T, hd):
    """Whole and partial blocks of 32 keys, scores far apart (the maxima move from
    block to block), and images whose output is zero next to others in a block of rows."""
    N, heads = 4, 3
    D = heads * hd
    g = torch.Generator().manual_seed(T * hd)
    v = torch.randn(N, T, 3 * D, generator=g)
    v[:, :, :D] *= 6.0
    v[1, :, 2 * D:] = 0.0
    v[3, :, 2 * D + hd: 2 * D + 2 * hd] = 0.0  # one head
    qb = synth.to_bf16_bits(v)
    y = torch.full((N, T, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(N * T, D)
    yo.buf.fill_(0x11)
    sp.sparoa_attention(ctx, sp.bits_to_device(qb).view(N, T, 3 * D), y, heads, y_occ=yo)
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), N * T, D), "attention")
    # (bf16 probabilities, 2^-9 of a value below 5)
    assert_close(y.float().cpu().numpy(), orc.attention(qb, N, T, heads, hd), what=f"attention {T} {hd}")


@pytest.mark.parametrize("N,H,W,C", [(1, 127, 1, 8), (1, 128, 1, 64), (2, 37, 41, 72), (32, 56, 56, 64), (1, 224, 224, 16),
                                     (150, 20, 20, 128), (3, 7, 7, 1280)])
def test_avgpool(sp, ctx, N, H, W, C):
    xb = _bits((N, H, W, C), H + C)
    xb.reshape(N, H, W, C)[..., ::5] = 0
    y = torch.empty(N, C, dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(N, C)
    sp.sparoa_avgpool_global(ctx, sp.bits_to_device(xb).view(N, H, W, C), y, y_occ=yo)
    assert_close(y.float().cpu().numpy(), orc.avgpool_global(xb, N, H, W, C), what="avgpool")
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), N, C), "avgpool")


@pytest.mark.parametrize("R,C", [(7, 1024), (1208, 1024), (1216, 768)])
def test_layernorm_counts_of_short_runs(sp, ctx, R, C):
    """One row a warp, so that a warp adds its column counts as early as it can:
    the same counters after every one of many calls, back to back."""
    xb = _bits((R, C), R)
    x = sp.bits_to_device(xb).view(R, C)
    y = torch.empty(R, C, dtype=torch.bfloat16, device="cuda")
    occ = [sp.OccupancyBuffer(R, C) for _ in range(64)]
    for yo in occ:
        sp.sparoa_layernorm(ctx, x, y, y_occ=yo)
    want = orc.stats(sp.device_to_bits(y).reshape(-1), R, C)
    for yo in occ:
        assert_occ_equal(yo.to_host(), want, f"layernorm {R}x{C}")


@pytest.mark.parametrize("T", [64, 197, 257])
@pytest.mark.parametrize("hd", [16, 32, 64])
def test_attention_large_scores(sp, ctx, T, hd):
    """Scores of 2^22 plus a few units, exact in fp32, whose maximum rises from one
    block of keys to the next: the weights depend on the differences alone.  Rounding
    s / sqrt(hd) and its maximum before the difference puts blocks 2^-5 apart
    (relative Frobenius error of such a softmax on the CPU: 6e-3 to 5e-2); with the
    difference first the probabilities' and the output's bf16 rounding is left, 2e-3
    to 2.5e-3."""
    g = torch.Generator().manual_seed(T + hd)
    v = torch.randn(1, T, 3 * hd, generator=g)
    q, k = torch.zeros(T, hd), torch.zeros(T, hd)
    q[:, 0] = k[:, 0] = 2048.0
    q[:, 1] = 1.0
    t = torch.arange(T)
    k[:, 1] = (2 * (t // 32) + (7 * t) % 5).float()
    v[0, :, :hd], v[0, :, hd:2 * hd] = q, k
    qb = synth.to_bf16_bits(v)
    y = torch.full((1, T, hd), float("nan"), dtype=torch.bfloat16, device="cuda")
    sp.sparoa_attention(ctx, sp.bits_to_device(qb).view(1, T, 3 * hd), y, 1)
    assert_close(y.float().cpu().numpy(), orc.attention(qb, 1, T, 1, hd), what=f"attention {T} {hd}")


@pytest.mark.parametrize("far", [1, 40])
def test_attention_weights_below_the_normal_range(sp, ctx, far):
    """Key 0 has a value of 2^125 and a weight of 2^-128.4 (key `far` scores 712 / 8
    higher, in the same block of keys or in a later one): fp32 and bf16 hold such
    weights as subnormals, and the output is 2^-3.4.  In the same block the weight
    is rounded to a multiple of 2^-133: within 2^-134 / 2^-128.4 = 2.1 %."""
    T, hd = 64, 64
    v = torch.zeros(1, T, 3 * hd)
    v[0, :, 0], v[0, :, hd] = 8.0, -1024.0
    v[0, 0, hd], v[0, far, hd] = 0.0, 89.0
    v[0, 0, 2 * hd] = 2.0 ** 125
    qb = synth.to_bf16_bits(v)
    y = torch.full((1, T, hd), float("nan"), dtype=torch.bfloat16, device="cuda")
    sp.sparoa_attention(ctx, sp.bits_to_device(qb).view(1, T, 3 * hd), y, 1)
    want = orc.attention(qb, 1, T, 1, hd).reshape(T, hd)
    got = y.float().cpu().numpy().reshape(T, hd)
    assert want[0, 0] > 0.09
    assert np.abs(got[:, 0] / want[:, 0] - 1).max() <= 0.021 + 2.0 ** -9
    assert not got[:, 1:].any()


@pytest.mark.parametrize("N,T,heads,hd", [(40, 17, 12, 64), (26, 64, 12, 16), (52, 100, 8, 32), (40, 129, 12, 16),
                                          (32, 225, 12, 16), (32, 300, 12, 16), (102, 300, 12, 16), (13, 500, 24, 64),
                                          (1, 500, 2, 64), (20, 48, 12, 32), (16, 385, 12, 32),
                                          (4, 384, 12, 64), (8, 380, 12, 32), (10, 330, 6, 16)])
def test_attention_splits(sp, ctx, N, T, heads, hd):
    """Every way a head's query tiles are shared out: a tile per warp, several in
    turn, one CTA a head and many, tiles that do not come out even."""
    D = heads * hd
    qb = _bits((N, T, 3 * D), T + N, 0.0)
    qb.reshape(N, T, 3 * D)[:, :, 2 * D: 2 * D + 5] = 0
    y = torch.full((N, T, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(N * T, D)
    yo.buf.fill_(0x11)
    sp.sparoa_attention(ctx, sp.bits_to_device(qb).view(N, T, 3 * D), y, heads, y_occ=yo)
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), N * T, D), "attention")
    assert_close(y.float().cpu().numpy(), orc.attention(qb, N, T, heads, hd), what=f"attention {N} {T} {heads} {hd}")


@pytest.mark.parametrize("R,C", [(1500, 1312), (3, 2056), (700, 4104), (40000, 8), (9000, 256)])
def test_layernorm_row_lengths(sp, ctx, R, C):
    xb = _bits((R, C), R + C)
    y = torch.full((R, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(R, C)
    yo.buf.fill_(0x77)
    sp.sparoa_layernorm(ctx, sp.bits_to_device(xb).view(R, C), y, y_occ=yo)
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), R, C), f"layernorm {R}x{C}")
    assert_close(y.float().cpu().numpy(), orc.layernorm(xb, R, C, None, 1e-6), what=f"layernorm {R}x{C}")


@pytest.mark.parametrize("N,H,W,C", [(8, 14, 14, 4096), (7, 8, 16, 64), (40, 16, 16, 264), (2, 300, 9, 8), (70, 9, 29, 64)])
def test_avgpool_kernels(sp, ctx, N, H, W, C):
    """Plain (many slices, small maps) and deep kernels around their lines, eight
    loads a round with remainders."""
    xb = _bits((N, H, W, C), H + C)
    y = torch.empty(N, C, dtype=torch.bfloat16, device="cuda")
    yo = sp.OccupancyBuffer(N, C)
    sp.sparoa_avgpool_global(ctx, sp.bits_to_device(xb).view(N, H, W, C), y, y_occ=yo)
    assert_close(y.float().cpu().numpy(), orc.avgpool_global(xb, N, H, W, C), what="avgpool")
    assert_occ_equal(yo.to_host(), orc.stats(sp.device_to_bits(y).reshape(-1), N, C), "avgpool")
