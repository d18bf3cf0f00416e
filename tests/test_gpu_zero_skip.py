"""What the zero-skip path leaves out is not multiplied: weights of infinity and
NaN that meet only unoccupied groups of the input (32 columns of a GEMM's 128-row
block, 64 channels of a convolution's tile) do not reach the output, which is bit
for bit that of the same weights with zeros there.  Over the one-tile kernel with
its cluster sizes (shares without an occupied block among them), the persistent
kernel's lean and general variants, and a single K block of two groups."""
import pytest
import torch

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


def _poison(w, cols):
    bad = w.clone()
    bad[..., cols] = float("inf")
    bad[..., cols[::3]] = float("nan")
    clean = w.clone()
    clean[..., cols] = 0.0
    return clean, bad


@pytest.mark.parametrize("M,K,N", [(1, 64, 64), (100, 64, 64), (128, 256, 64), (128, 512, 128), (128, 768, 512),
                                   (60, 1160, 1024), (128, 2304, 64), (300, 4608, 256), (128, 3584, 4800),
                                   (20000, 64, 96), (20000, 40, 64), (5000, 1000, 200), (2000, 768, 3072)])
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("empty", ["odd groups", "few", "most"])
def test_gemm(sp, ctx, M, K, N, f32, empty):
    g = torch.Generator().manual_seed(M + K + N)
    x = torch.randn(M, K, generator=g)
    groups = (K + 31) // 32
    gone = {"odd groups": range(1, groups, 2), "few": range(groups - 1, 0, -7), "most": range(1, groups)}[empty]
    cols = torch.tensor([c for q in gone for c in range(32 * q, min(32 * q + 32, K))])
    x[:, cols] = 0.0
    x = x.to(torch.bfloat16).cuda()
    clean, bad = _poison((torch.randn(N, K, generator=g) / K ** 0.5).to(torch.bfloat16), cols)
    out = []
    for w in (clean.cuda(), bad.cuda()):
        y = torch.full((M, N), float("nan"), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
        sp.sparoa_gemm(ctx, x, w, y, thr=sp.thresholds(force_path=2))
        out.append(y)
    assert torch.isfinite(out[1]).all()
    assert torch.equal(out[0], out[1])
    ref = x.double() @ clean.double().cuda().T
    assert (out[0].double() - ref).norm() <= 5e-3 * ref.norm()


@pytest.mark.parametrize("N,H,Cin,Cout,k,stride", [(1, 7, 512, 512, 3, 1), (1, 14, 256, 64, 3, 1), (2, 14, 128, 256, 3, 2),
                                                   (8, 28, 128, 128, 3, 1), (1, 28, 128, 256, 1, 2), (1, 20, 192, 24, 5, 1),
                                                   (32, 28, 128, 128, 3, 1), (40, 29, 192, 72, 3, 2)])
def test_conv(sp, ctx, N, H, Cin, Cout, k, stride):
    g = torch.Generator().manual_seed(H + Cin + Cout)
    x = torch.randn(N, H, H, Cin, generator=g)
    cols = torch.arange(64, 128)
    x[..., cols] = 0.0
    if N > 1:
        x[0] = 0.0  # tiles with nothing but the other images' values, or none at all
        x[0, :, :, 0] = 1.0
    x = x.to(torch.bfloat16).cuda()
    clean, bad = _poison((torch.randn(Cout, k, k, Cin, generator=g) / (k * k * Cin) ** 0.5).to(torch.bfloat16), cols)
    Ho = (H + 2 * (k // 2) - k) // stride + 1
    out = []
    for w in (clean.cuda(), bad.cuda()):
        y = torch.full((N, Ho, Ho, Cout), float("nan"), dtype=torch.bfloat16, device="cuda")
        sp.sparoa_conv2d(ctx, x, w, y, stride=stride, pad=k // 2, act=sp.ACT_RELU, thr=sp.thresholds(force_path=2))
        out.append(y)
    assert torch.isfinite(out[1]).all()
    assert torch.equal(out[0], out[1])
    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), clean.double().cuda().permute(0, 3, 1, 2),
                                     stride=stride, padding=k // 2).clamp(min=0).permute(0, 2, 3, 1)
    assert (out[0].double() - ref).norm() <= 5e-3 * ref.norm()
