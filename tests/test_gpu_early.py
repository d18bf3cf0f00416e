"""Weights and parameters written on the stream immediately before a call (kernels
load weights before their dependency wait where another kernel of the same call
lies between), back to back and without a synchronisation; and capture and replay
of the kernels that run as thread-block clusters.  Every output and occupancy is
bit for bit that of a call made with everything at rest."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    from paper_2511_19457_gb300 import sparoa
    return sparoa


def _same(a, b):
    return all(np.array_equal(a[k], b[k]) for k in a)


def _relu(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda").relu().to(torch.bfloat16)


def _gemm(M, K, N, **kw):
    def make(sp, ctx, g):
        x = _relu(g, M, K)
        w, bn = torch.empty(N, K, dtype=torch.bfloat16, device="cuda"), torch.empty(4, N, device="cuda")
        return x, w, bn, (M, N), lambda y, yo: sp.sparoa_gemm(ctx, x, w, y, bn=bn, act=sp.ACT_RELU, y_occ=yo, **kw)
    return make


def _conv(n, H, Cin, Cout, k, stride, pad, **kw):
    def make(sp, ctx, g):
        x = _relu(g, n, H, H, Cin)
        w = torch.empty(Cout, k, k, Cin, dtype=torch.bfloat16, device="cuda")
        bn = torch.empty(4, Cout, device="cuda")
        Ho = (H + 2 * pad - k) // stride + 1
        return x, w, bn, (n, Ho, Ho, Cout), lambda y, yo: sp.sparoa_conv2d(
            ctx, x, w, y, stride=stride, pad=pad, bn=bn, act=sp.ACT_RELU, y_occ=yo, **kw)
    return make


CASES = {
    "one tile": _gemm(128, 2304, 640),
    "one tile, one K block a share": _gemm(60, 256, 64),
    "persistent": _gemm(4096, 768, 768),
    "persistent, short K": _gemm(9000, 64, 96),
    "conv one tile": _conv(1, 14, 256, 256, 3, 1, 1),
    "conv persistent": _conv(16, 28, 128, 128, 3, 1, 1),
    "conv slab": _conv(4, 56, 64, 64, 3, 1, 1),
    "stem": _conv(4, 96, 3, 64, 7, 2, 3),
    "patches": _conv(2, 64, 3, 128, 16, 16, 0),
    "gather": _conv(2, 28, 24, 40, 3, 1, 1),
}


def _params(g, w, bn):
    return ((torch.randn(w.shape, generator=g, device="cuda") / w[0].numel() ** 0.5).to(torch.bfloat16),
            torch.rand(bn.shape, generator=g, device="cuda") + 0.5)


@pytest.mark.parametrize("name", list(CASES))
def test_parameters_written_just_before(sp, name):
    s = torch.cuda.Stream()
    g = torch.Generator(device="cuda").manual_seed(3)
    with torch.cuda.stream(s):
        ctx = sp.Context(0)
        x, w, bn, shape, call = CASES[name](sp, ctx, g)
        R, C = int(torch.tensor(shape[:-1]).prod()), shape[-1]
        sets = [_params(g, w, bn) for _ in range(6)]
        out = lambda: (torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda"), sp.OccupancyBuffer(R, C))
        want = []
        for wi, bi in sets:
            w.copy_(wi)
            bn.copy_(bi)
            s.synchronize()
            y, yo = out()
            s.synchronize()
            call(y, yo)
            s.synchronize()
            want.append((y, yo.to_host()))
        got = [out() for _ in sets * 4]
        busy = torch.randn(2048, 2048, device="cuda")
        s.synchronize()
        for i, (y, yo) in enumerate(got):
            if i % 3 == 0:
                busy = busy @ busy * 1e-3  # the stream falls behind the host
            w.copy_(sets[i % 6][0])
            bn.copy_(sets[i % 6][1])
            call(y, yo)
    torch.cuda.synchronize()
    for i, (y, yo) in enumerate(got):
        assert torch.equal(y, want[i % 6][0]), f"call {i}"
        assert _same(yo.to_host(), want[i % 6][1]), f"call {i}: occupancy"
    ctx.close()


@pytest.mark.parametrize("force", [1, 2])
def test_clusters_under_capture(sp, force):
    """A chain of one-tile convolutions (clusters of 2, 4 and 8) and a clustered
    average pool, captured once, replayed on new inputs."""
    s = torch.cuda.Stream()
    g = torch.Generator(device="cuda").manual_seed(7)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    with torch.cuda.stream(s):
        ctx = sp.Context(0)
        x = torch.empty(1, 28, 28, 128, **bf)
        ws = [(torch.randn(co, 3, 3, ci, generator=g, device="cuda") / (9 * ci) ** 0.5).to(torch.bfloat16)
              for ci, co in ((128, 128), (128, 256), (256, 256), (256, 512))]
        a = [torch.empty(1, 28, 28, 128, **bf), torch.empty(1, 14, 14, 256, **bf), torch.empty(1, 14, 14, 256, **bf),
             torch.empty(1, 7, 7, 512, **bf)]
        big = torch.empty(2, 56, 56, 64, **bf)
        pooled = torch.empty(2, 64, **bf)
        occ = [sp.OccupancyBuffer(t.numel() // t.shape[-1], t.shape[-1]) for t in a + [pooled]]

        def body():
            src, src_occ = x, None
            for i, st in enumerate((1, 2, 1, 2)):
                sp.sparoa_conv2d(ctx, src, ws[i], a[i], stride=st, pad=1, act=sp.ACT_RELU, x_occ=src_occ, y_occ=occ[i],
                                 thr=sp.thresholds(force_path=force))
                src, src_occ = a[i], occ[i]
            sp.sparoa_avgpool_global(ctx, big, pooled, y_occ=occ[4])

        def fill(seed):
            g.manual_seed(seed)
            x.copy_(torch.randn(x.shape, generator=g, device="cuda").relu())
            big.copy_(torch.randn(big.shape, generator=g, device="cuda"))

        results = []
        for seed in range(3):
            fill(seed)
            body()
            s.synchronize()
            results.append(([t.clone() for t in a + [pooled]], [o.to_host() for o in occ]))
        graph = torch.cuda.CUDAGraph()
        s.synchronize()
        with torch.cuda.graph(graph, stream=s):
            body()
        for seed in (2, 0, 1, 1):
            fill(seed)
            for o in occ:
                o.buf.fill_(0x5A)
            graph.replay()
            s.synchronize()
            for i, t in enumerate(a + [pooled]):
                assert torch.equal(t, results[seed][0][i]), (seed, i)
                assert _same(occ[i].to_host(), results[seed][1][i]), (seed, i)
    ctx.close()
