"""Timed cases: the operators, blocks and whole networks that a program runs through this library.

A case names a kind and its sizes.  ``prepare`` draws a case's inputs and
weights on the GPU, ``run`` is one pass through the public entry points (the
ctypes binding's calls; the caller's output tensors and occupancy blocks are
reused, as a serving loop does), ``exact`` the same computation in 64 bits with
plain torch.  Every tensor that is handed from one call to the next is bf16,
so ``exact`` rounds there too.

Kinds and what they stand for:
  fc         a fully connected head on a small batch, whole input features zero
  conv       one convolution of a CNN on an activation that no producer measured
  block      a ResNet basic block with a strided shortcut: three convolutions,
             each handing its output's occupancy to the next
  stem       the RGB stem convolution of a CNN and the max pool behind it
  invres     a MobileNetV2 inverted residual block: 1x1 expand, 3x3 depthwise,
             1x1 project (+ residual)
  mlp        a transformer MLP on ragged token counts: up + GELU, down + residual
  mlp_down   the down projection of a ReLU MLP on a sparse hidden activation
  attn       a pre-norm attention layer: layer norm, QKV, attention, projection
  light      the low-intensity operators on their own: statistics of an
             activation, batch norm + ReLU, global average pool
  net        a whole network through the graph walk: its logits
"""
import math

import torch

from paper_2511_19457_gb300 import sparoa as sp
from paper_2511_19457_gb300 import synth

_ctx = None


def _context():
    """The context that a program keeps for its lifetime."""
    global _ctx
    if _ctx is None:
        _ctx = sp.Context(0)
    return _ctx


def listed():
    return [
        # a classifier head at batch 64: one launch, latency
        {"name": "fc_b64", "kind": "fc", "M": 64, "K": 512, "N": 512, "f32": True},
        # the first ResNet-18 stage at batch 8, fresh activation: count, rule, convolution
        {"name": "conv3x3_b8", "kind": "conv", "B": 8, "H": 56, "W": 56, "cin": 64, "cout": 64, "k": 3, "stride": 1},
        # the downsampling basic block of ResNet-18's third stage at batch 8
        {"name": "block_s2_b8", "kind": "block", "B": 8, "H": 28, "W": 28, "cin": 128, "cout": 256},
        # ResNet-18's 7x7/2 stem and max pool at batch 32
        {"name": "stem7x7_b32", "kind": "stem", "B": 32, "H": 224, "W": 224, "cout": 64, "k": 7},
        # MobileNetV2's first stride-2 block (largest activations) and a stride-1 block with residual
        {"name": "invres_s2_b32", "kind": "invres", "B": 32, "H": 112, "W": 112, "cin": 16, "cout": 24, "stride": 2},
        {"name": "invres_s1_b32", "kind": "invres", "B": 32, "H": 56, "W": 56, "cin": 24, "cout": 24, "stride": 1},
        # ViT-B/16's MLP at batch 32 (32 x 197 tokens: no multiple of a tile)
        {"name": "mlp_6304", "kind": "mlp", "M": 6304, "d": 768, "hidden": 3072},
        # the MLP sweep's down projection, block zeros: the zero-skip path
        {"name": "mlp_down_4096", "kind": "mlp_down", "M": 4096, "K": 3072, "N": 768, "rho": 0.7, "structure": "block32"},
        # one ViT-B/16 attention layer at batch 32
        {"name": "attn_b32", "kind": "attn", "B": 32, "T": 197, "heads": 12, "hd": 64},
        # ResNet-18's first-stage activation at batch 32 through the memory-bound operators
        {"name": "light_b32", "kind": "light", "B": 32, "H": 56, "W": 56, "C": 64},
        # one image through ResNet-18 (latency) and a batch of 8 through ViT-B/16
        {"name": "resnet18_b1", "kind": "net", "net": "resnet18", "B": 1, "depth": 0},
        {"name": "vit_b16_b8", "kind": "net", "net": "vit", "B": 8, "depth": 12},
    ]


def _log(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(step, int(round(v / step)) * step)


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["fc", "conv", "conv", "block", "stem", "invres", "invres", "mlp", "mlp_down", "attn", "light",
                       "net"])
    if kind == "fc":
        return {"kind": kind, "M": _log(rng, 1, 128), "K": _log(rng, 64, 2048, 8), "N": _log(rng, 64, 1024, 8),
                "f32": rng.random() < 0.5}
    if kind == "conv":
        B, H, cin = _log(rng, 1, 32), _log(rng, 7, 56), _log(rng, 16, 512, 8)
        if B * H * H * cin > 16_000_000:
            cin = 64
        if rng.random() < 0.4:
            cin = 64
        same = rng.random() < 0.4
        return {"kind": kind, "B": B, "H": H, "W": max(7, H + rng.choice([-2, -1, 0, 0, 3])), "cin": cin,
                "cout": cin if same else _log(rng, 16, 512, 8), "k": rng.choice([1, 3, 3]),
                "stride": rng.choice([1, 1, 2])}
    if kind == "block":
        c = rng.choice([64, 96, 128, 192, 256])
        return {"kind": kind, "B": _log(rng, 1, 16), "H": rng.randint(7, 56), "W": rng.randint(7, 56), "cin": c,
                "cout": 2 * c}
    if kind == "stem":
        return {"kind": kind, "B": _log(rng, 1, 32), "H": rng.randint(64, 224), "W": rng.randint(64, 224),
                "cout": rng.choice([32, 64, 64, 96]), "k": rng.choice([3, 7])}
    if kind == "invres":
        H = _log(rng, 7, 112)
        top = 32 if H > 56 else (96 if H > 28 else 160)
        cin = _log(rng, 16, top, 8)
        stride = rng.choice([1, 2])
        return {"kind": kind, "B": _log(rng, 1, 32), "H": H, "W": max(7, H + rng.choice([-1, 0, 0, 1])), "cin": cin,
                "cout": cin if stride == 1 and rng.random() < 0.6 else _log(rng, 16, top, 8), "stride": stride}
    if kind == "mlp":
        d = rng.choice([192, 384, 512, 768])
        return {"kind": kind, "M": _log(rng, 128, 6304), "d": d, "hidden": 4 * d}
    if kind == "mlp_down":
        return {"kind": kind, "M": _log(rng, 256, 4096), "K": _log(rng, 768, 3072, 32), "N": _log(rng, 192, 768, 8),
                "rho": round(rng.uniform(0.5, 0.95), 2), "structure": rng.choice(["block32", "block32", "unstructured",
                                                                                  "token"])}
    if kind == "attn":
        return {"kind": kind, "B": _log(rng, 1, 32), "T": rng.randint(50, 257), "heads": rng.choice([3, 6, 12]),
                "hd": rng.choice([32, 64, 64])}
    if kind == "light":
        return {"kind": kind, "B": _log(rng, 1, 32), "H": _log(rng, 7, 112), "W": _log(rng, 7, 112),
                "C": _log(rng, 16, 144, 8)}
    if rng.random() < 0.5:
        return {"kind": "net", "net": "resnet18", "B": rng.randint(1, 8), "depth": 0}
    return {"kind": "net", "net": "vit", "B": rng.randint(1, 8), "depth": rng.randint(1, 6)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class _Draw:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def normal(self, *shape, scale=1.0):
        return (torch.randn(*shape, generator=self.g, device="cuda") * scale).to(torch.bfloat16)

    def relu(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda").relu_().to(torch.bfloat16)

    def weight(self, cout, k, cin, gain=2.0):
        return self.normal(cout, k, k, cin, scale=math.sqrt(gain / (cin * k * k)))

    def bn(self, c):
        u, n = torch.rand(2, c, generator=self.g, device="cuda"), torch.randn(2, c, generator=self.g, device="cuda")
        return torch.stack([0.5 + u[0], 0.2 * n[0], 0.2 * n[1], 0.5 + u[1]]).contiguous()

    def bias(self, c):
        return 0.02 * torch.randn(c, generator=self.g, device="cuda")


def _new(*shape, dtype=torch.bfloat16):
    return torch.empty(*shape, dtype=dtype, device="cuda")


def _size(n, k, stride, pad):
    return (n + 2 * pad - k) // stride + 1


def prepare(case, seed):
    s = {"case": case, "ctx": _context()}
    s.update(_inputs(case, seed))
    kind = case["kind"]
    if kind == "fc":
        s["y"] = _new(case["M"], case["N"], dtype=torch.float32 if case["f32"] else torch.bfloat16)
    elif kind == "conv":
        B, k, st = case["B"], case["k"], case["stride"]
        Ho, Wo = _size(case["H"], k, st, k // 2), _size(case["W"], k, st, k // 2)
        s["y"] = _new(B, Ho, Wo, case["cout"])
        s["yo"] = sp.OccupancyBuffer(B * Ho * Wo, case["cout"])
    elif kind == "block":
        B, co = case["B"], case["cout"]
        Ho, Wo = _size(case["H"], 3, 2, 1), _size(case["W"], 3, 2, 1)
        for n in ("a", "sc", "y"):
            s[n] = _new(B, Ho, Wo, co)
        s["xo"] = sp.OccupancyBuffer(B * case["H"] * case["W"], case["cin"])
        s["ao"] = sp.OccupancyBuffer(B * Ho * Wo, co)
        s["yo"] = sp.OccupancyBuffer(B * Ho * Wo, co)
    elif kind == "stem":
        B, k, co = case["B"], case["k"], case["cout"]
        Ho, Wo = _size(case["H"], k, 2, k // 2), _size(case["W"], k, 2, k // 2)
        Hp, Wp = _size(Ho, 3, 2, 1), _size(Wo, 3, 2, 1)
        s["a"], s["y"] = _new(B, Ho, Wo, co), _new(B, Hp, Wp, co)
        s["ao"], s["yo"] = sp.OccupancyBuffer(B * Ho * Wo, co), sp.OccupancyBuffer(B * Hp * Wp, co)
    elif kind == "invres":
        B, hid, co = case["B"], 6 * case["cin"], case["cout"]
        H, W = case["H"], case["W"]
        Ho, Wo = _size(H, 3, case["stride"], 1), _size(W, 3, case["stride"], 1)
        s["a"], s["b"], s["y"] = _new(B, H, W, hid), _new(B, Ho, Wo, hid), _new(B, Ho, Wo, co)
        s["xo"] = sp.OccupancyBuffer(B * H * W, case["cin"])
        s["ao"] = sp.OccupancyBuffer(B * H * W, hid)
        s["bo"] = sp.OccupancyBuffer(B * Ho * Wo, hid)
        s["yo"] = sp.OccupancyBuffer(B * Ho * Wo, co)
    elif kind == "mlp":
        s["h"], s["y"] = _new(case["M"], case["hidden"]), _new(case["M"], case["d"])
        s["ho"] = sp.OccupancyBuffer(case["M"], case["hidden"])
    elif kind == "mlp_down":
        s["y"] = _new(case["M"], case["N"])
        s["yo"] = sp.OccupancyBuffer(case["M"], case["N"])
    elif kind == "attn":
        B, T, D = case["B"], case["T"], case["heads"] * case["hd"]
        s["n"], s["qkv"], s["a"], s["y"] = _new(B * T, D), _new(B * T, 3 * D), _new(B * T, D), _new(B * T, D)
        s["no"], s["ao"] = sp.OccupancyBuffer(B * T, D), sp.OccupancyBuffer(B * T, D)
    elif kind == "light":
        B, H, W, C = case["B"], case["H"], case["W"], case["C"]
        s["y"], s["z"] = _new(B, H, W, C), _new(B, C)
        s["xo"], s["yo"] = sp.OccupancyBuffer(B * H * W, C), sp.OccupancyBuffer(B * H * W, C)
        s["zo"] = sp.OccupancyBuffer(B, C)
    else:
        s["y"] = _new(case["B"], 1000)
        s["graph"] = sp.Graph(s["ops"])
    if "xo" in s and kind != "light":  # the producer of x measured it
        sp.sparoa_op_stats(s["ctx"], s["x"], tuple(s["x"].shape), occ=s["xo"], host=False)
    return s


def _inputs(case, seed):
    d, kind = _Draw(seed), case["kind"]
    if kind == "fc":
        M, K, N = case["M"], case["K"], case["N"]
        x = d.relu(M, K) * (torch.rand(K, generator=d.g, device="cuda") >= 0.4)
        w = d.normal(N, K, scale=math.sqrt(1.0 / K))
        return {"x": x, "w": w, "wkn": w.t().contiguous(), "bias": d.bias(N)}
    if kind == "conv":
        B, H, W, ci, co, k = (case[n] for n in ("B", "H", "W", "cin", "cout", "k"))
        return {"x": d.relu(B, H, W, ci), "w": d.weight(co, k, ci), "bn": d.bn(co)}
    if kind == "block":
        ci, co = case["cin"], case["cout"]
        return {"x": d.relu(case["B"], case["H"], case["W"], ci), "w1": d.weight(co, 3, ci), "w2": d.weight(co, 3, co),
                "ws": d.weight(co, 1, ci), "bn1": d.bn(co), "bn2": d.bn(co), "bns": d.bn(co)}
    if kind == "stem":
        co = case["cout"]
        return {"x": d.normal(case["B"], case["H"], case["W"], 3), "w": d.weight(co, case["k"], 3), "bn": d.bn(co)}
    if kind == "invres":
        ci, co, hid = case["cin"], case["cout"], 6 * case["cin"]
        return {"x": d.normal(case["B"], case["H"], case["W"], ci), "w1": d.weight(hid, 1, ci),
                "wd": d.normal(hid, 3, 3, 1, scale=math.sqrt(2.0 / 9)), "w2": d.weight(co, 1, hid), "bn1": d.bn(hid),
                "bnd": d.bn(hid), "bn2": d.bn(co)}
    if kind == "mlp":
        M, D, h = case["M"], case["d"], case["hidden"]
        return {"x": d.normal(M, D), "r": d.normal(M, D), "w1": d.normal(h, D, scale=math.sqrt(1.0 / D)),
                "w2": d.normal(D, h, scale=math.sqrt(1.0 / h)), "b1": d.bias(h), "b2": d.bias(D)}
    if kind == "mlp_down":
        M, K, N, rho = case["M"], case["K"], case["N"], case["rho"]
        v = torch.randn(M, K, generator=d.g, device="cuda").abs_() + 1e-3
        if case["structure"] == "block32":
            keep = torch.rand((M + 127) // 128, (K + 31) // 32, generator=d.g, device="cuda") >= rho
            keep = keep.repeat_interleave(128, 0)[:M].repeat_interleave(32, 1)[:, :K]
        elif case["structure"] == "token":
            keep = torch.rand(M, 1, generator=d.g, device="cuda") >= rho
        else:
            keep = torch.rand(M, K, generator=d.g, device="cuda") >= rho
        return {"x": (v * keep).to(torch.bfloat16), "w": d.normal(N, K, scale=math.sqrt(2.0 / K)), "bias": d.bias(N)}
    if kind == "attn":
        D = case["heads"] * case["hd"]
        gb = torch.stack([1.0 + 0.1 * torch.randn(D, generator=d.g, device="cuda"), d.bias(D)]).contiguous()
        return {"x": d.normal(case["B"] * case["T"], D), "gb": gb, "wq": d.normal(3 * D, D, scale=math.sqrt(1.0 / D)),
                "wp": d.normal(D, D, scale=math.sqrt(1.0 / D)), "bq": d.bias(3 * D), "bp": d.bias(D)}
    if kind == "light":
        return {"x": d.normal(case["B"], case["H"], case["W"], case["C"]), "bn": d.bn(case["C"])}
    if case["net"] == "resnet18":
        ops, bits, shape = synth.resnet18(batch=case["B"], seed=seed)
    else:
        ops, bits, shape = synth.vit(batch=case["B"], seed=seed, depth=case["depth"])
    return {"ops": ops, "x": sp.bits_to_device(bits).view(*shape)}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c, kind, ctx = s["case"], s["case"]["kind"], s["ctx"]
    if kind == "fc":
        sp.sparoa_gemm(ctx, s["x"], s["w"], s["y"], W_kn=s["wkn"], bias=s["bias"])
        return {"y": s["y"]}
    if kind == "conv":
        sp.sparoa_conv2d(ctx, s["x"], s["w"], s["y"], stride=c["stride"], pad=c["k"] // 2, bn=s["bn"],
                         act=sp.ACT_RELU, y_occ=s["yo"])
        return {"y": s["y"], "occ": s["yo"].buf}
    if kind == "block":
        sp.sparoa_conv2d(ctx, s["x"], s["w1"], s["a"], stride=2, pad=1, bn=s["bn1"], act=sp.ACT_RELU, x_occ=s["xo"],
                         y_occ=s["ao"])
        sp.sparoa_conv2d(ctx, s["x"], s["ws"], s["sc"], stride=2, pad=0, bn=s["bns"], x_occ=s["xo"])
        sp.sparoa_conv2d(ctx, s["a"], s["w2"], s["y"], stride=1, pad=1, bn=s["bn2"], act=sp.ACT_RELU,
                         residual=s["sc"], x_occ=s["ao"], y_occ=s["yo"])
        return {"a": s["a"], "sc": s["sc"], "y": s["y"], "occ": s["yo"].buf}
    if kind == "stem":
        sp.sparoa_conv2d(ctx, s["x"], s["w"], s["a"], stride=2, pad=c["k"] // 2, bn=s["bn"], act=sp.ACT_RELU,
                         y_occ=s["ao"])
        sp.sparoa_maxpool2d(ctx, s["a"], s["y"], 3, 2, 1, y_occ=s["yo"])
        return {"a": s["a"], "a_occ": s["ao"].buf, "y": s["y"], "occ": s["yo"].buf}
    if kind == "invres":
        sp.sparoa_conv2d(ctx, s["x"], s["w1"], s["a"], bn=s["bn1"], act=sp.ACT_RELU6, x_occ=s["xo"], y_occ=s["ao"])
        sp.sparoa_conv2d(ctx, s["a"], s["wd"], s["b"], stride=c["stride"], pad=1, groups=6 * c["cin"], bn=s["bnd"],
                         act=sp.ACT_RELU6, x_occ=s["ao"], y_occ=s["bo"])
        sp.sparoa_conv2d(ctx, s["b"], s["w2"], s["y"], bn=s["bn2"], x_occ=s["bo"], y_occ=s["yo"],
                         residual=s["x"] if _skips(c) else None)
        return {"a": s["a"], "a_occ": s["ao"].buf, "b": s["b"], "b_occ": s["bo"].buf, "y": s["y"], "occ": s["yo"].buf}
    if kind == "mlp":
        sp.sparoa_gemm(ctx, s["x"], s["w1"], s["h"], bias=s["b1"], act=sp.ACT_GELU, y_occ=s["ho"])
        sp.sparoa_gemm(ctx, s["h"], s["w2"], s["y"], bias=s["b2"], residual=s["r"], x_occ=s["ho"])
        return {"h": s["h"], "h_occ": s["ho"].buf, "y": s["y"]}
    if kind == "mlp_down":
        sp.sparoa_gemm(ctx, s["x"], s["w"], s["y"], bias=s["bias"], y_occ=s["yo"])
        return {"y": s["y"], "occ": s["yo"].buf}
    if kind == "attn":
        B, T, D = c["B"], c["T"], c["heads"] * c["hd"]
        sp.sparoa_layernorm(ctx, s["x"], s["n"], gamma_beta=s["gb"], y_occ=s["no"])
        sp.sparoa_gemm(ctx, s["n"], s["wq"], s["qkv"], bias=s["bq"], x_occ=s["no"])
        sp.sparoa_attention(ctx, s["qkv"].view(B, T, 3 * D), s["a"], c["heads"], y_occ=s["ao"])
        sp.sparoa_gemm(ctx, s["a"], s["wp"], s["y"], bias=s["bp"], residual=s["x"], x_occ=s["ao"])
        return {"n": s["n"], "qkv": s["qkv"], "a": s["a"], "a_occ": s["ao"].buf, "y": s["y"]}
    if kind == "light":
        sp.sparoa_op_stats(ctx, s["x"], tuple(s["x"].shape), occ=s["xo"], host=False)
        sp.sparoa_bn_act(ctx, s["x"], s["y"], bn=s["bn"], act=sp.ACT_RELU, y_occ=s["yo"])
        sp.sparoa_avgpool_global(ctx, s["y"], s["z"], y_occ=s["zo"])
        return {"x_occ": s["xo"].buf, "y": s["y"], "occ": s["yo"].buf, "z": s["z"]}
    sp.sparoa_run_graph(ctx, s["graph"], s["x"], s["y"])
    return {"logits": s["y"]}


def _skips(c):
    return c["stride"] == 1 and c["cin"] == c["cout"]


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------
def _occ_bytes(R, C):
    T = (C + 63) // 64
    return 8 + 4 * C + 4 * T + 8 * R * ((T + 63) // 64) + 4 * ((R + 127) // 128) * ((C + 31) // 32)


def _conv_w(R, Ro, ci, co, k):
    """bytes (input, weights, BN, output, output occupancy) and FLOPs of one dense convolution"""
    return 2 * (R * ci + co * k * k * ci + Ro * co) + 16 * co + _occ_bytes(Ro, co), 2 * Ro * co * k * k * ci


def work(case):
    kind = case["kind"]
    if kind == "fc":
        M, K, N = case["M"], case["K"], case["N"]
        return {"bytes": 2 * (M * K + N * K) + 4 * N + M * N * (4 if case["f32"] else 2), "flops": 2 * M * N * K}
    if kind == "conv":
        k, st = case["k"], case["stride"]
        Ro = case["B"] * _size(case["H"], k, st, k // 2) * _size(case["W"], k, st, k // 2)
        b, f = _conv_w(case["B"] * case["H"] * case["W"], Ro, case["cin"], case["cout"], k)
        return {"bytes": b, "flops": f}
    if kind == "block":
        ci, co, R = case["cin"], case["cout"], case["B"] * case["H"] * case["W"]
        Ro = case["B"] * _size(case["H"], 3, 2, 1) * _size(case["W"], 3, 2, 1)
        b1, f1 = _conv_w(R, Ro, ci, co, 3)
        b2, f2 = _conv_w(Ro, Ro, co, co, 3)
        return {"bytes": b1 + b2 + 2 * (ci * co + 2 * Ro * co), "flops": f1 + f2 + 2 * Ro * ci * co}
    if kind == "stem":
        B, k, co = case["B"], case["k"], case["cout"]
        Ho, Wo = _size(case["H"], k, 2, k // 2), _size(case["W"], k, 2, k // 2)
        Rp = B * _size(Ho, 3, 2, 1) * _size(Wo, 3, 2, 1)
        b, f = _conv_w(B * case["H"] * case["W"], B * Ho * Wo, 3, co, k)
        return {"bytes": b + 2 * (B * Ho * Wo + Rp) * co + _occ_bytes(Rp, co), "flops": f}
    if kind == "invres":
        ci, co, hid, R = case["cin"], case["cout"], 6 * case["cin"], case["B"] * case["H"] * case["W"]
        Ro = case["B"] * _size(case["H"], 3, case["stride"], 1) * _size(case["W"], 3, case["stride"], 1)
        b1, f1 = _conv_w(R, R, ci, hid, 1)
        b2, f2 = _conv_w(Ro, Ro, hid, co, 1)
        bd = 2 * (R + Ro + 9) * hid + 16 * hid + _occ_bytes(Ro, hid)
        return {"bytes": b1 + b2 + bd + (2 * R * ci if _skips(case) else 0), "flops": f1 + f2 + 18 * Ro * hid}
    if kind == "mlp":
        M, D, h = case["M"], case["d"], case["hidden"]
        return {"bytes": 2 * (3 * M * D + 2 * M * h + 2 * D * h) + _occ_bytes(M, h), "flops": 4 * M * D * h}
    if kind == "mlp_down":
        M, K, N = case["M"], case["K"], case["N"]
        kept = 1.0 - case["rho"] if case["structure"] != "unstructured" else 1.0
        return {"bytes": 2 * (M * K + N * K + M * N) + _occ_bytes(M, N), "flops": 2 * M * N * K * kept}
    if kind == "attn":
        B, T, D = case["B"], case["T"], case["heads"] * case["hd"]
        R = B * T
        return {"bytes": 2 * R * D * (2 + 4 + 4 + 3) + 2 * 4 * D * D + 2 * _occ_bytes(R, D),
                "flops": 8 * R * D * D + 4 * B * T * T * D}
    if kind == "light":
        R, C = case["B"] * case["H"] * case["W"], case["C"]
        return {"bytes": 8 * R * C + 2 * case["B"] * C + 2 * _occ_bytes(R, C), "flops": 3 * R * C}
    if case["net"] == "resnet18":
        return {"bytes": 2 * 11_690_000 + case["B"] * 2 * 2 * 2_480_000, "flops": case["B"] * 2 * 1.814e9}
    L, B, D = case["depth"], case["B"], 768
    R = 197 * B
    per = 2 * R * D * (2 * 2 + 4 + 4 + 3 + 5 + 6) + 2 * 12 * D * D
    fl = 24 * R * D * D + 4 * B * 197 * 197 * D
    return {"bytes": L * per + 2 * 2 * D * D + B * 600_000, "flops": L * fl + 2 * B * 196 * D * D}


def tolerance(case):
    """About four times the distance from the 64-bit computation, which is the
    rounding of the bf16 outputs (2^-9 each) and, across calls, of the bf16
    tensors between them.  ``differ`` covers occupancy bytes: a value that
    rounds to either side of zero changes one bit or count."""
    if case["kind"] == "fc" and case["f32"]:  # fp32 out: the order of the sums (7e-8 seen)
        return {"rel": 2e-6, "max": 2e-5}
    if case["kind"] == "net":  # logits behind 20 (3e-3 seen) or 50 (1e-2 seen) bf16 operators
        return {"rel": 0.012, "max": 0.12} if case["net"] == "resnet18" else {"rel": 0.03, "max": 0.3}
    return {"rel": 8e-3, "max": 0.1, "differ": 2e-3}  # 1.6e-3 to 2.1e-3 seen


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _d(t):
    return t.double()


def _bf(t):
    return t.to(torch.bfloat16)


def _norm(v, bn):
    g, b, m, var = bn.double()
    return (v - m) * (g / torch.sqrt(var + 1e-5)) + b


def _conv64(x, w, stride, pad):
    """x [B, H, W, C], w [O, k, k, C] -> [B, Ho, Wo, O] in float64, a few images at a time"""
    O, k, _, C = w.shape
    B, H, W, _ = x.shape
    Ho, Wo = _size(H, k, stride, pad), _size(W, k, stride, pad)
    wm = w.double().permute(0, 3, 1, 2).reshape(O, C * k * k)
    out = torch.empty(B, Ho, Wo, O, dtype=torch.float64, device=x.device)
    step = max(1, int(6e7 // max(1, C * k * k * Ho * Wo)))
    for b in range(0, B, step):
        xi = x[b:b + step].double().permute(0, 3, 1, 2)
        cols = xi[:, :, ::stride, ::stride].reshape(xi.shape[0], C, -1) if k == 1 and pad == 0 else \
            torch.nn.functional.unfold(xi, k, padding=pad, stride=stride)
        out[b:b + step] = (wm @ cols).transpose(1, 2).reshape(-1, Ho, Wo, O)
    return out


def _dw64(x, w, stride):
    B, H, W, C = x.shape
    xp = torch.nn.functional.pad(_d(x), (0, 0, 1, 1, 1, 1))
    Ho, Wo = _size(H, 3, stride, 1), _size(W, 3, stride, 1)
    out = 0.0
    for r in range(3):
        for q in range(3):
            out = out + xp[:, r:r + (Ho - 1) * stride + 1:stride, q:q + (Wo - 1) * stride + 1:stride] * _d(w[:, r, q, 0])
    return out


def _pool64(x):
    v = torch.nn.functional.max_pool2d(_d(x).permute(0, 3, 1, 2), 3, 2, 1)
    return v.permute(0, 2, 3, 1).contiguous()


def _gelu64(v):
    return torch.nn.functional.gelu(v, approximate="tanh")


def _ln64(x, gb, eps):
    x = _d(x)
    m = x.mean(-1, keepdim=True)
    v = ((x - m) ** 2).mean(-1, keepdim=True)
    return (x - m) / torch.sqrt(v + eps) * gb[0].double() + gb[1].double()


def _attn64(qkv, B, T, heads, hd):
    q, k, v = _d(qkv).view(B, T, 3, heads, hd).permute(2, 0, 3, 1, 4)
    p = torch.softmax(q @ k.transpose(-1, -2) / math.sqrt(hd), -1)
    return (p @ v).permute(0, 2, 1, 3).reshape(B * T, heads * hd)


def exact(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    if kind == "fc":
        return {"y": _d(s["x"]) @ _d(s["w"]).t() + s["bias"].double()}
    if kind == "conv":
        y = _norm(_conv64(s["x"], s["w"], case["stride"], case["k"] // 2), s["bn"]).relu()
        return {"y": y, "occ": None}
    if kind == "block":
        a = _norm(_conv64(s["x"], s["w1"], 2, 1), s["bn1"]).relu()
        sc = _norm(_conv64(s["x"], s["ws"], 2, 0), s["bns"])
        y = (_norm(_conv64(_bf(a), s["w2"], 1, 1), s["bn2"]) + _d(_bf(sc))).relu()
        return {"a": a, "sc": sc, "y": y, "occ": None}
    if kind == "stem":
        a = _norm(_conv64(s["x"], s["w"], 2, case["k"] // 2), s["bn"]).relu()
        return {"a": a, "a_occ": None, "y": _pool64(_bf(a)), "occ": None}
    if kind == "invres":
        a = _norm(_conv64(s["x"], s["w1"], 1, 0), s["bn1"]).clamp(0, 6)
        b = _norm(_dw64(_bf(a), s["wd"], case["stride"]), s["bnd"]).clamp(0, 6)
        y = _norm(_conv64(_bf(b), s["w2"], 1, 0), s["bn2"])
        if _skips(case):
            y = y + _d(s["x"])
        return {"a": a, "a_occ": None, "b": b, "b_occ": None, "y": y, "occ": None}
    if kind == "mlp":
        h = _gelu64(_d(s["x"]) @ _d(s["w1"]).t() + s["b1"].double())
        y = _d(_bf(h)) @ _d(s["w2"]).t() + s["b2"].double() + _d(s["r"])
        return {"h": h, "h_occ": None, "y": y}
    if kind == "mlp_down":
        return {"y": _d(s["x"]) @ _d(s["w"]).t() + s["bias"].double(), "occ": None}
    if kind == "attn":
        n = _ln64(s["x"], s["gb"], 1e-6)
        qkv = _d(_bf(n)) @ _d(s["wq"]).t() + s["bq"].double()
        a = _attn64(_bf(qkv), case["B"], case["T"], case["heads"], case["hd"])
        y = _d(_bf(a)) @ _d(s["wp"]).t() + s["bp"].double() + _d(s["x"])
        return {"n": n, "qkv": qkv, "a": a, "a_occ": None, "y": y}
    if kind == "light":
        y = _norm(_d(s["x"]), s["bn"]).relu()
        return {"x_occ": None, "y": y, "occ": None, "z": _d(_bf(y)).mean((1, 2))}
    return {"logits": _net64(s["ops"], s["x"])}


def _net64(ops, x):
    """The operator list in float64, every value between operators rounded to bf16."""
    def dev(a):
        return torch.from_numpy(a).cuda()

    vals = [x]
    for op in ops:
        v, kind = vals[op["input"]], op["kind"]
        if kind == "conv":
            w = sp.bits_to_device(op["w"]).view(op["cout"], op["k"], op["k"], -1)
            r = _conv64(v, w, op["stride"], op["pad"])
        elif kind == "fc":
            r = _d(v).reshape(v.shape[0], -1) @ _d(sp.bits_to_device(op["w"]).view(op["cout"], -1)).t()
        elif kind == "maxpool":
            r = _pool64(v)
        elif kind == "avgpool":
            r = _d(v).mean((1, 2))
        elif kind == "layernorm":
            r = _ln64(v, dev(op["gamma_beta"]), 1e-5)  # the graph's eps field
        elif kind == "attention":
            B, T = v.shape[0], v.shape[1] * v.shape[2]
            r = _attn64(v.reshape(B * T, -1), B, T, op["heads"], v.shape[3] // 3 // op["heads"]).view(B, 1, T, -1)
        elif kind == "tokens":
            B, D = v.shape[0], v.shape[3]
            cls = _d(sp.bits_to_device(op["cls"])).view(1, 1, D).expand(B, 1, D)
            r = (torch.cat([cls, _d(v).reshape(B, -1, D)], 1) + dev(op["pos"]).double()).unsqueeze(1)
        else:  # select
            r = _d(v).reshape(v.shape[0], -1, v.shape[3])[:, op["index"]].view(v.shape[0], 1, 1, -1)
        if op.get("bias") is not None:
            r = r + dev(op["bias"]).double()
        if op.get("bn") is not None:
            r = _norm(r, dev(op["bn"]))
        if op.get("residual", -1) >= 0:
            r = r + _d(vals[op["residual"]])
        act = op.get("act", 0)
        r = r.relu() if act == 1 else r.clamp(0, 6) if act == 2 else _gelu64(r) if act == 3 else r
        vals.append(_bf(r))
    return r.reshape(x.shape[0], -1)
