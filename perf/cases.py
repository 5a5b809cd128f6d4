"""The calls by which this library's speed is measured.

Every case is work that a program around the library has it do through the
Python binding (paper_2609_34867_gb300.p4q): the visual-token selector between
the vision projector and the language model, the W4A4 linears of prefill and
decode, and the fused quantizers and the attention between them. The sizes are
those of the LLaVA-shaped workloads (workloads.py): one image or a batch, 576
tokens per image or five crops of 576, the 7B (4096 / 11008) and 13B (5120 /
13824) decoders; `draw` takes odd sizes from the same ranges.
"""
import math

import torch

from paper_2609_34867_gb300 import p4q
from paper_2609_34867_gb300 import workloads as wl

EPS = 1e-5  # RMSNorm epsilon of the decoders


def listed():
    return [
        # One decode step of one sequence through a 7B decoder layer: the four
        # fused linears with the norms and quantizers before them (down on the
        # re-quantized up block, the benchmark's dataflow), replayed as a CUDA
        # graph as decode loops are (latency and launches count).
        {"name": "decode-7b", "kind": "decode", "rows": 1, "d": 4096, "ffn": 11008},
        # The same for 24 sequences decoded together on the 13B decoder.
        {"name": "decode-13b-batch24", "kind": "decode", "rows": 24, "d": 5120, "ffn": 13824},
        # Prefill of one pruned image (64 kept tokens + 32 text tokens): one
        # projection with the quantizer of its input.
        {"name": "linear-one-image", "kind": "linear", "M": 96, "Kin": 4096, "N": 4096, "ws": False},
        # Prefill of 8 pruned LLaVA-1.5 images: an MLP projection, packed
        # weights resident, with a workspace.
        {"name": "linear-7b-b8", "kind": "linear", "M": 2048, "Kin": 4096, "N": 11008, "ws": True},
        # Prefill of 32 pruned LLaVA-NeXT images on the 13B decoder: the up
        # projection whose output the next linear's quantizer takes in one
        # pass (row maxima from the GEMM).
        {"name": "mlp-up-13b-b32", "kind": "chain", "M": 22528, "Kin": 5120, "N": 13824},
        # Input norm of a decoder layer with the quantizer of q/k/v, prefill.
        {"name": "rmsnorm-7b-b8", "kind": "rmsnorm", "M": 2048, "Kin": 4096},
        # SwiGLU of a fused gate|up output with the quantizer of down, prefill
        # of 16 pruned LLaVA-NeXT images.
        {"name": "swiglu-7b-b16", "kind": "swiglu", "M": 6144, "Kin": 11008},
        # The selector for one LLaVA-1.5 image (an interactive request).
        {"name": "select-one-image", "kind": "select", "B": 1, "N": 576, "d": 4096, "K": 64, "T": 32, "J": 3,
         "tower": False, "heavy": False},
        # The selector for a batch of LLaVA-1.5 images, the saliency taken
        # from the vision tower's final layer.
        {"name": "select-15-b8", "kind": "select", "B": 8, "N": 576, "d": 4096, "K": 192, "T": 64, "J": 3,
         "tower": True, "heavy": False},
        # The selector for a large batch of five-crop LLaVA-NeXT images on
        # heavy-tailed 13B features.
        {"name": "select-next-13b-b32", "kind": "select", "B": 32, "N": 2880, "d": 5120, "K": 640, "T": 64, "J": 3,
         "tower": False, "heavy": True},
        # Prefill attention on the pruned sequences, q|k|v one fused output.
        {"name": "attention-7b-b8", "kind": "attention", "B": 8, "m": 256, "H": 32, "Hkv": 32},
        {"name": "attention-13b-b32", "kind": "attention", "B": 32, "m": 704, "H": 40, "Hkv": 40},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("decode", "linear", "linear", "chain", "rmsnorm", "swiglu", "select", "select", "attention",
                       "attention"))
    d, ffn = rng.choice(((4096, 11008), (5120, 13824)))
    if kind == "decode":  # decode batches
        return {"kind": kind, "rows": _log_int(rng, 2, 64), "d": d, "ffn": ffn}
    if kind == "linear":  # prefill linears, every shape of the decoders, ragged row counts
        kin, n = rng.choice(wl.SWEEP_KN)
        m = _log_int(rng, 9, 8192)
        return {"kind": kind, "M": m, "Kin": kin, "N": n, "ws": rng.random() < 0.6}
    if kind == "chain":
        return {"kind": kind, "M": _log_int(rng, 256, 16384), "Kin": d, "N": ffn}
    if kind == "rmsnorm":
        return {"kind": kind, "M": _log_int(rng, 1, 16384), "Kin": d}
    if kind == "swiglu":
        return {"kind": kind, "M": _log_int(rng, 1, 6144), "Kin": ffn}
    if kind == "select":
        # whole crops or (images of other aspect ratios) any number of tokens
        n = 576 * rng.randint(1, 5) if rng.random() < 0.6 else rng.randint(200, 2880)
        b = _log_int(rng, 1, 16)
        tower = n % 576 == 0 and b * n <= 8 * 576 and rng.random() < 0.5
        return {"kind": kind, "B": b, "N": n, "d": d, "K": max(1, round(n * rng.uniform(0.05, 0.4))),
                "T": rng.randint(0, 96), "J": rng.randint(0, 5), "tower": tower, "heavy": rng.random() < 0.3}
    h = rng.choice((32, 40))
    return {"kind": kind, "B": _log_int(rng, 1, 32), "m": _log_int(rng, 33, 704), "H": h,
            "Hkv": rng.choice((h, h, 8))}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _gain(d, heavy):
    return torch.from_numpy(wl.channel_gain(d, heavy)).cuda()


def _features(g, shape, d, heavy=False):
    x = torch.randn(tuple(shape) + (d,), generator=g, device="cuda", dtype=torch.float32)
    return x.mul_(_gain(d, heavy)).half()


def _weight(g, n, kin):
    w = (torch.randn((n, kin), generator=g, device="cuda", dtype=torch.float32) * 0.02).half()
    return p4q.quant_weight(w)


def _codes_out(M, kin, expanded):
    o = {"q": torch.empty((M, kin // 2), dtype=torch.uint8, device="cuda"),
         "s": torch.empty((M,), dtype=torch.float32, device="cuda"), "u": None, "su": None}
    if expanded:
        o["u"] = torch.empty((M, kin), dtype=torch.uint8, device="cuda")
        o["su"] = torch.empty((M,), dtype=torch.int32, device="cuda")
    return o


def _half(*shape):
    return torch.empty(shape, dtype=torch.float16, device="cuda")


def _decode_inputs(c, seed):
    g, d, f, m = _gen(seed), c["d"], c["ffn"], c["rows"]
    s = {"x1": _features(g, (m,), d), "x2": _features(g, (m,), d), "a": _features(g, (m,), d),
         "w1": (1 + 0.1 * torch.randn((d,), generator=g, device="cuda")).half(),
         "w2": (1 + 0.1 * torch.randn((d,), generator=g, device="cuda")).half()}
    for name, n, k in (("qkv", 3 * d, d), ("o", d, d), ("gu", 2 * f, d), ("down", d, f)):
        s["W" + name] = _weight(g, n, k)
    return s


def _decode_calls(s):
    f = s["f"]
    p4q.p4q_rmsnorm_quant_expanded(s["x1"], s["w1"], EPS, s["c1"]["q"], s["c1"]["s"])
    p4q.p4q_w4a4_linear(s["c1"]["q"], s["c1"]["s"], *s["Wqkv"], s["Yqkv"])
    p4q.p4q_quant_act(s["a"], s["c2"]["q"], s["c2"]["s"])
    p4q.p4q_w4a4_linear(s["c2"]["q"], s["c2"]["s"], *s["Wo"], s["Yo"])
    p4q.p4q_rmsnorm_quant_expanded(s["x2"], s["w2"], EPS, s["c3"]["q"], s["c3"]["s"])
    p4q.p4q_w4a4_linear(s["c3"]["q"], s["c3"]["s"], *s["Wgu"], s["Ygu"])
    p4q.p4q_quant_act_ld(s["Ygu"][:, f:], s["c4"]["q"], s["c4"]["s"])
    p4q.p4q_w4a4_linear(s["c4"]["q"], s["c4"]["s"], *s["Wdown"], s["Ydown"])


def _select_inputs(c, seed):
    g, B, N, d = _gen(seed), c["B"], c["N"], c["d"]
    s = {"V": _features(g, (B, N), d, c["heavy"]), "Q": None, "A": None, "text": None}
    if c["J"]:
        rows = torch.randint(0, N, (B, c["J"]), generator=g, device="cuda")
        base = torch.gather(s["V"], 1, rows[:, :, None].expand(-1, -1, d)).float()
        s["Q"] = (base + 0.5 * torch.randn(base.shape, generator=g, device="cuda")).half()
    if c["T"]:
        s["text"] = torch.randn((B, c["T"], d), generator=g, device="cuda").half()
    if c["tower"]:
        C, H, dh = N // wl.CROP, wl.VIT_HEADS, wl.VIT_HEAD_DIM
        s["qc"] = (2 * torch.randn((B, C, H, dh), generator=g, device="cuda")).half()
        s["kc"] = torch.randn((B, C, H, dh), generator=g, device="cuda").half()
        s["k"] = torch.randn((B, N, H, dh), generator=g, device="cuda").half()
    else:
        z = 2 * torch.randn((B, N), generator=g, device="cuda")
        s["A"] = torch.cat([torch.softmax(t, 1) for t in z.split(wl.CROP, 1)], 1).contiguous()
    return s


def _attention_inputs(c, seed):
    n = (c["H"] + 2 * c["Hkv"]) * 128
    qkv = torch.randn((c["B"] * c["m"], n), generator=_gen(seed), device="cuda").half()
    h, hk = c["H"] * 128, c["Hkv"] * 128
    return qkv[:, :h], qkv[:, h:h + hk], qkv[:, h + hk:]


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"kind": kind}
    if kind == "decode":
        m, d, f = c["rows"], c["d"], c["ffn"]
        s.update(_decode_inputs(c, seed), f=f)
        for i, k in (("c1", d), ("c2", d), ("c3", d), ("c4", f)):
            s[i] = _codes_out(m, k, False)
        s.update(Yqkv=_half(m, 3 * d), Yo=_half(m, d), Ygu=_half(m, 2 * f), Ydown=_half(m, d))
        _decode_calls(s)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _decode_calls(s)
    elif kind == "linear":
        g = _gen(seed)
        s["X"] = _features(g, (c["M"],), c["Kin"])
        s["W"] = _weight(g, c["N"], c["Kin"])
        s["c"] = _codes_out(c["M"], c["Kin"], False)
        s["Y"] = _half(c["M"], c["N"])
        s["ws"] = p4q.linear_workspace(c["M"], c["N"], c["Kin"], "cuda") if c["ws"] else None
    elif kind == "chain":
        g, M, N = _gen(seed), c["M"], c["N"]
        X = _features(g, (M,), c["Kin"])
        s["x"] = _codes_out(M, c["Kin"], True)
        p4q.p4q_quant_act_expanded(X, s["x"]["q"], s["x"]["s"], s["x"]["u"], s["x"]["su"])
        s["W"] = _weight(g, N, c["Kin"])
        s["Wu"] = torch.empty((N, c["Kin"]), dtype=torch.uint8, device="cuda")
        s["Wsu"] = torch.empty((N,), dtype=torch.int32, device="cuda")
        s["Y"], s["c"] = _half(M, N), _codes_out(M, N, True)
        s["rm"] = torch.empty((1, M), dtype=torch.int32, device="cuda")
    elif kind == "rmsnorm":
        g = _gen(seed)
        s["X"] = _features(g, (c["M"],), c["Kin"])
        s["w"] = (1 + 0.1 * torch.randn((c["Kin"],), generator=g, device="cuda")).half()
        s["c"] = _codes_out(c["M"], c["Kin"], True)
    elif kind == "swiglu":
        s["gu"] = torch.randn((c["M"], 2 * c["Kin"]), generator=_gen(seed), device="cuda").half()
        s["c"] = _codes_out(c["M"], c["Kin"], True)
    elif kind == "select":
        B, N, d, K, M = c["B"], c["N"], c["d"], c["K"], c["B"] * (c["K"] + c["T"])
        s.update(_select_inputs(c, seed), K=K)
        if c["tower"]:
            s["A"] = torch.empty((B, N), dtype=torch.float32, device="cuda")
        s["idx"] = torch.empty((B, K), dtype=torch.int32, device="cuda")
        s["X"], s["c"] = _half(B, K + c["T"], d), _codes_out(M, d, False)
        s["ws"] = p4q.select_workspace(B, N, d, c["J"], K, "cuda")
    else:
        s["q"], s["k"], s["v"] = _attention_inputs(c, seed)
        s["o"] = _half(c["B"] * c["m"], c["H"] * 128)
        s["args"] = (c["B"], c["m"], c["H"], c["Hkv"])
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "decode":
        s["graph"].replay()
        return {"qkv": s["Yqkv"], "o": s["Yo"], "gu": s["Ygu"], "down": s["Ydown"]}
    if kind == "linear":
        c = s["c"]
        p4q.p4q_quant_act(s["X"], c["q"], c["s"])
        p4q.p4q_w4a4_linear_ws(c["q"], c["s"], *s["W"], s["Y"], s["ws"])
        return {"q": c["q"], "s": c["s"], "Y": s["Y"]}
    if kind == "chain":
        x, c = s["x"], s["c"]
        n = s["Y"].shape[1]
        p4q.p4q_expand_codes(s["W"][0], s["Wu"], s["Wsu"])
        p4q.p4q_w4a4_linear_expanded_rowmax(x["u"], x["su"], x["s"], s["Wu"], s["Wsu"], s["W"][1], s["Y"], [(0, n)],
                                            s["rm"])
        p4q.p4q_quant_act_expanded_rowmax(s["Y"], [(0, n)], s["rm"], None, [c["s"]], [c["u"]], [c["su"]])
        return {"Y": s["Y"], "s": c["s"], "u": c["u"], "su": c["su"]}
    if kind == "rmsnorm":
        c = s["c"]
        p4q.p4q_rmsnorm_quant_expanded(s["X"], s["w"], EPS, c["q"], c["s"], c["u"], c["su"])
        return c
    if kind == "swiglu":
        c, f = s["c"], s["gu"].shape[1] // 2
        p4q.p4q_swiglu_quant_expanded(s["gu"][:, :f], s["gu"][:, f:], c["q"], c["s"], c["u"], c["su"])
        return c
    if kind == "select":
        c = s["c"]
        if "k" in s:
            p4q.p4q_cls_saliency(s["qc"], s["kc"], s["k"], s["A"])
        p4q.p4q_select_gather_quant(s["V"], s["Q"], s["A"], s["text"], s["K"], s["idx"], s["X"], c["q"], c["s"],
                                    s["ws"])
        return {"idx": s["idx"], "X": s["X"], "q": c["q"], "s": c["s"], "A": s["A"]}
    p4q.p4q_causal_attention(s["q"], s["k"], s["v"], s["o"], *s["args"])
    return s["o"]


# ---------------------------------------------------------------- what a pass cannot do without
def _linear_work(M, K, N):
    return {"bytes": M * K / 2 + N * K / 2 + 4 * (M + N) + 2 * M * N, "flops": 2.0 * M * N * K}


def _add(*ws):
    return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}


def _split(c):
    kq = 300 * c["K"] // 1000 if c["J"] else 0
    ks = 200 * c["K"] // 1000
    return kq, ks, c["K"] - kq - ks


def work(case):
    c, kind = case, case["kind"]
    if kind == "decode":
        m, d, f = c["rows"], c["d"], c["ffn"]
        return _add(*[_linear_work(m, k, n) for k, n in ((d, 3 * d), (d, d), (d, 2 * f), (f, d))],
                    {"bytes": 2.0 * m * 3 * d + 4 * d + 2.0 * m * f, "flops": 0})
    if kind == "linear":
        w = _linear_work(c["M"], c["Kin"], c["N"])
        return _add(w, {"bytes": 2.0 * c["M"] * c["Kin"], "flops": 0})
    if kind == "chain":  # activations arrive as one byte per code, leave as fp16 and one byte per code
        M, K, N = c["M"], c["Kin"], c["N"]
        return {"bytes": M * K + N * K / 2 + 3.0 * M * N + 4 * (4 * M + 2 * N), "flops": 2.0 * M * N * K}
    if kind == "rmsnorm":
        return {"bytes": 3.5 * c["M"] * c["Kin"] + 2 * c["Kin"] + 8 * c["M"], "flops": 4.0 * c["M"] * c["Kin"]}
    if kind == "swiglu":
        return {"bytes": 5.5 * c["M"] * c["Kin"] + 8 * c["M"], "flops": 8.0 * c["M"] * c["Kin"]}
    if kind == "select":
        B, N, d, K, T = c["B"], c["N"], c["d"], c["K"], c["T"]
        kq, ks, kd = _split(c)
        b = B * (2.0 * N * d + 2 * c["J"] * d + 4 * N + 2 * T * d + (K + T) * (2.5 * d + 4) + 4 * K)
        if c["tower"]:
            b += B * N * wl.VIT_HEADS * wl.VIT_HEAD_DIM * 2
        # tokens x concepts, tokens x kept set of stages 1-2, stage 3's picks with each other
        return {"bytes": b, "flops": 2.0 * B * d * ((c["J"] + kq + ks) * N + kd * kd / 2)}
    B, m, H, hk = c["B"], c["m"], c["H"], c["Hkv"]
    return {"bytes": 2.0 * B * m * 128 * (2 * H + 2 * hk), "flops": 4.0 * 128 * B * H * m * (m + 1) / 2}


# ---------------------------------------------------------------- tolerances
def tolerance(case):
    kind = case["kind"]
    if kind == "swiglu":
        # scales to 32 bits; a code within 6e-6 of a .5 boundary may differ (1.5e-8
        # of the codes and 1.6e-4 of the row sums do from the 64-bit result)
        return {"rel": 3e-7, "max": 1e-6, "differ": 2e-3}
    if kind == "attention":
        # weights rounded to fp16 before the product with v, fp16 output (2.5e-4
        # and 3e-3 off the 64-bit result)
        return {"rel": 1e-3, "max": 1.2e-2}
    if kind == "select" and case["tower"]:
        # the saliency is a 32-bit softmax (2e-7 and 7e-7 off the 64-bit
        # result); the rest follows from whole numbers
        return {"rel": 1e-6, "max": 3e-6}
    # codes, scales, integer sums and the fp16 rounding of the linears are
    # fixed bit for bit by the interface (include/p4q.h)
    return "exact"


# ---------------------------------------------------------------- 64-bit results in plain torch
def _q4(x):
    """Codes (as float64 integers) and scales of rows x: the scale and the
    quotient rounded to fp32 as the interface states."""
    x = x.double()
    s = (x.abs().amax(-1) / 7).float()
    sd = s.double().unsqueeze(-1)
    q = torch.where(sd > 0, x / sd, torch.zeros_like(x)).float()
    return torch.round(q).double(), s


def _pack(codes):
    c = codes.to(torch.int32) & 15
    return (c[:, 0::2] | (c[:, 1::2] << 4)).to(torch.uint8)


def _expand(codes):
    """One byte per code (code + 8): the even four of each eight, then the odd four."""
    u = (codes + 8).to(torch.uint8).view(codes.shape[0], -1, 4, 2)
    return u.transpose(2, 3).reshape(codes.shape)


def _unpack(p):
    p = p.to(torch.int32)
    lo, hi = p & 15, p >> 4
    c = torch.stack((lo, hi), -1).view(p.shape[0], -1)
    return torch.where(c > 7, c - 16, c).float()


def _exact_linear(codes, s, W):
    """fp64 dequantized product; the integer dot products are exact in fp32."""
    wq, sw = W
    out = torch.empty((codes.shape[0], wq.shape[0]), dtype=torch.float64, device="cuda")
    a = codes.float()
    for n0 in range(0, wq.shape[0], 4096):
        out[:, n0:n0 + 4096] = (a @ _unpack(wq[n0:n0 + 4096]).t()).double() * sw[n0:n0 + 4096].double()
    return out.mul_(s.double().unsqueeze(1))


def _rounded_linear(codes, s, W):
    """The linear's fp16 output in the interface's roundings (a later quantizer's input)."""
    one = torch.ones_like(s)
    acc = torch.cat([_exact_linear(c, o, (W[0], torch.ones_like(W[1]))).float() for c, o in
                     zip(codes.split(4096), one.split(4096))])
    return acc.mul_(s.unsqueeze(1)).mul_(W[1]).half()


def _exact_weight(g, n, kin):
    w = (torch.randn((n, kin), generator=g, device="cuda", dtype=torch.float32) * 0.02).half()
    codes, s = _q4(w)
    return _pack(codes), s


def _exact_rmsnorm(x, w):
    ms = (x.double().square().sum(-1).float().double() / x.shape[-1]).float()
    r = (1 / ((ms.double() + torch.tensor(EPS).double()).float().double().sqrt().float().double())).float()
    t = (x.double() * r.double().unsqueeze(-1)).float().half()
    return (t.double() * w.double()).half()


def _exact_swiglu(g, u):
    h = g.double() / (1 + torch.exp(-g.double())) * u.double()
    a = h.abs().amax(-1)
    codes = torch.round(h * (7 / a).unsqueeze(-1))
    return codes, a / 7


def _exact_saliency(s, wanted):
    q, kc, k = s["qc"].double(), s["kc"].double(), s["k"].double()
    B, C, H, dh = q.shape
    k = k.view(B, C, -1, H, dh)
    l = torch.einsum("bchd,bcnhd->bchn", q, k) / math.sqrt(dh)
    l0 = (q * kc).sum(-1, keepdim=True) / math.sqrt(dh)
    p = torch.softmax(torch.cat((l0, l), -1), -1)[..., 1:]
    return p.mean(2).reshape(B, -1)


def _cosines(a, na, b, nb):
    """Cosines of code rows, each step rounded to fp32 as the interface states."""
    dot = (a.float() @ b.float().t()).double()
    n = (na[:, None] * nb[None, :]).float().double().sqrt().float().double()
    return torch.where(n > 0, dot / n, torch.zeros_like(dot)).float()


def _exact_select(c, s, A):
    kq, ks, kd = _split(c)
    kept = torch.zeros((c["B"], c["N"]), dtype=torch.bool, device="cuda")
    cos = torch.empty((c["B"], c["N"], c["N"]), dtype=torch.float32, device="cuda")
    for b in range(c["B"]):
        v, _ = _q4(s["V"][b])
        nv = v.square().sum(1)
        cos[b] = _cosines(v, nv, v, nv)
        if kq:
            q, _ = _q4(s["Q"][b])
            sc = _cosines(q, q.square().sum(1), v, nv)
            for j in range(c["J"]):
                n = kq // c["J"] + (1 if j < kq % c["J"] else 0)
                order = torch.sort(torch.where(kept[b], torch.full_like(sc[j], -9.0), sc[j]), descending=True,
                                   stable=True)[1]
                kept[b, order[:n]] = True
        a = torch.where(kept[b], torch.full_like(A[b], -9.0), A[b])
        kept[b, torch.sort(a, descending=True, stable=True)[1][:ks]] = True
    inf = torch.tensor(float("inf"), device="cuda")
    m = torch.where(kept[:, None, :], cos, -inf).amax(2)
    tok = torch.arange(c["N"], device="cuda")
    img = torch.arange(c["B"], device="cuda")
    for _ in range(kd):
        f = torch.where(kept, inf, m)
        pick = torch.where(f == f.amin(1, keepdim=True), tok, c["N"]).amin(1)
        kept[img, pick] = True
        m = torch.maximum(m, cos[img, pick])
    return kept.nonzero()[:, 1].view(c["B"], c["K"])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "decode":
        g, d, f, m = _gen(seed), c["d"], c["ffn"], c["rows"]
        x1, x2, a = _features(g, (m,), d), _features(g, (m,), d), _features(g, (m,), d)
        w1 = (1 + 0.1 * torch.randn((d,), generator=g, device="cuda")).half()
        w2 = (1 + 0.1 * torch.randn((d,), generator=g, device="cuda")).half()
        W = {name: _exact_weight(g, n, k) for name, n, k in (("qkv", 3 * d, d), ("o", d, d), ("gu", 2 * f, d),
                                                             ("down", d, f))}
        qkv = _exact_linear(*_q4(_exact_rmsnorm(x1, w1)), W["qkv"])
        o = _exact_linear(*_q4(a), W["o"])
        gu = _exact_linear(*_q4(_exact_rmsnorm(x2, w2)), W["gu"])
        down = _exact_linear(*_q4(_rounded_linear(*_q4(_exact_rmsnorm(x2, w2)), W["gu"])[:, f:]), W["down"])
        return {"qkv": qkv, "o": o, "gu": gu, "down": down}
    if kind in ("linear", "chain"):
        g = _gen(seed)
        codes, s = _q4(_features(g, (c["M"],), c["Kin"]))
        W = _exact_weight(g, c["N"], c["Kin"])
        Y = _exact_linear(codes, s, W)
        if kind == "linear":
            return {"q": _pack(codes), "s": s.double(), "Y": Y}
        codes, s = _q4(_rounded_linear(codes, s, W))
        return {"Y": Y, "s": s.double(), "u": _expand(codes), "su": (codes + 8).sum(1).to(torch.int32)}
    if kind == "rmsnorm":
        g = _gen(seed)
        X = _features(g, (c["M"],), c["Kin"])
        w = (1 + 0.1 * torch.randn((c["Kin"],), generator=g, device="cuda")).half()
        codes, s = _q4(_exact_rmsnorm(X, w))
        return {"q": _pack(codes), "s": s.double(), "u": _expand(codes), "su": (codes + 8).sum(1).to(torch.int32)}
    if kind == "swiglu":
        gu, f = torch.randn((c["M"], 2 * c["Kin"]), generator=_gen(seed), device="cuda").half(), c["Kin"]
        codes, s = _exact_swiglu(gu[:, :f], gu[:, f:])
        return {"q": _pack(codes), "s": s, "u": _expand(codes), "su": (codes + 8).sum(1).to(torch.int32)}
    if kind == "select":
        s = _select_inputs(c, seed)
        A = _exact_saliency(s, c) if c["tower"] else s["A"].double()
        idx = _exact_select(c, s, A.float())
        X = torch.gather(s["V"], 1, idx[:, :, None].expand(-1, -1, c["d"]))
        if c["T"]:
            X = torch.cat((X, s["text"]), 1)
        codes, sa = _q4(X.reshape(-1, c["d"]))
        return {"idx": idx, "X": X.double(), "q": _pack(codes), "s": sa.double(), "A": A}
    q, k, v = _attention_inputs(c, seed)
    B, m, H, hk = c["B"], c["m"], c["H"], c["Hkv"]
    mask = torch.ones((m, m), dtype=torch.bool, device="cuda").triu(1)
    out = torch.empty((B * m, H * 128), dtype=torch.float64, device="cuda")
    for b in range(B):
        r = slice(b * m, (b + 1) * m)
        qb = q[r].double().view(m, H, 128).transpose(0, 1)
        kb, vb = (t[r].double().view(m, hk, 128).transpose(0, 1).repeat_interleave(H // hk, 0) for t in (k, v))
        p = torch.softmax((qb @ kb.transpose(1, 2) / math.sqrt(128)).masked_fill(mask, float("-inf")), -1)
        out[r] = (p @ vb).transpose(0, 1).reshape(m, H * 128)
    return out
