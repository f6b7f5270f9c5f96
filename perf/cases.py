"""What a program does with this framework, as cases that can be timed and compared.

Every case goes through the public entry points of ``paper_2607_24981_gb300``: whole models (the
integer ViT encoder, the full detector), single layers of them (an encoder block, attention, linear
layers, a decoder layer, the two-stage query selection) and the stand-alone nonlinearities.  All
results are whole numbers (some carried in float16), so two correct implementations agree in every
element and the tolerance is exact everywhere.  ``exact`` restates each path in plain torch with
64-bit integers (matrix products in float64, exact below 2^53).

Weights are one fixed checkpoint per model (seed 2): a serving program keeps its model and gets new
images, so only the inputs follow the case's seed.
"""
import math

import numpy as np
import torch

import paper_2607_24981_gb300 as ilw
from paper_2607_24981_gb300 import synth

CKPT = 2  # the seed of every checkpoint
MODELS = {"tiny": "tiny_backbone_b8", "medium": "medium_backbone_b8"}
LEVELS = ((80, 80), (40, 40), (20, 20))


def listed():
    return [
        # the smallest model call: one encoder block on 256 tokens of width 192 (latency, launches)
        {"name": "block_256tok", "kind": "block", "B": 1, "T": 256, "d": 192, "H": 3, "F": 768, "win": 0, "mode": "literal"},
        # one camera frame through the Tiny encoder, recorded once as a CUDA graph (latency)
        {"name": "tiny_b1", "kind": "backbone", "model": "tiny", "B": 1, "hw": 640, "graph": True},
        # the Medium encoder at the batch its throughput is quoted on (graph)
        {"name": "medium_b8", "kind": "backbone", "model": "medium", "B": 8, "hw": 640, "graph": True},
        # one camera frame through the whole Medium detector, recorded as a CUDA graph (latency)
        {"name": "detector_b1", "kind": "detector", "B": 1, "graph": True},
        # the largest call: 16 images through the whole detector, called eagerly
        {"name": "detector_b16", "kind": "detector", "B": 16, "graph": False},
        # attention called as an operator on plain int8 q|k|v, a token count that fills no tile evenly
        {"name": "attention_i8", "kind": "attention", "B": 3, "T": 900, "H": 6, "dh": 64, "win": 0, "form": "i8"},
        # the decoder's widest linear layer with its fused SD-ShiftGELU, plain int8 in and out
        {"name": "linear_gelu_i8", "kind": "linear", "M": 4800, "N": 1024, "K": 256, "form": "i8", "epi": "gelu"},
        # one decoder layer on 4 images (self-attention, deformable cross-attention, FFN)
        {"name": "decoder_layer_b4", "kind": "decoder", "B": 4, "Q": 300},
        # two-stage query selection over the memory of 8 images
        {"name": "two_stage_b8", "kind": "two_stage", "B": 8, "K": 300},
        # the nonlinearities on their own, at the sizes of the nonlinearity sweep
        {"name": "shiftmax_400", "kind": "shiftmax", "rows": (1 << 27) // 400, "len": 400},
        {"name": "gelu_2p28", "kind": "gelu", "n": 1 << 28},
        {"name": "layernorm_384", "kind": "layernorm", "rows": 1 << 20, "C": 384, "in_bits": 32, "out_bits": 8, "iters": 10},
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["block", "backbone", "detector", "attention", "linear", "decoder", "two_stage", "shiftmax", "gelu",
                       "layernorm"])
    if kind == "block":  # square token grids, windowed or global, widths of the Tiny and Medium models
        d, H = rng.choice([(192, 3), (384, 6), (256, 4), (128, 2)])
        win = rng.choice([0, 2])
        g = 2 * rng.randint(4, 28)
        return {"kind": kind, "B": _log(rng, 1, 16), "T": g * g, "d": d, "H": H, "F": 4 * d, "win": win,
                "mode": rng.choice(["literal", "calibrated"])}
    if kind == "backbone":  # image sizes that give even token grids
        return {"kind": kind, "model": rng.choice(["tiny", "medium"]), "B": _log(rng, 1, 16), "hw": 32 * rng.randint(8, 24),
                "graph": rng.random() < 0.5}
    if kind == "detector":
        return {"kind": kind, "B": _log(rng, 1, 16), "graph": rng.random() < 0.5}
    if kind == "attention":
        win = rng.choice([0, 0, 2, 4])
        if win:
            T = (win * rng.randint(4, 56 // win)) ** 2
        else:
            T = _log(rng, 17, 2500)
        return {"kind": kind, "B": _log(rng, 1, 8), "T": T, "H": rng.randint(1, 8), "dh": rng.choice([32, 64]), "win": win,
                "form": rng.choice(["i8", "f16"])}
    if kind == "linear":
        form, epi = rng.choice(["i8", "f16"]), rng.choice(["i8", "i16_res", "gelu", "raw32"])
        return {"kind": kind, "M": _log(rng, 1, 30000), "N": rng.choice([4, 80, 192, 256, 384, 576, 768, 1000, 1024, 1152, 1536]),
                "K": 16 * _log(rng, 4, 96), "form": form, "epi": epi}
    if kind == "decoder":
        return {"kind": kind, "B": _log(rng, 1, 16), "Q": rng.randint(50, 400)}
    if kind == "two_stage":
        return {"kind": kind, "B": _log(rng, 1, 16), "K": rng.randint(50, 500)}
    if kind == "shiftmax":  # any row length, odd ones among them
        n = _log(rng, 8, 2048)
        return {"kind": kind, "rows": _log(rng, 500, (1 << 27) // n), "len": n}
    if kind == "gelu":
        return {"kind": kind, "n": _log(rng, 1000, 1 << 28)}
    C = rng.choice([rng.randint(16, 1024), 64 * rng.randint(1, 12)])
    return {"kind": kind, "rows": _log(rng, 100, (1 << 28) // C), "C": C, "in_bits": rng.choice([16, 32]),
            "out_bits": rng.choice([8, 16]), "iters": rng.choice([10, 20])}


# ------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator("cuda").manual_seed(int(seed))


def _uniform(g, shape, lo, hi, dtype):
    return torch.randint(lo, hi + 1, shape, generator=g, device="cuda", dtype=dtype)


def _normal(g, shape, std, dtype):
    """Rounded normal values, clipped to the int8 range: what a calibrated layer hands on."""
    return torch.empty(shape, device="cuda").normal_(0.0, std, generator=g).round_().clamp_(-127, 127).to(dtype)


def _laplace(g, shape, scale, dtype):
    u = torch.rand(shape, generator=g, device="cuda").sub_(0.5).clamp_(-0.4999999, 0.4999999)
    return (-scale * u.sign() * torch.log1p(-2 * u.abs())).round_().clamp_(-127, 127).to(dtype)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _model_params(model, hw):
    cfg = dict(synth.CONFIGS[MODELS[model]])
    return cfg, synth.patch_embed_params(CKPT, cfg["d"], T=(hw // 16) ** 2), synth.backbone_params(CKPT, cfg)


def _detector_params():
    cfg = synth.CONFIGS["medium_detector_b16"]
    bcfg, pe, blocks = _model_params("medium", 640)
    n = cfg["dec_layers"]
    return dict(cfg=cfg, pe=pe, blocks=blocks, pp=synth.projector_params(CKPT, len(cfg["taps"]), bcfg["d"], cfg["N"]),
                dps=[synth.decoder_params(CKPT, i, cfg["N"], cfg["Hd"], cfg["Fd"], 3, cfg["P"]) for i in range(n)],
                tsp=synth.two_stage_params(CKPT), hp=synth.head_params(CKPT), pq=synth.query_pos_params(CKPT),
                rps=synth.refine_params(CKPT, n - 1))


def _linear_params(case):
    return synth.gemm_params(CKPT, "perf.linear", case["N"], case["K"], 40.0, 2000.0 if case["epi"] == "gelu" else 40.0)


GELU = {"I0": 1000, "k_inter": 16, "k_out": 8}
GELU_OUT = (3 << 29, 38)   # dyadic output scale of the fused SD-ShiftGELU
RES = (1 << 30, 31)        # dyadic scale of the residual term
SMX = {"I0": 6000, "k_inter": 16, "k_out": 8, "s_d": -1, "m_p": 4, "M_hw": 31}
ATT_OUT = (3 << 29, 38)


def _inputs(case, seed):
    """The tensors of a case's inputs, from the seed alone."""
    g, kind = _gen(seed), case["kind"]
    if kind == "block":
        return {"x": _laplace(g, (case["B"] * case["T"], case["d"]), 20.0, torch.int16)}
    if kind == "backbone":
        return {"img": _uniform(g, (case["B"], 3, case["hw"], case["hw"]), -127, 127, torch.int8)}
    if kind == "detector":
        img = _uniform(g, (case["B"], 3, 640, 640), -127, 127, torch.int8)
        return {"img": img, "tgt": _uniform(g, (case["B"] * 300, 256), -(1 << 11), 1 << 11, torch.int16)}
    if kind == "attention":
        qkv = _normal(g, (case["B"] * case["T"], 3 * case["H"] * case["dh"]), 40.0, torch.int8)
        return {"qkv": qkv if case["form"] == "i8" else qkv.half()}
    if kind == "linear":
        A = _normal(g, (case["M"], case["K"]), 40.0, torch.int8)
        r = {"A": A if case["form"] == "i8" else A.half()}
        if case["epi"] == "i16_res":
            r["res"] = _uniform(g, (case["M"], case["N"]), -3000, 3000, torch.int16)
        return r
    if kind == "decoder":
        B, Q, S = case["B"], case["Q"], sum(h * w for h, w in LEVELS)
        return {"tgt": _uniform(g, (B * Q, 256), -(1 << 11), 1 << 11, torch.int16),
                "pos": _uniform(g, (B * Q, 256), -(1 << 11), 1 << 11, torch.int16),
                "refs": _uniform(g, (B, Q, 2), 0, (1 << 16) - 1, torch.int32), "mem": _normal(g, (B * S, 256), 40.0, torch.int8)}
    if kind == "two_stage":
        return {"mem": _normal(g, (case["B"] * 8400, 256), 40.0, torch.int8)}
    if kind == "shiftmax":
        return {"X": _uniform(g, (case["rows"], case["len"]), -(1 << 15), 1 << 15, torch.int32)}
    if kind == "gelu":
        return {"X": _uniform(g, (case["n"],), -(1 << 12), 1 << 12, torch.int32)}
    lim = 3000 if case["in_bits"] == 16 else 1 << 14
    return {"X": _uniform(g, (case["rows"], case["C"]), -lim, lim, torch.int16 if case["in_bits"] == 16 else torch.int32)}


# ------------------------------------------------------------------------------------------ the pass
def prepare(case, seed):
    s, kind = dict(_inputs(case, seed), case=case), case["kind"]
    if kind == "block":
        B, T, d, F = case["B"], case["T"], case["d"], case["F"]
        s["bw"] = ilw.BlockWeights(synth.block_params(CKPT, 0, d, case["H"], F, case["win"], case["mode"]))
        s["ws"] = torch.empty(ilw.block_workspace_bytes(B, T, d, F), dtype=torch.uint8, device="cuda")
        s["out"] = torch.empty_like(s["x"])
    elif kind == "backbone":
        _, pe, blocks = _model_params(case["model"], case["hw"])
        s["net"] = ilw.Backbone(pe, blocks, case["B"], (case["hw"], case["hw"]))
        if case["graph"]:
            s["graph"] = s["net"].capture(s["img"])
    elif kind == "detector":
        p = _detector_params()
        c = p.pop("cfg")
        s["net"] = ilw.Detector(p["pe"], p["blocks"], c["taps"], p["pp"], p["dps"], case["B"], c["Q"], c["levels"], c["grid"],
                                tsp=p["tsp"], hp=p["hp"], pq=p["pq"], rps=p["rps"])
        if case["graph"]:
            s["graph"] = ilw.Graphed(lambda: s["net"].forward(s["img"], s["tgt"]))
    elif kind == "attention":
        s["out"] = torch.empty((case["B"] * case["T"], case["H"] * case["dh"]), dtype=s["qkv"].dtype, device="cuda")
    elif kind == "linear":
        W, b, m, sh = _linear_params(case)
        s["Wp"], s["b"], s["m"], s["s"] = ilw.pack_weight(_dev(W)), _dev(b), _dev(m), _dev(sh)
    elif kind == "decoder":
        s["dw"] = ilw.DecoderWeights(synth.decoder_params(CKPT, 0))
        s["ws"] = torch.empty(ilw.decoder_workspace_bytes(case["B"], case["Q"], 8400, 256, 1024, 8, 3, 4), dtype=torch.uint8,
                              device="cuda")
        s["out"] = torch.empty_like(s["tgt"])
    elif kind == "two_stage":
        s["ts"] = ilw.TwoStage(synth.two_stage_params(CKPT))
    elif kind == "shiftmax":
        s["out"] = torch.empty(s["X"].shape, dtype=torch.uint8, device="cuda")
    elif kind == "gelu":
        s["out"] = torch.empty_like(s["X"])
    else:
        s["beta"], s["mult"], s["shift"] = (_dev(a) for a in synth.ln_params(CKPT, "perf.ln", case["C"],
                                                                              32.0 if case["out_bits"] == 8 else 2048.0))
        s["out"] = torch.empty(s["X"].shape, dtype=torch.int8 if case["out_bits"] == 8 else torch.int16, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "block":
        return ilw.block_forward(s["bw"], s["x"], case["B"], case["T"], s["ws"], out=s["out"])
    if kind == "backbone":
        return s["graph"].replay() if case["graph"] else s["net"].forward(s["img"])
    if kind == "detector":  # decoder output, class scores, boxes
        return s["graph"].replay() if case["graph"] else s["net"].forward(s["img"], s["tgt"])
    if kind == "attention":
        return ilw.shiftmax_attn(s["qkv"], case["B"], case["T"], case["H"], case["dh"], case["win"], SMX, *ATT_OUT, out=s["out"])
    if kind == "linear":
        a = (s["A"], s["Wp"], case["N"], s["b"], s["m"], s["s"])
        if case["epi"] == "gelu":
            return ilw.gemm(*a, 8 if case["form"] == "i8" else ilw.I8_IN_F16, gelu=GELU, m_g=GELU_OUT[0], s_g=GELU_OUT[1])
        if case["epi"] == "i16_res":
            return ilw.gemm(*a, 16, res=s["res"], m_r=RES[0], s_r=RES[1])
        if case["epi"] == "raw32":
            return ilw.gemm(s["A"], s["Wp"], case["N"], s["b"], None, None, 32)
        return ilw.gemm(*a, 8 if case["form"] == "i8" else ilw.I8_IN_F16)
    if kind == "decoder":
        return ilw.decoder_layer_forward(s["dw"], s["tgt"], s["pos"], s["mem"], LEVELS, s["refs"], case["B"], case["Q"], s["ws"],
                                         out=s["out"])
    if kind == "two_stage":  # best logits, token indices, reference logits, boxes
        return s["ts"].forward(s["mem"], case["B"], 8400, case["K"])
    if kind == "shiftmax":
        return ilw.shiftmax_rows(s["X"], SMX, out=s["out"])
    if kind == "gelu":
        return ilw.sdshiftgelu(s["X"], {"I0": 600, "k_inter": 16, "k_out": 8}, out=s["out"])
    return ilw.int_layernorm(s["X"], s["beta"], s["mult"], s["shift"], case["iters"], case["out_bits"], out=s["out"])


# ------------------------------------------------------------------------------------------ work
def _block_work(M, d, F, keys):
    """(weight bytes, flops) of one encoder block on M tokens, each attending to `keys` tokens."""
    return 2 * (4 * d * d + 2 * d * F), 2 * M * (4 * d * d + 2 * d * F) + 4 * M * keys * d


def _backbone_work(model, B, hw):
    cfg = synth.CONFIGS[MODELS[model]]
    d, F, T = cfg["d"], cfg["F"], (hw // 16) ** 2
    by, fl = B * 3 * hw * hw + 2 * 768 * d + 2 * T * d, 2 * B * T * 768 * d
    for i in range(cfg["layers"]):
        wb, f = _block_work(B * T, d, F, T if i in cfg["global_layers"] else T // 4)
        by, fl = by + wb, fl + f
    return by, fl, 2 * B * T * d


def _decoder_work(B, Q, d=256, F=1024, H=8, LP=12, S=8400):
    w = 2 * (4 * d * d + d * d + 3 * H * LP * d + d * d + 2 * d * F)
    flops = 2 * B * Q * (5 * d * d + 3 * H * LP * d + 2 * d * F) + 2 * B * S * d * d + 4 * B * Q * Q * d + 2 * B * Q * LP * d
    return w, flops


def work(case):
    kind = case["kind"]
    if kind == "block":
        M = case["B"] * case["T"]
        wb, fl = _block_work(M, case["d"], case["F"], case["T"] if not case["win"] else case["T"] // case["win"] ** 2)
        return {"bytes": wb + 4 * M * case["d"], "flops": fl}
    if kind == "backbone":
        by, fl, out = _backbone_work(case["model"], case["B"], case["hw"])
        return {"bytes": by + out, "flops": fl}
    if kind == "detector":
        B = case["B"]
        by, fl, _ = _backbone_work("medium", B, 640)
        wd, fd = _decoder_work(B, 300)
        by += 2 * 3 * 4 * 384 * 256 + 3 * wd + 2 * B * 300 * 256 * 2 + B * 300 * 84 * 4
        fl += 2 * 3 * B * 1600 * 4 * 384 * 256 + 3 * fd + 2 * B * 8400 * 256 * 80 + 2 * B * 300 * (8 * 256 * 256 + 80 * 256)
        return {"bytes": by, "flops": fl}
    if kind == "attention":
        M, d = case["B"] * case["T"], case["H"] * case["dh"]
        keys = case["T"] if not case["win"] else case["T"] // case["win"] ** 2
        return {"bytes": 4 * M * d * (1 if case["form"] == "i8" else 2), "flops": 4 * M * keys * d}
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        ab = 1 if case["form"] == "i8" else 2
        ob = {"raw32": 4, "i16_res": 4}.get(case["epi"], ab)  # i16_res: a 16-bit residual in and 16 bits out
        return {"bytes": M * K * ab + 2 * N * K + M * N * ob, "flops": 2 * M * N * K}
    if kind == "decoder":
        w, fl = _decoder_work(case["B"], case["Q"])
        return {"bytes": w + case["B"] * (8400 * 256 + case["Q"] * (3 * 512 + 8)), "flops": fl}
    if kind == "two_stage":
        B, K = case["B"], case["K"]
        return {"bytes": B * 8400 * 256 + 2 * 256 * 340 + B * K * 32, "flops": 2 * B * 8400 * 256 * 80 + 2 * B * K * 256 * 260}
    if kind == "shiftmax":
        return {"bytes": 5 * case["rows"] * case["len"], "flops": 35 * case["rows"] * case["len"]}
    if kind == "gelu":
        return {"bytes": 8 * case["n"], "flops": 20 * case["n"]}
    return {"bytes": (case["in_bits"] + case["out_bits"]) // 8 * case["rows"] * case["C"], "flops": 10 * case["rows"] * case["C"]}


def tolerance(case):
    return "exact"  # every output is a whole number that the method defines exactly


# ------------------------------------------------------------------------------------------ 64 bits
def _rq(v, m, s):
    """Dyadic requantisation (v m + 2^(s-1)) >> s; m, s numbers or per-column tensors."""
    if isinstance(s, torch.Tensor):
        return (v * m + (torch.ones_like(s) << (s - 1))) >> s
    return (v * m + (1 << (s - 1))) >> s


def _sat(v, bits):
    lim = (1 << (bits - 1)) - 1
    return v.clamp(-lim, lim)


def _i64(a):
    return (_dev(a) if isinstance(a, np.ndarray) else a).to(torch.int64)


def _lin(x, W, b):
    """x [M, K] int64 times W [N, K], plus the bias: every partial sum is far below 2^53."""
    return (x.double() @ _i64(W).double().T).to(torch.int64) + _i64(b)


def _shiftexp(I, I0, k):
    n = torch.minimum(-(I + (I >> 1) - (I >> 4)), torch.full_like(I, k * I0))
    q = n // I0
    return (I0 + ((q * I0 - n) >> 1)) << (k - q)


def _shiftmax(x, p):
    """Constrained Shiftmax over the last dimension."""
    e = _shiftexp(x - x.amax(-1, keepdim=True), p["I0"], p["k_inter"])
    S = e.sum(-1, keepdim=True)
    bits = torch.where(S > 1, torch.frexp((S - 1).double())[1].to(torch.int64), torch.zeros_like(S))  # ceil(log2 S)
    sd = (bits + p["m_p"] - p["M_hw"]).clamp(min=0) if p["s_d"] < 0 else torch.full_like(S, p["s_d"])
    F = ((1 << 31) - 1) // (S >> sd).clamp(1, (1 << 31) - 1)
    return (e * F) >> (32 - p["k_out"] + sd)


def _gelu(x, I0, k, k_out):
    z = x + (x >> 1) + (x >> 3) + (x >> 4)
    e, top = _shiftexp(-z.abs(), I0, k), I0 << k
    F = ((1 << 31) - 1) // (top + e)
    return x * ((torch.where(z >= 0, torch.full_like(e, top), e) * F) >> (32 - k_out))


def _sigmoid(x, I0, k, k_out):
    e, top = _shiftexp(-x.abs(), I0, k), I0 << k
    F = ((1 << 31) - 1) // (top + e)
    return (torch.where(x >= 0, torch.full_like(e, top), e) * F) >> (32 - k_out)


def _ln(x, beta, mult, shift, iters, bits):
    C = x.shape[-1]
    mu = torch.div(2 * x.sum(-1, keepdim=True) + C, 2 * C, rounding_mode="floor")
    y = x - mu
    V = (y * y).sum(-1, keepdim=True)
    r = torch.full_like(V, 1 << 16)
    for _ in range(iters):
        r = torch.where(r == 0, r, (r + V // r.clamp(min=1)) >> 1)
    n = (y * (((1 << 31) - 1) // r.clamp(min=1))) >> 1
    return _sat(_rq(n + _i64(beta), _i64(mult), _i64(shift)), bits)


def _attn(qkv, B, T, H, dh, win, smx, m_o, s_o):
    """qkv [B T, 3 H dh] -> [B T, H dh]; win > 1: win x win windows of the square token grid."""
    d = H * dh
    t = qkv.view(B, T, 3, H, dh)
    if win > 1:
        g = math.isqrt(T)
        w = g // win
        t = t.view(B, win, w, win, w, 3, H, dh).transpose(2, 3).reshape(B * win * win, w * w, 3, H, dh)
    out = torch.empty((t.shape[0], t.shape[1], H, dh), dtype=torch.int64, device=qkv.device)
    for i in range(t.shape[0]):
        q, k, v = (t[i, :, j].permute(1, 0, 2).double() for j in range(3))  # [H, n, dh]
        for h in range(H):
            P = _shiftmax((q[h] @ k[h].T).to(torch.int64), smx)
            out[i, :, h] = _sat(_rq((P.double() @ v[h]).to(torch.int64), m_o, s_o), 8)
    if win > 1:
        out = out.view(B, win, win, w, w, H, dh).transpose(2, 3).reshape(B, T, H, dh)
    return out.reshape(B * T, d)


def _block(bp, x, B, T):
    d, H = bp["d"], bp["H"]

    def lin(a, n, bits):
        r = _rq(_lin(a, bp["w_" + n], bp["b_" + n]), _i64(bp["m_" + n]), _i64(bp["s_" + n]))
        return _sat(r, bits) if bits else r

    a = _ln(x, bp["ln1_beta"], bp["ln1_mult"], bp["ln1_shift"], bp["ln_iters"], 8)
    o = _attn(lin(a, "qkv", 8), B, T, H, d // H, bp["win_side"], bp["smx"], bp["m_o"], bp["s_o"])
    x1 = _sat(lin(o, "proj", 0) + _rq(x, bp["m_r1"], bp["s_r1"]), 16)
    a = _ln(x1, bp["ln2_beta"], bp["ln2_mult"], bp["ln2_shift"], bp["ln_iters"], 8)
    g = _gelu(lin(a, "fc1", 16), bp["gelu_I0"], bp["gelu_k_inter"], bp["gelu_k_out"])
    return _sat(lin(_sat(_rq(g, bp["m_g"], bp["s_g"]), 8), "fc2", 0) + _rq(x1, bp["m_r2"], bp["s_r2"]), 16)


def _patch(pe, img):
    B, _, hw, _ = img.shape
    n = hw // 16
    a = _i64(img).view(B, 3, n, 16, n, 16).permute(0, 2, 4, 1, 3, 5).reshape(B * n * n, 768)
    r = _rq(_lin(a, pe["w"], pe["b"]), _i64(pe["m"]), _i64(pe["s"]))
    return _sat(r + _rq(_i64(pe["pos"]), pe["m_pos"], pe["s_pos"]).repeat(B, 1), 16)


def _backbone(pe, blocks, img, taps=()):
    """The last block's output, and those of the tapped blocks."""
    x, kept = _patch(pe, img), []
    for i, bp in enumerate(blocks):
        x = _block(bp, x, img.shape[0], (img.shape[2] // 16) ** 2)
        kept += [x] if i in taps else []
    return x, kept


def _projector(pp, taps, B, grid=40):
    """Each level: requantised taps through their branches, each branch rescaled, summed, resampled."""
    t = [_sat(_rq(x, *ms), 8) for x, ms in zip(taps, pp["taps"])]
    mem = []
    for lv, (h, w) in zip(pp["levels"], LEVELS):
        acc = sum(_rq(_lin(x, W, np.zeros(W.shape[0], np.int64)), m, s) for x, W, m, s in zip(t, lv["w"], lv["m_b"], lv["s_b"]))
        y = _sat(_rq(acc + _i64(lv["b"]), _i64(lv["m"]), _i64(lv["s"])), 8).view(B, grid, grid, -1)
        iy, ix = torch.arange(h, device="cuda") * grid // h, torch.arange(w, device="cuda") * grid // w
        mem.append(y[:, iy][:, :, ix].reshape(B, h * w, -1))
    return torch.cat(mem, 1).reshape(-1, mem[0].shape[-1])


def _deform(value, refs, off, w, B, Q, H, P, m, s):
    """Nearest-neighbour sampling; value [B, S, H, dh], off [B, Q, H, L, P, 2] in Q8 pixels, w [B, Q, H, L, P]."""
    out, start = 0, 0
    b, h = torch.arange(B, device="cuda").view(B, 1, 1, 1), torch.arange(H, device="cuda").view(1, 1, H, 1)
    for l, (hl, wl) in enumerate(LEVELS):
        ix = (((refs[..., 0] * wl) >> 8).view(B, Q, 1, 1) + off[:, :, :, l, :, 0]) >> 8
        iy = (((refs[..., 1] * hl) >> 8).view(B, Q, 1, 1) + off[:, :, :, l, :, 1]) >> 8
        ok = (ix >= 0) & (ix < wl) & (iy >= 0) & (iy < hl)
        v = value[b, start + iy.clamp(0, hl - 1) * wl + ix.clamp(0, wl - 1), h]  # [B, Q, H, P, dh]
        out = out + (v * (w[:, :, :, l] * ok).unsqueeze(-1)).sum(3)
        start += hl * wl
    return _sat(_rq(out, m, s), 8).reshape(B * Q, -1)


def _decoder(dp, tgt, pos, mem, refs, B, Q):
    d, H, L, P, it = dp["d"], dp["H"], dp["L"], dp["P"], dp["ln_iters"]

    def lin(a, n, bits=0, p=None):
        r = _rq(_lin(a, dp["w_" + n], dp["b_" + n]), _i64(dp["m_" + (p or n)]), _i64(dp["s_" + (p or n)]))
        return _sat(r, bits) if bits else r

    def to8(x, k):
        return _rq(x, dp["m_" + k], dp["s_" + k])

    def ln(x, i):
        return _ln(x, dp[f"ln{i}_beta"], dp[f"ln{i}_mult"], dp[f"ln{i}_shift"], it, 16)

    qk = lin(_sat(to8(tgt, "q1") + to8(pos, "q2"), 8), "qk", 8)
    o = _attn(torch.cat([qk, lin(_sat(to8(tgt, "v1"), 8), "v", 8)], 1), B, Q, H, d // H, 0, dp["smx"], dp["m_o"], dp["s_o"])
    t1 = ln(_sat(lin(o, "o", p="oc") + to8(tgt, "r1"), 16), 1)
    c = _sat(to8(t1, "c1") + to8(pos, "c2"), 8)
    off = lin(c, "off", 16).view(B, Q, H, L, P, 2)
    w = _shiftmax(lin(c, "att", 16).view(B, Q, H, L * P), dp["smx_w"]).view(B, Q, H, L, P)
    sm = _deform(lin(mem, "val", 8).view(B, -1, H, d // H), refs, off, w, B, Q, H, P, dp["m_s"], dp["s_s"])
    t2 = ln(_sat(lin(sm, "o2") + to8(t1, "r2"), 16), 2)
    g = _gelu(lin(_sat(to8(t2, "f"), 8), "fc1", 16), dp["gelu_I0"], dp["gelu_k_inter"], dp["gelu_k_out"])
    return ln(_sat(lin(_sat(to8(g, "g"), 8), "fc2") + to8(t2, "r3"), 16), 3)


def _box_mlp(p, a):
    """Raw box deltas of the 3-layer MLP (ReLU on the int8 hidden outputs)."""
    for n in ("b1", "b2"):
        a = _sat(_rq(_lin(a, p["w_" + n], p["b_" + n]), _i64(p["m_" + n]), _i64(p["s_" + n])), 8).clamp(min=0)
    return _lin(a, p["w_b3"], p["b_b3"])


def _two_stage(tp, mem, B, K):
    best = _lin(mem, tp["w_enc"], tp["b_enc"]).amax(1).view(B, -1)
    vals, idx = torch.sort(best, dim=1, descending=True, stable=True)  # ties keep the lower index first
    vals, idx = vals[:, :K], idx[:, :K]
    sel = mem.view(B, -1, mem.shape[1])[torch.arange(B, device="cuda").unsqueeze(1), idx].reshape(B * K, -1)
    h = _sat(_rq(_lin(sel, tp["w_p1"], tp["b_p1"]), _i64(tp["m_p1"]), _i64(tp["s_p1"])), 8).clamp(min=0)
    ref = _sat(_rq(_lin(h, tp["w_p2"], tp["b_p2"]), tp["m_d"], tp["s_d"])
               + _rq(_i64(tp["anchor16"])[idx.reshape(-1)], tp["m_a"], tp["s_a"]), 16)
    return vals, idx, ref, _sigmoid(ref, tp["ref_I0"], tp["k_inter"], 17)


def _detector(p, img, tgt):
    B, Q = img.shape[0], p["cfg"]["Q"]
    _, taps = _backbone(p["pe"], p["blocks"], img, p["cfg"]["taps"])
    mem = _projector(p["pp"], taps, B)
    _, _, ref, boxes = _two_stage(p["tsp"], mem, B, Q)
    x, pq, hp = _i64(tgt), p["pq"], p["hp"]
    for i, dp in enumerate(p["dps"]):
        b8 = _sat(_rq(boxes, pq["m_box"], pq["s_box"]), 8)
        h = _sat(_rq(_lin(b8, pq["w_q1"], pq["b_q1"]), _i64(pq["m_q1"]), _i64(pq["s_q1"])), 8).clamp(min=0)
        pos = _sat(_rq(_lin(h, pq["w_q2"], pq["b_q2"]), _i64(pq["m_q2"]), _i64(pq["s_q2"])), 16)
        x = _decoder(dp, x, pos, mem, boxes.view(B, Q, 4)[..., :2], B, Q)
        if i + 1 < len(p["dps"]):
            rp = p["rps"][i]
            dl = _box_mlp(rp, _sat(_rq(x, rp["m_in"], rp["s_in"]), 8))
            ref = _sat(_rq(dl, rp["m_d"], rp["s_d"]) + _rq(ref, rp["m_ref"], rp["s_ref"]), 16)
            boxes = _sigmoid(ref, rp["box_I0"], rp["k_inter"], 17)
    a = _sat(_rq(x, hp["m_in"], hp["s_in"]), 8)
    scores = _sigmoid(_lin(a, hp["w_cls"], hp["b_cls"]), hp["cls_I0"], hp["k_inter"], hp["cls_k_out"])
    z = _rq(_box_mlp(hp, a), hp["m_d"], hp["s_d"]) + _rq(ref, hp["m_ref"], hp["s_ref"])
    return x.to(torch.int16), scores.to(torch.int32), _sigmoid(z, hp["box_I0"], hp["k_inter"], 17).to(torch.int32)


def _by_rows(f, X, step):
    return torch.cat([f(X[i:i + step].to(torch.int64)) for i in range(0, X.shape[0], step)])


def exact(case, seed):
    """run()'s outputs in 64-bit integers, without this framework's code.  (Sums over a whole Medium model at
    batch 16 take some seconds of device time.)"""
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "block":
        bp = synth.block_params(CKPT, 0, case["d"], case["H"], case["F"], case["win"], case["mode"])
        return _block(bp, _i64(x["x"]), case["B"], case["T"]).to(torch.int16)
    if kind == "backbone":
        _, pe, blocks = _model_params(case["model"], case["hw"])
        return _backbone(pe, blocks, x["img"])[0].to(torch.int16)
    if kind == "detector":
        return _detector(_detector_params(), x["img"], x["tgt"])
    if kind == "attention":
        r = _attn(_i64(x["qkv"]), case["B"], case["T"], case["H"], case["dh"], case["win"], SMX, *ATT_OUT)
        return r.to(torch.int8) if case["form"] == "i8" else r.double()
    if kind == "linear":
        W, b, m, s = _linear_params(case)
        acc = _lin(_i64(x["A"]), W, b)
        if case["epi"] == "raw32":
            return acc.to(torch.int32)
        r = _rq(acc, _i64(m), _i64(s))
        if case["epi"] == "i16_res":
            return _sat(r + _rq(_i64(x["res"]), *RES), 16).to(torch.int16)
        if case["epi"] == "gelu":
            r = _rq(_gelu(_sat(r, 16), GELU["I0"], GELU["k_inter"], GELU["k_out"]), *GELU_OUT)
        r = _sat(r, 8)
        return r.to(torch.int8) if case["form"] == "i8" else r.double()
    if kind == "decoder":
        return _decoder(synth.decoder_params(CKPT, 0), _i64(x["tgt"]), _i64(x["pos"]), _i64(x["mem"]), _i64(x["refs"]), case["B"],
                        case["Q"]).to(torch.int16)
    if kind == "two_stage":
        vals, idx, ref, boxes = _two_stage(synth.two_stage_params(CKPT), _i64(x["mem"]), case["B"], case["K"])
        return vals.to(torch.int32), idx.to(torch.int32), ref.to(torch.int16), boxes.to(torch.int32)
    if kind == "shiftmax":
        return _by_rows(lambda t: _shiftmax(t, SMX).to(torch.uint8), x["X"], max(1, (1 << 24) // case["len"]))
    if kind == "gelu":
        return _by_rows(lambda t: _gelu(t, 600, 16, 8).to(torch.int32), x["X"], 1 << 24)
    beta, mult, shift = synth.ln_params(CKPT, "perf.ln", case["C"], 32.0 if case["out_bits"] == 8 else 2048.0)
    dt = torch.int8 if case["out_bits"] == 8 else torch.int16
    return _by_rows(lambda t: _ln(t, beta, mult, shift, case["iters"], case["out_bits"]).to(dt), x["X"],
                    max(1, (1 << 24) // case["C"]))
