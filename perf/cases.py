"""The calls whose speed matters to a user of the library: what they are, their inputs, one pass of each.

Every kind of call below is one way in which a program runs the compensated MXFP4 layer:

  linear   one layer on M tokens: quantise, multiply (or both in one call for a few tokens)
  stack    a decode step: the seven linears of some decoder blocks, captured once in a CUDA graph and replayed
  block    a prefill step: the seven linears of one decoder block, each quantised and multiplied
  ffn      a gated FFN whose producer writes the down projection's quantised input
  moe      one projection of stacked experts on routed tokens
  mxfp8    attention projections in the second format, prepared as one layer
  load     bringing one layer up from a weight matrix on the GPU, and its first rows

Sizes are those of the repository's configurations (Qwen3-4B-shaped blocks, Qwen3-30B-A3B-shaped experts, the tiny
linear) and of its tests; `draw` spreads them over the ranges in between.
"""
import math

import numpy as np
import torch

from paper_2609_22106_b200 import binding as prq, synth

# (name, input channels, output features) of a Qwen3-4B-shaped decoder block's linears
BLOCK = (("q", 2560, 4096), ("k", 2560, 1024), ("v", 2560, 1024), ("o", 4096, 2560),
         ("gate", 2560, 9728), ("up", 2560, 9728), ("down", 9728, 2560))
# which of them read the same activation
SHARED = (("q", "k", "v"), ("o",), ("gate", "up"), ("down",))
QKV = (4096, 1024, 1024)


def listed():
    return [
        # the smallest call there is (the tiny linear of the tests): launches and host work only
        {"name": "tiny_16", "kind": "linear", "M": 16, "N": 256, "K": 256, "k": 32, "mode": "permute", "y": "f32",
         "form": "two", "buffers": True},
        # one token through the down projection, activation folded into its producer: the one-launch decode call
        {"name": "down_1", "kind": "linear", "M": 1, "N": 2560, "K": 9728, "k": 256, "mode": "identity", "y": "bf16",
         "form": "fused", "buffers": True},
        # decode steps of a model: one sequence (one-launch calls), and a served batch (layers batched per launch)
        {"name": "decode_1", "kind": "stack", "M": 1, "layers": 4, "k": 256, "form": "fused"},
        {"name": "decode_64", "kind": "stack", "M": 64, "layers": 4, "k": 256, "form": "multi"},
        # a short prompt of odd length through the o projection, called as the README does (no buffers handed over)
        {"name": "o_387", "kind": "linear", "M": 387, "N": 2560, "K": 4096, "k": 128, "mode": "permute", "y": "bf16",
         "form": "two", "buffers": False},
        # the benchmark's layer: down projection, 2048 tokens, fp32 output
        {"name": "down_2048", "kind": "linear", "M": 2048, "N": 2560, "K": 9728, "k": 256, "mode": "identity", "y": "f32",
         "form": "two", "buffers": True},
        # a prefill chunk of 4096 tokens through one decoder block, scale and permutation applied online
        {"name": "block_4096", "kind": "block", "M": 4096, "k": 128, "k_down": 256},
        # a ragged prefill chunk through a gated FFN with the activation inside the producer
        {"name": "ffn_3000", "kind": "ffn", "M": 3000, "H": 2560, "C": 9728, "k_gu": 128, "k": 256},
        # routed experts at decode and at prefill
        {"name": "moe_64", "kind": "moe", "T": 64, "E": 128, "N": 2048, "K": 768, "k": 64, "mode": "permute"},
        {"name": "moe_8192", "kind": "moe", "T": 8192, "E": 128, "N": 2048, "K": 768, "k": 64, "mode": "permute"},
        # the attention linears' format
        {"name": "mxfp8_qkv_4096", "kind": "mxfp8", "M": 4096, "N": 6144, "K": 2560, "mode": "permute", "y": "bf16"},
        # start-up of a server: one layer of the model is prepared on the GPU and takes its first rows
        {"name": "load_down", "kind": "load", "N": 2560, "K": 9728, "k": 256, "search": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cols(rng, lo, hi, unit=32):
    return max(1, _log(rng, lo, hi) // unit) * unit


def _tail(rng, K, most=256):
    return rng.choice([k for k in (0, 32, 64, 128, 256) if k <= min(K, most)])


def draw(rng):
    kind = rng.choice(("linear",) * 5 + ("stack",) * 2 + ("block", "ffn", "moe", "moe", "mxfp8", "load"))
    if kind == "linear":
        K = _cols(rng, 256, 9728)
        c = {"kind": kind, "M": _log(rng, 1, 4096), "N": _log(rng, 64, 9728), "K": K, "k": _tail(rng, K),
             "mode": rng.choice(("identity", "permute")), "y": rng.choice(("f32", "bf16")), "form": "two",
             "buffers": rng.random() < 0.7}
        if c["M"] <= prq.FUSED_MAX_M and c["mode"] == "identity":
            c["form"] = "fused"
        return c
    if kind == "stack":
        form = rng.choice(("fused", "multi"))
        return {"kind": kind, "M": _log(rng, 1, prq.FUSED_MAX_M if form == "fused" else 128), "layers": rng.randint(2, 4),
                "k": rng.choice((0, 128, 256)), "form": form}
    if kind == "block":
        return {"kind": kind, "M": _log(rng, 256, 4000), "k": rng.choice((0, 128, 256)), "k_down": rng.choice((0, 128, 256))}
    if kind == "ffn":
        H = _cols(rng, 512, 2560)
        return {"kind": kind, "M": _log(rng, 1, 4000), "H": H, "C": _cols(rng, 1024, 9728, 256), "k_gu": _tail(rng, H),
                "k": rng.choice((0, 256))}
    if kind == "moe":
        K = _cols(rng, 256, 1024)
        return {"kind": kind, "T": _log(rng, 8, 8192), "E": rng.choice((16, 32, 64, 128)), "N": _cols(rng, 512, 2048, 8),
                "K": K, "k": _tail(rng, K, 128), "mode": rng.choice(("permute", "identity"))}
    if kind == "mxfp8":
        return {"kind": kind, "M": _log(rng, 16, 4096), "N": _cols(rng, 512, 6144, 8), "K": _cols(rng, 512, 4096),
                "mode": rng.choice(("permute", "identity")), "y": rng.choice(("f32", "bf16"))}
    K = _cols(rng, 512, 9728)
    return {"kind": kind, "N": _log(rng, 256, 2560), "K": K, "k": _tail(rng, K), "search": rng.random() < 0.3}


# ---- inputs -------------------------------------------------------------------------------------------------

class _Source:
    """Seeded tensors on the GPU with the distributions of the synthetic layers: weights N(0, 0.02^2), activations
    Student-t(3) times a lognormal gain per channel, one channel in a hundred times 30."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda")

    def gain(self, K):
        gain = torch.exp(self.normal(K))
        loud = torch.randperm(K, generator=self.g, device="cuda")[: round(0.01 * K)]
        gain[loud] *= 30.0
        return gain

    def rows(self, M, gain):
        out = torch.empty((M, gain.numel()), dtype=torch.bfloat16, device="cuda")
        step = max(1, (1 << 24) // gain.numel())
        for r in range(0, M, step):
            n = min(M, r + step) - r
            chi2 = self.normal(3, n, gain.numel()).square_().sum(0)
            out[r:r + n] = self.normal(n, gain.numel()) / torch.sqrt(chi2 / 3) * gain
        return out

    def weight(self, *shape):
        return (self.normal(*shape) * 0.02).to(torch.bfloat16)


def _amax(src, gain, T=512):
    return src.rows(T, gain).abs().amax(0).float().cpu().numpy()


def _bits(t):
    return t.view(torch.int16).cpu().numpy().view(np.uint16)


class _Layer:
    """A prepared layer with the buffers a program keeps for it (or without them, `buffers` False)."""

    def __init__(self, w, M, y_dtype, buffers=True, workspace=True):
        self.w, self.M, self.y_dtype = w, M, y_dtype
        self.act = self.ws = self.y = None
        if buffers:
            codes, sf = (torch.zeros(prq.act_bytes(M, w.K, w.k_tail, w.n_experts, b), dtype=torch.uint8, device="cuda")
                         for b in (prq.BUF_CODES, prq.BUF_SCALES_SF))
            self.act = (codes, None, sf)
            self.ws = prq.new_workspace(w, M) if workspace else None
        if buffers or w.N % 8:
            # rows of y start on 16 bytes
            self.y = torch.empty((M, -(-w.N // 8) * 8), dtype=torch.float32 if y_dtype == prq.F32 else torch.bfloat16,
                                 device="cuda")[:, : w.N]

    def forward(self, x, mode):
        codes, _, sf = prq.quantize_act(self.w, x, mode, out=self.act)
        return prq.linear(self.w, codes, sf, self.M, self.y_dtype, workspace=self.ws, out=self.y)


_MODE = {"identity": prq.ACT_IDENTITY, "permute": prq.ACT_SCALE_PERM}
_DTYPE = {"f32": prq.F32, "bf16": prq.BF16}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, _Source(seed), seed)


def _prepare_linear(c, src, seed):
    gain = src.gain(c["K"])
    w = prq.prepare_weights_device(src.weight(c["N"], c["K"]), _amax(src, gain), 0.5, c["k"])
    return {"case": c, "layer": _Layer(w, c["M"], _DTYPE[c["y"]], c["buffers"]), "x": src.rows(c["M"], gain)}


def _block_layers(src, M, k, k_down):
    """The seven linears of a decoder block and the activations they read (the ones that share one: one tensor)."""
    layers, x = {}, {}
    for names in SHARED:
        K = next(K for n, K, _ in BLOCK if n == names[0])
        gain = src.gain(K)
        amax = _amax(src, gain)
        x[names] = src.rows(M, gain)
        for name, _, N in BLOCK:
            if name in names:
                w = prq.prepare_weights_device(src.weight(N, K), amax, 0.5, k_down if name == "down" else k)
                layers[name] = _Layer(w, M, prq.BF16)
    return layers, x


def _stack_step(s):
    for layers, x in s["stack"]:
        for names in SHARED:
            group = [layers[n] for n in names]
            if s["case"]["form"] == "fused":
                for l in group:
                    prq.linear_fused(l.w, x[names], prq.ACT_IDENTITY, prq.BF16, out=l.y)
            elif len(group) == 1:
                group[0].forward(x[names], prq.ACT_SCALE_PERM)
            else:
                ws = [l.w for l in group]
                acts = prq.quantize_act_multi(ws, x[names], prq.ACT_SCALE_PERM, out=[(l.act[0], l.act[2]) for l in group])
                prq.linear_multi(ws, acts, s["case"]["M"], prq.BF16, out=[l.y for l in group])


def _prepare_stack(c, src, seed):
    s = {"case": c, "stack": [_block_layers(src, c["M"], c["k"], c["k"]) for _ in range(c["layers"])]}
    _stack_step(s)
    torch.cuda.synchronize()
    s["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s["graph"]):
        _stack_step(s)
    s["y"] = [l.y for layers, _ in s["stack"] for l in layers.values()]
    return s


def _prepare_block(c, src, seed):
    layers, x = _block_layers(src, c["M"], c["k"], c["k_down"])
    return {"case": c, "layers": layers, "x": x}


def _prepare_ffn(c, src, seed):
    M, H, C = c["M"], c["H"], c["C"]
    gain_in, gain_mid = src.gain(H), src.gain(C)
    w_down = prq.prepare_weights_device(src.weight(H, C), _amax(src, gain_mid), 0.5, c["k"])
    # the down projection's scaling and permutation go into its producers' rows
    perm = torch.from_numpy(w_down.get(prq.FIELD_PERM)).cuda().long()
    inv_s = torch.from_numpy(w_down.get(prq.FIELD_INV_S)).cuda()
    up = (src.weight(C, H).float()[perm] * inv_s[perm][:, None]).to(torch.bfloat16)
    gate = src.weight(C, H)[perm]
    both = torch.cat([gate.view(C // 32, 32, H), up.view(C // 32, 32, H)], 1).reshape(2 * C, H).contiguous()
    w_gu = prq.prepare_weights_device(both, _amax(src, gain_in), 0.5, c["k_gu"], gated_producer=True)
    mid = tuple(torch.zeros(prq.act_bytes(M, C, c["k"], 1, b), dtype=torch.uint8, device="cuda")
                for b in (prq.BUF_CODES, prq.BUF_SCALES_SF))
    return {"case": c, "gu": _Layer(w_gu, M, prq.BF16, workspace=False), "down": _Layer(w_down, M, prq.BF16), "mid": (mid[0], None, mid[1]),
            "x": src.rows(M, gain_in)}


def _routing(c, seed):
    """Row boundaries of the experts for T tokens, eight experts each with Zipf popularity."""
    return synth.zipf_routing(seed, c["T"], c["E"])[1]


def _prepare_moe(c, src, seed):
    gain = src.gain(c["K"])
    amax = np.stack([_amax(src, gain, 64) for _ in range(c["E"])])
    w = prq.prepare_weights_device(src.weight(c["E"], c["N"], c["K"]), amax, 0.5, c["k"])
    M = 8 * c["T"]
    return {"case": c, "layer": _Layer(w, M, prq.BF16, workspace=False), "x": src.rows(M, gain), "offsets": torch.from_numpy(_routing(c, seed)).cuda()}


def _prepare_mxfp8(c, src, seed):
    gain = src.gain(c["K"])
    total = sum(QKV)
    Ns = [c["N"] * n // total // 8 * 8 for n in QKV[1:]]
    Ns = [c["N"] - sum(Ns)] + Ns
    w = prq.prepare_weights_stacked([_bits(src.weight(n, c["K"])) for n in Ns], _amax(src, gain), 0.5, 0, fmt=prq.FMT_MXFP8)
    x = src.rows(c["M"], gain)
    return {"case": c, "w": w, "x": x, "act": prq.quantize_act(w, x, _MODE[c["mode"]]), "ws": prq.new_workspace(w, c["M"]),
            "y": torch.empty((c["M"], c["N"]), dtype=torch.float32 if c["y"] == "f32" else torch.bfloat16, device="cuda")}


def _prepare_load(c, src, seed):
    gain = src.gain(c["K"])
    return {"case": c, "W": src.weight(c["N"], c["K"]), "amax": _amax(src, gain), "x": src.rows(16, gain)}


_PREPARE = {"linear": _prepare_linear, "stack": _prepare_stack, "block": _prepare_block, "ffn": _prepare_ffn,
            "moe": _prepare_moe, "mxfp8": _prepare_mxfp8, "load": _prepare_load}


# ---- one pass -----------------------------------------------------------------------------------------------

def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "linear":
        l = s["layer"]
        if c["form"] == "fused":
            return prq.linear_fused(l.w, s["x"], prq.ACT_IDENTITY, l.y_dtype, out=l.y)
        return l.forward(s["x"], _MODE[c["mode"]])
    if kind == "stack":
        s["graph"].replay()
        return s["y"]
    if kind == "block":
        return [s["layers"][n].forward(s["x"][names], prq.ACT_SCALE_PERM) for names in SHARED for n in names]
    if kind == "ffn":
        gu, down = s["gu"], s["down"]
        codes, _, sf = prq.quantize_act(gu.w, s["x"], prq.ACT_SCALE_PERM, out=gu.act)
        codes, _, sf, _ = prq.linear_gated(gu.w, codes, sf, gu.M, down.w, out=s["mid"])
        return prq.linear(down.w, codes, sf, down.M, prq.BF16, workspace=down.ws, out=down.y)
    if kind == "moe":
        l = s["layer"]
        codes, _, sf = prq.quantize_act(l.w, s["x"], _MODE[c["mode"]], expert_offsets=s["offsets"], out=l.act)
        return prq.linear_grouped(l.w, codes, sf, s["offsets"], l.M, prq.BF16, out=l.y)
    if kind == "mxfp8":
        codes, _, sf = prq.quantize_act(s["w"], s["x"], _MODE[c["mode"]], out=s["act"])
        return prq.linear(s["w"], codes, sf, c["M"], _DTYPE[c["y"]], workspace=s["ws"], out=s["y"])
    w = prq.prepare_weights_device(s["W"], s["amax"], 0.5, c["k"], scale_search=c["search"])
    codes, _, sf = prq.quantize_act(w, s["x"], prq.ACT_SCALE_PERM)
    y = torch.empty((16, -(-w.N // 8) * 8), dtype=torch.float32, device="cuda")[:, : w.N]
    return {"y": prq.linear(w, codes, sf, 16, prq.F32, out=y), "perm": w.get(prq.FIELD_PERM), "inv_s": w.get(prq.FIELD_INV_S)}


# ---- the same results in 64 bits ------------------------------------------------------------------------------

def _mx(v, elem_exp, rounded, search=False):
    """Blocks of 32 along the last axis: power-of-two scale (floor of the largest magnitude's exponent less `elem_exp`),
    elements through `rounded`; with `search` the neighbouring scales too, the smaller one first, if strictly better."""
    b = v.double().reshape(*v.shape[:-1], -1, 32)
    e0 = (torch.frexp(b.abs().amax(-1, keepdim=True))[1] - 1 - elem_exp).clamp(min=-127)
    best = torch.ldexp(rounded(torch.ldexp(b, -e0)), e0)
    if search:
        err = (b - best).square().sum(-1, keepdim=True)
        for step in (-1, 1):
            e = e0 + step
            q = torch.ldexp(rounded(torch.ldexp(b, -e)), e)
            d = (b - q).square().sum(-1, keepdim=True)
            better = (d < err) & (e >= -127)
            best, err = torch.where(better, q, best), torch.where(better, d, err)
    return best.reshape(v.shape)


def _e2m1(a):
    m = a.abs()
    m = torch.where(m < 2, (m * 2).round() / 2, torch.where(m < 4, m.round(), (m / 2).round() * 2)).clamp(max=6)
    return torch.copysign(m, a)


def _e4m3(a):
    return a.clamp(-448, 448).float().to(torch.float8_e4m3fn).double()


def _exact_scales(amax):
    s = torch.from_numpy(amax).cuda().double().clamp(min=1e-5).sqrt().float()
    return s, (1.0 / s.double()).float()


def _exact_layer(W, amax, k, search=False):
    """(weights in the permuted order, residual of the tail, permutation, reciprocal scales)"""
    s, inv_s = _exact_scales(amax)
    W0 = W.float() * s
    err = (W0.double() - _mx(W0, 2, _e2m1)).square().sum(0)
    tail = torch.sort(err, descending=True, stable=True)[1][:k]
    picked = torch.zeros(W.shape[1], dtype=torch.bool, device="cuda")
    picked[tail] = True
    perm = torch.cat([torch.nonzero(~picked)[:, 0], torch.nonzero(picked)[:, 0]])
    Wt = W0[:, perm]
    Q = _mx(Wt, 2, _e2m1, search)
    R = _mx((Wt.double() - Q)[:, W.shape[1] - k:], 2, _e2m1, search) if k else Q[:, :0]
    return Q, R, perm, inv_s


def _exact_linear(layer, x, mode):
    Q, R, perm, inv_s = layer
    a = _mx((x.float() * inv_s)[:, perm] if mode == "permute" else x, 2, _e2m1)
    return a @ Q.T + a[:, a.shape[1] - R.shape[1]:] @ R.T


def _exact_block(src, M, k, k_down, mode):
    out = []
    for names in SHARED:
        K = next(K for n, K, _ in BLOCK if n == names[0])
        gain = src.gain(K)
        amax = _amax(src, gain)
        x = src.rows(M, gain)
        for name, _, N in BLOCK:
            if name in names:
                out.append(_exact_linear(_exact_layer(src.weight(N, K), amax, k_down if name == "down" else k), x, mode))
    return out


def exact(c, seed):
    """What `run` returns for the same inputs: the layer's quantisation rules and the products of the quantised
    operands in 64 bits, with torch alone."""
    src, kind = _Source(seed), c["kind"]
    if kind == "linear":
        gain = src.gain(c["K"])
        layer = _exact_layer(src.weight(c["N"], c["K"]), _amax(src, gain), c["k"])
        return _exact_linear(layer, src.rows(c["M"], gain), c["mode"])
    if kind == "stack":
        mode = "identity" if c["form"] == "fused" else "permute"
        return [y for _ in range(c["layers"]) for y in _exact_block(src, c["M"], c["k"], c["k"], mode)]
    if kind == "block":
        return _exact_block(src, c["M"], c["k"], c["k_down"], "permute")
    if kind == "ffn":
        H, C = c["H"], c["C"]
        gain_in, gain_mid = src.gain(H), src.gain(C)
        down = _exact_layer(src.weight(H, C), _amax(src, gain_mid), c["k"])
        perm, inv_s = down[2], down[3]
        up = (src.weight(C, H).float()[perm] * inv_s[perm][:, None]).to(torch.bfloat16)
        gate = src.weight(C, H)[perm]
        both = torch.cat([gate.view(C // 32, 32, H), up.view(C // 32, 32, H)], 1).reshape(2 * C, H)
        layer = _exact_layer(both, _amax(src, gain_in), c["k_gu"])
        gu = _exact_linear(layer, src.rows(c["M"], gain_in), "permute").view(c["M"], C // 32, 2, 32)
        h = torch.nn.functional.silu(gu[:, :, 0]) * gu[:, :, 1]
        return _exact_linear(down, h.reshape(c["M"], C).to(torch.bfloat16), "identity")
    if kind == "moe":
        gain = src.gain(c["K"])
        amax = np.stack([_amax(src, gain, 64) for _ in range(c["E"])])
        W = src.weight(c["E"], c["N"], c["K"])
        x, off = src.rows(8 * c["T"], gain), _routing(c, seed)
        return torch.cat([_exact_linear(_exact_layer(W[e], amax[e], c["k"]), x[off[e]:off[e + 1]], c["mode"])
                          for e in range(c["E"]) if off[e + 1] > off[e]])
    if kind == "mxfp8":
        gain = src.gain(c["K"])
        Ns = [c["N"] * n // sum(QKV) // 8 * 8 for n in QKV[1:]]
        Ns = [c["N"] - sum(Ns)] + Ns
        W = torch.cat([src.weight(n, c["K"]) for n in Ns])
        s, inv_s = _exact_scales(_amax(src, gain))
        x = src.rows(c["M"], gain)
        return _mx(x.float() * inv_s if c["mode"] == "permute" else x, 8, _e4m3) @ _mx(W.float() * s, 8, _e4m3).T
    gain = src.gain(c["K"])
    layer = _exact_layer(src.weight(c["N"], c["K"]), _amax(src, gain), c["k"], c["search"])
    y = _exact_linear(layer, src.rows(16, gain), "permute")
    return {"y": y, "perm": layer[2].int().cpu().numpy(), "inv_s": layer[3].double().cpu().numpy()}


# ---- what a pass cannot do without, and how far results may be apart ------------------------------------------

def _layer_work(M, N, K, k, y_bytes, x_bytes=2.0, w_bytes=17 / 32):
    return {"bytes": w_bytes * N * (K + k) + x_bytes * M * K + y_bytes * M * N, "flops": 2.0 * M * N * (K + k)}


def _sum(works):
    works = list(works)
    return {"bytes": sum(w["bytes"] for w in works), "flops": sum(w["flops"] for w in works)}


def work(c):
    kind = c["kind"]
    if kind == "linear":
        return _layer_work(c["M"], c["N"], c["K"], c["k"], 4 if c["y"] == "f32" else 2)
    if kind in ("stack", "block"):
        n = c.get("layers", 1)
        k_down = c.get("k_down", c["k"])
        one = _sum(_layer_work(c["M"], N, K, k_down if name == "down" else c["k"], 2, 0) for name, K, N in BLOCK)
        x = sum(2 * c["M"] * next(K for n_, K, _ in BLOCK if n_ == names[0]) for names in SHARED)
        return {"bytes": n * (one["bytes"] + x), "flops": n * one["flops"]}
    if kind == "ffn":
        C = c["C"]
        return _sum((_layer_work(c["M"], 2 * C, c["H"], c["k_gu"], 0), _layer_work(c["M"], c["H"], C, c["k"], 2, 0)))
    if kind == "moe":
        rows = 8 * c["T"]
        live = int(np.count_nonzero(np.diff(_routing(c, 1))))
        return {"bytes": 17 / 32 * live * c["N"] * (c["K"] + c["k"]) + 2.0 * rows * (c["K"] + c["N"]),
                "flops": 2.0 * rows * c["N"] * (c["K"] + c["k"])}
    if kind == "mxfp8":
        return _layer_work(c["M"], c["N"], c["K"], 0, 4 if c["y"] == "f32" else 2, w_bytes=33 / 32)
    return {"bytes": c["N"] * (2.0 * c["K"] + 17 / 32 * (c["K"] + c["k"])), "flops": 8.0 * c["N"] * (c["K"] + c["k"])}


def tolerance(c):
    # Against sums in float64 of the same operands: MXFP4's products lie on so coarse a grid that the fp32 sums come out
    # the same; E4M3's show 4e-7 (largest 3e-6), and in bf16 7e-5 (one unit in the last place where a sum lies next to a
    # rounding boundary).  The gated producer rounds silu(gate) * up to bf16 and then to four bits: where a code moves,
    # a row of few tokens shows it (3000 rows: 1e-5 in all, 3e-3 at most).
    if c["kind"] == "load" or c.get("y") == "f32":
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.0}
    if c["kind"] == "mxfp8":
        return {"rel": 3e-4, "max": 1.6e-2}
    if c["kind"] == "ffn":
        return {"rel": 2e-3, "max": 5e-2}
    return {"rel": 1e-4, "max": 1e-2}
