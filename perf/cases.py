"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values; `kind` says which public entry point it goes through:

  step   one pass through the linear layers of `blocks` LLaMA-shaped transformer blocks, four launch units per block
         (q|k|v fused, o, gate|up fused, down), through eora_linear_forward_fused / eora_linear_forward.  With few
         tokens (decoding) the program keeps a CUDA graph of the pass, as serving programs and the benchmark do; with
         many (prefill) it makes the calls.  Several blocks, so that the weights of a pass come from HBM as in a model.
  layer  one eora_linear_forward of one layer.
  multi  one eora_linear_forward_multi: a batch of requests, each with its own adapter on a shared backbone.
  host   one eora_linear_forward_fused_host of a q|k|v group: activations in pinned host memory.
  solve  one offline EoRA solve (Algorithm 1, steps 1-6) of a layer.
"""
from __future__ import annotations

import math

import torch

import paper_2410_21271_b200 as E
from paper_2410_21271_b200 import traffic

DEV = "cuda:0"
AB_CODE = {"f16": E.EORA_AB_F16, "q4": E.EORA_AB_Q4, "q3": E.EORA_AB_Q3, "q8": E.EORA_AB_Q8}
X_CODE = {"f16": E.EORA_X_F16, "bf16": E.EORA_X_BF16}
Y_CODE = {"f16": E.EORA_Y_F16, "bf16": E.EORA_Y_BF16, "f32": E.EORA_Y_F32}
TORCH = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    llama8b = {"hidden": 4096, "kv": 1024, "inter": 14336}
    base = {"w": "q4", "group": 128, "ab": "f16", "rank": 128, "x": "f16", "y": "f16"}
    return [
        # the smallest call there is in an LLaMA3-8B layer set: one key projection for one token
        {**base, "name": "k layer, 1 token", "kind": "layer", "d_in": 4096, "d_out": 1024, "m": 1},
        # batch-1 decoding, 3-bit backbone: the paper's latency table and the benchmark's headline
        {**base, **llama8b, "name": "decode 3-bit, 1 token", "kind": "step", "w": "q3", "m": 1, "blocks": 4},
        # batch-1 decoding with a 2:4 sparse fp16 backbone
        {**base, **llama8b, "name": "decode 2:4, 1 token", "kind": "step", "w": "sp24", "m": 1, "blocks": 2},
        # a small batch of requests decoding together
        {**base, **llama8b, "name": "decode 3-bit, 8 tokens", "kind": "step", "w": "q3", "m": 8, "blocks": 4},
        # a medium batch, adapters quantised like the backbone
        {**base, **llama8b, "name": "decode 4-bit, 16 tokens", "kind": "step", "ab": "q4", "m": 16, "blocks": 4},
        # a large decode batch with the largest adapters, 8 bits per channel
        {**base, **llama8b, "name": "decode 4-bit, 64 tokens", "kind": "step", "ab": "q8", "rank": 512, "m": 64, "blocks": 3},
        # several task adapters on one backbone, a ragged batch of requests (one of them without an adapter)
        {**base, "name": "4 adapters, 7 tokens", "kind": "multi", "rank": 64, "d_in": 4096, "d_out": 4096, "adapters": 4, "m": 7},
        # a caller whose activations live in pinned host memory
        {**base, "name": "q|k|v from host, 1 token", "kind": "host", "w": "q3", "hidden": 4096, "kv": 1024, "m": 1},
        # a short prompt (or a chunk of a long one) of a bf16 model, an odd number of tokens
        {**base, **llama8b, "name": "prompt of 333, bf16", "kind": "step", "x": "bf16", "y": "bf16", "rank": 64, "m": 333, "blocks": 1},
        # prefill of the benchmark's length through a whole block
        {**base, **llama8b, "name": "prefill 4-bit, 2048 tokens", "kind": "step", "m": 2048, "blocks": 1},
        # prefill through a 2:4 sparse down projection
        {**base, "name": "prefill 2:4 down, 2048", "kind": "layer", "w": "sp24", "d_in": 14336, "d_out": 4096, "m": 2048},
        # the offline half: the low-rank pair of a q-shaped layer at the paper's rank
        {"name": "solve 4096 x 4096", "kind": "solve", "d": 4096, "k": 4096, "n": 2048, "rank": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(v, q):
    return max(q, int(round(v / q)) * q)


def draw(rng):
    kind = rng.choices(["step", "layer", "multi", "host", "solve"], [45, 25, 8, 8, 14])[0]
    if kind == "solve":
        d, k = _log_int(rng, 512, 4096), _log_int(rng, 512, 4096)
        d, k = (d, k) if rng.random() < 0.3 else (_mult(d, 128), _mult(k, 128))
        return {"kind": kind, "d": d, "k": k, "n": rng.choice([512, 1000, 2048, _log_int(rng, 256, 2048)]), "rank": rng.choice([32, 64, 100, 128, 128, 256])}
    w = rng.choices(["q4", "q3", "sp24", "sq4"], [4, 4, 2, 1])[0]
    ab = rng.choices(["f16", "q4", "q3", "q8"], [5, 2, 1, 2])[0]
    x, y = rng.choice([("f16", "f16"), ("f16", "f16"), ("bf16", "bf16"), ("f16", "f32")])
    c = {"kind": kind, "w": w, "group": rng.choice([128, 128, 128, 64]), "ab": ab, "x": x, "y": y}
    c["rank"] = rng.choice([64, 128, 128, 256, 512]) if ab in ("q4", "q3") else rng.choice([0, 24, 64, 128, 128, 256, 512])
    if kind in ("multi", "host"):
        c["rank"] = c["rank"] or 64
    # decoding batches are small numbers, prompts anything up to the benchmark's length
    m = _log_int(rng, 1, 64) if rng.random() < 0.65 else _log_int(rng, 65, 2048)
    if kind == "step":
        hidden = _mult(_log_int(rng, 1024, 4096), 128)
        c.update(hidden=hidden, kv=_mult(hidden / rng.choice([1, 2, 4, 8]), 128), inter=min(14336, _mult(hidden * rng.uniform(2.5, 3.6), 128)), m=m)
        c["blocks"] = 1 if m > 64 else rng.choice([2, 3, 4])
    elif kind == "layer":
        c.update(d_in=_mult(_log_int(rng, 1024, 14336), 128), d_out=_mult(_log_int(rng, 512, 14336), 32), m=m)
    elif kind == "multi":
        c.update(d_in=_mult(_log_int(rng, 1024, 8192), 128), d_out=_mult(_log_int(rng, 1024, 8192), 32), adapters=rng.randint(2, 8), m=_log_int(rng, 1, 32))
        c["rank"] = min(c["rank"], 128)
    else:
        hidden = _mult(_log_int(rng, 1024, 5120), 128)
        c.update(hidden=hidden, kv=_mult(hidden / rng.choice([1, 2, 4, 8]), 128), m=_log_int(rng, 1, 16))
    return c


# ------------------------------------------------------------------------------------------------------- inputs
class _Gen:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(seed)

    def words(self, *shape):
        return torch.randint(-2**31, 2**31, shape, dtype=torch.int32, device=DEV, generator=self.g)

    def ints(self, hi, *shape):
        return torch.randint(0, hi, shape, dtype=torch.int64, device=DEV, generator=self.g)

    def normal(self, *shape, std=1.0, dtype=torch.float16):
        return (torch.randn(shape, device=DEV, generator=self.g) * std).to(dtype)

    def scales(self, *shape):
        return (0.002 + torch.randn(shape, device=DEV, generator=self.g).abs() * 1e-3).to(torch.float16)


def _pack(codes, bits):
    """Integer codes [count][C] -> LSB-first bit stream along axis 0, int32 [bits * count / 32][C]."""
    count, cols = codes.shape
    per = 8 if bits == 4 else 32
    c = codes.to(torch.int64).reshape(count // per, per, cols)
    words = torch.zeros((count // per, per * bits // 32 + 1, cols), dtype=torch.int64, device=codes.device)
    for e in range(per):
        i, off = divmod(bits * e, 32)
        v = c[:, e] << off
        words[:, i] |= v & 0xFFFFFFFF
        words[:, i + 1] |= v >> 32
    words = words[:, :-1].reshape(-1, cols)
    return torch.where(words >= 2**31, words - 2**32, words).to(torch.int32)


def _positions(g, n, k):
    """2:4 position words of n rows: per quad two random places p0 < p1."""
    pairs = torch.tensor([p0 | p1 << 2 for p0 in range(4) for p1 in range(p0 + 1, 4)], device=DEV)
    nib = pairs[g.ints(6, n, k // 32, 8)]
    words = (nib << (4 * torch.arange(8, device=DEV))).sum(-1)
    return torch.where(words >= 2**31, words - 2**32, words).to(torch.int32)


def _backbone(g, c, k, n):
    """(codes or values, scales, zeros or positions, positions of the combined format) as the library takes them."""
    w, grp = c["w"], c["group"]
    if w == "sp24":
        return g.normal(n, k // 2, std=0.02), None, _positions(g, n, k), None
    bits = 3 if w == "q3" else 4
    kept = k // 2 if w == "sq4" else k
    return g.words(bits * kept // 32, n), g.scales(k // grp, n), g.words(k // grp, bits * n // 32), _positions(g, n, k) if w == "sq4" else None


def _adapter_matrix(g, ab, rows, cols):
    """One matrix of a pair with entries ~ N(0, 0.02^2): fp16, or the codes, scales and zero-points that round-to-nearest
    quantisation of such a matrix gives (range of a group about +-2.7 standard deviations)."""
    if ab == "f16":
        return g.normal(rows, cols, std=0.02), None, None
    bits = {"q4": 4, "q3": 3, "q8": 8}[ab]
    top = 2**bits - 1
    groups = 1 if ab == "q8" else rows // min(128, rows)
    reach = 3.7 if ab == "q8" else 2.7
    codes = torch.clamp(torch.round(top / 2 + torch.randn((rows, cols), device=DEV, generator=g.g) * (top / (2 * reach))), 0, top).to(torch.int64)
    scales = (0.02 * 2 * reach / top * (1 + 0.1 * torch.randn((groups, cols), device=DEV, generator=g.g))).to(torch.float16)
    zeros = top // 2 + g.ints(2, groups, cols)
    if ab == "q8":
        return codes.to(torch.uint8), scales.reshape(-1), zeros.to(torch.uint8).reshape(-1)
    return _pack(codes, bits), scales, _pack(zeros.t().contiguous(), bits).t().contiguous()


def _layer(g, c, k, n, max_m, adapters=1):
    """The config and weight structs of one layer (one weight struct per adapter) and the buffers behind them."""
    cfg = E.eora_linear_config()
    cfg.d_in, cfg.d_out, cfg.rank, cfg.max_m = k, n, c["rank"], max_m
    cfg.w_format = {"sp24": E.EORA_W_SPARSE24, "sq4": E.EORA_W_SPARSE24_Q4}.get(c["w"], E.EORA_W_QUANT)
    cfg.w_bits, cfg.w_group = 3 if c["w"] == "q3" else 4, c["group"]
    cfg.ab_format, cfg.ab_group = AB_CODE[c["ab"]], 128
    cfg.x_dtype, cfg.y_dtype, cfg.kernel_policy = X_CODE[c["x"]], Y_CODE[c["y"]], E.EORA_POLICY_AUTO
    back = _backbone(g, c, k, n)
    wts, keep = [], [back]
    for _ in range(adapters):
        t = E.eora_linear_weights()
        t.w_codes, t.w_scales, t.w_zeros, t.w_meta = [None if b is None else b.data_ptr() for b in back]
        if c["rank"]:
            a, b = _adapter_matrix(g, c["ab"], k, c["rank"]), _adapter_matrix(g, c["ab"], c["rank"], n)
            t.a, t.a_scales, t.a_zeros, t.b, t.b_scales, t.b_zeros = [None if v is None else v.data_ptr() for v in (*a, *b)]
            keep += [a, b]
        wts.append(t)
    return cfg, wts, keep


class _Handle:
    """Owns a library handle."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        if torch is not None and self.h:
            torch.cuda.synchronize()
            E.eora_linear_destroy(self.h)
            self.h = None


def _x(g, c, m, k):
    return g.normal(m, k, dtype=TORCH[c["x"]])


def _y(c, m, n):
    return torch.empty((m, n), dtype=TORCH[c["y"]], device=DEV)


def _fused(g, c, k, outs, m):
    parts = [_layer(g, c, k, n, m) for n in outs]
    return _Handle(E.eora_linear_create_fused([p[0] for p in parts], [p[1][0] for p in parts]))


def _single(g, c, k, n, m):
    cfg, wts, _keep = _layer(g, c, k, n, m)
    return _Handle(E.eora_linear_create(cfg, wts[0]))


def _quantised_copy(w):
    """Round-to-nearest 3-bit copy of a weight in groups of 128 along its inputs (the last group may be shorter)."""
    d, k = w.shape
    pad = -k % 128
    g = torch.nn.functional.pad(w, (0, pad)).reshape(d, -1, 128)
    lo, hi = g.amin(-1, keepdim=True), g.amax(-1, keepdim=True)
    s = (hi - lo).clamp_min(1e-8) / 7
    return (torch.round((g - lo) / s) * s + lo).reshape(d, -1)[:, :k].contiguous()


def prepare(case, seed):
    c, g = case, _Gen(seed)
    if c["kind"] == "solve":
        d, k, n = c["d"], c["k"], c["n"]
        w = g.normal(d, k, std=0.02, dtype=torch.float32)
        # calibration activations: channels of different size (a few large), directions with a power-law spectrum
        q = min(k, n)
        z = torch.randn((q, n), device=DEV, generator=g.g) / torch.arange(1, q + 1, device=DEV).pow(0.75)[:, None]
        x = torch.randn((k, q), device=DEV, generator=g.g) @ z + 0.02 * torch.randn((k, n), device=DEV, generator=g.g)
        x *= torch.exp(0.5 * torch.randn((k, 1), device=DEV, generator=g.g))
        return {"case": c, "w": w, "w_hat": _quantised_copy(w), "x": x.contiguous()}
    if c["kind"] == "layer":
        return {"case": c, "h": _single(g, c, c["d_in"], c["d_out"], c["m"]), "x": _x(g, c, c["m"], c["d_in"]), "y": _y(c, c["m"], c["d_out"])}
    if c["kind"] == "multi":
        cfg, wts, _keep = _layer(g, c, c["d_in"], c["d_out"], c["m"], c["adapters"])
        ids = g.ints(c["adapters"] + 1, c["m"]).tolist()
        return {"case": c, "h": _Handle(E.eora_linear_create_multi(cfg, wts)), "ids": [i - 1 for i in ids],
                "x": _x(g, c, c["m"], c["d_in"]), "y": _y(c, c["m"], c["d_out"])}
    if c["kind"] == "host":
        outs = [c["hidden"], c["kv"], c["kv"]]
        return {"case": c, "h": _fused(g, c, c["hidden"], outs, c["m"]), "x": _x(g, c, c["m"], c["hidden"]).cpu().pin_memory(),
                "ys": [torch.empty((c["m"], n), dtype=TORCH[c["y"]]).pin_memory() for n in outs]}
    # step
    h, kv, f, m = c["hidden"], c["kv"], c["inter"], c["m"]
    units = []
    for _ in range(c["blocks"]):
        units.append((_fused(g, c, h, [h, kv, kv], m), _x(g, c, m, h), [_y(c, m, n) for n in (h, kv, kv)]))
        units.append((_single(g, c, h, h, m), _x(g, c, m, h), [_y(c, m, h)]))
        units.append((_fused(g, c, h, [f, f], m), _x(g, c, m, h), [_y(c, m, f) for _ in range(2)]))
        units.append((_single(g, c, f, h, m), _x(g, c, m, f), [_y(c, m, h)]))
    s = {"case": c, "units": units, "ys": [u[2] for u in units], "graph": None}
    if m <= 64:                                   # decoding: a graph of the step, kept for every token that follows
        _calls(units, m)                          # first use outside the capture
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _calls(units, m)
    return s


# ---------------------------------------------------------------------------------------------------- the calls
def _calls(units, m):
    for hd, x, ys in units:
        if len(ys) > 1:
            E.eora_linear_forward_fused(hd.h, x, m, ys)
        else:
            E.eora_linear_forward(hd.h, x, m, ys[0])


def run(s):
    c = s["case"]
    if c["kind"] == "step":
        if s["graph"] is not None:
            s["graph"].replay()
        else:
            _calls(s["units"], c["m"])
        return s["ys"]
    if c["kind"] == "layer":
        E.eora_linear_forward(s["h"].h, s["x"], c["m"], s["y"])
        return s["y"]
    if c["kind"] == "multi":
        E.eora_linear_forward_multi(s["h"].h, s["x"], c["m"], s["ids"], s["y"])
        return s["y"]
    if c["kind"] == "host":
        E.eora_linear_forward_fused_host(s["h"].h, s["x"], c["m"], s["ys"])
        return s["ys"]
    b, a, sigma = E.solve(s["w"], s["w_hat"], s["x"], c["rank"])
    # B' and A are unique up to one sign per rank-one pair, their product (the compensation) is unique
    return {"compensation": b @ a, "sigma": sigma}


# --------------------------------------------------------------------------------------------------- accounting
def _groups(c):
    """(d_in, [d_out ...], adapters) of every launch unit of a pass."""
    if c["kind"] == "step":
        h, kv, f = c["hidden"], c["kv"], c["inter"]
        return [(h, [h, kv, kv], 1), (h, [h], 1), (h, [f, f], 1), (f, [h], 1)] * c["blocks"]
    if c["kind"] == "host":
        return [(c["hidden"], [c["hidden"], c["kv"], c["kv"]], 1)]
    return [(c["d_in"], [c["d_out"]], c.get("adapters", 1))]


def work(case):
    c = case
    if c["kind"] == "solve":
        d, k, n, r = c["d"], c["k"], c["n"], c["rank"]
        # the projected error (W - W^) X~ and the two sides of its rank-r part
        return {"bytes": 4 * (2 * d * k + k * n + d * r + r * k + r), "flops": 2 * d * k * n + 2 * r * d * (k + n)}
    yb = 4 if c["y"] == "f32" else 2
    b = f = 0
    for k, outs, adapters in _groups(c):
        b += 2 * c["m"] * k
        for n in outs:
            b += traffic.backbone_bytes(c["w"], k, n, c["group"]) + adapters * traffic.adapter_bytes(c["ab"], k, n, c["rank"]) + yb * c["m"] * n
            f += traffic.forward_flops(k, n, c["rank"], c["m"])
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["kind"] == "solve":
        # rounding of the fp32 products over the relative gap between the singular values on both sides of the cut (1 %)
        return {"rel": 1e-3}
    # the rounding of the output, of weights that are dequantised to fp16 (2.8e-4) and of t = X.A where it is held in fp16
    return {"rel": {"f16": 1e-3, "bf16": 6e-3, "f32": 6e-4}[case["y"]]}
