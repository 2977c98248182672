"""The workloads that users of this library run, as measurable cases.

A case is one call, or the calls of one layer, of the rotated 4-bit inference
path, through the tensor-level entry points of ``paper_2405_16406_gb300.spinq``
with the output and workspace buffers that a serving loop keeps:

  linear        per-token int4 activation quantizer (with or without the online
                rotation), then the W4A4 GEMM;
  down          the same in one call (``rotated_linear``), optionally with the
                random-sign rotation;
  linear8       the 8-bit linears: W4A8 (int8 codes in two planes) and FP8;
  kv            RoPE (optional), R3 on Q and K, the 4-bit KV-cache quantizer;
  attention     decode attention over the 4-bit cache;
  decode_layer  one decoder layer at decode: kv + attention + the four linears
                (QKV, output, gate/up, down), captured once into a CUDA graph
                and replayed for every token, as decode loops do;
  weights       offline weight preparation: merge the rotation, quantize per
                channel;
  cayley        one Cayley SGD step on a batch of rotations (learning R2).

Sizes are those of the repository's benchmark and tests: layers of 4096 /
14336 and 3072 / 8192, 2048 to 8192 tokens at prefill, 1 to 256 at decode, a
cache of 8 x 4096 tokens; ``draw`` spreads over the same ranges.
"""
from __future__ import annotations

import math

import torch

from paper_2405_16406_gb300 import spinq

DEV = "cuda"

# The online rotation of each reduction length: (n_small, n_pow2).
HAD = {256: (1, 256), 2048: (1, 2048), 3072: (12, 256), 4096: (1, 4096), 8192: (1, 8192), 10240: (20, 512),
       14336: (28, 512)}

# hidden, ffn, query heads, kv heads, head_dim of the decoder layers.
LAYERS = {"h4096": (4096, 14336, 32, 8, 128), "h3072": (3072, 8192, 48, 12, 64)}


def listed():
    return [
        # one token through one projection, called eagerly: the smallest call
        {"name": "linear_1tok", "kind": "linear", "M": 1, "K": 3072, "N": 8192, "rot": True, "sym": True, "clip": 1.0},
        # single-stream decode
        {"name": "decode_layer_b1", "kind": "decode_layer", "layer": "h4096", "B": 1, "S": 2048},
        # batched decode of the smaller layer
        {"name": "decode_layer_b16", "kind": "decode_layer", "layer": "h3072", "B": 16, "S": 1024},
        # a busy server's batch, not a round number
        {"name": "decode_layer_b77", "kind": "decode_layer", "layer": "h4096", "B": 77, "S": 513},
        # prefill, gate/up: asymmetric codes, R1 merged (no online rotation)
        {"name": "gate_up_2048", "kind": "linear", "M": 2048, "K": 4096, "N": 14336, "rot": False, "sym": False,
         "clip": 1.0},
        # prefill, down: online R4 = H28 (x) H512 in the one-call form
        {"name": "down_2048", "kind": "down", "M": 2048, "K": 14336, "N": 4096, "signed": False, "sym": True,
         "clip": 1.0},
        # prefill of the KV cache: RoPE, R3, KV4 (the largest traffic)
        {"name": "kv_8x4096", "kind": "kv", "rope": True, "B": 8, "S": 4096, "Hq": 32, "Hkv": 8, "D": 128},
        # decode attention over long, ragged contexts
        {"name": "attention_8x4096", "kind": "attention", "B": 8, "S": 4096, "Hq": 32, "Hkv": 8, "D": 128},
        # the W4A8 setting, down projection
        {"name": "w4a8_down_2048", "kind": "linear8", "fmt": "w4a8", "M": 2048, "K": 14336, "N": 4096, "rot": True,
         "sym": True},
        # the FP8 setting on a ragged prompt
        {"name": "fp8_gate_up_1531", "kind": "linear8", "fmt": "fp8", "M": 1531, "K": 4096, "N": 14336, "rot": False,
         "sym": True},
        # weight preparation of a down projection: R4 merged into W
        {"name": "merge_down", "kind": "weights", "fmt": "int4", "N": 4096, "K": 14336, "rot": True},
        # learning R2: one 128 x 128 rotation per layer
        {"name": "cayley_32", "kind": "cayley", "batch": 32, "n": 128, "iters": 2},
    ]


def _log(rng, lo, hi):
    """A whole number of [lo, hi], uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["linear", "linear", "down", "linear8", "kv", "attention", "decode_layer", "decode_layer",
                       "weights", "cayley"])
    K, N = rng.choice([(3072, 8192), (8192, 3072), (4096, 14336), (14336, 4096), (4096, 6144), (4096, 4096),
                       (10240, 4096), (2048, 8192), (256, 512)])
    if kind == "linear":
        return {"kind": kind, "M": _log(rng, 1, 4096), "K": K, "N": N, "rot": rng.random() < 0.5,
                "sym": rng.random() < 0.5, "clip": rng.choice([1.0, 1.0, 0.9])}
    if kind == "down":
        K, N = rng.choice([(14336, 4096), (8192, 3072), (10240, 4096), (3072, 3072)])
        return {"kind": kind, "M": _log(rng, 16, 3000), "K": K, "N": N, "signed": rng.random() < 0.3,
                "sym": rng.random() < 0.7, "clip": rng.choice([1.0, 1.0, 0.95])}
    if kind == "linear8":
        fmt = rng.choice(["w4a8", "fp8"])
        return {"kind": kind, "fmt": fmt, "M": _log(rng, 16, 2048), "K": K, "N": N, "rot": rng.random() < 0.5,
                "sym": fmt == "fp8" or rng.random() < 0.5}
    if kind in ("kv", "attention"):
        Hkv = rng.choice([2, 4, 8, 12])
        D = rng.choice([64, 128])
        c = {"kind": kind, "B": _log(rng, 1, 16), "S": _log(rng, 33, 4096), "Hq": Hkv * rng.choice([1, 2, 4]),
             "Hkv": Hkv, "D": D}
        while c["B"] * c["S"] > 8 * 4096:
            c["B"] = (c["B"] + 1) // 2
        if kind == "kv":
            c["rope"] = rng.random() < 0.7
        return c
    if kind == "decode_layer":
        return {"kind": kind, "layer": rng.choice(sorted(LAYERS)), "B": _log(rng, 1, 256), "S": _log(rng, 65, 1024)}
    if kind == "weights":
        return {"kind": kind, "fmt": rng.choice(["int4", "int4", "w4a8", "fp8"]), "N": 16 * _log(rng, 8, 256), "K": K,
                "rot": rng.random() < 0.7}
    return {"kind": kind, "batch": _log(rng, 1, 152), "n": rng.choice([32, 64, 128, 128]), "iters": rng.choice([1, 2, 2, 4])}


# ---------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _acts(g, M, K, share=0.01, factor=30.0):
    """Activations: N(0, 1) with a few outlier channels common to all tokens."""
    x = torch.randn(M, K, generator=g, device=DEV)
    n = max(1, int(K * share))
    x[:, torch.randperm(K, generator=g, device=DEV)[:n]] *= factor
    return x.half()


def _weight(g, N, K):
    return torch.randn(N, K, generator=g, device=DEV) * 0.02


def _int4(w):
    """Round-to-nearest per-channel int4: codes [N, K] (int8) and scales."""
    scale = w.abs().amax(1).clamp_min(1e-12) / 7
    return (w / scale[:, None]).round().clamp(-8, 7).to(torch.int8), scale


def _pack(q):
    return (q[:, 0::2].to(torch.uint8) & 15) | ((q[:, 1::2].to(torch.uint8) & 15) << 4)


def _weight4(g, N, K):
    q, scale = _int4(_weight(g, N, K))
    return spinq.WeightCodes(_pack(q), scale, q.sum(1, dtype=torch.int32))


def _weight8(g, N, K, fmt):
    w = _weight(g, N, K)
    if fmt == "w4a8":
        q, scale = _int4(w)
        return spinq.WeightCodes(q.float().to(torch.float8_e4m3fn).view(torch.uint8), scale, q.sum(1, dtype=torch.int32))
    scale = w.abs().amax(1) / 448
    return spinq.WeightCodes((w / scale[:, None]).to(torch.float8_e4m3fn).view(torch.uint8), scale,
                             torch.zeros(N, dtype=torch.int32, device=DEV))


def _act_out(M, width, sym):
    return spinq.ActCodes(torch.empty(M, width, dtype=torch.uint8, device=DEV), torch.empty(M, device=DEV),
                          None if sym else torch.empty(M, device=DEV))


def _half(*shape):
    return torch.empty(*shape, dtype=torch.float16, device=DEV)


def _kv_out(B, S, Hq, Hkv, D):
    def f32():
        return torch.empty(B, S, Hkv, device=DEV)

    def codes():
        return torch.empty(B, S, Hkv, D // 2, dtype=torch.uint8, device=DEV)

    return spinq.KVCodes(_half(B, S, Hq, D), codes(), f32(), f32(), codes(), f32(), f32())


def _qkv(g, B, S, Hq, Hkv, D):
    """Q, K, V: N(0, 1) with two large channels (as keys have)."""
    out = []
    for h in (Hq, Hkv, Hkv):
        t = torch.randn(B, S, h, D, generator=g, device=DEV)
        t[..., 3] *= 20
        t[..., D - 5] *= 20
        out.append(t.half())
    return out


def _rope_table(max_pos, D):
    ang = torch.arange(max_pos, device=DEV, dtype=torch.float64)[:, None] * (
        10000.0 ** (-torch.arange(0, D, 2, device=DEV, dtype=torch.float64) / D))[None]
    return torch.stack([ang.cos(), ang.sin()], -1)


def _cache4(g, B, S, Hkv, D):
    """Asymmetric int4 codes, scales and zeros of N(0, 1) rows."""
    t = torch.randn(B, S, Hkv, D, generator=g, device=DEV)
    lo, hi = t.amin(-1), t.amax(-1)
    scale = (hi - lo) / 15
    u = ((t - lo[..., None]) / scale[..., None]).round().clamp(0, 15).to(torch.uint8)
    return u[..., 0::2] | (u[..., 1::2] << 4), scale, lo


def _cache(g, B, S, Hkv, D):
    return spinq.KVCodes(None, *_cache4(g, B, S, Hkv, D), *_cache4(g, B, S, Hkv, D))


def _lens(g, B, S):
    return torch.randint(max(1, S // 2), S + 1, (B,), generator=g, device=DEV, dtype=torch.int32)


def _layer_linears(layer):
    """(name, K, N, rotated, symmetric) of a decoder layer's projections."""
    hid, ffn, Hq, Hkv, D = LAYERS[layer]
    return [("qkv", hid, (Hq + 2 * Hkv) * D, False, False), ("o", Hq * D, hid, False, False),
            ("gate_up", hid, 2 * ffn, False, False), ("down", ffn, hid, True, True)]


def _signs(g, K):
    return (torch.randint(0, 2, (K,), generator=g, device=DEV) * 2 - 1).float()


def _rotations(g, batch, n):
    """Orthonormal matrices: products of two random-sign Hadamard rotations."""
    h = torch.ones(1, 1, device=DEV)
    while h.shape[0] < n:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    s = (torch.randint(0, 2, (batch, 2, n), generator=g, device=DEV) * 2 - 1).float()
    return ((h * s[:, 0, None, :]) @ (h * s[:, 1, None, :]) / n).contiguous()


def _inputs(c, seed):
    """The inputs of a case, from the seed alone."""
    g, k = _gen(seed), c["kind"]
    if k in ("linear", "down"):
        w = _weight4(g, c["N"], c["K"])
        share, factor = (0.005, 100.0) if k == "down" else (0.01, 30.0)
        return {"x": _acts(g, c["M"], c["K"], share, factor), "w": w,
                "signs": _signs(g, c["K"]) if c.get("signed") else None}
    if k == "linear8":
        return {"w": _weight8(g, c["N"], c["K"], c["fmt"]), "x": _acts(g, c["M"], c["K"])}
    if k == "kv":
        q, kk, v = _qkv(g, c["B"], c["S"], c["Hq"], c["Hkv"], c["D"])
        pos = torch.arange(c["S"], device=DEV, dtype=torch.int32).repeat(c["B"], 1)
        return {"q": q, "k": kk, "v": v, "pos": pos, "table": _rope_table(c["S"], c["D"])}
    if k == "attention":
        return {"q": torch.randn(c["B"], c["Hq"], c["D"], generator=g, device=DEV).half(),
                "cache": _cache(g, c["B"], c["S"], c["Hkv"], c["D"]), "lens": _lens(g, c["B"], c["S"])}
    if k == "decode_layer":
        _, _, Hq, Hkv, D = LAYERS[c["layer"]]
        B, S = c["B"], c["S"]
        q, kk, v = _qkv(g, B, 1, Hq, Hkv, D)
        lens = _lens(g, B, S)
        return {"q": q, "k": kk, "v": v, "lens": lens, "pos": (lens - 1)[:, None].contiguous(),
                "table": _rope_table(S, D), "cache": _cache(g, B, S, Hkv, D),
                "lin": [(_acts(g, B, K), _weight4(g, N, K)) for _, K, N, _, _ in _layer_linears(c["layer"])]}
    if k == "weights":
        return {"w": _weight(g, c["N"], c["K"]).half()}
    n = c["n"]
    return {"R": _rotations(g, c["batch"], n), "grad": torch.randn(c["batch"], n, n, generator=g, device=DEV) / n}


# ---------------------------------------------------------------- calls


class _State:
    """One case's pass, and what has to live as long as it: a replayed graph
    reads and writes the buffers it was captured on."""

    def __init__(self, run, keep=None):
        self.run, self.keep = run, keep


def _linear_pass(x, w, had, sym, clip):
    M, K = x.shape
    N = w.codes.shape[0]
    out, y = _act_out(M, K // 2, sym), _half(M, N)
    ws = spinq.gemm_workspace(M, N, K)

    def run():
        a = spinq.rotate_quant_act(x, had, symmetric=sym, clip=clip, out=out)
        spinq.w4a4_gemm_splitk(a, w, workspace=ws, y=y)
        return [out.codes, out.scale, out.zero, y]

    return run


def prepare(case, seed):
    c, i, k = case, _inputs(case, seed), case["kind"]
    if k == "linear":
        return _State(_linear_pass(i["x"], i["w"], HAD[c["K"]] if c["rot"] else None, c["sym"], c["clip"]))
    if k == "down":
        x, w, had = i["x"], i["w"], HAD[c["K"]]
        y = _half(c["M"], c["N"])
        ws = torch.empty(spinq.spinq_rotated_linear_workspace_bytes(c["M"], c["K"]), dtype=torch.uint8, device=DEV)
        signs = None if i["signs"] is None else spinq.sign_mask(i["signs"])
        return _State(lambda: spinq.rotated_linear(x, had, w, signs=signs, symmetric=c["sym"], clip=c["clip"], y=y,
                                                   workspace=ws))
    if k == "linear8":
        x, w, had, y = i["x"], i["w"], HAD[c["K"]] if c["rot"] else None, _half(c["M"], c["N"])
        w4a8 = c["fmt"] == "w4a8"
        out = _act_out(c["M"], c["K"] * (2 if w4a8 else 1), c["sym"])
        fmt = spinq.SPINQ_FMT_INT8_PLANES if w4a8 else spinq.SPINQ_FMT_E4M3

        def run8():
            a = spinq.rotate_quant_act8(x, had, fmt, symmetric=c["sym"], out=out)
            (spinq.w4a8_gemm if w4a8 else spinq.fp8_gemm)(a, w, y=y)
            return [out.codes, out.scale, out.zero, y]

        return _State(run8)
    if k == "kv":
        out = _kv_out(c["B"], c["S"], c["Hq"], c["Hkv"], c["D"])
        table = i["table"].float().contiguous()

        def run_kv():
            if c["rope"]:
                o = spinq.rope_rotate_quant_kv(i["q"], i["k"], i["v"], i["pos"], table, out=out)
            else:
                o = spinq.rotate_quant_kv(i["q"], i["k"], i["v"], out=out)
            return [o.q_out, o.k_codes, o.k_scale, o.k_zero, o.v_codes, o.v_scale, o.v_zero]

        return _State(run_kv)
    if k == "attention":
        q, cache, lens, out = i["q"], i["cache"], i["lens"], torch.empty_like(i["q"])
        ws = _attention_ws(c["B"], c["S"], c["Hq"], c["Hkv"], c["D"])
        return _State(lambda: spinq.decode_attention_kv4(q, cache, lens=lens, out=out, workspace=ws))
    if k == "decode_layer":
        return _State(*_decode_layer(c, i))
    if k == "weights":
        w, had = i["w"], HAD[c["K"]] if c["rot"] else None

        def run_w():
            if c["fmt"] == "int4":
                o = spinq.quant_weight(w, had)
            else:
                o = spinq.quant_weight8(w, had, spinq.SPINQ_FMT_INT4_BYTES if c["fmt"] == "w4a8" else spinq.SPINQ_FMT_E4M3)
            return [o.codes, o.scale, None if c["fmt"] == "fp8" else o.rowsum]

        return _State(run_w)
    R, grad, out = i["R"], i["grad"], torch.empty_like(i["R"])
    return _State(lambda: spinq.cayley_step(R, grad, ALPHA, iters=c["iters"], out=out, want_y=True))


ALPHA = 0.5  # Cayley learning rate (gradients of norm about one)


def _attention_ws(B, S, Hq, Hkv, D):
    need = spinq.spinq_decode_attention_workspace_bytes(B, S, Hq, Hkv, D)
    return torch.empty(max(need, 16), dtype=torch.uint8, device=DEV)


def _decode_layer(c, i):
    """One decoder layer's calls for B new tokens, captured into a CUDA graph.
    The residual, the norms, SiLU and the append to the cache are the model's
    own operations and stay outside, so every projection has its input in hand."""
    _, _, Hq, Hkv, D = LAYERS[c["layer"]]
    B, S = c["B"], c["S"]
    kv, table = _kv_out(B, 1, Hq, Hkv, D), i["table"].float().contiguous()
    att, ws = _half(B, Hq, D), _attention_ws(B, S, Hq, Hkv, D)
    lins = [_linear_pass(x, w, HAD[K] if rot else None, sym, 1.0)
            for (x, w), (_, K, _, rot, sym) in zip(i["lin"], _layer_linears(c["layer"]))]

    def calls():
        spinq.rope_rotate_quant_kv(i["q"], i["k"], i["v"], i["pos"], table, out=kv)
        spinq.decode_attention_kv4(kv.q_out.view(B, Hq, D), i["cache"], lens=i["lens"], out=att, workspace=ws)
        outs = [kv.q_out, kv.k_codes, kv.k_scale, kv.k_zero, kv.v_codes, kv.v_scale, kv.v_zero, att]
        for f in lins:
            outs += f()
        return outs

    calls()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        outs = calls()

    def run():
        graph.replay()
        return outs

    return run, calls


def run(state):
    return state.run()


# ---------------------------------------------------------------- work


def _linear_work(M, N, K, w_bytes, a_bytes):
    """fp16 rows in, codes and scales out and in again as one hand-over, the
    weights once, fp16 outputs."""
    return {"bytes": 2 * M * K + a_bytes * M * K + 8 * M + w_bytes * N * K + 8 * N + 2 * M * N, "flops": 2 * M * N * K}


def _kv_work(B, S, Hq, Hkv, D, rope):
    T = B * S
    return T * Hq * 4 * D + 2 * T * Hkv * (2 * D + D // 2 + 8) + (4 * T + 4 * S * D if rope else 0)


def _attention_work(B, S, Hq, Hkv, D):
    t = 0.75 * B * S   # lens are uniform in [S / 2, S]
    return {"bytes": t * Hkv * (D + 16) + 4 * B * Hq * D, "flops": 4 * t * Hq * D}


def work(case):
    c, k = case, case["kind"]
    if k in ("linear", "down"):
        return _linear_work(c["M"], c["N"], c["K"], 0.5, 0.5 if k == "linear" else 0.0)
    if k == "linear8":
        return _linear_work(c["M"], c["N"], c["K"], 1.0, 2.0 if c["fmt"] == "w4a8" else 1.0)
    if k == "kv":
        return {"bytes": _kv_work(c["B"], c["S"], c["Hq"], c["Hkv"], c["D"], c["rope"]), "flops": 0}
    if k == "attention":
        return _attention_work(c["B"], c["S"], c["Hq"], c["Hkv"], c["D"])
    if k == "decode_layer":
        _, _, Hq, Hkv, D = LAYERS[c["layer"]]
        total = _attention_work(c["B"], c["S"], Hq, Hkv, D)
        total["bytes"] += _kv_work(c["B"], 1, Hq, Hkv, D, True)
        for _, K, N, _, _ in _layer_linears(c["layer"]):
            w = _linear_work(c["B"], N, K, 0.5, 0.5)
            total = {m: total[m] + w[m] for m in total}
        return total
    if k == "weights":
        return {"bytes": c["N"] * c["K"] * (2.5 if c["fmt"] == "int4" else 3) + 8 * c["N"], "flops": 0}
    n = c["n"]
    return {"bytes": 16 * c["batch"] * n * n, "flops": (4 + c["iters"]) * 2 * c["batch"] * n ** 3}


# ---------------------------------------------------------------- 64 bits


def _gf27_char():
    """The quadratic character chi(a_i - a_j) of GF(27) = GF(3)[t] / (t^3 + 2t + 1),
    element i = c0 + 3 c1 + 9 c2."""
    def dig(i):
        return [i % 3, i // 3 % 3, i // 9]

    def num(d):
        return d[0] + 3 * d[1] + 9 * d[2]

    def mul(a, b):
        p = [0] * 5
        for x in range(3):
            for y in range(3):
                p[x + y] += a[x] * b[y]
        for e in (4, 3):   # t^3 = t + 2
            p[e - 2] += p[e]
            p[e - 3] += 2 * p[e]
        return [v % 3 for v in p[:3]]

    squares = {num(mul(dig(i), dig(i))) for i in range(1, 27)}
    return [[0 if i == j else 1 if num([(x - y) % 3 for x, y in zip(dig(i), dig(j))]) in squares else -1
             for j in range(27)] for i in range(27)]


def _small_hadamard(n):
    if n == 1:
        return torch.ones(1, 1, dtype=torch.float64, device=DEV)
    q = n - 1
    if q == 27:
        chi = _gf27_char()
    else:
        squares = {x * x % q for x in range(1, q)}
        chi = [[0 if i == j else 1 if (i - j) % q in squares else -1 for j in range(q)] for i in range(q)]
    rows = [[1] + [1] * q] + [[-1] + [chi[i][j] + (i == j) for j in range(q)] for i in range(q)]
    return torch.tensor(rows, dtype=torch.float64, device=DEV)


def _rotate(x, had):
    """x (H_s (x) H_P) / sqrt(K) over the last dimension."""
    ns, P = had
    shape, K = x.shape, ns * P
    t = x.reshape(-1, ns, P)
    h = 1
    while h < P:
        t = t.reshape(-1, P // (2 * h), 2, h)
        t = torch.stack([t[:, :, 0] + t[:, :, 1], t[:, :, 0] - t[:, :, 1]], 2)
        h *= 2
    t = t.reshape(-1, ns, P)
    if ns > 1:
        t = torch.einsum("rip,ij->rjp", t, _small_hadamard(ns))
    return (t / math.sqrt(K)).reshape(shape)


def _quant(x, bits, sym, clip=1.0):
    """Eq. 1 per row: dequantized values, scale, zero."""
    if sym:
        qmax = 2 ** (bits - 1) - 1
        scale = clip * x.abs().amax(-1) / qmax
        return (x / scale[..., None]).round().clamp(-qmax - 1, qmax) * scale[..., None], scale, None
    lo, hi = clip * x.amin(-1), clip * x.amax(-1)
    scale = (hi - lo) / (2 ** bits - 1)
    u = ((x - lo[..., None]) / scale[..., None]).round().clamp(0, 2 ** bits - 1)
    return u * scale[..., None] + lo[..., None], scale, lo


def _nibbles(codes, signed):
    u = torch.stack([codes & 15, codes >> 4], -1).reshape(*codes.shape[:-1], -1).to(torch.float64)
    return torch.where(u > 7, u - 16, u) if signed else u


def _exact_linear(x, w, had, sym, clip):
    x = x.double()
    a, scale, zero = _quant(_rotate(x, had) if had else x, 4, sym, clip)
    return [None, scale, zero, a @ (_nibbles(w.codes, True) * w.scale.double()[:, None]).T]


def _exact_kv(i, Hq, Hkv, D, rope):
    out = []
    for name in ("q", "k", "v"):
        t = i[name].double()
        if name != "v":
            if rope:
                cs = i["table"][i["pos"].long()][:, :, None]   # [B, S, 1, D/2, 2]
                a, b = t[..., : D // 2], t[..., D // 2:]
                t = torch.cat([a * cs[..., 0] - b * cs[..., 1], a * cs[..., 1] + b * cs[..., 0]], -1)
            t = _rotate(t, (1, D))
        if name == "q":
            out.append(t)
        else:
            _, scale, zero = _quant(t, 4, False)
            out += [None, scale, zero]
    return out


def _exact_attention(q, cache, lens):
    """q [B, Hq, D] in 64 bits over the dequantized cache."""
    outs = []
    Hkv = cache.k_codes.shape[2]
    for b in range(q.shape[0]):
        n = int(lens[b])
        k, v = (_nibbles(codes[b, :n], False) * s[b, :n, :, None].double() + z[b, :n, :, None].double()
                for codes, s, z in ((cache.k_codes, cache.k_scale, cache.k_zero),
                                    (cache.v_codes, cache.v_scale, cache.v_zero)))
        qq = q[b].double().reshape(Hkv, -1, q.shape[-1])
        p = torch.softmax(torch.einsum("hgd,thd->hgt", qq, k) / math.sqrt(q.shape[-1]), -1)
        outs.append(torch.einsum("hgt,thd->hgd", p, v).reshape(q.shape[1:]))
    return torch.stack(outs)


def exact(case, seed):
    c, i, k = case, _inputs(case, seed), case["kind"]
    if k == "linear":
        return _exact_linear(i["x"], i["w"], HAD[c["K"]] if c["rot"] else None, c["sym"], c["clip"])
    if k == "down":
        x = i["x"].double()
        if i["signs"] is not None:
            x = x * i["signs"].double()
        return _exact_linear(x, i["w"], HAD[c["K"]], c["sym"], c["clip"])[3]
    if k == "linear8":
        x, w = i["x"].double(), i["w"]
        x = _rotate(x, HAD[c["K"]]) if c["rot"] else x
        if c["fmt"] == "w4a8":
            a, scale, zero = _quant(x, 8, c["sym"])
        else:
            scale, zero = x.abs().amax(-1) / 448, None
            a = (x / scale[:, None]).float().to(torch.float8_e4m3fn).double() * scale[:, None]
        wd = w.codes.view(torch.float8_e4m3fn).double() * w.scale.double()[:, None]
        return [None, scale, zero, a @ wd.T]
    if k == "kv":
        return _exact_kv(i, c["Hq"], c["Hkv"], c["D"], c["rope"])
    if k == "attention":
        return _exact_attention(i["q"], i["cache"], i["lens"])
    if k == "decode_layer":
        _, _, Hq, Hkv, D = LAYERS[c["layer"]]
        outs = _exact_kv(i, Hq, Hkv, D, True)
        outs.append(_exact_attention(outs[0].reshape(c["B"], Hq, D), i["cache"], i["lens"]))
        for (x, w), (_, K, _, rot, sym) in zip(i["lin"], _layer_linears(c["layer"])):
            outs += _exact_linear(x, w, HAD[K] if rot else None, sym, 1.0)
        return outs
    if k == "weights":
        x = i["w"].double()
        x = _rotate(x, HAD[c["K"]]) if c["rot"] else x
        return [None, x.abs().amax(1) / (448 if c["fmt"] == "fp8" else 7), None]
    R, G = i["R"].double(), -i["grad"].double()
    Rt = R.transpose(1, 2)
    Gh = G @ Rt - 0.5 * R @ Rt @ G @ Rt
    Y = Gh - Gh.transpose(1, 2)
    out = R + ALPHA * Y @ R
    for _ in range(c["iters"]):
        out = R + 0.5 * ALPHA * Y @ (R + out)
    return [out, Y]
