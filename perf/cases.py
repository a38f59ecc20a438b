"""Measured cases: training steps and evaluations of low-rank decomposed layers through the library's C ABI.

A case is one of three kinds:
  "linear"  one decomposed fully connected layer: forward + backward under a freeze mask ("train"), the same with the
            gradients added to the caller's buffers ("accumulate": micro-batches), or the forward alone ("eval");
  "block"   the six decomposed layers of a transformer block (query / key / value as one group, output projection, two
            feed-forward layers), forward, then backward with the weight gradients on a second stream beside the next
            layer's data pass;
  "tucker"  one Tucker-2 decomposed k x k convolution, forward + backward under a freeze mask.
Factors, activations and incoming gradients are drawn on the device from the seed: X and dY ~ N(0, 1), factors scaled so
that the intermediates and outputs stay at unit scale.
"""
from __future__ import annotations

import math

import torch

from paper_2309_03824_b200 import binding as b

DTYPES = {"bf16": (b.LRD_BF16, torch.bfloat16), "f32": (b.LRD_F32, torch.float32)}
MASKS = {"none": b.LRD_FREEZE_NONE, "U": b.LRD_FREEZE_U, "V": b.LRD_FREEZE_V}
TUCKER_MASKS = {"none": b.LRD_TK_FREEZE_NONE, "factors": b.LRD_TK_FREEZE_FACTORS, "core": b.LRD_TK_FREEZE_CORE}


def _linear(mode, M, K, N, r, dtype, freeze):
    return {"kind": "linear", "mode": mode, "M": M, "K": K, "N": N, "r": r, "dtype": dtype, "freeze": freeze}


def _block(M, d, r, freeze):
    """A block of model width d: four d -> d layers of rank r, d -> 4 d and 4 d -> d of rank 2 r."""
    return {"kind": "block", "M": M, "d": d, "r": r, "dtype": "bf16", "freeze": freeze}


def _tucker(B, H, W, C, S, r1, r2, k, stride, dtype, freeze):
    return {"kind": "tucker", "B": B, "H": H, "W": W, "C": C, "S": S, "r1": r1, "r2": r2, "k": k, "stride": stride,
            "dtype": dtype, "freeze": freeze}


def listed():
    cases = [
        # evaluating a decomposed feed-forward layer on a short batch: one launch, all latency
        ("eval_small", _linear("eval", 64, 768, 3072, 384, "bf16", "U")),
        # a small fp32 layer trained with nothing frozen, rank as the compression ratio gives it
        ("fc_f32_small", _linear("train", 256, 512, 512, 40, "f32", "none")),
        # an attention projection on one short sequence batch: the smallest bf16 training step
        ("attn_small", _linear("train", 128, 768, 768, 192, "bf16", "U")),
        # the same projection at an ordinary batch of 32 x 128 tokens, the other mask
        ("attn", _linear("train", 4096, 768, 768, 192, "bf16", "V")),
        # the expanding feed-forward layer at that batch
        ("ffn_1", _linear("train", 4096, 768, 3072, 384, "bf16", "U")),
        # a wide layer on 8192 tokens, quantized rank, nothing frozen: the largest
        ("wide_quantized", _linear("train", 8192, 4096, 4096, 512, "bf16", "none")),
        # the same layer with a rank as the ratio gives it, factors stored packed
        ("wide_packed_rank", _linear("train", 8192, 4096, 4096, 250, "bf16", "V")),
        # gradient accumulation over micro-batches of an odd number of tokens
        ("micro_batch", _linear("accumulate", 1021, 1024, 4096, 512, "bf16", "V")),
        # one step of a whole transformer block at 32 x 128 tokens
        ("block", _block(4096, 768, 192, "V")),
        # a residual network's 3 x 3 convolution, decomposed, core frozen
        ("conv", _tucker(64, 14, 14, 256, 256, 96, 96, 3, 1, "bf16", "core")),
        # its downsampling block: the same convolution with stride 2, 1 x 1 factors frozen
        ("conv_stride2", _tucker(64, 28, 28, 256, 256, 96, 96, 3, 2, "bf16", "factors")),
        # the last stage on 7 x 7 images at the rank of the compression formula (odd), nothing frozen
        ("conv_packed_rank", _tucker(64, 7, 7, 512, 512, 309, 309, 3, 1, "bf16", "none")),
    ]
    return [dict(c, name=n) for n, c in cases]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rank(rng, r, top):
    """A rank near r: as it is (odd ones among them) or rounded to a multiple of 8, 16, 32 or 64."""
    m = rng.choice([1, 8, 16, 32, 32, 64, 64])
    return max(min(m, top), min((r + m // 2) // m * m, top // m * m if top >= m else top))


def _draw_linear(rng):
    dtype = "f32" if rng.random() < 0.15 else "bf16"
    if dtype == "f32":
        M, K, N = _log(rng, 64, 1024), 8 * _log(rng, 16, 96), 8 * _log(rng, 16, 96)
    else:
        M, K, N = _log(rng, 64, 8192), 8 * _log(rng, 32, 512), 8 * _log(rng, 32, 512)
    r = _rank(rng, int(K * N / (K + N) / math.exp(rng.uniform(math.log(1.5), math.log(8.0)))) + 1, min(K, N, 1024))
    mode = rng.choice(["train"] * 6 + ["accumulate", "eval"])
    return _linear(mode, M, K, N, r, dtype, "U" if mode == "eval" else rng.choice(["U", "V", "U", "V", "none"]))


def _draw_block(rng):
    d = 64 * rng.randint(6, 16)
    return _block(_log(rng, 512, 8192), d, 32 * max(2, round(d / 4 / 32)), rng.choice(["U", "V"]))


def _draw_tucker(rng):
    C = 8 * _log(rng, 8, 64)
    S = rng.choice([C, C, 8 * _log(rng, 8, 64)])
    H = rng.choice([7, 14, 28, rng.randint(5, 32)])
    W = rng.choice([H, H, H, rng.randint(5, 32)])
    dtype = "f32" if rng.random() < 0.1 else "bf16"
    pixels = _log(rng, 1000, 4000 if dtype == "f32" else 50000)
    B = max(1, pixels // (H * W))
    r = b.lrd_tucker_rank(C, S, 3, math.exp(rng.uniform(math.log(2.0), math.log(5.0))))[0]
    r = _rank(rng, max(r, 8), min(C, S))
    return _tucker(B, H, W, C, S, r, r, rng.choice([3] * 8 + [1, 5]), rng.choice([1, 1, 2]), dtype, rng.choice(["factors", "core", "factors", "core", "none"]))


def draw(rng):
    top = max(work(c)["flops"] for c in listed())
    while True:
        c = rng.choice([_draw_linear, _draw_linear, _draw_linear, _draw_block, _draw_tucker, _draw_tucker])(rng)
        if work(c)["flops"] <= top:
            return c


# ---- states -------------------------------------------------------------------------------------------------------
def _normal(g, tdt, *shape, std=1.0):
    return torch.randn(*shape, device="cuda", generator=g).mul_(std).to(tdt)


def _empty(tdt, *shape):
    return torch.empty(*shape, dtype=tdt, device="cuda")


def _workspace(nbytes):
    return torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")


def _layer(g, M, K, N, r, dtype, freeze, mode="train", X=None):
    code, tdt = DTYPES[dtype]
    f = MASKS[freeze]
    L = {"desc": b.linear_desc(M, K, N, r, code), "f": f}
    L["X"] = _normal(g, tdt, M, K) if X is None else X
    L["V"], L["U"] = _normal(g, tdt, K, r, std=K ** -0.5), _normal(g, tdt, N, r, std=r ** -0.5)
    L["bias"] = _normal(g, tdt, N, std=0.1)
    L["Y"] = _empty(tdt, M, N)
    L["Z"] = None if freeze == "U" else _empty(tdt, M, r)
    fwd = b.lrd_linear_workspace_bytes(L["desc"], f, 0)
    if mode == "eval":
        L["ws"] = _workspace(fwd)
        return L
    L["dY"], L["dX"] = _normal(g, tdt, M, N), _empty(tdt, M, K)
    L["dU"], L["db"] = (None, None) if freeze == "U" else (_empty(tdt, N, r), _empty(tdt, N))
    L["dV"] = None if freeze == "V" else _empty(tdt, K, r)
    L["ws"] = _workspace(max(fwd, b.lrd_linear_workspace_bytes(L["desc"], f, 2 if mode == "accumulate" else 1)))
    return L


def _layer_outputs(L):
    return [L[k] for k in ("Y", "Z", "dX", "dU", "dV", "db") if L.get(k) is not None]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "linear":
        L = _layer(g, case["M"], case["K"], case["N"], case["r"], case["dtype"], case["freeze"], case["mode"])
        if case["mode"] == "accumulate":         # what the earlier micro-batches of this step have left
            for k in ("dU", "dV", "db"):
                if L[k] is not None:
                    L[k] = _normal(g, L[k].dtype, *L[k].shape, std=case["M"] ** 0.5)
        return dict(L, case=case)
    if case["kind"] == "block":
        M, d, r, dt, f = case["M"], case["d"], case["r"], case["dtype"], case["freeze"]
        X = _normal(g, DTYPES[dt][1], M, d)
        qkv = [_layer(g, M, d, d, r, dt, f, X=X) for _ in range(3)]
        rest = [_layer(g, M, d, d, r, dt, f), _layer(g, M, d, 4 * d, 2 * r, dt, f), _layer(g, M, 4 * d, d, 2 * r, dt, f)]
        return {"case": case, "qkv": qkv, "rest": rest, "stream": torch.cuda.Stream()}
    code, tdt = DTYPES[case["dtype"]]
    f = TUCKER_MASKS[case["freeze"]]
    B, H, W, C, S, r1, r2, k, s = (case[n] for n in ("B", "H", "W", "C", "S", "r1", "r2", "k", "stride"))
    Ho, Wo = (H - 1) // s + 1, (W - 1) // s + 1
    T = {"case": case, "f": f, "desc": b.tucker2_desc(B, H, W, C, S, r1, r2, code, k=k, stride=s, pad=(k - 1) // 2)}
    T["X"], T["dY"] = _normal(g, tdt, B, H, W, C), _normal(g, tdt, B, Ho, Wo, S)
    T["A"], T["G"] = _normal(g, tdt, C, r1, std=C ** -0.5), _normal(g, tdt, r2, k, k, r1, std=(k * k * r1) ** -0.5)
    T["Bm"], T["bias"] = _normal(g, tdt, S, r2, std=r2 ** -0.5), _normal(g, tdt, S, std=0.1)
    T["Y"], T["dX"] = _empty(tdt, B, Ho, Wo, S), _empty(tdt, B, H, W, C)
    core, factors = case["freeze"] != "core", case["freeze"] != "factors"
    T["Z1"], T["dG"] = (_empty(tdt, B, H, W, r1), _empty(tdt, r2, k, k, r1)) if core else (None, None)
    T["Z2"], T["dA"], T["dB"], T["db"] = (_empty(tdt, B, Ho, Wo, r2), _empty(tdt, C, r1), _empty(tdt, S, r2), _empty(tdt, S)) if factors else (None,) * 4
    T["ws"] = _workspace(max(b.lrd_tucker2_workspace_bytes(T["desc"], f, i) for i in (0, 1)))
    return T


# ---- one pass -----------------------------------------------------------------------------------------------------
def _forward(L):
    b.lrd_linear_fwd(L["desc"], L["X"], L["V"], L["U"], L["bias"], L["Y"], L["Z"], L["f"], L["ws"])


def _run_linear(L):
    mode = L["case"]["mode"]
    _forward(L)
    if mode == "eval":
        return [L["Y"]]
    backward = b.lrd_linear_bwd if mode == "train" else b.lrd_linear_bwd_accumulate
    backward(L["desc"], L["dY"], None if L["f"] == b.LRD_FREEZE_V else L["X"], L["V"], L["U"], L["Z"], L["dX"], L["dU"], L["dV"],
             L["db"], L["f"], L["ws"])
    return _layer_outputs(L)


def _each(layers, key):
    v = [L[key] for L in layers]
    return None if all(x is None for x in v) else v


def _run_block(S):
    qkv, rest, side = S["qkv"], S["rest"], S["stream"]
    f = qkv[0]["f"]
    descs, ws = [L["desc"] for L in qkv], [L["ws"] for L in qkv]
    b.lrd_linear_group_fwd(descs, _each(qkv, "X"), _each(qkv, "V"), _each(qkv, "U"), _each(qkv, "bias"), _each(qkv, "Y"), _each(qkv, "Z"), f, ws)
    for L in rest:
        _forward(L)
    main = torch.cuda.current_stream()
    for L in reversed(rest):
        b.lrd_linear_bwd_data(L["desc"], L["dY"], L["V"], L["U"], L["dX"], f, L["ws"])
        side.wait_stream(main)
        b.lrd_linear_bwd_weights(L["desc"], L["dY"], None if f == b.LRD_FREEZE_V else L["X"], L["Z"], L["dU"], L["dV"], L["db"], f, L["ws"],
                                 stream=side.cuda_stream)
    b.lrd_linear_group_bwd(descs, _each(qkv, "dY"), None if f == b.LRD_FREEZE_V else _each(qkv, "X"), _each(qkv, "V"), _each(qkv, "U"),
                           _each(qkv, "Z"), _each(qkv, "dX"), _each(qkv, "dU"), _each(qkv, "dV"), _each(qkv, "db"), f, ws)
    main.wait_stream(side)
    return [_layer_outputs(L) for L in qkv + rest]


def _run_tucker(T):
    X = None if T["f"] == b.LRD_TK_FREEZE_FACTORS else T["X"]
    b.lrd_tucker2_fwd(T["desc"], T["X"], T["A"], T["G"], T["Bm"], T["bias"], T["Y"], T["Z1"], T["Z2"], T["f"], T["ws"])
    b.lrd_tucker2_bwd(T["desc"], T["dY"], X, T["A"], T["G"], T["Bm"], T["Z1"], T["Z2"], T["dX"], T["dA"], T["dG"], T["dB"], T["db"], T["f"],
                      T["ws"])
    return [T[k] for k in ("Y", "Z1", "Z2", "dX", "dA", "dG", "dB", "db") if T[k] is not None]


def run(state):
    return {"linear": _run_linear, "block": _run_block, "tucker": _run_tucker}[state["case"]["kind"]](state)


# ---- work and tolerance -------------------------------------------------------------------------------------------
def _linear_work(M, K, N, r, freeze, mode, e):
    flops, values = 2 * M * r * (K + N), M * K + (K + N) * r + N + M * N
    if mode != "eval":
        dU, dV = freeze != "U", freeze != "V"
        flops += 2 * M * r * (K + N) + 2 * M * r * (N * dU + K * dV)
        values += M * N + (K + N) * r + M * K                                  # dY, the factors again, dX
        values += dU * (2 * M * r + N * r + N) + dV * (M * K + K * r)          # Z written and read, dU, db; X again, dV
        if mode == "accumulate":
            values += dU * (N * r + N) + dV * K * r
    return flops, values * e


def work(case):
    e = 2 if case["dtype"] == "bf16" else 4
    f = case["freeze"]
    if case["kind"] == "linear":
        flops, nbytes = _linear_work(case["M"], case["K"], case["N"], case["r"], f, case["mode"], e)
    elif case["kind"] == "block":
        M, d, r = case["M"], case["d"], case["r"]
        parts = [_linear_work(M, K, N, q, f, "train", e) for K, N, q in [(d, d, r)] * 4 + [(d, 4 * d, 2 * r), (4 * d, d, 2 * r)]]
        flops, nbytes = sum(p[0] for p in parts), sum(p[1] for p in parts)
        nbytes -= 2 * M * d * e * (2 if f != "V" else 1)                       # query, key and value read one X
    else:
        B, H, W, C, S, r1, r2, k, s = (case[n] for n in ("B", "H", "W", "C", "S", "r1", "r2", "k", "stride"))
        P, Po = B * H * W, B * ((H - 1) // s + 1) * ((W - 1) // s + 1)
        ends, core, weights = 2 * (P * C * r1 + Po * r2 * S), 2 * Po * k * k * r1 * r2, C * r1 + k * k * r1 * r2 + S * r2
        g_ends, g_core = f != "factors", f != "core"
        flops = (2 + g_ends) * ends + (2 + g_core) * core
        nbytes = e * (2 * (P * C + Po * S + weights) + S + g_core * (2 * P * r1 + k * k * r1 * r2)
                      + g_ends * (2 * Po * r2 + P * C + C * r1 + S * r2 + S))
    return {"bytes": nbytes, "flops": flops}


# Against the same passes in fp64 the outputs are off by at most 2.9e-3 in bf16 (each product rounds its result once; a
# Tucker-2 layer chains three) and 1.1e-6 in fp32 (sums over up to some 3000 pixels): about four times that.
REL = {"bf16": 1e-2, "f32": 5e-6}


def tolerance(case):
    return {"rel": REL[case["dtype"]]}
