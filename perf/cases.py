"""The work this library is measured on: what a program that serves a Spark Transformer has it do.

Six kinds of work, each through the public entry points of `paper_2506_06644_b200.binding`:

* ``topk``    statistical top-k of rows (threshold and counts; ordered lists; dense result)
* ``ffn``     the Spark FFN of 1 to 64 tokens (fp32, bf16, FP8 weights)
* ``attn``    Spark attention of one new token per sequence over its own cache (bf16, FP8 slice, FP8 cache)
* ``gemv``    a dense projection (LM head, QKV, output projection) of 1 to 64 tokens
* ``decode``  one token per sequence through a stack of layers, replayed from a CUDA graph as a serving loop does
* ``prefill`` a prompt through a stack of layers in chunks, one or several chunks in flight

Operators called on their own use a context with its default settings (other kernels of the caller may run beside
them); decode and prefill own the GPU and switch launch overlap on, as the benchmark does.  Shapes are the
repository's (`synth.GEMMA2_2B`, `GEMMA2_9B`, `TINY`, the paper's FFN width 13824) and generic ones.
"""
from __future__ import annotations

import math

import torch

from paper_2506_06644_b200 import binding as S
from paper_2506_06644_b200 import synth

SHAPES = {"2b": synth.GEMMA2_2B, "9b": synth.GEMMA2_9B, "tiny": synth.TINY}
# FFN shapes: d, d_ff, r.  The last two are generic (a neuron count that divides nothing; a power of two).
FFN_SHAPES = {"2b": (2304, 9216, 1024), "2b-wide": (2304, 13824, 1024), "9b": (3584, 14336, 1792), "tiny": (256, 1024, 128),
              "ragged": (512, 3000, 256), "pow2": (2048, 8192, 1024)}
HEADS = {"2b": (8, 4, 256, 128), "9b": (16, 8, 256, 128), "tiny": (4, 2, 64, 32), "gqa8": (8, 1, 128, 64)}
K_ATTN = 256


def listed():
    return [
        # the check every new user runs first: 64 rows of 1024 scores, 8 % kept, ordered lists (one short launch)
        dict(name="topk-64x1024-lists", kind="topk", rows=64, n=1024, k=82, dist="normal", out="lists"),
        # the standalone operator at its full size, heavy-tailed rows, the dense result of Eq. 10 (1 GB in, 1 GB out)
        dict(name="topk-4096x65536-dense", kind="topk", rows=4096, n=65536, k=5243, dist="student", out="dense"),
        # a tiny fp32 model, one token: what a unit test or an embedded predictor calls (latency only)
        dict(name="ffn-tiny-fp32-1", kind="ffn", shape="tiny", tokens=1, dtype="f32", k=82),
        # a small verify batch of speculative decoding at the 2B shape
        dict(name="ffn-2b-bf16-4", kind="ffn", shape="2b", tokens=4, dtype="bf16", k=737),
        # a serving batch that does not fill a tile, at the 9B shape
        dict(name="ffn-9b-bf16-45", kind="ffn", shape="9b", tokens=45, dtype="bf16", k=1147),
        # one chat sequence of ordinary length
        dict(name="attn-2b-bf16-1x4096", kind="attn", heads="2b", batch=1, cap=4096, window=0, storage="bf16"),
        # eight long documents of different lengths, caches of 32768 rows
        dict(name="attn-2b-bf16-8x32768", kind="attn", heads="2b", batch=8, cap=32768, window=0, storage="bf16"),
        # the 9B heads with the whole cache in FP8, three sequences of odd lengths
        dict(name="attn-9b-fp8kv-3x16001", kind="attn", heads="9b", batch=3, cap=16001, window=0, storage="fp8kv"),
        # the LM head of a 2B decoding step: the largest dense matrix of the model, one token
        dict(name="gemv-lm-head-2b-1", kind="gemv", n_in=2304, n_out=256000, tokens=1),
        # the headline: one token through all 26 layers of the 2B shape behind 8192 tokens, local 4096 / global layers
        dict(name="decode-2b-1x8192", kind="decode", shape="2b", layers=26, batch=1, ctx=8192, storage="bf16"),
        # the same model serving eight sequences
        dict(name="decode-2b-8x8192", kind="decode", shape="2b", layers=26, batch=8, ctx=8192, storage="bf16"),
        # a prompt that does not divide by the chunk, eight layers, 64-token chunks from an empty cache
        dict(name="prefill-2b-4000", kind="prefill", shape="2b", layers=8, tokens=4000, start=0, chunk=64, inflight=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["topk", "ffn", "attn", "gemv", "decode", "prefill"])
    if kind == "topk":
        n = _log(rng, 512, 65536)
        rows = _log(rng, 16, 4096)
        return dict(kind=kind, rows=rows, n=n, k=max(1, int(n * rng.choice([0.02, 0.08, 0.25]))),
                    dist=rng.choice(["normal", "laplace", "student"]), out=rng.choice(["stats", "lists", "dense"]))
    if kind == "ffn":
        shape = rng.choice(list(FFN_SHAPES))
        dtype = rng.choice(["bf16", "bf16", "bf16", "fp8"] + (["f32"] if shape in ("tiny", "ragged") else []))
        tokens = rng.randint(1, 4) if dtype == "fp8" else _log(rng, 1, 64)
        return dict(kind=kind, shape=shape, tokens=tokens, dtype=dtype, k=max(1, int(FFN_SHAPES[shape][1] * rng.uniform(0.05, 0.12))))
    if kind == "attn":
        heads = rng.choice(["2b", "2b", "9b", "9b", "tiny", "gqa8"])
        storage = rng.choice(["bf16", "bf16", "fp8k", "fp8kv"])
        return dict(kind=kind, heads=heads, batch=_log(rng, 1, 8), cap=_log(rng, 300, 32768), window=rng.choice([0, 0, 4096]), storage=storage)
    if kind == "gemv":
        # widths of the 2B and 9B model and attention outputs, one that divides nothing; from a projection's rows to a vocabulary's
        return dict(kind=kind, n_in=rng.choice([2048, 2304, 3584, 4096, 1000]), n_out=_log(rng, 1000, 256000), tokens=_log(rng, 1, 64))
    if kind == "decode":
        shape, batch, ctx = rng.choice(["2b", "2b", "9b", "tiny"]), _log(rng, 1, 16), _log(rng, 128, 8192)
        storage = rng.choice(["bf16", "bf16", "fp8"]) if batch <= 4 else "bf16"
        return dict(kind=kind, shape=shape, layers=rng.randint(2, 12), batch=batch, ctx=ctx, storage=storage)
    shape = rng.choice(["2b", "2b", "9b", "tiny"])
    return dict(kind="prefill", shape=shape, layers=rng.randint(2, 4 if shape == "9b" else 8), tokens=_log(rng, 100, 4000 if shape != "9b" else 2000),
                start=rng.choice([0, 0, rng.randint(1, 2000)]), chunk=rng.choice([64, 64, 48]), inflight=rng.choice([1, 1, 2]) if shape != "tiny" else 1)


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _bf16(g, *shape, scale=1.0):
    return (torch.randn(*shape, device="cuda", generator=g) * scale).to(torch.bfloat16)


def _fp8_rows(t):
    """E4M3 codes and one scale per row (the library's storage rule)."""
    tf = t.float()
    sc = tf.abs().amax(dim=-1).clamp_min(1e-30) / 448.0
    return (tf / sc[..., None]).to(torch.float8_e4m3fn).view(torch.uint8), sc


def _rows(g, dist, rows, ld):
    if dist == "normal":
        return torch.randn(rows, ld, device="cuda", generator=g)
    if dist == "laplace":
        u = torch.rand(rows, ld, device="cuda", generator=g) - 0.5
        return -torch.sign(u) * torch.log((1 - 2 * u.abs()).clamp_min(1e-30))
    z = torch.randn(rows, ld, device="cuda", generator=g)      # Student-t with four degrees of freedom
    chi = torch.zeros(rows, ld, device="cuda")
    for _ in range(4):
        chi += torch.randn(rows, ld, device="cuda", generator=g) ** 2
    return z / torch.sqrt(chi / 4)


def _lengths(batch, cap):
    """Sequence lengths of an attention batch: the longest fills the cache, the others are shorter by odd steps."""
    return [max(1, cap - (b * cap) // (2 * batch) - b) for b in range(batch)]


def _prepare_topk(c, g):
    rows, n = c["rows"], c["n"]
    ld = (n + 3) // 4 * 4
    s = dict(ctx=S.SparkContext(), x=_rows(g, c["dist"], rows, ld), ld=ld, theta=torch.zeros(rows, device="cuda"),
             count=torch.zeros(rows, dtype=torch.int32, device="cuda"), cap=0, idx=None, val=None, y=None)
    if c["out"] == "lists":
        s["cap"] = (min(n, 2 * c["k"] + 64) + 3) // 4 * 4
        s["idx"] = torch.zeros(rows, s["cap"], dtype=torch.int32, device="cuda")
        s["val"] = torch.zeros(rows, s["cap"], device="cuda")
    elif c["out"] == "dense":
        s["y"] = torch.zeros(rows, ld, device="cuda")
    return s


def _run_topk(c, s):
    S.spark_stat_topk(s["ctx"], s["x"], c["rows"], c["n"], s["ld"], c["k"], S.SPARK_FILL_ZERO, s["theta"], s["count"], s["idx"], s["val"],
                      s["cap"], s["y"])
    return {k: s[k] for k in ("theta", "count", "idx", "val", "y") if s[k] is not None}


def _prepare_ffn(c, g):
    d, d_ff, r = FFN_SHAPES[c["shape"]]
    B = c["tokens"]
    x = torch.randn(B, d, device="cuda", generator=g)
    s = dict(ctx=S.SparkContext(max_batch=B, max_dff=d_ff, max_d=d), x=x / x.pow(2).mean(dim=1, keepdim=True).sqrt(),
             y=torch.zeros(B, d, device="cuda"), theta=torch.zeros(B, device="cuda"))
    w = [torch.randn(d_ff, cols, device="cuda", generator=g) * d ** -0.5 for cols in (r, d - r, d)]
    if c["dtype"] == "fp8":
        s["w"] = [t for m in w for t in _fp8_rows(m)]
    else:
        s["w"] = [m if c["dtype"] == "f32" else m.to(torch.bfloat16) for m in w]
    return s


def _run_ffn(c, s):
    d, d_ff, r = FFN_SHAPES[c["shape"]]
    if c["dtype"] == "fp8":
        S.spark_ffn_decode_fp8(s["ctx"], s["x"], c["tokens"], *s["w"], d, d_ff, r, c["k"], S.SPARK_GELU_TANH, s["y"], s["theta"], None, None)
    else:
        S.spark_ffn_decode(s["ctx"], s["x"], c["tokens"], *s["w"], S.SPARK_F32 if c["dtype"] == "f32" else S.SPARK_BF16, d, d_ff, r, c["k"],
                           S.SPARK_GELU_TANH, s["y"], s["theta"], None, None)
    return {k: s[k] for k in ("y", "theta")}


def _prepare_attn(c, g):
    n_q, n_kv, hd, r = HEADS[c["heads"]]
    B, cap = c["batch"], c["cap"]
    k1, k2, v = (_bf16(g, B, n_kv, cap, w) for w in (r, hd - r, hd))
    s = dict(ctx=S.SparkContext(max_batch=B, max_cap=cap, n_q=n_q, hd=hd), q=torch.randn(B, n_q, hd, device="cuda", generator=g) * hd ** -0.5,
             lens=torch.tensor(_lengths(B, cap), dtype=torch.int32, device="cuda"), o=torch.zeros(B, n_q, hd, device="cuda"),
             theta=torch.zeros(B, n_q, device="cuda"))
    if c["storage"] == "bf16":
        s["kv"] = [k1, k2, v]
    elif c["storage"] == "fp8k":
        s["kv"] = [*_fp8_rows(k1), k2, v]
    else:
        s["kv"] = [*_fp8_rows(k1), *_fp8_rows(k2), *_fp8_rows(v)]
    return s


def _run_attn(c, s):
    n_q, n_kv, hd, r = HEADS[c["heads"]]
    tail = (c["batch"], n_q, n_kv, hd, r, c["cap"], s["lens"], c["window"], K_ATTN, 0, s["o"], s["theta"], None, None, 0)
    if c["storage"] == "bf16":
        S.spark_attn_decode(s["ctx"], s["q"], *s["kv"], S.SPARK_BF16, *tail)
    elif c["storage"] == "fp8k":
        S.spark_attn_decode_fp8k(s["ctx"], s["q"], *s["kv"], *tail)
    else:
        S.spark_attn_decode_fp8kv(s["ctx"], s["q"], *s["kv"], *tail)
    return {k: s[k] for k in ("o", "theta")}


def _prepare_gemv(c, g):
    n_in, n_out = c["n_in"], c["n_out"]
    B = c["tokens"]
    return dict(ctx=S.SparkContext(max_batch=B, max_d=n_in), W=_bf16(g, n_out, n_in, scale=n_in ** -0.5),
                x=torch.randn(B, n_in, device="cuda", generator=g), y=torch.zeros(B, n_out, device="cuda"))


def _run_gemv(c, s):
    n_in, n_out = c["n_in"], c["n_out"]
    S.spark_dense_gemv(s["ctx"], s["x"], c["tokens"], s["W"], S.SPARK_BF16, n_in, n_out, None, s["y"])
    return s["y"]


def _layer_weights(g, sh, fp8):
    nqkv, nqo = (sh.n_q + 2 * sh.n_kv) * sh.hd, sh.n_q * sh.hd
    w = dict(norm1=1.0 + 0.1 * torch.randn(sh.d, device="cuda", generator=g), norm2=1.0 + 0.1 * torch.randn(sh.d, device="cuda", generator=g),
             Wqkv=_bf16(g, nqkv, sh.d, scale=sh.d ** -0.5), Wo=_bf16(g, sh.d, nqo, scale=nqo ** -0.5),
             K1t=_bf16(g, sh.d_ff, sh.r_ff, scale=sh.d ** -0.5), K2t=_bf16(g, sh.d_ff, sh.d - sh.r_ff, scale=sh.d ** -0.5),
             Vt=_bf16(g, sh.d_ff, sh.d, scale=sh.d ** -0.5))
    if fp8:
        for name, scale in (("K1t", "K1s"), ("K2t", "K2s"), ("Vt", "Vs")):
            w[name], w[scale] = _fp8_rows(w[name])
    return w


def _layer_cfg(sh, layer, cap, flags):
    # local (4096) and global attention layers alternate
    return dict(d=sh.d, d_ff=sh.d_ff, r_ff=sh.r_ff, k_ff=sh.k_ff, n_q=sh.n_q, n_kv=sh.n_kv, hd=sh.hd, r_attn=sh.r_attn, k_attn=sh.k_attn,
                window=4096 if layer % 2 == 0 and cap > 4096 else 0, cap=cap, rms_eps=1e-6, rope_base=10000.0, flags=flags)


def _prepare_decode(c, g):
    sh, B, L = SHAPES[c["shape"]], c["batch"], c["layers"]
    fp8 = c["storage"] == "fp8"
    cap = c["ctx"] + 1
    lead = (L, B, sh.n_kv, cap)
    k1, k2, v = (torch.empty(*lead, w, dtype=torch.bfloat16, device="cuda") for w in (sh.r_attn, sh.hd - sh.r_attn, sh.hd))
    k1q = torch.empty(*lead, sh.r_attn, dtype=torch.uint8, device="cuda") if fp8 else None
    k1s = torch.empty(*lead, device="cuda") if fp8 else None
    layers, new = [], [k1q if fp8 else k1, k2, v] + ([k1s] if fp8 else [])
    for l in range(L):
        for t in (k1, k2, v):
            t[l].copy_(torch.randn(t[l].shape, device="cuda", generator=g))
        cache = dict(k1c=k1[l], k2c=k2[l], vc=v[l])
        if fp8:
            codes, scales = _fp8_rows(k1[l])
            k1q[l].copy_(codes)
            k1s[l].copy_(scales)
            cache.update(k1c=k1q[l], k1s=k1s[l])
        flags = (S.SPARK_FFN_FP8 | S.SPARK_K1C_FP8) if fp8 else 0
        layers.append(S.make_layer(_layer_weights(g, sh, fp8), _layer_cfg(sh, l, cap, flags), cache))
    cfg = dict(n_q=sh.n_q, n_kv=sh.n_kv, hd=sh.hd, d=sh.d)
    s = dict(ctx=S.SparkContext(max_batch=B, max_dff=sh.d_ff, max_cap=cap, n_q=sh.n_q, hd=sh.hd, max_d=sh.d), stack=S.make_stack(layers),
             x=torch.randn(B, sh.d, device="cuda", generator=g), h=torch.zeros(B, sh.d, device="cuda"),
             lens=torch.full((B,), cap, dtype=torch.int32, device="cuda"), scratch=torch.empty(S.layer_scratch_floats(cfg, B), device="cuda"))
    s["ctx"].set_launch_overlap(True)
    s["new_rows"] = [t[:, :, :, cap - 1] for t in new]         # the cache rows that a step writes
    # one step as a graph: the token's embedding comes in, the stack runs
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())

    def step():
        s["h"].copy_(s["x"])
        S.spark_stack_decode(s["ctx"], s["stack"], s["lens"], s["h"], B, s["scratch"])

    with torch.cuda.stream(side):
        step()
        side.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=side):
            step()
    return s


def _run_decode(c, s):
    s["graph"].replay()
    return [s["h"]] + s["new_rows"]


def _prepare_prefill(c, g):
    sh, L = SHAPES[c["shape"]], c["layers"]
    cap = c["start"] + c["tokens"]
    k1, k2, v = (_bf16(g, L, sh.n_kv, cap, w) for w in (sh.r_attn, sh.hd - sh.r_attn, sh.hd))
    layers = [S.make_layer(_layer_weights(g, sh, False), _layer_cfg(sh, l, cap, S.SPARK_SHARED_CACHE), dict(k1c=k1[l], k2c=k2[l], vc=v[l]))
              for l in range(L)]
    ctxs = [S.SparkContext(max_batch=c["chunk"], max_dff=sh.d_ff, max_cap=cap, n_q=sh.n_q, hd=sh.hd, max_d=sh.d) for _ in range(c["inflight"])]
    for ctx in ctxs:
        ctx.set_launch_overlap(True)
    x = torch.randn(c["tokens"], sh.d, device="cuda", generator=g)
    return dict(ctxs=ctxs, streams=[torch.cuda.Stream() for _ in ctxs[1:]], layers=layers, x=x, h=torch.empty_like(x), caches=(k1, k2, v))


def _run_prefill(c, s):
    s["h"].copy_(s["x"])
    S.spark_prefill(s["ctxs"][0], s["layers"], s["h"], c["start"], chunk=c["chunk"], more_ctx=s["ctxs"][1:], more_streams=s["streams"])
    return [s["h"]] + [t[:, :, c["start"]:] for t in s["caches"]]      # the outputs and every cache row the prompt wrote


_PREPARE = dict(topk=_prepare_topk, ffn=_prepare_ffn, attn=_prepare_attn, gemv=_prepare_gemv, decode=_prepare_decode, prefill=_prepare_prefill)
_RUN = dict(topk=_run_topk, ffn=_run_ffn, attn=_run_attn, gemv=_run_gemv, decode=_run_decode, prefill=_run_prefill)


def prepare(case, seed):
    s = _PREPARE[case["kind"]](case, _gen(seed))
    s["case"] = case
    torch.cuda.synchronize()
    return s


def run(state):
    return _RUN[state["case"]["kind"]](state["case"], state)


# ---- what a pass cannot do without ------------------------------------------------------------------------------------
def _ffn_work(d, d_ff, r, k, tokens, width):
    active = min(1.0, k / d_ff)
    union = d_ff * (1.0 - (1.0 - active) ** tokens)            # rows some token needs, the tokens' sets independent
    nbytes = (d_ff * r + union * (2 * d - r)) * width + 8 * tokens * d + (d_ff + 2 * union) * 4 * (width == 1)
    return nbytes, 2.0 * tokens * (d_ff * r + active * d_ff * (2 * d - r))


def _attn_work(n_q, n_kv, hd, r, lens, k, storage):
    slice_w = 2 * r if storage == "bf16" else r + 4
    row_w = 2 * (2 * hd - r) if storage != "fp8kv" else 2 * hd - r + 8
    keep = [min(k, n) for n in lens]
    union = [n * (1.0 - (1.0 - m / n) ** (n_q // n_kv)) for n, m in zip(lens, keep)]      # rows some head of the group keeps
    nbytes = sum(n_kv * (n * slice_w + u * row_w) for n, u in zip(lens, union)) + 8 * len(lens) * n_q * hd
    return nbytes, 2.0 * n_q * sum(n * r + m * (2 * hd - r) for n, m in zip(lens, keep))


def work(case):
    c = case
    if c["kind"] == "topk":
        per = 4.0 * c["n"] + 8 + {"stats": 0, "lists": 8 * min(c["n"], c["k"]), "dense": 4 * c["n"]}[c["out"]]
        return {"bytes": c["rows"] * per, "flops": 5.0 * c["rows"] * c["n"]}
    if c["kind"] == "ffn":
        b, f = _ffn_work(*FFN_SHAPES[c["shape"]], c["k"], c["tokens"], {"f32": 4, "bf16": 2, "fp8": 1}[c["dtype"]])
        return {"bytes": b, "flops": f}
    if c["kind"] == "attn":
        lens = [min(n, c["window"]) if c["window"] else n for n in _lengths(c["batch"], c["cap"])]
        b, f = _attn_work(*HEADS[c["heads"]], lens, K_ATTN, c["storage"])
        return {"bytes": b, "flops": f}
    if c["kind"] == "gemv":
        n_in, n_out = c["n_in"], c["n_out"]
        return {"bytes": 2.0 * n_in * n_out + 4.0 * c["tokens"] * (n_in + n_out), "flops": 2.0 * c["tokens"] * n_in * n_out}
    sh = SHAPES[c["shape"]]
    proj = sh.d * (2 * sh.n_q + 2 * sh.n_kv) * sh.hd
    tokens = c["batch"] if c["kind"] == "decode" else c["tokens"]
    storage = "bf16" if c["kind"] == "prefill" or c["storage"] == "bf16" else "fp8k"
    fb, ff = _ffn_work(sh.d, sh.d_ff, sh.r_ff, sh.k_ff, tokens, 2 if storage == "bf16" else 1)
    nbytes = flops = 0.0
    for l in range(c["layers"]):
        cap = c["ctx"] + 1 if c["kind"] == "decode" else c["start"] + tokens
        window = _layer_cfg(sh, l, cap, 0)["window"] or cap
        if c["kind"] == "decode":
            ab, af = _attn_work(sh.n_q, sh.n_kv, sh.hd, sh.r_attn, [min(window, cap)] * tokens, sh.k_attn, storage)
        else:                                                  # every row of the cache is read or written once, every token looks back
            ab = 4.0 * sh.n_kv * sh.hd * cap
            af = 2.0 * sh.n_q * sum(min(n, window) * sh.r_attn + min(n, window, sh.k_attn) * (2 * sh.hd - sh.r_attn)
                                    for n in range(c["start"] + 1, cap + 1))
        nbytes += 2.0 * proj + fb + ab + 4.0 * tokens * sh.n_kv * sh.hd
        flops += 2.0 * tokens * proj + ff + af
    return {"bytes": nbytes + 8.0 * tokens * sh.d, "flops": flops}


def tolerance(case):
    """About four times what the library shows against the same arithmetic in 64 bits (operators), or against itself with
    its sums in another order (stacks of layers)."""
    c = case
    if c["kind"] == "topk":          # sums in fp64; a value one rounding step from the threshold shifts its row's list
        return {"rel": 1e-6, "max": 1e-3, "differ": 1e-3}
    if c["kind"] in ("ffn", "gemv"):
        # from five tokens on with bf16 weights the inputs enter the tensor cores as two bf16 terms (16 bits): 7e-6 measured
        split = c["tokens"] >= 5 and c.get("dtype", "bf16") == "bf16"
        return {"rel": 3e-5, "max": 2e-4} if split else {"rel": 2e-6, "max": 1e-5}
    if c["kind"] == "attn":
        # an FP8 slice meets the query with 16 bits, so a token at the threshold may fall on either side of it, which moves its
        # head's result by the token's share of the weights; without that 3e-7 measured
        return {"rel": 2e-6, "max": 1e-5} if c["storage"] == "bf16" else {"rel": 1e-2, "max": 0.5}
    # Stacks: a stored bf16 row that rounds the other way, or a token at an attention threshold, is carried on by the layers
    # above.  Up to four tokens (fp32 inputs) a step shows 1e-4 (one rounding step of a row: 8e-3 of its value), from five on
    # (two-term inputs) 9e-3 after 26 layers; a prompt 4e-3 after eight layers, 1.5e-2 at the tiny shape (a head keeps 16 tokens).
    if c["kind"] == "decode" and c["batch"] <= 4:
        return {"rel": 4e-4, "max": 0.03, "differ": 4e-3}
    if c["shape"] == "tiny":
        return {"rel": 0.03, "max": 0.99}
    return {"rel": 0.03, "max": 0.3} if c["kind"] == "decode" else {"rel": 0.017, "max": 0.16}
