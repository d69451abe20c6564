"""What is timed: the calls a user of this library makes, over the sizes they make them at.

Three kinds of case.

  "layer"     the four quantised projections of a transformer layer (qkv, o, gate/up, down), `layers` of
              them one after another on one stream, each with weights, transforms and activations of its
              own; "w4a4" through batq_linear_w4a4, "w4a8" through batq_linear_w4a8.  With `graph` the
              calls are captured once and a pass replays the graph, which is how a server runs a decode
              step; without it they are made one by one, as a prefill or an uncaptured step makes them.
  "linear"    one such projection alone.
  "quantise"  the activation quantiser alone (transform, clip, MXFP4 or MXFP8), as for a tensor that feeds
              several weights, or for the key/value cache taken head by head.
"""
from __future__ import annotations

import math

import torch

from paper_2603_16590_b200 import binding as B
from paper_2603_16590_b200 import synth

LLAMA8B = {"hidden": 4096, "qkv": 6144, "inter": 14336}      # synth.LLAMA8B_PREFILL
QWEN2VL7B = {"hidden": 3584, "qkv": 4608, "inter": 18944}    # synth.QWEN2VL7B_PREFILL


def _layer(name, fmt, tokens, shape, layers=1, graph=False, vision=0.0):
    return {"name": name, "kind": "layer", "format": fmt, "tokens": tokens, **shape, "layers": layers,
            "graph": graph, "vision": vision, "geometry": "baseline", "gr": 4, "gc": 8, "clip": True}


def _linear(name, fmt, tokens, n, m, out):
    return {"name": name, "kind": "linear", "format": fmt, "tokens": tokens, "n": n, "m": m, "out": out,
            "geometry": "baseline", "gr": 4, "gc": 8, "clip": True}


def _quantise(name, fmt, rows, n, layout, clip=True):
    return {"name": name, "kind": "quantise", "format": fmt, "rows": rows, "n": n, "layout": layout,
            "geometry": "baseline", "gr": 4, "gc": 8, "clip": clip}


def listed():
    return [
        # the smallest call: one small layer on one 128-token tile, fp32 out; launches and latency
        _linear("small_layer_128", "w4a4", 128, 1024, 1024, "f32"),
        # one user's next token, the calls made one by one
        _layer("decode_1_calls", "w4a4", 1, LLAMA8B),
        # a decode step of a small batch, captured: four layers, weights from HBM
        _layer("decode_4_graph", "w4a4", 4, LLAMA8B, layers=4, graph=True),
        _layer("decode_16_graph", "w4a4", 16, LLAMA8B, layers=4, graph=True),
        # the same with 8-bit activations
        _layer("decode_8_w4a8_graph", "w4a8", 8, LLAMA8B, layers=4, graph=True),
        # a busy server's decode batch, uneven
        _layer("batch_75_calls", "w4a4", 75, LLAMA8B),
        # a chunk of a prompt, not a multiple of any tile
        _layer("prefill_333", "w4a4", 333, LLAMA8B),
        # the prefill that the library's headline figure is quoted on
        _layer("prefill_2048", "w4a4", 2048, LLAMA8B),
        # a long prompt with image tokens: the largest pass
        _layer("prefill_8192_vision", "w4a4", 8192, QWEN2VL7B, vision=0.75),
        # prefill with 8-bit activations
        _layer("prefill_2048_w4a8", "w4a8", 2048, LLAMA8B),
        # a large activation tensor, quantised once for several weights
        _quantise("quantise_32768x8192", "mxfp4", 32768, 8192, "mma"),
        # an 8-bit key/value cache: 4096 tokens x 8 heads of 128 channels
        _quantise("kv_cache_32768x128", "mxfp8", 32768, 128, "rowmajor", clip=False),
    ]


_MOST_FLOPS = 3.8e12   # of a drawn pass: what the largest listed one has


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "linear", "quantise"])
    case = {"kind": kind}
    # transform: mostly the default 4 x 8 factors, sometimes the other sizes of the ablation
    gr, gc = rng.choice([(4, 8), (4, 8), (4, 8), (8, 4), (1, 32)])
    tail = {"geometry": "baseline" if (gr, gc) == (1, 32) else rng.choice(["baseline", "paper", "naive"]),
            "gr": gr, "gc": gc, "clip": rng.random() < 0.8}
    if kind == "quantise":
        fmt = rng.choice(["mxfp4", "mxfp8"])
        n = 32 * _log_int(rng, 2, 256)
        rows = _log_int(rng, 1, 32768)
        return {**case, "format": fmt, "rows": rows, "n": n, "layout": rng.choice(["mma", "rowmajor"]), **tail}
    fmt = rng.choice(["w4a4", "w4a4", "w4a8"])
    step = 128 if fmt == "w4a8" else 32   # the 8-bit GEMM wants n % 128 == 0
    if kind == "linear":
        n = step * _log_int(rng, 512 // step, 16384 // step)
        m = 8 * _log_int(rng, 32, 4096)
        tokens = min(_log_int(rng, 1, 8192), round(_MOST_FLOPS / (2 * n * m)))
        return {**case, "format": fmt, "tokens": tokens, "n": n, "m": m, "out": rng.choice(["bf16", "bf16", "f32"]), **tail}
    hidden = step * _log_int(rng, 1024 // step, 5120 // step)
    inter = step * _log_int(rng, round(2.5 * hidden) // step, 18944 // step)
    qkv = hidden + 256 * rng.randint(1, 8)
    decode = rng.random() < 0.5
    tokens = _log_int(rng, 1, 128) if decode else _log_int(rng, 129, 6000)
    tokens = min(tokens, round(_MOST_FLOPS / (2 * hidden * (qkv + hidden + 3 * inter))))
    graph = decode and rng.random() < 0.6
    return {**case, "format": fmt, "tokens": tokens, "hidden": hidden, "qkv": qkv, "inter": inter,
            "layers": 2 if graph else 1, "graph": graph, "vision": rng.choice([0.0, 0.0, 0.75]), **tail}


def _projections(case):
    """[(n, m)] of one pass, in order."""
    if case["kind"] == "linear":
        return [(case["n"], case["m"])]
    h, q, f = case["hidden"], case["qkv"], case["inter"]
    return [(h, q), (h, h), (h, 2 * f), (f, h)] * case["layers"]


def _activations(gen, rows, n, vision):
    """N(0,1) with 1 % of the channels x 50 and one row in 64 x 100; the first `vision` of the rows are
    Student-t(3) draws without outlier rows (the distributions of synth.make_activations)."""
    x = torch.randn((rows, n), generator=gen, device="cuda")
    nv = int(rows * vision)
    for at in range(0, nv, 1024):
        part = x[at:min(at + 1024, nv)]
        chi = torch.randn((3,) + tuple(part.shape), generator=gen, device="cuda").square_().mean(0).sqrt_()
        part /= chi
    channels = torch.randperm(n, generator=gen, device="cuda")[:max(1, n // (200 if nv else 100))]
    x[nv:, channels] *= 50.0
    if nv == 0 and rows >= 32:
        x[torch.randperm(rows, generator=gen, device="cuda")[:round(rows / 64)]] *= 100.0
    return x.to(torch.bfloat16)


def _factors(case, n, seed):
    return synth.make_transform(n, seed, case["geometry"], clip=case["clip"], gr=case["gr"], gc=case["gc"])


def _transform(case, n, t):
    return B.batq_transform_create(n, t.left, t.right, t.clip_lo, t.clip_hi, gr=case["gr"], gc=case["gc"])


def _inputs(case, seed):
    """(factors, weight or None, activations) of every call of a pass, in order."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "quantise":
        yield _factors(case, case["n"], seed), None, _activations(gen, case["rows"], case["n"], 0.0)
        return
    for i, (n, m) in enumerate(_projections(case)):
        weight = (torch.randn((m, n), generator=gen, device="cuda") * 0.02).to(torch.bfloat16)
        yield _factors(case, n, seed * 64 + i), weight, _activations(gen, case["tokens"], n, case.get("vision", 0.0))


def prepare(case, seed):
    if case["kind"] == "quantise":
        rows, n = case["rows"], case["n"]
        (t, _, x), = _inputs(case, seed)
        fp8 = case["format"] == "mxfp8"
        layout = B.SF_MMA if case["layout"] == "mma" else B.SF_ROWMAJOR
        return {"run": _run_quantise, "fn": B.batq_quantize_act_mxfp8 if fp8 else B.batq_quantize_act,
                "t": _transform(case, n, t), "x": x, "layout": layout,
                "codes": torch.zeros((rows, n if fp8 else n // 2), dtype=torch.uint8, device="cuda"),
                "scales": torch.zeros(B.batq_sf_bytes(rows, n, layout), dtype=torch.uint8, device="cuda")}
    tokens, a8 = case["tokens"], case["format"] == "w4a8"
    out = torch.float32 if case.get("out") == "f32" else torch.bfloat16
    calls, need = [], 0
    for (n, m), (t, weight, x) in zip(_projections(case), _inputs(case, seed)):
        t = _transform(case, n, t)
        w = B.batq_prepare_weight(t, weight)
        need = max(need, B.batq_linear_w4a8_workspace_bytes(w, tokens) if a8 else B.batq_linear_workspace_bytes(w, tokens))
        calls.append((t, w, x, torch.zeros((tokens, m), dtype=out, device="cuda")))
    del weight
    state = {"run": _run_calls, "fn": B.batq_linear_w4a8 if a8 else B.batq_linear_w4a4, "calls": calls,
             "workspace": B.aligned_workspace(need), "out": [c[3] for c in calls]}
    if case.get("graph"):
        _run_calls(state)   # first launches outside the capture
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _run_calls(state)
        state.update(graph=graph, run=_run_graph)
    return state


def _run_quantise(state):
    state["fn"](state["t"], state["x"], state["codes"], state["scales"], state["layout"])
    return state["codes"], state["scales"]


def _run_calls(state):
    fn, workspace = state["fn"], state["workspace"]
    for t, w, x, y in state["calls"]:
        fn(t, w, x, y, workspace)
    return state["out"]


def _run_graph(state):
    state["graph"].replay()
    return state["out"]


def run(state):
    return state["run"](state)


def work(case):
    """Bytes: bf16 activations in; 17/32 byte a weight; results out.  Flops: two per weight and token, and
    24 an activation for the two contractions of a 4 x 8 block transform (2 (gr + gc) in general)."""
    per = 2.0 * (case["gr"] + case["gc"])
    if case["kind"] == "quantise":
        elems = case["rows"] * case["n"]
        return {"bytes": elems * (2 + (1 if case["format"] == "mxfp8" else 0.5) + 1 / 32), "flops": elems * per}
    s, ob = case["tokens"], 4 if case.get("out") == "f32" else 2
    proj = _projections(case)
    return {"bytes": sum(2 * s * n + n * m * 17 / 32 + ob * s * m for n, m in proj),
            "flops": sum(2.0 * s * n * m + per * s * n for n, m in proj)}


def tolerance(case):
    """Four times the largest difference seen between two correct computations of the same case: the
    block transform's fp32 sums in another order (the tensor-core and the streaming ALU quantiser) flip
    4.8e-7 of the codes of the largest tensor (rel 1.1e-4), each to its neighbour, and move a whole
    layer's bf16 results by up to 9e-4; tile shapes and K splits of the GEMM changed nothing."""
    if case["kind"] == "quantise":
        return {"rel": 5e-4, "differ": 2e-6}
    return {"rel": 4e-3}


def _block_transform(v, left, right):
    """vec(L^T V R) of every 32-element block of the rows of v, 64 bits."""
    k, gr, gc = v.shape[1] // 32, left.shape[-1], right.shape[-1]
    v = v.view(-1, k, gr, gc)
    v = torch.matmul(v, right)                        # [rows, k, gr, gc] x [1 or k, gc, gc]
    return torch.matmul(left.transpose(-1, -2), v).reshape(-1, k, 32)


def _mx(v, emax):
    """The values that MXFP4 (emax 2) or MXFP8 E4M3 (emax 8) keeps of blocks v [rows, k, 32]: shared scale
    2^(floor(log2 amax) - emax), elements to the nearest, ties to even, saturating."""
    e = (torch.frexp(v.abs().amax(-1, keepdim=True))[1] - 1 - emax).clamp(-127, 127)
    u = torch.ldexp(v, -e)
    low, bits, top = (0, 1, 6.0) if emax == 2 else (-6, 3, 448.0)   # exponent of the subnormals, mantissa bits, maximum
    step = (torch.frexp(u)[1] - 1).clamp_min(low) - bits
    u = torch.ldexp(torch.round(torch.ldexp(u, -step)), step).clamp(-top, top)
    return torch.ldexp(u, e).reshape(v.shape[0], -1)


def exact(case, seed):
    """The results in 64 bits; nothing for codes and scale bytes, which are whole numbers."""
    if case["kind"] == "quantise":
        return None
    emax, out = 8 if case["format"] == "w4a8" else 2, []
    for t, weight, x in _inputs(case, seed):
        left, right = (torch.from_numpy(f).cuda().double() for f in (t.left, t.right))
        inverse_left, inverse_right = (torch.linalg.inv(f).transpose(-1, -2) for f in (left, right))
        w = torch.cat([_mx(_block_transform(p.double(), inverse_left, inverse_right), 2) for p in weight.split(2048)])
        y = []
        for p in x.split(2048):
            v = _block_transform(p.double(), left, right)
            if t.clip_lo is not None:
                lo, hi = (torch.from_numpy(c).cuda().double()[:, None] for c in (t.clip_lo, t.clip_hi))
                v = torch.minimum(torch.maximum(v, lo * v.amin(-1, keepdim=True)), hi * v.amax(-1, keepdim=True))
            y.append(_mx(v, emax) @ w.T)
        out.append(torch.cat(y))
    return out
