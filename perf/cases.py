"""The work that users of the MUXQ layer have it do, as cases that can be timed and compared.

Three kinds of work:

  linear    muxq_linear called once per layer on activations that are on the GPU: prompts (M > 16 token rows, the
            tensor-core path) and single decode steps (M <= 16, the weight-streaming path).  Layers are the four
            projections of a transformer block of width d (d -> 3d, d -> d, d -> 4d, 4d -> d) or one d -> d layer.
  list      muxq_chain_run: the projections of all blocks at a decode step in one persistent launch.
  weights   muxq_quantize(is_weight = 1): what loading a model costs per block.

Activations are N(0, 1) with a few outlier channels times 40 to 80, or heavy-tailed (Student-t with 4 degrees of
freedom, times 0.05) with outlier channels times 60; weights are N(0, 0.02)."""
import math

import torch

import paper_2604_04701_b200 as mx

_PROMPT = {"kind": "linear", "linears": "block", "blocks": 1, "vector": False, "bias": False, "out": "f16",
           "bulk": "normal", "graph": False}
_STEP = dict(_PROMPT, outliers=8)
_LIST = {"kind": "list", "linears": "block", "vector": False, "bias": False, "out": "f16", "bulk": "normal",
         "outliers": 8, "dependent": False}


def listed():
    return [
        # one small projection on a short prompt: the smallest call, latency and launches count
        dict(_PROMPT, name="single_128", linears="one", width=768, tokens=128, outliers=4),
        # a prompt of odd length through a block whose width is no multiple of 64 or 128, fp32 results for a residual
        # stream kept in fp32, per-token / per-channel scales, bias
        dict(_PROMPT, name="prompt_1003_ragged", width=1040, tokens=1003, vector=True, bias=True, out="f32", outliers=7),
        # eight prompts of 1024 tokens through a block of the small width, per-tensor scales
        dict(_PROMPT, name="small_8192", width=768, tokens=8192, outliers=6),
        # the same tokens at the large width, per-token / per-channel scales, with bias and many outlier channels
        dict(_PROMPT, name="large_8192_vector_bias", width=1280, tokens=8192, vector=True, bias=True, outliers=32),
        # the largest prompt batch: a block of the large width at 16384 tokens
        dict(_PROMPT, name="large_16384", width=1280, tokens=16384, outliers=8),
        # one decode step of one sequence through 36 blocks, one call per layer, captured once in a graph and replayed
        dict(_STEP, name="step_1_graph", width=1280, tokens=1, blocks=36, graph=True),
        # one decode step of 16 sequences through 12 blocks of the small width, one plain call per layer
        dict(_STEP, name="step_16_calls", width=768, tokens=16, blocks=12),
        # the same as lists in one launch: one sequence, four (medium width), sixteen
        dict(_LIST, name="list_1", width=1280, tokens=1, blocks=36),
        dict(_LIST, name="list_4", width=1024, tokens=4, blocks=24),
        dict(_LIST, name="list_16", width=1280, tokens=16, blocks=36),
        # loading the weights of one block of the large width, per output channel
        {"name": "weights_large", "kind": "weights", "linears": "block", "width": 1280, "vector": True},
    ]


_MOST_FLOPS = 2 * 16384 * 12 * 1280 ** 2


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("prompt", "prompt", "prompt", "step", "list", "list", "weights"))
    if kind == "weights":
        return {"kind": "weights", "linears": "block", "width": 16 * rng.randint(24, 96), "vector": rng.random() < 0.5}
    vector, bias = rng.random() < 0.4, rng.random() < 0.4
    out = rng.choice(("f16", "f16", "f32"))
    if kind == "list":
        case = dict(_LIST, width=64 * rng.randint(8, 20), tokens=rng.randint(1, 16), vector=vector, bias=bias)
        if rng.random() < 0.25:  # every layer reads the one before it
            return dict(case, blocks=rng.randint(2, 8), outliers=rng.choice((0, 2, 8)), dependent=True)
        return dict(case, blocks=rng.randint(2, 36), out=out, outliers=rng.choice((0, 2, 8, 32)))
    if kind == "step":
        return dict(_STEP, width=16 * rng.randint(32, 80), tokens=rng.randint(1, 16), blocks=rng.randint(1, 24),
                    vector=vector, bias=bias, out=out, outliers=rng.choice((0, 2, 8, 32)), graph=rng.random() < 0.5)
    one = rng.random() < 0.25
    width = 16 * rng.randint(24, 96)
    most = min(16384, _MOST_FLOPS // (2 * width * width * (1 if one else 12)))
    return dict(_PROMPT, linears="one" if one else "block", width=width, tokens=_log_uniform(rng, 17, most),
                vector=vector, bias=bias, out=out, bulk=rng.choice(("normal", "normal", "t4")),
                outliers=rng.choice((0, 2, 6, 8, 32)))


def _shapes(case):
    d = case["width"]
    return [(d, d)] if case["linears"] == "one" else [(d, 3 * d), (d, d), (d, 4 * d), (4 * d, d)]


def _params(case):
    return mx.MuxqParams(gran=mx.MUXQ_PER_VECTOR if case["vector"] else mx.MUXQ_PER_TENSOR)


def _activations(gen, count, tokens, K, outliers, bulk, mult=(40.0, 80.0)):
    """[count, tokens, K] fp16, each of the `count` matrices with outlier channels of its own."""
    if bulk == "t4":
        x = torch.randn(count, tokens, K, device="cuda", generator=gen)
        u = torch.rand(2, count, tokens, K, device="cuda", generator=gen).clamp_(min=1e-7)
        x = 0.05 * x / (-0.5 * (u[0] * u[1]).log()).sqrt()
        lo, hi = 60.0, 60.0
    else:
        x = torch.randn(count, tokens, K, device="cuda", generator=gen)
        lo, hi = mult
    if outliers:
        channels = torch.rand(count, K, device="cuda", generator=gen).argsort(dim=1)[:, :outliers]
        by = lo + (hi - lo) * torch.rand(count, outliers, device="cuda", generator=gen)
        x *= torch.ones(count, K, device="cuda").scatter_(1, channels, by)[:, None, :]
    return x.half()


def _weight(gen, K, N, sigma=0.02, large=0):
    w = torch.randn(K, N, device="cuda", generator=gen) * sigma
    if large:  # output channels that become outlier channels of the next layer
        w[:, torch.randperm(N, device="cuda", generator=gen)[:large]] *= 10.0
    return w.half()


def _out_dtype(case):
    return torch.float32 if case["out"] == "f32" else torch.float16


def _out_kind(case):
    return mx.MUXQ_OUT_F32 if case["out"] == "f32" else mx.MUXQ_OUT_F16


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    p, shapes = _params(case), _shapes(case)
    load = mx.Workspace(mx.muxq_small_workspace_bytes(max(N for _, N in shapes)))
    if case["kind"] == "weights":
        return {"kind": "weights", "p": p, "ws": load, "w": [_weight(gen, K, N) for K, N in shapes]}
    tokens, blocks, dependent = case["tokens"], case["blocks"], case.get("dependent", False)
    if dependent:  # a layer's output feeds the next: keep its magnitude, and outlier channels in every layer
        shapes = [(case["width"], 4 * case["width"]), (4 * case["width"], case["width"])]
    y = [torch.empty(blocks, tokens, N, dtype=_out_dtype(case), device="cuda") for _, N in shapes]
    x = [_activations(gen, blocks, tokens, K, case["outliers"], case["bulk"], (10.0, 10.0) if dependent else (40.0, 80.0))
         for K, _ in shapes]
    layers = []
    for b in range(blocks):
        for i, (K, N) in enumerate(shapes):
            sigma = 1.0 / math.sqrt(K + 99.0 * case["outliers"]) if dependent else 0.02
            w_q, s_w = mx.muxq_quantize(_weight(gen, K, N, sigma, case["outliers"] if dependent else 0), p, True, load)
            bias = 0.1 * torch.randn(N, device="cuda", generator=gen) if case["bias"] else None
            first = not layers
            xi = x[i][b] if first or not dependent else layers[-1][3]
            layers.append((xi, w_q, s_w, y[i][b], mx.MUXQ_LAYER_WAIT_PREV if dependent and not first else 0, bias))
    state = {"kind": case["kind"], "p": p, "out_kind": _out_kind(case), "y": y, "layers": layers, "graph": None}
    if case["kind"] == "list":
        state["chain"] = mx.Chain(layers, p, state["out_kind"])
        return state
    state["ws"] = mx.Workspace(max(mx.muxq_workspace_bytes(tokens, K, N, p) for K, N in shapes))
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _calls(state)
            side.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                _calls(state)
        torch.cuda.synchronize()
        state["graph"] = graph
    return state


def _calls(state):
    for x, w_q, s_w, y, _, bias in state["layers"]:
        mx.muxq_linear(x, w_q, s_w, state["p"], state["ws"], state["out_kind"], out=y, bias=bias)


def run(state):
    if state["kind"] == "weights":
        return [mx.muxq_quantize(w, state["p"], True, state["ws"]) for w in state["w"]]
    if state["kind"] == "list":
        state["chain"].run()
    elif state["graph"] is not None:
        state["graph"].replay()
    else:
        _calls(state)
    return state["y"]


def work(case):
    """Inputs once, outputs once: X fp16, W_q int8 (fp16 W in, int8 W_q out for the weights), scales, bias, Y."""
    b = f = 0.0
    shapes = _shapes(case)
    if case["kind"] == "weights":
        return {"bytes": sum(3.0 * K * N + 4.0 * (N if case["vector"] else 1) for K, N in shapes), "flops": 0.0}
    tokens, blocks = case["tokens"], case["blocks"]
    if case.get("dependent"):
        shapes = [(case["width"], 4 * case["width"]), (4 * case["width"], case["width"])]
    out = 4.0 if case["out"] == "f32" else 2.0
    for K, N in shapes:
        b += 2.0 * tokens * K + 1.0 * K * N + out * tokens * N
        b += (4.0 * N if case["vector"] else 4.0) + (4.0 * N if case["bias"] else 0.0)
        f += 2.0 * tokens * K * N
    return {"bytes": b * blocks, "flops": f * blocks}


def tolerance(case):
    """The codes and accumulators are whole numbers and the same for every correct implementation; what may differ is the
    rounding of the last two products and of the cast.  Against the same products in 64 bits: fp32 results 3.4e-8 (largest
    8.1e-8), fp16 results 5e-6 to 1.3e-5 (one unit in the last place on one value in ten thousand, largest 9.8e-4).  Where a
    layer reads the fp16 result of the one before it, such a unit can move a code, and that grows along the list; the
    interface pins both roundings (scales first, then the accumulator), so these lists have one right answer."""
    if case["kind"] == "weights" or case.get("dependent"):
        return "exact"
    return {"rel": 1.4e-7, "max": 4e-7} if case["out"] == "f32" else {"rel": 5e-5, "max": 4e-3}
