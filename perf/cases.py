"""What is timed: the calls that a program serving a model with a compressed KV cache makes.

A case names one path and its sizes:
  encode         append new tokens' keys and values to one layer's packed cache
  encode_hidden  the same, straight from the layer input
  decode         one decode step: every layer's attention of one new token per sequence
  decode_sw      the same with the attention sink and the recent window kept in bf16
  prefill        a chunk of new query tokens, causal over the packed cache
  group_encode, group_decode   encode and decode with one transform per group of kv-heads

The head counts, contexts and bit budgets are those of the workloads of this repository
(a Llama-3.1-8B-shaped layer with 8 kv-heads and 32 query heads, a Qwen-2.5-7B-shaped one with 4
and 28) and odd ones around them.  Keys and values follow the repository's input model: a random
orthogonal basis, a power-law spectrum, four outlier coordinates on the keys, bf16.  Plans are
"stream" (every kv-head's keys and values have the same budget), "global" (one pool of bits over
layers and heads whose spectra differ, so every stream has another record layout) or "wide" (a
global pool with channels of up to 16 bits).
"""
import functools
import math

import numpy as np
import torch

import paper_2608_14191_gb300 as aatc

D = 128
DEV = "cuda"
SINK = 4


def listed():
    return [
        # one flush of the recent window while a sequence is generated: 16 tokens, latency only
        dict(name="append_flush", path="encode", n_kv=8, n_q=32, batch=1, n_tokens=16, start=4099, layers=1,
             plan="stream", bits=2.75),
        # the prompt of one long request, one layer
        dict(name="encode_prompt", path="encode", n_kv=8, n_q=32, batch=1, n_tokens=32768, start=0, layers=1,
             plan="stream", bits=2.75),
        # several requests of a ragged length appended to caches that hold tokens already
        dict(name="encode_ragged", path="encode", n_kv=4, n_q=28, batch=5, n_tokens=3001, start=77, layers=1,
             plan="global", bits=3.0),
        # the same prompt encoded from the layer input
        dict(name="encode_hidden", path="encode_hidden", n_kv=8, n_q=32, batch=1, n_tokens=16384, start=0, layers=1,
             plan="stream", bits=2.75, d_model=4096),
        # the first tokens after a short prompt: a small cache, latency only
        dict(name="decode_short", path="decode", n_kv=8, n_q=32, batch=1, n_ctx=1001, layers=1, plan="stream",
             bits=2.75),
        # one decode step of a long request through some layers of the model
        dict(name="decode_step", path="decode", n_kv=8, n_q=32, batch=1, n_ctx=32768, layers=4, plan="stream",
             bits=2.75),
        # a batch of requests, seven query heads to a kv-head
        dict(name="decode_batch", path="decode", n_kv=4, n_q=28, batch=16, n_ctx=8192, layers=1, plan="stream",
             bits=2.75),
        # the global allocation: every layer and head has its own record layout
        dict(name="decode_global", path="decode", n_kv=8, n_q=32, batch=1, n_ctx=20011, layers=4, plan="global",
             bits=2.75),
        # the inference policy with a bf16 sink and window around the packed tokens
        dict(name="decode_sink_window", path="decode_sw", n_kv=8, n_q=32, batch=2, n_ctx=16021, n_full=139, layers=1,
             plan="stream", bits=2.0),
        # prefill of a batch of prompts, one layer
        dict(name="prefill_prompt", path="prefill", n_kv=4, n_q=28, batch=4, n_queries=8192, n_ctx=8192, layers=1,
             plan="stream", bits=2.75),
        # a ragged chunk at the end of a long context (chunked prefill, a follow-up turn)
        dict(name="prefill_chunk", path="prefill", n_kv=8, n_q=32, batch=1, n_queries=333, n_ctx=30011, layers=1,
             plan="stream", bits=2.75),
        # a decode step with one transform per four kv-heads
        dict(name="group_decode", path="group_decode", n_kv=8, n_q=32, g_h=4, batch=1, n_ctx=16384, layers=1,
             plan="stream", bits=2.75),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["encode", "encode", "encode_hidden", "decode", "decode", "decode", "decode_sw", "prefill",
                       "prefill", "group_encode", "group_decode"])
    n_kv, group = rng.choice([(8, 4), (8, 4), (4, 7), (2, 4), (4, 2), (8, 1), (1, 8), (3, 5)])
    plans = ["stream", "global"] + (["wide"] if path in ("encode", "decode") else [])
    c = dict(path=path, n_kv=n_kv, n_q=n_kv * group, layers=1, plan=rng.choice(plans),
             bits=rng.choice([1.5, 2.0, 2.25, 2.5, 2.75, 3.0, 3.5, 4.0]))
    if path in ("group_encode", "group_decode"):
        c["n_kv"], c["g_h"], group = rng.choice([(8, 4, 4), (8, 2, 4), (4, 4, 2), (4, 2, 7)])
        c.update(n_q=c["n_kv"] * group, plan="stream", bits=rng.choice([2.0, 2.5, 2.75, 3.0]))
    if path in ("encode", "group_encode", "encode_hidden"):
        c["n_tokens"] = _log_int(rng, 1, 16384 if path == "encode_hidden" else 32768)
        c["batch"] = max(1, min(_log_int(rng, 1, 32), 32768 // c["n_tokens"]))
        c["start"] = rng.choice([0, rng.randrange(1, 1000)])
        if path == "encode_hidden":
            c["d_model"] = rng.choice([512, 1536, 2048, 4096])
            c["batch"] = max(1, min(c["batch"], 16384 // c["n_tokens"]))
        return c
    c["n_ctx"] = _log_int(rng, 1, 65536)
    c["batch"] = max(1, min(_log_int(rng, 1, 32), 131072 // c["n_ctx"]))
    if path == "decode":
        c["layers"] = rng.choice([1, 1, 2, 3])
    if path == "decode_sw":
        c["n_full"] = _log_int(rng, 1, 400)
        c["n_ctx"] = max(c["n_ctx"], SINK + 1)
    if path == "prefill":
        c["batch"] = max(1, min(c["batch"], 32768 // c["n_ctx"]))
        c["n_queries"] = min(c["n_ctx"], _log_int(rng, 1, 8192))
        while c["batch"] * c["n_queries"] * c["n_ctx"] * c["n_q"] > 3.5e9:
            c["n_queries"] = max(1, c["n_queries"] // 2)
    return c


# ---------------------------------------------------------------- the model behind the inputs
def _width(case):
    return D * case.get("g_h", 1)


def _allocate(g, total, b_max):
    """Integer reverse water-filling: the `total` largest marginal gains of g 4^-b over all channels."""
    flat = g.reshape(-1)
    gains = flat[:, None] * 4.0 ** -np.arange(b_max)[None, :]
    order = np.argsort(-gains.reshape(-1), kind="stable")[:total]
    return np.bincount(order // b_max, minlength=flat.size).reshape(g.shape).astype(np.uint8)


@functools.lru_cache(maxsize=24)
def _model(n_layers, n_streams, n, plan, bits):
    """Per stream (layer, head or group, keys | values): the mixing matrix of its vectors and the
    basis, widths and scales of its plan, channels by falling variance."""
    rng = np.random.default_rng([n_layers, n_streams, n, int(bits * 64), len(plan)])
    shape = (n_layers, n_streams, 2)
    mix, basis = np.empty(shape + (n, n), np.float32), np.empty(shape + (n, n), np.float32)
    var = np.empty(shape + (n,))
    for i in np.ndindex(shape):
        q, r = np.linalg.qr(rng.standard_normal((n, n)))
        exponent = 1.5 if plan == "stream" else rng.uniform(1.1, 2.1)
        m = q * np.sign(np.diag(r)) * np.sqrt(np.arange(1, n + 1) ** -exponent)
        if i[2] == 0 and n == D:
            m[rng.choice(n, 4, replace=False)] *= 8.0
        w, u = np.linalg.eigh(m @ m.T)
        mix[i], basis[i], var[i] = m, u[:, ::-1], np.maximum(w[::-1], 1e-30)
    widths = np.empty(shape + (n,), np.uint8)
    if plan == "stream":
        for i in np.ndindex(shape):
            widths[i] = _allocate(var[i], round(bits * n), 8)
    else:
        b_max = 16 if plan == "wide" else 8
        for kind in (0, 1):
            widths[:, :, kind] = _allocate(var[:, :, kind], round(bits * n) * n_layers * n_streams, b_max)
    scales = (2.5758293 * np.sqrt(var)).astype(np.float32)          # the 99th percentile of |h|
    return mix, np.ascontiguousarray(basis), widths, scales


def _model_of(case):
    return _model(case["layers"], case["n_kv"] // case.get("g_h", 1), _width(case), case["plan"], case["bits"])


@functools.lru_cache(maxsize=8)
def _hidden_model(n_kv, d_model, plan, bits):
    """Variances of the layer input, the encode operand (W U)^T of every stream, and the plan."""
    rng = np.random.default_rng([n_kv, d_model, int(bits * 64), len(plan)])
    std = np.sqrt(np.arange(1, d_model + 1) ** -1.0)
    std[rng.choice(d_model, 4, replace=False)] *= 20.0
    std = rng.permutation(std)
    operand = np.empty((n_kv, 2, D, d_model), np.float32)
    basis = np.empty((1, n_kv, 2, D, D), np.float32)
    var = np.empty((1, n_kv, 2, D))
    for h in range(n_kv):
        for kind in (0, 1):
            w = rng.standard_normal((d_model, D), np.float32) / math.sqrt(d_model)
            k = w * std[:, None].astype(np.float32)
            e, u = np.linalg.eigh((k.T @ k).astype(np.float64))
            basis[0, h, kind], var[0, h, kind] = u[:, ::-1], np.maximum(e[::-1], 1e-30)
            operand[h, kind] = (w @ basis[0, h, kind]).T
    widths = np.empty((1, n_kv, 2, D), np.uint8)
    for kind in (0, 1):
        if plan == "stream":
            for h in range(n_kv):
                widths[0, h, kind] = _allocate(var[0, h, kind], round(bits * D), 8)
        else:
            widths[0, :, kind] = _allocate(var[0, :, kind], round(bits * D) * n_kv, 8)
    scales = (2.5758293 * np.sqrt(var)).astype(np.float32)
    return std.astype(np.float32), operand, basis, widths, scales


def _generator(seed):
    g = torch.Generator(DEV)
    g.manual_seed(int(seed))
    return g


def _tokens(case, layer, batch, n, gen):
    """K and V of one layer: bf16 [batch][n][n_kv][128], drawn from the streams' models."""
    mix = torch.from_numpy(_model_of(case)[0][layer]).to(DEV)          # [streams][2][n][n]
    w = _width(case)
    out = []
    for kind in (0, 1):
        x = torch.empty((batch, n, case["n_kv"], D), dtype=torch.bfloat16, device=DEV)
        xs = x.view(batch * n, -1, w)
        for s in range(xs.shape[1]):
            z = torch.randn((batch * n, w), generator=gen, device=DEV)
            xs[:, s] = (z @ mix[s, kind].T).to(torch.bfloat16)
        out.append(x)
    return out


def _plan(case):
    if case["path"] == "encode_hidden":
        basis, widths, scales = _hidden_model(case["n_kv"], case["d_model"], case["plan"], case["bits"])[2:]
    else:
        basis, widths, scales = _model_of(case)[1:]
    dims = aatc.dims(case["layers"], case["n_kv"], case["n_q"], b_max=16 if case["plan"] == "wide" else 8)
    if "g_h" in case:
        return aatc.GroupPlan(dims, case["g_h"], basis, widths, scales)
    return aatc.Plan(dims, basis, widths, scales)


def _inputs(case, seed):
    """The tensors of one pass, from the seed alone."""
    g = _generator(seed)
    c = case
    if c["path"] in ("encode", "group_encode"):
        return dict(kv=_tokens(c, 0, c["batch"], c["n_tokens"], g))
    if c["path"] == "encode_hidden":
        std, operand = _hidden_model(c["n_kv"], c["d_model"], c["plan"], c["bits"])[:2]
        x = torch.randn((c["batch"], c["n_tokens"], c["d_model"]), generator=g, device=DEV)
        return dict(x=(x * torch.from_numpy(std).to(DEV)).to(torch.bfloat16),
                    a_hat=torch.from_numpy(operand).to(DEV).to(torch.bfloat16)[None].contiguous())
    got = dict(kv=[_tokens(c, layer, c["batch"], c["n_ctx"], g) for layer in range(c["layers"])])
    rows = (c["batch"], c["n_queries"]) if c["path"] == "prefill" else (c["layers"], c["batch"])
    got["q"] = torch.randn(rows + (c["n_q"], D), generator=g, device=DEV).to(torch.bfloat16)
    if c["path"] == "decode_sw":
        got["full"] = _tokens(c, 0, c["batch"], c["n_full"], g)
    return got


def _capacity(case):
    used = case["start"] + case["n_tokens"] if "n_tokens" in case else case["n_ctx"]
    return (used + 511) // 256 * 256


def prepare(case, seed):
    got = _inputs(case, seed)
    plan, cap = _plan(case), _capacity(case)
    state = dict(case=case, plan=plan, cap=cap, **got)
    if "n_tokens" in case:
        state["cache"] = plan.new_cache(case["batch"], cap, DEV).zero_()
        return state
    state["caches"] = []
    for layer, (k, v) in enumerate(state.pop("kv")):
        cache = plan.new_cache(case["batch"], cap, DEV).zero_()
        aatc.encode(plan, layer, k, v, cache, 0, cap)
        state["caches"].append(cache)
    # what a serving loop allocates once: the outputs and the workspace of its calls
    if case["path"] in ("decode", "decode_sw", "group_decode"):
        state["out"] = torch.empty((case["layers"], case["batch"], case["n_q"], D), device=DEV)
        n = plan.workspace_bytes(case["batch"], case["n_ctx"])
        state["workspace"] = torch.empty(max(1, n // 4), device=DEV)
    return state


def run(state):
    c, plan, cap = state["case"], state["plan"], state["cap"]
    if "n_tokens" in c:
        cache = state["cache"]
        if c["path"] == "encode_hidden":
            aatc.encode_hidden(plan, 0, state["x"], state["a_hat"], cache, c["start"], cap)
        else:
            aatc.encode(plan, 0, state["kv"][0], state["kv"][1], cache, c["start"], cap)
        n_alpha = c["batch"] * c["n_kv"] * 2 * cap // 128 * 128
        return dict(words=cache[:-n_alpha], alpha=cache[-n_alpha:].view(torch.float32))
    if c["path"] == "prefill":
        return aatc.prefill_attention(plan, 0, state["q"], c["n_ctx"] - c["n_queries"], state["caches"][0],
                                      c["n_ctx"], cap)
    out, q, ws = state["out"], state["q"], state["workspace"]
    if c["path"] == "decode_sw":
        aatc.decode_attention_sw(plan, 0, q[0], state["caches"][0], SINK, c["n_ctx"], cap, state["full"][0],
                                 state["full"][1], c["n_full"], out=out[0], workspace=ws)
        return out
    for layer in range(c["layers"]):
        aatc.decode_attention(plan, layer, q[layer], state["caches"][layer], c["n_ctx"], cap, out=out[layer],
                              workspace=ws)
    return out


# ---------------------------------------------------------------- work, tolerance, 64-bit results
def _record_bytes(case, layer):
    """Packed bytes of one token: every stream's code bits and a 32-bit scale (one per stream)."""
    widths = (_hidden_model(case["n_kv"], case["d_model"], case["plan"], case["bits"])[3]
              if case["path"] == "encode_hidden" else _model_of(case)[2])
    return float(widths[layer].astype(np.int64).sum()) / 8 + 4 * widths[layer][..., 0].size


def work(case):
    c = case
    w = _width(c)
    if "n_tokens" in c:
        tokens = c["batch"] * c["n_tokens"]
        packed = tokens * _record_bytes(c, 0)
        if c["path"] == "encode_hidden":
            m = c["d_model"]
            return dict(bytes=tokens * m * 2 + c["n_kv"] * 2 * D * m * 2 + packed,
                        flops=2.0 * tokens * m * c["n_kv"] * 2 * D)
        return dict(bytes=tokens * c["n_kv"] * 2 * D * 2 + packed, flops=2.0 * tokens * c["n_kv"] * 2 * D * w)
    if c["path"] == "prefill":
        rows = c["batch"] * c["n_queries"] * c["n_q"]
        first = c["n_ctx"] - c["n_queries"]
        pairs = c["batch"] * c["n_q"] * sum(range(first + 1, c["n_ctx"] + 1))
        return dict(bytes=rows * D * 6 + c["batch"] * c["n_ctx"] * _record_bytes(c, 0), flops=4.0 * pairs * D)
    tokens = c["batch"] * (c["n_ctx"] - (SINK if c["path"] == "decode_sw" else 0))
    size = sum(tokens * _record_bytes(c, layer) for layer in range(c["layers"]))
    size += c["layers"] * c["batch"] * c["n_q"] * D * 6
    full = c["batch"] * c.get("n_full", 0)
    return dict(bytes=size + full * c["n_kv"] * D * 4,
                flops=4.0 * c["n_q"] * (c["layers"] * tokens * w // c["n_kv"] * c["n_kv"] + full * D))


def tolerance(case):
    if "n_tokens" in case:
        # words: only codes within fp32 rounding of a decision threshold; scales: one fp32 maximum
        return {"rel": 1e-5, "max": 1e-4, "differ": 1e-5}
    if case["path"] == "prefill":
        return {"rel": 1e-3, "max": 6e-2}          # softmax weights as f16 tensor-core operands
    return {"rel": 1e-4, "max": 2.5e-3}              # fp32 sums over operands of about 22 bits


def _coefficients(x, operand, widths, scales):
    """h = x U in 64 bits with the bf16 operand, the token scale, the channel scales and widths."""
    h = x.double() @ operand.double()
    b = torch.from_numpy(widths.astype(np.float64)).to(DEV)
    s = torch.from_numpy(scales.astype(np.float64)).to(DEV)
    alpha = torch.where(b > 0, h.abs() / s, torch.zeros_like(h)).amax(-1)
    return h, alpha, s, b


def _dequantized(h, alpha, s, b):
    f = torch.where(b > 0, s * torch.exp2(1.0 - b), torch.zeros_like(s))
    step = alpha[:, None] * f
    t = torch.floor(torch.where(step > 0, h / torch.where(step > 0, step, torch.ones_like(step)),
                                torch.zeros_like(h)) + 0.5)
    half = torch.exp2(b - 1.0)
    code = torch.where(b > 0, torch.minimum(torch.maximum(t, -half), half - 1), torch.zeros_like(t))
    return code * step


def _bf16_operand(u):
    return torch.from_numpy(u).to(DEV).to(torch.bfloat16)


def _stream_values(case, kv, layer):
    """Per stream and kind: 64-bit tokens rebuilt from their codes, [2][streams][batch n][n]."""
    _, basis, widths, scales = _model_of(case)
    w = _width(case)
    got = []
    for kind in (0, 1):
        xs = kv[layer][kind].reshape(-1, case["n_kv"] * D // w, w)
        one = []
        for s in range(xs.shape[1]):
            h = _coefficients(xs[:, s], _bf16_operand(basis[layer, s, kind]), widths[layer, s, kind],
                              scales[layer, s, kind])
            one.append(_dequantized(*h) @ torch.from_numpy(basis[layer, s, kind]).to(DEV).double().T)
        got.append(one)
    return got


def exact(case, seed):
    c = case
    got = _inputs(c, seed)
    if "n_tokens" in c:
        cap = _capacity(c)
        alpha = torch.zeros((c["batch"], c["n_kv"], 2, cap), dtype=torch.float64, device=DEV)
        for h in range(c["n_kv"]):
            for kind in (0, 1):
                if c["path"] == "encode_hidden":
                    _, _, _, widths, scales = _hidden_model(c["n_kv"], c["d_model"], c["plan"], c["bits"])
                    x, op, s = got["x"].reshape(-1, c["d_model"]), got["a_hat"][0, h, kind].T, h
                else:
                    w = _width(c)
                    s = h * D // w                     # a group's streams share one scale
                    _, basis, widths, scales = _model_of(c)
                    x = got["kv"][kind].reshape(c["batch"] * c["n_tokens"], -1, w)[:, s]
                    op = _bf16_operand(basis[0, s, kind])
                a = _coefficients(x, op, widths[0, s, kind], scales[0, s, kind])[1]
                alpha[:, h, kind, c["start"]:c["start"] + c["n_tokens"]] = a.view(c["batch"], c["n_tokens"])
        return dict(words=None, alpha=alpha.reshape(-1))
    rows = (c["batch"], c["n_queries"], c["n_q"], D) if c["path"] == "prefill" else got["q"].shape
    out = torch.zeros(rows, dtype=torch.float64, device=DEV)
    group, w, n = c["n_q"] // c["n_kv"], _width(c), c["n_ctx"]
    first = SINK if c["path"] == "decode_sw" else 0
    for layer in range(c["layers"]):
        keys, values = _stream_values(c, got["kv"], layer)
        for b in range(c["batch"]):
            for h in range(c["n_kv"]):
                part = slice(h * D % w, h * D % w + D)
                k, v = (t[h * D // w].view(c["batch"], n, w)[b, first:, part] for t in (keys, values))
                heads = slice(h * group, (h + 1) * group)
                if c["path"] == "decode_sw":
                    k, v = (torch.cat([t, f[b, :, h].double()]) for t, f in zip((k, v), got["full"]))
                if c["path"] != "prefill":
                    p = torch.softmax(got["q"][layer, b, heads].double() @ k.T / math.sqrt(D), -1)
                    out[layer, b, heads] = p @ v
                    continue
                for q0 in range(0, c["n_queries"], 1024):
                    q = got["q"][b, q0:q0 + 1024, heads].double()          # [rows][group][128]
                    pos = n - c["n_queries"] + q0 + torch.arange(q.shape[0], device=DEV)
                    end = int(pos[-1]) + 1
                    s = torch.einsum("rgd,td->rgt", q, k[:end]) / math.sqrt(D)
                    s.masked_fill_(torch.arange(end, device=DEV)[None, None] > pos[:, None, None], -math.inf)
                    out[b, q0:q0 + 1024, heads] = torch.softmax(s, -1) @ v[:end]
    return out
