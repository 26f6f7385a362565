"""Performance cases of the HybridKV path: what a serving program has the library do for one model.

Four kinds, all through the binding of the C ABI with device buffers the caller owns:

* ``decode``    one autoregressive step: one attention call per layer over that layer's compressed cache.
                ``call`` says how the program issues it: ``eager`` (a call per layer), ``graph`` (the same
                calls captured once in a CUDA graph and replayed every step) or ``host`` (queries and
                outputs in pinned host memory, one call for the whole step, waited for).
* ``prefill``   one layer's prompt: its K/V compressed into caller-owned memory, then the first step over it.
* ``generate``  a short request: every layer's prompt compressed, then a few tokens, each layer's new key and
                value appended before its attention call.
* ``classify``  static / dynamic labels of one layer's heads from the text tokens' queries.

Head geometries are 28 query / 4 KV heads and 16 / 2, head_dim 128, as in the benchmark and the tests.  Inputs
are drawn on the GPU from the seed: keys are per-frame means plus noise (video and image prompts have correlated
keys), three chunks per layer lie along a direction the decode queries lean towards (cosine 0.6), text spans
separate the visual blocks.
"""
import math
import random

import numpy as np
import torch

from paper_2604_05887_b200 import binding as hkv

HEAD_DIM = 128
WINDOW = 32          # observation window of every workload
TAIL_TEXT = 64       # the user's question at the end of the prompt
TOPK_FRACTION, THETA = 0.05, 0.9

_BASE = dict(q_heads=28, kv_heads=4, chunk=32, budget=0.1, static=0.5, ragged=False, block=1024, span=16,
             out="bf16", score="sum", causal=False)


def _case(name, kind, **fields):
    return dict(_BASE, name=name, kind=kind, **fields)


def listed():
    return [
        # the smallest call: one layer of a single short prompt (latency and launch cost)
        _case("decode_1l_b1_2k", "decode", call="eager", layers=1, batch=1, tokens=2048, block=1920),
        # an interactive user with an image-block prompt: a whole model's step, batch 1
        _case("decode_28l_b1_16k", "decode", call="eager", layers=28, batch=1, tokens=16384),
        # the benchmark's step: video-like prompts of different lengths, replayed as one graph
        _case("decode_28l_b4_32k_graph", "decode", call="graph", layers=28, batch=4, tokens=32768, ragged=True,
              chunk=64, static=0.6, block=500, span=11),
        # the longest contexts, a small share of them kept: many chunk means scored per retained token
        _case("decode_28l_b8_50k", "decode", call="eager", layers=28, batch=8, tokens=50000, budget=0.05, static=0.4),
        # a throughput batch at a large budget: bytes decide
        _case("decode_1l_b16_32k_half", "decode", call="eager", layers=1, batch=16, tokens=32768, budget=0.5),
        # the 16 / 2 geometry with the options a research user turns on: float32 output, group maximum, small chunks
        _case("decode_8l_b3_5k_f32", "decode", call="eager", layers=8, batch=3, tokens=5003, ragged=True, q_heads=16,
              kv_heads=2, chunk=16, budget=0.2, out="f32", score="max"),
        # queries and outputs in host memory, the step waited for (end to end)
        _case("decode_28l_b2_9k_host", "decode", call="host", layers=28, batch=2, tokens=9001, ragged=True),
        # one layer of the benchmark's prompts, compressed
        _case("prefill_b4_32k", "prefill", batch=4, tokens=32768, ragged=True, chunk=64, static=0.6, block=500, span=11),
        # the largest prompts
        _case("prefill_b8_50k", "prefill", batch=8, tokens=50000, budget=0.05, static=0.4),
        # a short request of one user from prompt to answer: small prefills, appends, small steps
        _case("generate_4l_b1_4k", "generate", layers=4, batch=1, tokens=4099, steps=8, causal=True),
        # head labels before the compression of the benchmark's prompts
        _case("classify_b4_32k_256t", "classify", batch=4, tokens=32768, ragged=True, block=500, span=11, text=256),
        # a single long prompt with a short question
        _case("classify_b1_50k_48t", "classify", batch=1, tokens=50000, text=48),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    # kinds in the proportions of the list
    kind = rng.choice(["decode"] * 7 + ["prefill"] * 2 + ["generate"] + ["classify"] * 2)
    c = dict(_BASE, kind=kind)
    c["q_heads"], c["kv_heads"] = rng.choice([(28, 4), (28, 4), (16, 2)])
    c["ragged"] = rng.random() < 0.5
    c["block"], c["span"] = rng.choice([(1024, 16), (500, 11)])
    c["static"] = round(rng.uniform(0.2, 0.8), 2)
    c["causal"] = rng.random() < 0.2
    c["tokens"] = _log_int(rng, 1500, 50000)
    c["batch"] = _log_int(rng, 1, 16)
    if kind == "classify":
        c["batch"] = _log_int(rng, 1, 4)
        c["text"] = _log_int(rng, 24, 256)
        return c
    c["chunk"] = rng.choice([16, 24, 32, 64, 128])
    c["budget"] = round(math.exp(rng.uniform(math.log(0.05), math.log(0.5))), 3)
    c["out"] = rng.choice(["bf16", "bf16", "bf16", "f32"])
    c["score"] = rng.choice(["sum", "sum", "sum", "max"])
    if kind == "decode":
        c["layers"] = _log_int(rng, 1, 28)
        c["call"] = rng.choice(["eager", "eager", "graph", "host"])
    elif kind == "prefill":
        c["batch"] = _log_int(rng, 1, 8)
    else:
        c["layers"], c["steps"] = _log_int(rng, 1, 8), _log_int(rng, 2, 16)
        c["batch"], c["tokens"] = _log_int(rng, 1, 4), _log_int(rng, 1500, 16384)
    return c


def _cost(case):
    """Rough seconds at the memory and tensor rates, for the limit on drawn cases."""
    w = work(case)
    return w["bytes"] / 6e12 + w["flops"] / 1e15


def draw(rng):
    """A case of the listed ranges that moves and computes no more than the largest listed one of its kind."""
    largest = {}
    for c in listed():
        largest[c["kind"]] = max(largest.get(c["kind"], 0.0), _cost(c))
    largest["generate"] = largest["prefill"]
    while True:
        c = _draw_once(rng)
        if _cost(c) <= largest[c["kind"]] and c.get("layers", 1) * c["batch"] * c["tokens"] <= 28 * 8 * 50000:
            return c


# ---------------------------------------------------------------------------------------------
# geometry that follows from the case alone
# ---------------------------------------------------------------------------------------------
def _seq_lens(case):
    """The full length first; a ragged batch goes down to three quarters of it."""
    B, C = case["batch"], case["tokens"]
    if not case["ragged"] or B == 1:
        return [C] * B
    return [C - (C // 4) * b // (B - 1) for b in range(B)]


def _budget_tokens(case):
    return [max(1, math.ceil(case["budget"] * c - 1e-9)) for c in _seq_lens(case)]


def _n_static(case):
    return int(math.floor(case["static"] * case["batch"] * case["kv_heads"] + 0.5))


def _head_types(case, layer):
    """Exactly the static fraction of the layer's (sequence, head) pairs, spread over them by the layer's number;
    0 = static, 1 = dynamic."""
    n, H = case["batch"] * case["kv_heads"], case["kv_heads"]
    flat = [0] * _n_static(case) + [1] * (n - _n_static(case))
    random.Random(layer).shuffle(flat)
    return [flat[b * H:(b + 1) * H] for b in range(case["batch"])]


def _flags(case):
    return ((hkv.HKV_OUT_F32 if case["out"] == "f32" else 0) | (hkv.HKV_GROUP_MAX if case["score"] == "max" else 0) |
            (hkv.HKV_CAUSAL_WINDOW if case["causal"] else 0))


def _config(case):
    return hkv.make_config(case["batch"], case["q_heads"], case["kv_heads"], HEAD_DIM, case["tokens"], case["chunk"],
                           WINDOW, 0.0, _flags(case), case.get("steps", 0))


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
class _State:
    """Device buffers and handles of one case."""

    def __init__(self):
        self.handles = []

    def close(self):
        while self.handles:
            hkv.hkv_cache_destroy(self.handles.pop())

    def __del__(self):
        self.close()


def _is_text(case):
    """Text spans between the visual blocks and the question at the end."""
    m = torch.zeros(case["batch"], case["tokens"], dtype=torch.uint8)
    for b, c in enumerate(_seq_lens(case)):
        for s in range(0, c, case["block"] + case["span"]):
            m[b, s:min(c, s + case["span"])] = 1
        m[b, max(0, c - TAIL_TEXT):c] = 1
    return m.cuda()


def _directions(case, g):
    u = torch.randn(case["batch"], case["kv_heads"], HEAD_DIM, device="cuda", generator=g)
    return u / u.norm(dim=-1, keepdim=True)


def _keys_values(case, g, rng, u):
    B, H, C, cs = case["batch"], case["kv_heads"], case["tokens"], case["chunk"]
    k = torch.randn(B, H, C, HEAD_DIM, device="cuda", dtype=torch.bfloat16, generator=g)
    v = torch.randn(B, H, C, HEAD_DIM, device="cuda", dtype=torch.bfloat16, generator=g)
    period = case["block"] + case["span"]
    mean = torch.randn(B, H, -(-C // period), HEAD_DIM, device="cuda", generator=g).mul_(math.sqrt(0.5)).bfloat16()
    for f in range(mean.shape[2]):
        k[:, :, f * period:(f + 1) * period] += mean[:, :, f:f + 1]
    n_chunks = min(_seq_lens(case)) // cs
    for c in rng.sample(range(n_chunks), min(3, n_chunks)):
        k[:, :, c * cs:(c + 1) * cs] += (4.0 * u).bfloat16()[:, :, None]
    return k, v


def _queries(case, g, u, n):
    """n steps' queries [n, B, Hq, d] at cosine about 0.6 to the planted direction of their KV head."""
    G = case["q_heads"] // case["kv_heads"]
    x = torch.randn(n, case["batch"], case["q_heads"], HEAD_DIM, device="cuda", generator=g)
    return (0.8 * x + 0.6 * math.sqrt(HEAD_DIM) * u.repeat_interleave(G, dim=1)).bfloat16()


def _out_buffer(case, n):
    dt = torch.float32 if case["out"] == "f32" else torch.bfloat16
    return torch.empty(n, case["batch"], case["q_heads"], HEAD_DIM, device="cuda", dtype=dt)


def _layer_inputs(case, g, rng, u, layer):
    """One layer's compression inputs in the order hkv_compress takes them, without the two buffers."""
    k, v = _keys_values(case, g, rng, u)
    q_obs = torch.randn(case["batch"], WINDOW, case["q_heads"], HEAD_DIM, device="cuda", dtype=torch.bfloat16, generator=g)
    lens, H = _seq_lens(case), case["kv_heads"]
    return [k, v, q_obs, None, _is_text(case), np.array(lens, np.int32), np.array(_head_types(case, layer), np.uint8),
            np.array([[t] * H for t in _budget_tokens(case)], np.int32)]


def _buffers(cfg, inputs):
    cache_bytes, ws_bytes = hkv.hkv_plan(cfg, *inputs[5:])
    return [torch.empty(n, dtype=torch.uint8, device="cuda") for n in (cache_bytes, ws_bytes)]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = random.Random(seed)
    s = _State()
    s.kind, s.call = case["kind"], case.get("call", "")
    if s.kind == "classify":
        return _prepare_classify(case, g, s)
    cfg, n = _config(case), case.get("layers", 1)
    if s.kind == "decode":
        s.keep, qs = [], []
        for layer in range(n):
            u = _directions(case, g)
            inputs = _layer_inputs(case, g, rng, u, layer)
            cache, ws = _buffers(cfg, inputs)
            s.handles.append(hkv.hkv_compress(cfg, *inputs, cache, ws))
            s.keep.append(cache)
            qs.append(_queries(case, g, u, 1)[0])
        s.q, s.out = torch.stack(qs), _out_buffer(case, n)
        s.layers = [(h, s.q[i], s.out[i]) for i, h in enumerate(s.handles)]
        if s.call == "host":
            s.q_host = s.q.cpu().pin_memory()
            s.out_host = torch.empty(s.out.shape, dtype=s.out.dtype, pin_memory=True)
        elif s.call == "graph":
            _steps(s)          # the first step after a compression is not the one to record
            torch.cuda.synchronize()
            s.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s.graph):
                _steps(s)
        return s
    s.cfg, s.steps, s.layers = cfg, case.get("steps", 1), []
    for layer in range(n):
        u = _directions(case, g)
        inputs = _layer_inputs(case, g, rng, u, layer)
        q = _queries(case, g, u, s.steps)
        new = [torch.randn(s.steps, case["batch"], case["kv_heads"], HEAD_DIM, device="cuda", dtype=torch.bfloat16, generator=g)
               for _ in range(2)]
        s.layers.append((inputs, _buffers(cfg, inputs), q, new, _out_buffer(case, s.steps)))
    s.out = [layer[4] for layer in s.layers]
    if s.kind == "prefill":
        # where the compression leaves the window scores of the static heads (they are among its results)
        inputs, (cache, ws) = s.layers[0][:2]
        h = hkv.hkv_compress(cfg, *inputs, cache, ws)
        s.handles.append(h)
        s.scores = []
        for b, c in enumerate(inputs[5]):
            for head, kind in enumerate(inputs[6][b]):
                if kind == 0:
                    off = hkv.hkv_window_scores_offset(h, b, head)
                    s.scores.append(ws[off:off + 4 * c].view(torch.float32))
        torch.cuda.synchronize()
        s.close()
    return s


def _prepare_classify(case, g, s):
    B, H, G, C, T = case["batch"], case["kv_heads"], case["q_heads"] // case["kv_heads"], case["tokens"], case["text"]
    s.cfg, s.lens = _config(case), np.array(_seq_lens(case), np.int32)
    s.n_text = np.array([max(1, T - (3 * b if case["ragged"] else 0)) for b in range(B)], np.int32)
    s.k = _keys_values(case, g, random.Random(0), _directions(case, g))[0]
    # heads from diffuse to sharply focused: noise plus a share of one of four keys of the head
    anchors = torch.randint(int(min(s.lens)), (B, H, 4), device="cuda", generator=g)
    pick = torch.randint(4, (B, H, T * G), device="cuda", generator=g)
    rows = anchors.gather(2, pick)[..., None].expand(-1, -1, -1, HEAD_DIM)
    focus = (torch.arange(B * H, device="cuda") % 4).view(B, H, 1, 1) / 3.0
    x = torch.randn(B, H, T * G, HEAD_DIM, device="cuda", generator=g) + 1.5 * focus * s.k.gather(2, rows).float()
    s.q_text = x.view(B, H, T, G, HEAD_DIM).permute(0, 2, 1, 3, 4).reshape(B, T, H * G, HEAD_DIM).bfloat16().contiguous()
    s.ws = torch.empty(hkv.hkv_classify_workspace(s.cfg, T)[1], dtype=torch.uint8, device="cuda")
    s.scores = torch.empty(B, H, dtype=torch.float64, device="cuda")
    s.types = torch.empty(B, H, dtype=torch.uint8, device="cuda")
    return s


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def _steps(s):
    for handle, q, out in s.layers:
        hkv.hkv_decode_attn(handle, q, out)


def run(s):
    if s.kind == "classify":
        hkv.hkv_classify_heads(s.cfg, s.k, s.q_text, s.lens, s.n_text, TOPK_FRACTION, THETA, s.ws, s.scores, s.types)
        return {"scores": s.scores, "types": s.types}
    if s.kind == "decode":
        if s.call == "graph":
            s.graph.replay()
        elif s.call == "host":
            hkv.hkv_decode_step_host(s.handles, s.q_host, s.out_host, s.q, s.out)
            torch.cuda.current_stream().synchronize()     # the program reads the outputs on the host
            return s.out_host
        else:
            _steps(s)
        return s.out
    handles = [hkv.hkv_compress(s.cfg, *inputs, *buffers) for inputs, buffers, _, _, _ in s.layers]
    for t in range(s.steps):
        for h, (_, _, q, new, out) in zip(handles, s.layers):
            if s.kind == "generate":
                hkv.hkv_append(h, new[0][t], new[1][t])
            hkv.hkv_decode_attn(h, q[t], out[t])
    for h in handles:
        hkv.hkv_cache_destroy(h)
    return {"out": s.out, "window_scores": s.scores} if s.kind == "prefill" else s.out


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _totals(case):
    """Over all layers: tokens of static heads, of dynamic heads, tokens they keep / attend, chunk means."""
    lens, kept, cs = _seq_lens(case), _budget_tokens(case), case["chunk"]
    sta = dyn = sta_kept = dyn_kept = means = 0
    for layer in range(case.get("layers", 1)):
        for c, t, heads in zip(lens, kept, _head_types(case, layer)):
            d = sum(heads)
            sta, dyn = sta + c * (len(heads) - d), dyn + c * d
            sta_kept, dyn_kept = sta_kept + min(c, t) * (len(heads) - d), dyn_kept + min(c, -(-t // cs) * cs) * d
            means += -(-c // cs) * d
    return sta, dyn, sta_kept, dyn_kept, means


def work(case):
    row, B, Hq, G, d = 2 * HEAD_DIM, case["batch"], case["q_heads"], case["q_heads"] // case["kv_heads"], HEAD_DIM
    if case["kind"] == "classify":
        rows = [max(1, case["text"] - (3 * b if case["ragged"] else 0)) * Hq for b in range(B)]
        return {"bytes": sum(_seq_lens(case)) * case["kv_heads"] * row + sum(rows) * row + 9.0 * B * case["kv_heads"],
                "flops": 2.0 * d * sum(r * c for r, c in zip(rows, _seq_lens(case)))}
    sta, dyn, sta_kept, dyn_kept, means = _totals(case)
    n, steps = case.get("layers", 1), case.get("steps", 1)
    out = 4 if case["out"] == "f32" else 2
    step_bytes = 2 * row * (sta_kept + dyn_kept) + row * means + n * B * Hq * d * (2 + out)
    step_flops = 4.0 * d * G * (sta_kept + dyn_kept) + 2.0 * d * G * means
    if case["kind"] == "decode":
        return {"bytes": step_bytes, "flops": step_flops}
    # prefill: the static heads' keys once, their kept values; all of the dynamic heads' K/V; the cache written
    fill_bytes = (row * sta + row * sta_kept + 2 * row * dyn + 2 * row * (sta_kept + dyn) + row * means + 4 * sta +
                  n * (WINDOW * B * Hq * row + sum(_seq_lens(case))))
    fill_flops = 2.0 * d * WINDOW * G * sta
    return {"bytes": fill_bytes + steps * step_bytes, "flops": fill_flops + steps * step_flops}


def tolerance(case):
    # attention: bf16 inputs, probabilities in bf16 for the product with V, bf16 or float32 output
    # labels: float32 softmax arithmetic summed over tens of thousands of entries; heads may not change their label
    return {"rel": 2e-5} if case["kind"] == "classify" else {"rel": 1e-2}
