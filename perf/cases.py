"""What a user of the library has it do, as timed cases: whole calls through the C ABI's Python binding.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)` one more of the same ranges; `prepare`
makes what a serving program holds before the call (pools, activations, weights, plans), `run` is one pass.  Kinds:

  step     one attention step of one layer over a ragged batch, the chunk's K/V appended in the same call
  prompt   one request's prompt processed chunk by chunk, then (optionally) one draft-verification call
  rope     append with the rotation fused, rotation of q, attention with 16-bit output: three calls of one layer
  layer    the QKV projection with rotation and append in its epilogue, then attention with 16-bit output
  host     one step whose activations and results live in pinned host memory
  serve    one inference step of a pipeline stage: plan the batch, run `layers` layers with it, free the plan

Request lengths come from the case's own `shape` number, values and page placement from the seed.
"""
from __future__ import annotations

import random

import numpy as np
import torch

from paper_2503_18989_b200 import binding as B
from paper_2503_18989_b200.workloads import PAGE_SIZE, random_tree_masks

DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16}


def _case(kind, dtype="fp16", heads=32, group=1, dim=128, layout="paged", prefill=0, chunk_lo=0, chunk_hi=0,
          chunk_any=False, pre_lo=0, pre_hi=0, pre_step=1, verify=0, draft_lo=1, draft_hi=8, ver_lo=0, ver_hi=0, tree=False,
          out16=False, prompt=0, chunk=0, draft=0, layers=1, hidden=0, shape=1, name=None):
    c = dict(kind=kind, dtype=dtype, heads=heads, group=group, dim=dim, layout=layout, prefill=prefill, chunk_lo=chunk_lo,
             chunk_hi=chunk_hi, chunk_any=chunk_any, pre_lo=pre_lo, pre_hi=pre_hi, pre_step=pre_step, verify=verify,
             draft_lo=draft_lo, draft_hi=draft_hi, ver_lo=ver_lo, ver_hi=ver_hi, tree=tree, out16=out16, prompt=prompt,
             chunk=chunk, draft=draft, layers=layers, hidden=hidden, shape=shape)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a single device in its decode phase: four draft tokens against one 700-token cache, the smallest call there is
        _case("step", name="verify_one_device", verify=1, draft_lo=4, draft_hi=4, ver_lo=700, ver_hi=700),
        # the five dependent calls of a short prompt on a small model with a contiguous cache (workload `tiny`)
        _case("prompt", name="tiny_prompt", heads=8, dim=64, layout="contiguous", prompt=256, chunk=64, draft=4),
        # one device's 2048-token prompt in chunks of 256 on a 7B-shaped layer (workload `llama7b_chunked`)
        _case("prompt", name="prompt_2048_by_256", prompt=2048, chunk=256),
        # prompt chunks of 30 devices at once (workload `ragged_prefill`)
        _case("step", name="ragged_prefill_fp16", prefill=30, chunk_lo=64, chunk_hi=512, pre_hi=4096, pre_step=16, shape=3),
        # draft verification for 30 devices at once, the common decode-phase step (workload `spec_verify`)
        _case("step", name="spec_verify_fp16", verify=30, ver_lo=512, ver_hi=4096, shape=4),
        # 13B-shaped batch of prompt chunks and drafts together (workload `mixed_13b`, the benchmark's default)
        _case("step", name="mixed_13b_bf16", dtype="bf16", heads=40, prefill=8, chunk_lo=512, chunk_hi=512, pre_hi=8192,
              verify=32, draft_lo=4, draft_hi=4, ver_lo=1024, ver_hi=8192, shape=5),
        # grouped query heads and token trees (what the benchmark's --q-group 4 --tree asks for), long contexts
        _case("step", name="verify_tree_gqa_bf16", dtype="bf16", heads=8, group=4, verify=16, draft_lo=4, draft_hi=8,
              ver_lo=1024, ver_hi=8192, tree=True, out16=True, shape=6),
        # chunk sizes as the chunk-size controller picks them (any integer), odd prefixes, K and q rotated by the library
        _case("rope", name="odd_chunks_rope_bf16", dtype="bf16", heads=40, prefill=6, chunk_lo=17, chunk_hi=600, chunk_any=True,
              pre_hi=3000, verify=3, ver_lo=300, ver_hi=3000, out16=True, shape=7),
        # one decoder layer up to the output projection, decode phase: 32 devices x 4 drafts, 13B shape (the weights dominate)
        _case("layer", name="layer_verify_13b_bf16", dtype="bf16", heads=40, hidden=5120, verify=32, draft_lo=4, draft_hi=4,
              ver_lo=512, ver_hi=2048, out16=True, shape=8),
        # the same for prompt chunks of a 7B-shaped layer: the projection is a large dense contraction
        _case("layer", name="layer_prefill_7b_fp16", hidden=4096, prefill=12, chunk_lo=128, chunk_hi=512, pre_hi=2048,
              out16=True, shape=9),
        # activations in pinned host memory, copies in the call (the benchmark's end-to-end arm), small mixed batch
        _case("host", name="host_mixed_fp16", prefill=4, chunk_lo=64, chunk_hi=256, pre_hi=1024, verify=12, ver_lo=256,
              ver_hi=2048, shape=10),
        # one decode-phase inference step of a pipeline stage of 8 layers: a new plan each step, used by every layer
        _case("serve", name="serve_verify_8_layers", layers=8, verify=12, ver_lo=512, ver_hi=2048, shape=11),
    ]


# ------------------------------------------------------------------ shapes
def _log_int(rng, lo, hi):
    """A whole number of [lo, hi], spread evenly over the logarithm."""
    lo1 = max(1, lo)
    return max(lo, min(hi, int(round(lo1 * (hi / lo1) ** rng.random()))))


def _calls(case):
    """Per call of the pass: (prefix lengths, chunk lengths)."""
    if case["kind"] == "prompt":
        out = [([p], [min(case["chunk"], case["prompt"] - p)]) for p in range(0, case["prompt"], case["chunk"])]
        if case["draft"]:
            out.append(([case["prompt"]], [case["draft"]]))
        return out
    rng = random.Random(case["shape"])
    reqs = []
    pow2 = [c for c in (32, 64, 128, 256, 512) if case["chunk_lo"] <= c <= case["chunk_hi"]]
    for _ in range(case["prefill"]):
        step = case["pre_step"]
        p = rng.randint((case["pre_lo"] + step - 1) // step, case["pre_hi"] // step) * step
        c = rng.randint(case["chunk_lo"], case["chunk_hi"]) if case["chunk_any"] else rng.choice(pow2)
        reqs.append((p, c))
    for _ in range(case["verify"]):
        reqs.append((rng.randint(case["ver_lo"], case["ver_hi"]), rng.randint(case["draft_lo"], case["draft_hi"])))
    rng.shuffle(reqs)                       # devices arrive in no particular order
    return [([p for p, _ in reqs], [c for _, c in reqs])]


def draw(rng):
    most = [work(c) for c in listed()]
    top_b, top_f = max(w["bytes"] for w in most), max(w["flops"] for w in most)
    while True:
        c = _draw(rng)
        w = work(c)
        if w["bytes"] <= top_b and w["flops"] <= top_f:
            return c


def _draw(rng):
    kind = rng.choice(["step", "step", "step", "prompt", "rope", "layer", "host", "serve"])
    dtype = rng.choice(["fp16", "bf16"])
    heads, group, dim = rng.choice([(32, 1, 128), (32, 1, 128), (40, 1, 128), (40, 1, 128), (8, 4, 128), (8, 1, 64), (32, 1, 64)])
    layout = rng.choice(["paged", "paged", "paged", "contiguous"])
    shape = rng.randrange(1 << 20)
    base = dict(dtype=dtype, heads=heads, group=group, dim=dim, layout=layout, shape=shape)
    if kind == "prompt":
        chunk = _log_int(rng, 32, 512)
        return _case(kind, prompt=_log_int(rng, chunk, min(3000, 8 * chunk)), chunk=chunk, draft=rng.choice([0, rng.randint(1, 8)]), **base)
    pre = dict(chunk_lo=rng.choice([17, 64, 128]), chunk_hi=_log_int(rng, 128, 600), chunk_any=rng.random() < 0.6,
               pre_hi=_log_int(rng, 256, 8192), pre_step=rng.choice([1, 16]))
    lo = _log_int(rng, 64, 1024)
    ver = dict(draft_hi=rng.randint(1, 8), ver_lo=lo, ver_hi=_log_int(rng, lo, 8192), tree=rng.random() < 0.25)
    mix = rng.choice(["prefill", "verify", "both"])
    if kind == "serve":
        return _case(kind, layers=rng.randint(2, 8), verify=_log_int(rng, 1, 16), **dict(ver, ver_hi=min(ver["ver_hi"], 2048)), **base)
    n_pre = _log_int(rng, 1, 12 if kind == "host" else 30) if mix != "verify" else 0
    n_ver = _log_int(rng, 1, 32) if mix != "prefill" else 0
    more = {}
    if kind == "layer":
        more = dict(hidden=heads * group * dim, out16=True)
    elif kind == "rope":
        more = dict(out16=True)
    elif kind == "step":
        more = dict(out16=rng.random() < 0.4)
    return _case(kind, prefill=n_pre, verify=n_ver, **pre, **ver, **more, **base)


# ------------------------------------------------------------------ what a serving program holds
def _randn(shape, dtype, gen, scale=1.0):
    x = torch.randn(shape, dtype=DTYPES[dtype], device="cuda", generator=gen)
    return x if scale == 1.0 else x.mul_(scale)


class _Call:
    """One batch: its descriptor arrays, activations and result buffers, and (unless planned in the pass) its plan."""


def _strides(case):
    d, h = case["dim"], case["heads"]
    if case["layout"] == "paged":           # [page][head][slot][d]
        return PAGE_SIZE * h * d, d, PAGE_SIZE * d
    return PAGE_SIZE * h * d, h * d, d      # [token][head][d]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    host_rng = np.random.Generator(np.random.PCG64(int(seed)))
    kind, dtype, h, d = case["kind"], case["dtype"], case["heads"], case["dim"]
    hq = h * case["group"]
    calls = _calls(case)

    # pages: every request owns distinct ones, anywhere in the pool (in order for a contiguous cache); the last call of a
    # prompt is the longest
    need = [(p + c + PAGE_SIZE - 1) // PAGE_SIZE for p, c in zip(*calls[-1])]
    num_pages = sum(need) + (0 if kind == "prompt" else max(8, len(need)))
    order = np.arange(num_pages) if case["layout"] == "contiguous" else host_rng.permutation(num_pages)
    table = np.full((len(need), max(need)), -1, dtype=np.int32)
    at = 0
    for r, n in enumerate(need):
        table[r, :n] = order[at:at + n]
        at += n

    sp, st, sh = _strides(case)
    s = {"case": case, "stream": torch.cuda.current_stream().cuda_stream, "table": table}
    s["pools"] = [tuple(_randn((num_pages * sp,), dtype, gen) for _ in range(2)) for _ in range(case["layers"])]
    s["caches"] = [B.make_cache_desc(dtype, num_pages, h, d, sp, st, sh, k, v, PAGE_SIZE) for k, v in s["pools"]]
    if kind == "layer":
        s["w"] = _randn(((hq + 2 * h) * d, case["hidden"]), dtype, gen, case["hidden"] ** -0.5)

    s["calls"] = []
    for prefix, chunk in calls:
        c = _Call()
        c.prefix, c.chunk = np.asarray(prefix, dtype=np.int32), np.asarray(chunk, dtype=np.int32)
        c.cu = np.concatenate([[0], np.cumsum(c.chunk)]).astype(np.int32)
        c.tree = random_tree_masks(case["shape"], chunk) if case["tree"] else None
        t = int(c.cu[-1])
        if kind == "layer":
            c.x = _randn((t, case["hidden"]), dtype, gen)
            c.q = torch.empty((t, hq, d), dtype=DTYPES[dtype], device="cuda")
        else:
            c.q = _randn((t, hq, d), dtype, gen)
            c.k = [_randn((t, h, d), dtype, gen) for _ in range(case["layers"])]
            c.v = [_randn((t, h, d), dtype, gen) for _ in range(case["layers"])]
        if kind == "rope":
            c.q_rot = torch.empty_like(c.q)
        out_type = DTYPES[dtype] if case["out16"] else torch.float32
        c.out = [torch.zeros((t, hq, d), dtype=out_type, device="cuda") for _ in range(case["layers"])]
        c.lse = [torch.zeros((t, hq), dtype=torch.float32, device="cuda") for _ in range(case["layers"])]
        c.plan = c.ws = None
        c.ws_bytes = 0
        if kind != "serve":
            c.plan = _plan(s, c)
            c.ws_bytes = B.hat_plan_workspace_bytes(c.plan)
            c.ws = torch.empty((max(c.ws_bytes, 256),), dtype=torch.uint8, device="cuda")
        if kind == "host":
            c.q, c.k[0], c.v[0], c.out[0], c.lse[0] = (x.cpu().pin_memory() for x in (c.q, c.k[0], c.v[0], c.out[0], c.lse[0]))
            c.staging_bytes = B.hat_plan_staging_bytes(c.plan)
            c.staging = torch.empty((max(c.staging_bytes, 256),), dtype=torch.uint8, device="cuda")
        s["calls"].append(c)
    return s


def _plan(s, c):
    return B.hat_plan_create(s["caches"][0], s["case"]["heads"] * s["case"]["group"], c.cu, c.prefix, c.chunk, s["table"], tree_mask=c.tree)


# ------------------------------------------------------------------ one pass
def _attend(s, c, layer, plan, q, new_kv):
    call = B.hat_chunk_attention_out16 if s["case"]["out16"] else B.hat_chunk_attention
    call(s["caches"][layer], plan, q, c.k[layer] if new_kv else None, c.v[layer] if new_kv else None, c.out[layer], c.lse[layer],
         0.0, c.ws, c.ws_bytes, s["stream"])


def run(s):
    case, stream = s["case"], s["stream"]
    kind = case["kind"]
    c = s["calls"][0]
    if kind in ("step", "prompt"):
        for c in s["calls"]:
            _attend(s, c, 0, c.plan, c.q, True)
    elif kind == "rope":
        B.hat_kv_append_rope(s["caches"][0], c.plan, c.k[0], c.v[0], 10000.0, False, stream)
        B.hat_rope_q(c.plan, c.q, c.q_rot, 10000.0, False, stream)
        _attend(s, c, 0, c.plan, c.q_rot, False)
    elif kind == "layer":
        B.hat_qkv_rope_append(s["caches"][0], c.plan, c.x, case["hidden"], s["w"], c.q, 10000.0, False, stream)
        _attend(s, c, 0, c.plan, c.q, False)
    elif kind == "host":
        B.hat_chunk_attention_host(s["caches"][0], c.plan, c.q, c.k[0], c.v[0], c.out[0], c.lse[0], 0.0, c.staging, c.staging_bytes,
                                   c.ws, c.ws_bytes, stream)
    else:                                   # serve
        plan = _plan(s, c)
        need = B.hat_plan_workspace_bytes(plan)
        if c.ws is None or need > c.ws_bytes:
            c.ws_bytes = max(need, 256)
            c.ws = torch.empty((c.ws_bytes,), dtype=torch.uint8, device="cuda")
        for layer in range(case["layers"]):
            _attend(s, c, layer, plan, c.q, True)
        plan.close()
    got = {"out": [x for c in s["calls"] for x in c.out], "lse": [x for c in s["calls"] for x in c.lse]}
    # appended rows are copies, bit for bit, unless the library computed them (rotation, projection)
    computed = kind in ("rope", "layer")
    got["pools"] = [p if computed else p.view(torch.int16) for kv in s["pools"] for p in kv]
    if kind == "rope":
        got["q"] = c.q_rot
    elif kind == "layer":
        got["q"] = c.q
    return got


# ------------------------------------------------------------------ what one pass cannot do without
def work(case):
    h, d, hq = case["heads"], case["dim"], case["heads"] * case["group"]
    out_size = 2 if case["out16"] else 4
    byts = flops = 0
    for prefix, chunk in _calls(case):
        t = sum(chunk)
        cached = sum(p for p, c in zip(prefix, chunk) if c)
        pairs = sum(c * p + c * (c + 1) // 2 for p, c in zip(prefix, chunk))
        flops += 4 * d * hq * pairs
        byts += 2 * cached * h * d * 2 + t * hq * d * (2 + out_size) + t * hq * 4     # cached K/V, q, out, lse
        byts += 2 * t * h * d * 2                                                     # the chunk's K/V into the pools
        if case["kind"] == "layer":
            f = (hq + 2 * h) * d
            flops += 2 * t * case["hidden"] * f
            byts += t * case["hidden"] * 2 + f * case["hidden"] * 2                   # x, weights
        else:
            byts += 2 * t * h * d * 2                                                 # k_new, v_new
        if case["kind"] == "rope":
            byts += t * hq * d * 2                                                    # the rotated q
    return {"bytes": case["layers"] * byts, "flops": case["layers"] * flops}


def tolerance(case):
    # fp32 results carry the softmax weights' rounding to fp16 (2^-12 on average; bf16 weights keep a second term and
    # stay below that); 16-bit results add their own last bit, 2^-9 for bf16
    if case["dtype"] == "bf16" and (case["out16"] or case["kind"] in ("rope", "layer")):
        return {"rel": 1e-2}
    return {"rel": 1e-3}
