"""Workloads of the D2O path that performance work is measured on: what a serving program has the library do for a
prompt and for generated tokens, through the public binding, from one short prompt to batches that fill the GPU.

A case names one use of the library (`kind`) and its sizes:

  stats     d2o_layer_stats(_layers): column sums and densities of the prompt attention, with or without the row
            normalisers of the caller's own attention kernel (`lse`)
  prompt    the whole prompt stage of one batch: column sums, budgets, compression (`ragged`: every sequence has its
            own prompt length); the layers share the cache equally
  compress  d2o_prefill_compress_layers with column sums and densities already in the context
  decode    generated tokens; `mode` says how the program calls: "layer" (a model that runs layer by layer), "step"
            (one call per token), "chain" (tokens whose inputs are known, one call), "host" (the same from pinned host
            memory)
  full      d2o_full_decode_step: attention of one token over uncompressed caches

Shapes are the 7B-like (32 query heads, 32 KV heads, d = 128, fp16), the 8B-like (32 / 8, d = 128, bf16) and the small
fp32 stacks of `workloads.CONFIGS`; inputs come from the generators of `workloads`.

Cache rows of 16-bit types are returned as the bit patterns of their elements, next to their positions: where two
candidates for eviction tie to rounding, or a merged element lies between two representable values, a correct
implementation may take either; the share of elements that differ tells that from an error, a norm does not.
"""
from __future__ import annotations

import math

import torch

from paper_2406_13035_b200 import binding as B
from paper_2406_13035_b200 import workloads as W

DEV = "cuda:0"
TORCH_DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BITS = {"f32": torch.float32, "f16": torch.int16, "bf16": torch.int16}
MANY = 1 << 24                      # generated tokens a context accepts: passes go on where the last one stopped


def _case(kind, shape, layers, batch, prompt, **more):
    q, kv, d, dtype = shape
    return dict(kind=kind, dtype=dtype, layers=layers, batch=batch, q_heads=q, kv_heads=kv, d_head=d, prompt=prompt,
                **more)


SMALL = (8, 8, 64, "f32")
MHA = (32, 32, 128, "f16")
GQA = (32, 8, 128, "bf16")


def listed():
    return [
        # one layer of a small fp32 model: the shortest call of the prompt stage
        dict(_case("stats", SMALL, 1, 1, 1024, lse=False), name="stats fp32 small"),
        # a 4096-token prompt whose attention kernel hands over its row normalisers
        dict(_case("stats", MHA, 8, 1, 4096, lse=True), name="stats 7b lse"),
        # a prompt as long as its user made it: no multiple of anything
        dict(_case("stats", GQA, 2, 1, 6001, lse=False), name="stats 8b odd"),
        # a long document
        dict(_case("stats", GQA, 2, 1, 32768, lse=False), name="stats 8b long"),
        # time to first token of one chat prompt, every layer
        dict(_case("prompt", MHA, 32, 1, 1200, rho=0.2, ragged=False), name="prompt 7b chat"),
        # a serving batch of prompts of different lengths
        dict(_case("prompt", GQA, 8, 8, 4096, rho=0.1, ragged=True), name="prompt 8b ragged"),
        # eviction and merging of a large batch, four layers at a time
        dict(_case("compress", GQA, 4, 16, 8192, rho=0.1, window=64), name="compress 8b batch"),
        # interactive generation: one sequence, the model calls once per layer
        dict(_case("decode", GQA, 32, 1, 4096, rho=0.4, window=0, mode="layer", tokens=4), name="decode 8b by layer"),
        # one sequence, one call per token over all layers
        dict(_case("decode", MHA, 32, 1, 2048, rho=0.4, window=0, mode="step", tokens=8), name="decode 7b by token"),
        # throughput: sixteen sequences, known inputs
        dict(_case("decode", GQA, 32, 16, 2048, rho=0.4, window=64, mode="chain", tokens=16), name="decode 8b batch"),
        # four multi-turn sessions, inputs and outputs in pinned host memory
        dict(_case("decode", MHA, 32, 4, 2048, rho=0.5, window=1000, mode="host", tokens=16), name="decode 7b host"),
        # the uncompressed baseline of the same model, eight sequences
        dict(_case("full", MHA, 4, 8, 2048), name="full cache 7b"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _prompt_length(rng, lo, hi, heads, d):
    """Half of the programs pad their prompts to 64 tokens, half do not; attention work (two sweeps over the logits of
    `heads` heads) stays within that of the longest listed case of either sort."""
    padded = rng.random() < 0.5
    most = math.sqrt((1.75e13 if padded else 6e11) / (2.0 * heads * d))
    p = max(100, min(_log(rng, lo, hi), int(most)))
    return -(-p // 64) * 64 if padded else p


def draw(rng):
    kind = rng.choice(["stats", "stats", "prompt", "compress", "decode", "decode", "decode", "full"])
    shape = rng.choice([SMALL, MHA, MHA, GQA, GQA, (32, 4, 128, "bf16"), (16, 8, 64, "f16")])
    q, kv, d, dtype = shape
    small = dtype == "f32"                                  # fp32 stacks stay small: fewer layers, shorter prompts
    if kind == "full":
        return _case(kind, shape, _log(rng, 1, 4), _log(rng, 1, 8), _log(rng, 100, 2047))
    if kind == "stats":
        layers, batch = _log(rng, 1, 8), _log(rng, 1, 4)
        prompt = _prompt_length(rng, 100, 2000 if small else 16000, layers * batch * q, d)
        return _case(kind, shape, layers, batch, prompt, lse=rng.random() < 0.4 and prompt <= 4096)
    if kind == "prompt":
        batch = _log(rng, 1, 8)
        layers = _log(rng, 2, 8) if small or batch > 2 else _log(rng, 8, 32)
        prompt = _prompt_length(rng, 200, 1000 if small else 4096, layers * batch * q, d)
        return _case(kind, shape, layers, batch, prompt, rho=round(rng.uniform(0.1, 0.4), 3),
                     ragged=batch > 1 and rng.random() < 0.5)
    if kind == "compress":
        layers, batch = _log(rng, 1, 4), _log(rng, 1, 8)
        prompt = _log(rng, 300, 1000 if small else 8192)
        return _case(kind, shape, layers, batch, prompt, rho=round(rng.uniform(0.1, 0.3), 3),
                     window=rng.choice([0, 32]))
    mode = rng.choice(["layer", "layer", "step", "step", "chain", "host"])
    layers = _log(rng, 1, 8) if small else _log(rng, 8, 32)
    batch = 1 if mode == "layer" and rng.random() < 0.5 else _log(rng, 1, 12)
    prompt = _log(rng, 300, 1000 if small else 2048)
    return _case(kind, shape, layers, batch, prompt, rho=round(rng.uniform(0.2, 0.5), 3), window=rng.choice([0, 32]),
                 mode=mode, tokens=4 if mode == "layer" else 8)


# ------------------------------------------------------------------------------------------------ inputs
def _workload(c, seed):
    return W.Workload("case", batch=c["batch"], n_layers=c["layers"], n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"],
                      d_head=c["d_head"], dtype=c["dtype"], prompt_len=c["prompt"], decode_steps=0, rho=c.get("rho", 1.0),
                      temp_first=1.0, temp_last=0.25, seed=seed % (1 << 31))


def _mean_budget(c):
    return max(16, int(c["rho"] * c["prompt"]))


def _context(c, equal):
    """`equal`: every layer gets the same share of the cache; else Eq. 5 with the densities of the context."""
    S, P = _mean_budget(c), c["prompt"]
    lo, hi = (8, 0) if equal else (max(8, S // 3), min(P, 4 * S))
    window = c.get("window", 0)
    cfg = B.make_config(n_layers=c["layers"], batch=c["batch"], n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"],
                        d_head=c["d_head"], dtype=c["dtype"], prompt_len=P,
                        max_new_tokens=MANY if c["kind"] == "decode" else 0,
                        rho=max(c["rho"], 16.5 / P), n_sink=1, window=window, beta=0.7,
                        density_temp=1e30 if equal else 1.0, min_budget=lo, max_budget=hi)
    ctx = B.D2OContext(cfg, DEV)
    for t in _state(ctx, c).values():
        t.zero_()                                           # rows that no slice fills, and the padding of ragged prompts
    ctx.colsum(0).zero_()
    for layer in range(1, c["layers"]):
        ctx.colsum(layer).zero_()
    return ctx


def _state(ctx, c):
    """The cache as the library keeps it (device views): rows (16-bit types as bit patterns), positions, scores, lengths, thresholds."""
    v = B.D2OView()
    assert ctx.lib.d2o_get_view(ctx.handle, 0, v) == 0
    n, d, sl = v.pool_rows, c["d_head"], c["layers"] * c["batch"] * c["kv_heads"]

    def at(ptr, count, dtype, shape):
        off = ptr - ctx.state.data_ptr()
        size = torch.empty(0, dtype=dtype).element_size()
        return ctx.state[off:off + count * size].view(dtype).view(shape)

    return {"k": at(v.k_cache, n * d, BITS[c["dtype"]], (n, d)), "v": at(v.v_cache, n * d, BITS[c["dtype"]], (n, d)),
            "pos": at(v.pos, n, torch.int32, (n,)), "score": at(v.score, n, torch.float32, (n,)),
            "len": at(v.len, sl, torch.int32, (sl,)), "tau": at(v.tau, sl, torch.float32, (sl,))}


def _blocks(q, k, rows):
    """Softmax rows `rows` of the causal attention of a batch of heads q, k [n, P, d], as fp32 logits [n, rows, P]."""
    P, d = k.shape[-2], k.shape[-1]
    x = torch.matmul(q[:, rows].float() / math.sqrt(d), k.float().transpose(1, 2))
    later = torch.arange(P, device=k.device)[None, :] > rows[:, None]
    return x.masked_fill_(later, float("-inf"))


def _row_lse(q, k):
    """Natural-log row normalisers [B, Hq, P] of the causal attention, as an attention kernel returns them."""
    b, hq, P, _ = q.shape
    g = hq // k.shape[1]
    out = torch.empty(b, hq, P, device=q.device)
    step = max(1, (1 << 28) // (P * g))
    for i in range(b):
        for h in range(k.shape[1]):
            for r in range(0, P, step):
                rows = torch.arange(r, min(P, r + step), device=q.device)
                x = _blocks(q[i, h * g:(h + 1) * g], k[i, h:h + 1].expand(g, -1, -1), rows)
                out[i, h * g:(h + 1) * g, r:r + step] = torch.logsumexp(x, -1)
    return out


def _sampled_colsum(q, k, stride=16):
    """Column sums [B, Hq, P] of the causal attention estimated from every stride-th query."""
    b, hq, P, _ = q.shape
    g = hq // k.shape[1]
    rows = torch.arange(stride - 1, P, stride, device=q.device)
    rows = torch.cat([rows, torch.tensor([P - 1], device=q.device)])
    out = torch.empty(b, hq, P, device=q.device)
    for i in range(b):
        x = _blocks(q[i], k[i].repeat_interleave(g, 0), rows)
        out[i] = torch.softmax(x, -1).sum(1) * (P / rows.numel())
    return out


def _densities(c, seed):
    """A density profile over the layers and sequences: weights exp(-F) that differ by factors, more in depth than
    between sequences."""
    g = torch.Generator().manual_seed(seed % (1 << 31))
    depth = 0.5 * torch.randn(1, c["layers"], 1, generator=g, dtype=torch.float64)
    own = 0.15 * torch.randn(c["batch"], c["layers"], c["q_heads"], generator=g, dtype=torch.float64)
    return 5.0 + depth + own


def _tokens(c, wl, streams, count):
    """q, k, v of `count` generated tokens: [count, L, B, H, d], continuing the prompts."""
    qs, ks, vs = [], [], []
    for layer, s in enumerate(streams):
        g = torch.Generator(device=DEV).manual_seed(wl.seed + 977 * (layer + 1))
        k = s._keys(count, g)
        v = torch.randn(k.shape, generator=g, device=DEV)
        xi = torch.randn(c["batch"], c["q_heads"], count, c["d_head"], generator=g, device=DEV)
        eta, _ = W._ar1(xi, s.eta)
        q = (s.m_q[:, :, None, :] + eta) / s.temp
        for out, t in ((qs, q), (ks, k), (vs, v)):
            out.append(t.to(TORCH_DTYPE[c["dtype"]]).permute(2, 0, 1, 3))
    return [torch.stack(x, 1).contiguous() for x in (qs, ks, vs)]


def prepare(case, seed):
    c = dict(case)
    wl = _workload(c, seed)
    if c["kind"] == "full":
        return _prepare_full(c, seed)
    L, kind = c["layers"], c["kind"]
    streams = [W.LayerStream(wl, layer, DEV) for layer in range(L)]
    st = {"case": c}
    if kind == "stats":
        st["ctx"] = ctx = _context(dict(c, rho=0.5), True)
        st["q"], st["k"] = zip(*[s.prompt()[:2] for s in streams])
        st["lse"] = [_row_lse(q, k) for q, k in zip(st["q"], st["k"])] if c["lse"] else None
        st["colsum"] = [ctx.colsum(layer) for layer in range(L)]
        st["density"] = ctx.density()
        return st
    equal = kind == "prompt"
    st["ctx"] = ctx = _context(c, equal)
    st["state"] = _state(ctx, c)
    if equal:
        if c["ragged"]:
            g = torch.Generator().manual_seed(seed % (1 << 31))
            lens = (c["prompt"] * (0.3 + 0.7 * torch.rand(c["batch"], generator=g))).int().clamp(min=100)
            lens[0] = c["prompt"]
            ctx.d2o_set_prompt_lens(lens)
        st["q"], st["k"], st["v"] = zip(*[s.prompt() for s in streams])
        st["colsum"] = [ctx.colsum(layer) for layer in range(L)]
        st["density"] = ctx.density()
        return st
    keys, values = [], []
    for layer, s in enumerate(streams):
        q, k, v = s.prompt()
        ctx.d2o_layer_stats(layer, q[:, :, :], k)
        ctx.colsum(layer).copy_(_sampled_colsum(q, k))      # the same scores whatever the library's rounding
        keys.append(k)
        values.append(v)
        del q
    ctx.density().copy_(_densities(c, seed))                # a measured profile of the model fixes the budgets
    ctx.d2o_layer_budgets()
    if kind == "compress":
        st["k"], st["v"] = keys, values
        return st
    ctx.d2o_prefill_compress_layers(0, L, keys, values)
    del keys, values
    n, count = c["tokens"], 64 if c["mode"] == "host" else 256
    q, k, v = _tokens(c, wl, streams, count)
    st["turn"], st["turns"] = 0, count // n
    st["out"] = torch.zeros(n, *q.shape[1:], dtype=q.dtype, device=DEV)
    if c["mode"] == "host":
        q, k, v, st["out"] = (t.cpu().pin_memory() for t in (q, k, v, st["out"]))
    if c["mode"] == "layer":                                # a model holds one tensor per layer and token
        st["calls"] = [[(layer, q[t, layer:layer + 1], k[t, layer:layer + 1], v[t, layer:layer + 1],
                         st["out"][t % n, layer:layer + 1]) for layer in range(L)] for t in range(count)]
    st["q"], st["k"], st["v"] = q, k, v
    torch.cuda.synchronize()
    return st


def _prepare_full(c, seed):
    g = torch.Generator(device=DEV).manual_seed(seed % (1 << 31))
    L, n, d, group, dt = c["layers"], c["batch"] * c["kv_heads"], c["d_head"], c["q_heads"] // c["kv_heads"], TORCH_DTYPE[c["dtype"]]
    P = c["prompt"]

    def rand(*shape):
        return torch.randn(*shape, generator=g, device=DEV).to(dt)

    return {"case": c, "k_cache": [rand(n, P + 16, d) for _ in range(L)], "v_cache": [rand(n, P + 16, d) for _ in range(L)],
            "q": [rand(n, group, d) for _ in range(L)], "k": [rand(n, d) for _ in range(L)],
            "v": [rand(n, d) for _ in range(L)], "out": [torch.zeros(n, group, d, dtype=dt, device=DEV) for _ in range(L)]}


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    c = state["case"]
    kind, L = c["kind"], c["layers"]
    if kind == "full":
        for l in range(L):
            B.d2o_full_decode_step(state["k_cache"][l], state["v_cache"][l], c["prompt"], state["q"][l], state["k"][l],
                                   state["v"][l], state["out"][l])
        return {"out": state["out"], "k": state["k_cache"], "v": state["v_cache"]}
    ctx = state["ctx"]
    if kind == "stats":
        if L == 1:
            ctx.d2o_layer_stats(0, state["q"][0], state["k"][0], state["lse"][0] if state["lse"] else None)
        else:
            ctx.d2o_layer_stats_layers(0, L, state["q"], state["k"], state["lse"])
        return {"colsum": state["colsum"], "density": state["density"]}
    if kind == "prompt":
        ctx.d2o_layer_stats_layers(0, L, state["q"], state["k"])
        budgets = ctx.d2o_layer_budgets()
        ctx.d2o_prefill_compress_layers(0, L, state["k"], state["v"])
        s = state["state"]
        return {"colsum": state["colsum"], "density": state["density"], "budgets": budgets, "k": s["k"], "v": s["v"],
                "pos": s["pos"], "len": s["len"], "tau": s["tau"]}
    if kind == "compress":
        ctx.d2o_prefill_compress_layers(0, L, state["k"], state["v"])
        return state["state"]
    n, t0, out = c["tokens"], state["turn"] * c["tokens"], state["out"]
    state["turn"] = (state["turn"] + 1) % state["turns"]
    if c["mode"] == "layer":
        for t in range(t0, t0 + n):
            for layer, q, k, v, o in state["calls"][t]:
                ctx.d2o_decode_step(layer, layer + 1, q, k, v, o)
    else:
        q, k, v = (state[x][t0:t0 + n] for x in "qkv")
        if c["mode"] == "step":
            for t in range(n):
                ctx.d2o_decode_step(0, L, q[t], k[t], v[t], out[t])
        elif c["mode"] == "chain":
            ctx.d2o_decode_steps(0, L, n, q, k, v, out)
        else:
            ctx.d2o_decode_steps_host(0, L, n, q, k, v, out)
    s = state["state"]
    return {"out": out, "k": s["k"], "v": s["v"], "pos": s["pos"], "score": s["score"], "len": s["len"], "tau": s["tau"]}


# ------------------------------------------------------------------------------------------------ what it takes
def work(case):
    """Prompt attention: its logits twice (the row normalisers come before the column sums), once with `lse`; queries
    and keys read once.  Compression: prompt keys and values read, the caches written, similarities evicted x retained.
    Decode: every cache row and its score, position and norm once per token."""
    c = case
    e = 4 if c["dtype"] == "f32" else 2
    L, b, hq, hkv, d, P = c["layers"], c["batch"], c["q_heads"], c["kv_heads"], c["d_head"], c["prompt"]
    if c["kind"] == "full":
        n = b * hkv
        return {"bytes": float(L * (2 * n * (P + 1) * d * e + 2 * n * d * e + 2 * b * hq * d * e)),
                "flops": float(L * 4 * b * hq * (P + 1) * d)}
    size = 1.0
    if c.get("ragged"):
        size = 0.65                                          # mean prompt over the longest one
    out = {"bytes": 0.0, "flops": 0.0}
    if c["kind"] in ("stats", "prompt"):
        sweeps = 1 if c.get("lse") else 2
        square = 0.46 if c.get("ragged") else 1.0           # the same for squares
        out["bytes"] += L * b * ((hq + hkv) * P * d * e + hq * P * 4) * size + (L * b * hq * P * 4 if c.get("lse") else 0)
        out["flops"] += float(sweeps * L * b * hq * P) * P * d * square
    if c["kind"] in ("prompt", "compress"):
        S, Pm = c["rho"] * P * size, P * size
        out["bytes"] += L * b * hkv * (2 * Pm * d * e + 2 * S * d * e + 12 * S) + L * b * hq * Pm * 4
        out["flops"] += L * b * hkv * 2.0 * (Pm - S) * S * d
    if c["kind"] == "decode":
        rows, n = L * b * hkv * c["rho"] * P, c["tokens"]
        out["bytes"] += n * (rows * (2 * d * e + 16) + L * b * (2 * hq + 2 * hkv) * d * e)
        out["flops"] += n * 4.0 * L * b * hq * c["rho"] * P * d
    return out


def tolerance(case):
    """About four times what the library's own alternatives (CUDA-core against tensor-core kernels, other numbers of
    warps per cache slice and so other orders of the sums) differ by on the listed cases: column sums 7e-7 (2e-5 with
    the caller's normalisers, which do not share the rounding of the logits), 9e-4 of the merged fp16 elements by one
    unit, outputs 7e-6 with single 16-bit roundings of 8e-3."""
    f32 = case["dtype"] == "f32"
    if case["kind"] == "stats":
        return {"rel": 1e-4, "max": 2e-4} if case["lse"] else {"rel": 1e-5, "max": 1e-4}
    if case["kind"] == "full":
        return {"rel": 1e-5, "max": 1e-4} if f32 else {"rel": 3e-5, "max": 3e-2}
    if case["kind"] in ("prompt", "compress"):
        return {"rel": 2e-5, "max": 1e-3, "differ": 5e-3}
    return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3} if f32 else {"rel": 3e-5, "max": 3e-2, "differ": 1e-3}
