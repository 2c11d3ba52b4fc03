"""Performance cases of the R-KV compression library: what a decode loop has it do, through the public entry points.

Kinds of case:
  compress  one firing of the periodic compression on device caches (Compressor.compress).  Between two firings a decode
            loop fills the buffer part of every cache with new tokens; a pass puts one block of new keys there (values do
            not take part in the scores: the buffer's values stay as they are), sets the lengths and fires.
  step      one decode step through the whole model, layer by layer: push_query, decode attention, append.
  host      one firing for caches that live in pinned host memory (Compressor.compress_host), results awaited.

Shapes are those of the repository's configurations (rkv_inputs), layers folded into the batch where the layers fire
together.  Keys: N(0, 1) with four outlier channels per (layer, KV head) scaled by 8, a share of the token spans noisy
copies of an earlier span; queries and values N(0, 1).
"""
from __future__ import annotations

import math

import torch

import paper_2505_24133_b200 as rkv

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32, "fp8": torch.float8_e4m3fn}
ESIZE = {"bf16": 2, "f32": 4, "fp8": 1}
FRESH = 8           # blocks of new keys a state holds; passes take them in turn
HOST_RING = 3       # host-resident caches a state holds; passes take them in turn
CHUNK = 1 << 29     # elements of keys made at a time


def _case(name, kind, layers, batch, kv_heads, q_heads, budget, buffer=128, dim=128, dtype="bf16", alpha=8, beta=1,
          threshold=0.5, pool_w=4, ragged=False, paged=False, flags=0, span=32, copies=0.30, sigma=0.05):
    c = dict(kind=kind, layers=layers, batch=batch, kv_heads=kv_heads, q_heads=q_heads, dim=dim, budget=budget, buffer=buffer,
             alpha=alpha, dtype=dtype, beta=beta, threshold=threshold, pool_w=pool_w, ragged=ragged, paged=paged, flags=flags,
             span=span, copies=copies, sigma=sigma)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one fp32 head of 96 tokens, all latency and launches
        _case("tiny_f32", "compress", 1, 1, 1, 4, 64, 32, dtype="f32", span=1, copies=0.17),
        # a single conversation: all 32 layers of an 8-KV-head model at batch 1
        _case("llama8b_b1", "compress", 32, 1, 8, 32, 1024),
        # the same model serving 16 sequences with a long budget
        _case("llama8b_b16", "compress", 32, 16, 8, 32, 4096),
        # seven query heads per KV head, many short caches, heavy redundancy
        _case("qwen7b_b64", "compress", 28, 64, 4, 28, 2048, span=64, copies=0.50, sigma=0.02),
        # the largest configuration: 12288 heads of 4224 tokens, 26.6 GB of cache
        _case("qwen14b_b32", "compress", 48, 32, 8, 40, 4096),
        # caches stored as 8-bit codes
        _case("llama8b_b16_fp8", "compress", 32, 16, 8, 32, 4096, dtype="fp8"),
        # heads of 64 dimensions
        _case("llama1b_b64_d64", "compress", 16, 64, 8, 32, 2048, dim=64),
        # continuous batching on a paged pool: sequences of different lengths, some still below the budget, an odd budget,
        # one query head per KV head, several partners kept per token
        _case("mha7b_ragged_paged", "compress", 32, 4, 32, 32, 1000, 152, beta=4, ragged=True, paged=True),
        # heads of 256 dimensions
        _case("wide_d256", "compress", 16, 4, 4, 16, 1024, dim=256),
        # one token of a single conversation through 32 layers: small launches, one after the other
        _case("step_llama8b_b1", "step", 32, 1, 8, 32, 1024),
        # one token of 16 long sequences through 32 layers
        _case("step_llama8b_b16", "step", 32, 16, 8, 32, 4096),
        # a conversation whose caches were moved out to host memory
        _case("host_llama8b_b1", "host", 32, 1, 8, 32, 1024),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["compress"] * 7 + ["step"] * 2 + ["host"])
    dtype = rng.choice(["bf16"] * 6 + ["fp8"] * 2 + ["f32"])
    dim = rng.choice([128] * 6 + [64] * 2 + [256])
    if kind == "step" and (dim == 256 or (dim == 64 and dtype != "bf16")):
        dim = 128
    kv_heads = rng.choice([1, 2, 4, 8, 8, 16, 32])
    group = rng.choice([1, 2, 3, 4, 4, 5, 7, 8])
    alpha = rng.choice([8, 8, 8, 8, 4, 12])
    buffer = rng.choice([32, 64, 128, 128, 128, 200, 512])
    # fp32 caches and 256 dimensions are small-cache options; the others go up to the largest cache the library takes
    slow = dtype == "f32" or dim == 256
    budget = int(_log(rng, 64, 1024 if slow else 7600))
    paged = rng.random() < 0.25
    if paged:                                   # pages of 128 rows: a whole number of them per head
        buffer += -(budget + buffer) % 128
    cap = budget + buffer
    most = 256 * 1152 if slow else 256 * 1152 if kind == "host" else 512 * 8 * 4224
    heads = max(1.0, _log(rng, kv_heads * cap, max(most, kv_heads * cap + 1)) / (cap * kv_heads))
    layers = rng.choice([1, 2, 16, 28, 32])
    layers = min(layers, max(1, int(heads)))
    batch = max(1, int(heads / layers))
    return _case(None, kind, layers, batch, kv_heads, kv_heads * group, budget, buffer, dim, dtype, alpha,
                 beta=rng.choice([1, 1, 1, 1, 2, 8]), threshold=rng.choice([0.5, 0.5, 0.5, 0.5, 0.35, 0.9]),
                 pool_w=rng.choice([4, 4, 4, 4, 0, 7]), ragged=kind == "compress" and rng.random() < 0.3,
                 paged=paged and kind != "host",
                 flags=rng.choice([0] * 6 + [rkv.RKV_FLAG_MEAN_THEN_POOL, rkv.RKV_FLAG_HEAD_MEAN, rkv.RKV_FLAG_GQA_MEAN_POOL]),
                 span=rng.choice([1, 16, 32, 64]), copies=rng.choice([0.1, 0.3, 0.5]), sigma=rng.choice([0.02, 0.05, 0.2]))


# ---------------------------------------------------------------------------------------------------- inputs
def _keys(c, tokens, gen):
    """[layers * batch, kv_heads, tokens, dim] keys of the case's type."""
    L, B, H, d, sp = c["layers"], c["batch"], c["kv_heads"], c["dim"], c["span"]
    dev = gen.device
    out = torch.empty(L * B, H, tokens, d, dtype=DTYPES[c["dtype"]], device=dev)
    scale = torch.ones(L, H, d, device=dev)
    if c["dtype"] != "f32":
        scale.scatter_(-1, torch.rand(L, H, d, generator=gen, device=dev).argsort(-1)[..., :4], 8.0)
    spans = -(-tokens // sp)
    step = max(1, CHUNK // (H * tokens * d))
    for s0 in range(0, L * B, step):
        n = min(step, L * B - s0)
        layer = torch.arange(s0, s0 + n, device=dev) // B
        k = torch.randn(n, H, tokens, d, generator=gen, device=dev).mul_(scale[layer][:, :, None])
        # every span but the first may be a copy of an earlier one (of that one's own source if it is a copy itself)
        at = torch.arange(spans, device=dev).expand(n, spans)
        src = torch.where((torch.rand(n, spans, generator=gen, device=dev) < c["copies"]) & (at > 0),
                          (torch.rand(n, spans, generator=gen, device=dev) * at).long(), at)
        for _ in range(14):
            src = src.gather(1, src)
        tok = (src[:, :, None] * sp + torch.arange(sp, device=dev)).reshape(n, -1)[:, :tokens].clamp_(max=tokens - 1)
        seq, pos = (tok != torch.arange(tokens, device=dev)).nonzero(as_tuple=True)
        block = k[seq, :, tok[seq, pos]]
        k[seq, :, pos] = block.add_(torch.randn(block.shape, generator=gen, device=dev), alpha=c["sigma"])
        out[s0:s0 + n] = k.to(out.dtype)
    return out


def _normal(shape, c, gen, query=False):
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    x = torch.randn(shape, generator=gen, device=gen.device, dtype=dt)
    return x if query or c["dtype"] != "fp8" else x.to(torch.float8_e4m3fn)


def _desc(c, batch):
    d = rkv.rkv_desc_default()
    d.batch, d.n_kv_heads, d.n_q_heads, d.head_dim = batch, c["kv_heads"], c["q_heads"], c["dim"]
    d.dtype = {"bf16": rkv.RKV_BF16, "f32": rkv.RKV_F32, "fp8": rkv.RKV_FP8_E4M3}[c["dtype"]]
    return d


def _bits(t):
    """The bit patterns: what is moved has to stay the same to the bit."""
    return t.view({1: torch.uint8, 2: torch.int16, 4: torch.int32}[t.element_size()])


def prepare(case, seed):
    c = dict(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    Bf, H, Hq, d = c["layers"] * c["batch"], c["kv_heads"], c["q_heads"], c["dim"]
    budget, buffer, cap = c["budget"], c["buffer"], c["budget"] + c["buffer"]
    s = {"case": c, "turn": 0}
    if c["kind"] == "host":
        s["comp"] = _compressor(c, Bf, host_staging=True)
        s["full"] = torch.full((Bf,), cap, dtype=torch.int32)
        s["ring"] = []
        for _ in range(HOST_RING):
            dev = [_keys(c, cap, gen), _normal((Bf, H, cap, d), c, gen), _normal((Bf, Hq, c["alpha"], d), c, gen, True)]
            host = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True) for t in dev]
            for a, b in zip(host, dev):
                a.copy_(b)
            host += [torch.empty(Bf, dtype=torch.int32, pin_memory=True),
                     torch.zeros(Bf, H, budget, dtype=torch.int32, pin_memory=True)]
            s["ring"].append(host)
        return s
    blocks = FRESH if c["kind"] == "compress" else 1
    everything = _keys(c, cap + (blocks - 1) * buffer, gen)
    k = everything[:, :, :cap].contiguous()
    fresh = [everything[:, :, budget + i * buffer:cap + i * buffer].contiguous() for i in range(blocks)]
    del everything
    v = _normal((Bf, H, cap, d), c, gen)
    s["q"] = _normal((Bf, Hq, c["alpha"], d), c, gen, True)
    table = None
    if c["paged"]:                              # the pages of a head lie anywhere in the pool
        tiles = cap // 128
        table = torch.randperm(Bf * H * tiles, generator=gen, device="cuda").view(Bf, H, tiles)
        flat = table.flatten()
        pool = torch.empty(Bf * H * tiles, 128, d, dtype=k.dtype, device="cuda")
        _bits(pool)[flat] = _bits(k).view(-1, 128, d)
        k, pool = pool, torch.empty_like(pool)
        _bits(pool)[flat] = _bits(v).view(-1, 128, d)
        v = pool
        row = torch.arange(budget, cap, device="cuda")
        s["rows"] = (table[:, :, row // 128] * 128 + row % 128).flatten()
        table = table.to(torch.int32)
    s["k"], s["v"] = k, v
    if c["kind"] == "step":
        return _prepare_step(s, c, gen, table)
    s["fresh"] = fresh
    s["comp"] = _compressor(c, Bf, block_table=table, pool_pages=k.shape[0] if c["paged"] else 0)
    s["full"] = torch.full((Bf,), cap, dtype=torch.int32, device="cuda")
    if c["ragged"]:                             # every sequence at a point of its own; a quarter still below the budget
        u = torch.rand(Bf, generator=gen, device="cuda")
        s["full"] = torch.where(u < 0.25, budget * (0.5 + 2 * u), budget + 1 + (buffer - 1) * (u - 0.25) / 0.75).to(torch.int32)
    s["lens"] = s["full"].clone()
    return s


def _compressor(c, Bf, **more):
    return rkv.Compressor(Bf, c["kv_heads"], c["q_heads"], c["budget"], c["buffer"], c["alpha"], 0.1, dtype=DTYPES[c["dtype"]],
                          pool_w=c["pool_w"], beta=c["beta"], sim_threshold=c["threshold"], flags=c["flags"],
                          head_dim=c["dim"], **more)


def _prepare_step(s, c, gen, table):
    L, B, H, Hq, d = c["layers"], c["batch"], c["kv_heads"], c["q_heads"], c["dim"]
    s["q_new"] = _normal((L, B, Hq, d), c, gen, True)
    s["k_new"], s["v_new"] = _normal((L, B, H, d), c, gen), _normal((L, B, H, d), c, gen)
    s["out"] = torch.zeros(L, B, Hq, d, device="cuda")
    s["start"] = torch.full((L, B), c["budget"], dtype=torch.int32, device="cuda")
    s["lens"] = s["start"].clone()
    desc = _desc(c, B)
    space = torch.empty(max(256, rkv.rkv_decode_workspace_bytes(desc, c["budget"], c["buffer"])), dtype=torch.uint8, device="cuda")
    s["keep"], s["layers"] = [space, table], []
    for i in range(L):
        desc = _desc(c, B)
        desc.workspace, desc.workspace_bytes = space.data_ptr(), space.numel()
        part = slice(i * B, (i + 1) * B)
        k, v = s["k"], s["v"]
        if table is not None:
            desc.block_table, desc.pool_pages = table[part].data_ptr(), k.shape[0]
        else:
            k, v = k[part], v[part]
        s["layers"].append((desc, k, v, s["q"][part], s["q_new"][i], s["k_new"][i], s["v_new"][i], s["lens"][i], s["out"][i]))
    return s


# ---------------------------------------------------------------------------------------------------- passes
def run(state):
    s = state
    c, turn = s["case"], s["turn"]
    s["turn"] += 1
    budget, buffer = c["budget"], c["buffer"]
    if c["kind"] == "host":
        k, v, q, lens, idx = s["ring"][turn % HOST_RING]
        lens.copy_(s["full"])
        s["comp"].compress_host(k, v, q, lens, idx)
        torch.cuda.current_stream().synchronize()         # the caller reads the host buffers next
        return {"idx": idx, "k": _bits(k), "v": _bits(v), "lens": lens}
    if c["kind"] == "step":
        if turn % buffer == 0:                            # the buffers are full: the next segment begins
            s["lens"].copy_(s["start"])
        slot = turn % c["alpha"]
        for desc, k, v, q, q_new, k_new, v_new, lens, out in s["layers"]:
            rkv.rkv_push_query(desc, q, q_new, c["alpha"], slot)
            rkv.rkv_decode_attention(desc, k, v, q_new, lens, out, budget, buffer)
            rkv.rkv_append(desc, k, v, k_new, v_new, lens, budget, buffer)
        return {"out": s["out"], "k": _bits(s["k"]), "v": _bits(s["v"]), "q": _bits(s["q"]), "lens": s["lens"]}
    fresh = s["fresh"][turn % FRESH]
    if c["paged"]:
        _bits(s["k"]).view(-1, c["dim"]).index_copy_(0, s["rows"], _bits(fresh).view(-1, c["dim"]))
    else:
        s["k"][:, :, budget:].copy_(fresh)
    s["lens"].copy_(s["full"])
    idx = s["comp"].compress(s["k"], s["v"], s["q"], s["lens"])
    return {"idx": idx, "k": _bits(s["k"]), "v": _bits(s["v"]), "lens": s["lens"]}


def work(case):
    c = case
    heads, d, cap = c["layers"] * c["batch"] * c["kv_heads"], c["dim"], c["budget"] + c["buffer"]
    group, row = c["q_heads"] // c["kv_heads"], c["dim"] * ESIZE[c["dtype"]]
    q_row = d * (4 if c["dtype"] == "f32" else 2)
    if c["kind"] == "step":
        # keys and values read once, the group's queries read and kept, the new rows kept, the output written
        n = c["budget"] + c["buffer"] / 2
        return {"bytes": heads * (2 * n * row + group * (2 * q_row + 4 * d) + 4 * row), "flops": heads * 4.0 * n * group * d}
    # all keys read; the kept rows of both caches read and written (the keys' read counted already); the index list
    n, share = cap - c["alpha"], 1.0
    if c["ragged"]:
        n, share = c["budget"] + c["buffer"] / 2 - c["alpha"], 0.75
    keys, kept = n * row, c["budget"] * row
    byt = keys + 3.0 * kept + group * c["alpha"] * q_row + 4 * c["budget"]
    if c["kind"] == "host":
        byt = 2.0 * cap * row + 2.0 * kept + group * c["alpha"] * q_row + 4 * c["budget"]
    # logits, norms, the sum of the normalised keys and its product with every key; one similarity per kept partner
    flops = n * d * (2.0 * group * c["alpha"] + 6.0 + 2.0 * c["beta"])
    return {"bytes": heads * share * byt, "flops": heads * share * flops}


def tolerance(case):
    if case["kind"] == "step":
        # fp32 sums of bf16 products, softmax weights to fp32 accuracy; what is moved is moved bit for bit
        return {"rel": 5e-5, "differ": 0.0}
    # index lists and moved bytes.  Two candidates whose scores agree to fp32 rounding may change places at the k-th
    # score, which shifts the part of that one head's list (and rows) between them
    return {"rel": 0.0, "differ": 0.01}
