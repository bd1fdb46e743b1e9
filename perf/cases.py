"""Workloads of the library as its users run them, for timing and for comparing two builds.

A case is one pass of a real use of the C ABI through its Python binding: a run of macro-steps
over a paged smashed-KV cache (bf16 or FP8 rows), the layer front followed by its attention, the
micro-step decoder, a prompt chunk, or the compositional embedder.  Inputs are drawn on the GPU
from a seed; slot counts, chunk lengths and patch sizes belong to the case (they fix its work).

Appending passes begin by rolling the counters back (ham_kv_set_lengths, the call that drops the
slots of a rejected macro-step), so that a pass can be repeated on one cache.  Passes with
"graph" replay a CUDA graph of the same calls, as a serving loop does with a launch-bound macro-step;
the others make the calls one by one.  Calls that turn q in place (ham_kv_append, ham_prefill)
find it turned once more in a repeated pass: values of the same size and distribution.
"""
import math

import numpy as np
import torch

from paper_2505_20438_gb300 import ham

ROPE_BASE = 10000.0
MAX_TOKENS = 4          # tokens a slot stands for, at most


# -------------------------------------------------------------------------------------------
# the cases
# -------------------------------------------------------------------------------------------
def _decode(name=None, **kw):
    c = dict(kind="decode", path="step", batch=8, kv_heads=8, group=4, head_dim=128, page_slots=16,
             layers=4, steps=4, lo=4096, hi=4096, kv="bf16", pos="slot", q_rot=False, out="bf16",
             scale=1.0, graph=False, read=False, lens=1, hidden=0)
    c.update(kw)
    return dict(c, name=name) if name else c


def _prefill(name=None, **kw):
    c = dict(kind="prefill", batch=4, kv_heads=8, group=4, head_dim=128, page_slots=16, rows_lo=4096,
             rows_hi=4096, lo=0, hi=0, pos="slot", ntok=False, out="bf16", scale=1.0, lens=1)
    c.update(kw)
    return dict(c, name=name) if name else c


def _embed(name=None, **kw):
    c = dict(kind="embed", batch=64, hidden=2048, heads=32, patch=4, vocab=0, lens=1)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest cache (8/2 heads of 64, 255 slots in two 128-slot pages) stepped by the two
        # separate calls, the host reading the counters after each macro-step: what one call costs.
        _decode("two_calls_b1_s255", path="split", batch=1, kv_heads=2, group=4, head_dim=64,
                page_slots=128, layers=1, steps=1, lo=255, hi=255, read=True),
        # The micro-step decoder of one macro-step: four layers, three micro-steps over four context
        # entries of a batch of 8 (Llama-3.2-1B heads), captured once.
        _decode("micro_b8", path="micro", head_dim=64, layers=4, steps=3, lo=4, hi=4, graph=True,
                q_rot=True),
        # One conversation at a time: macro-steps of a 32-layer stack at batch 1, captured.
        _decode("stack_b1_s2048", batch=1, layers=32, lo=2048, hi=2048, graph=True,
                scale=128 ** -0.5),
        # The small serving batch of a Llama-8B layer at 4096 slots.
        _decode("step_b8_s4096", graph=True, scale=128 ** -0.5),
        # A ragged serving batch: 64 sequences of 512 to 8192 slots, positions by token count.
        _decode("step_ragged_b64", batch=64, layers=1, steps=2, lo=512, hi=8192, pos="token", lens=2),
        # Long context: few sequences, 65,536 slots each.
        _decode("step_long_b4_s65536", batch=4, layers=1, steps=2, lo=65536, hi=65536),
        # The same serving batch over 8-bit rows, at twice the length.
        _decode("step_fp8_b8_s8192", lo=8192, hi=8192, kv="fp8", graph=True),
        # A layer from its normalised input: projection, RoPE and append, then the attention, called
        # one by one for the layers of a small batch.
        _decode("front_b8_h4096", path="front", hidden=4096, steps=1, lo=2048, hi=2048),
        # The tokens of a macro-step fused into one state for 64 sequences (Llama-3.2-1B width).
        _embed("embed_b64_h2048"),
        # Four fresh prompts of 4096 tokens through one layer.
        _prefill("prefill_b4_s4096", scale=128 ** -0.5),
        # Chunks of unequal length over caches of unequal length, explicit token counts.
        _prefill("prefill_chunk_ragged", batch=6, rows_lo=65, rows_hi=1023, lo=500, hi=6000,
                 page_slots=32, pos="token", ntok=True, lens=3),
        # A short question after a long document: 64 rows over 65,536 cached slots.
        _prefill("prefill_b1_c64_s65536", batch=1, rows_lo=64, rows_hi=64, lo=65536, hi=65536),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "fp8", "split", "micro", "front", "embed", "prefill", "prefill",
                       "short_chunk"])
    lens = rng.randrange(1 << 20)
    d = rng.choice([64, 128, 128])
    heads = dict(kv_heads=rng.choice([2, 4, 8, 8]), group=rng.choice([1, 2, 4, 4, 8]), head_dim=d,
                 page_slots=rng.choice([16, 16, 32, 64, 128]), lens=lens,
                 scale=rng.choice([1.0, d ** -0.5]))
    pos = rng.choice(["slot", "slot", "token", "given"])
    out = rng.choice(["bf16", "bf16", "f32"])
    if kind == "micro":
        return _decode(path="micro", batch=_log_int(rng, 1, 100), layers=rng.randint(2, 6),
                       steps=rng.randint(1, 4), lo=1, hi=rng.randint(1, 8), pos=pos, out=out,
                       q_rot=rng.random() < 0.5, graph=True, **dict(heads, page_slots=16))
    if kind == "embed":
        hd = rng.choice([32, 64, 128])
        hidden = 128 * rng.randint(4, 32)
        return _embed(batch=_log_int(rng, 1, 300), hidden=hidden, heads=hidden // hd,
                      patch=rng.choice([4, 4, 2, 8]), lens=lens,
                      vocab=_log_int(rng, 1000, 60000) if rng.random() < 0.4 else 0)
    if kind in ("prefill", "short_chunk"):
        if kind == "prefill":
            batch, rows = _log_int(rng, 1, 8), _log_int(rng, 17, 4096)
            cached = rng.choice([0, 0, _log_int(rng, 16, 16384)])
        else:
            batch, rows = rng.randint(1, 2), _log_int(rng, 1, 200)
            cached = _log_int(rng, 2048, 65536)
        # (row, attended slot) pairs x heads x head_dim within the largest listed chunk's
        hq_d = heads["kv_heads"] * heads["group"] * d
        while batch * rows * (cached + rows / 2) * 4 * hq_d > 4e11:
            if batch > 1:
                batch -= 1
            else:
                rows //= 2
        lo = max(1, int(rows * rng.uniform(0.2, 1.0)))
        c_lo = int(cached * rng.uniform(0.2, 1.0))
        return _prefill(batch=batch, rows_lo=lo, rows_hi=rows, lo=c_lo, hi=cached, pos=pos,
                        ntok=rng.random() < 0.5, out=out, **heads)
    batch = _log_int(rng, 1, 100)
    layers, steps = rng.choice([1, 2, 4, 8]), rng.randint(1, 4)
    if kind == "fp8":
        heads["head_dim"] = 128
        heads["scale"] = 1.0
    hidden = 0
    if kind == "front":
        hidden = 256 * _log_int(rng, 2, 32)
    if kind in ("front", "split"):
        steps = min(steps, 2)
    per_slot = heads["kv_heads"] * heads["head_dim"] * 4
    most = int(min(65536, 1.0e9 / (per_slot * batch * layers * steps), 2.5e9 / (per_slot * batch * layers)))
    hi = _log_int(rng, 32, max(33, most))
    lo = max(1, int(hi * rng.uniform(0.1, 1.0)))
    path = kind if kind in ("front", "split") else "step"
    return _decode(path=path, batch=batch, layers=layers, steps=steps, lo=lo, hi=hi, pos=pos, out=out,
                   kv="fp8" if kind == "fp8" or (kind == "front" and heads["head_dim"] == 128
                                                 and rng.random() < 0.3) else "bf16",
                   q_rot=path == "step" and rng.random() < 0.5, read=rng.random() < 0.3 and path == "split",
                   graph=path == "step" and rng.random() < 0.6, hidden=hidden, **heads)


# -------------------------------------------------------------------------------------------
# what a case fixes (lengths) and what a seed fixes (values)
# -------------------------------------------------------------------------------------------
def _lengths(c, salt, lo, hi, n):
    g = np.random.Generator(np.random.PCG64([c["lens"], salt]))
    return g.integers(lo, hi + 1, size=n).astype(np.int64)


def _slots(c):
    return _lengths(c, 1, c["lo"], c["hi"], c["batch"])


def _rows(c):
    return _lengths(c, 2, c["rows_lo"], c["rows_hi"], c["batch"])


def _patches(c):
    g = np.random.Generator(np.random.PCG64([c["lens"], 3]))
    return np.minimum(g.geometric(0.5, size=c["batch"]), c["patch"]).astype(np.int64)


def _gen(seed, *what):
    x = np.random.SeedSequence([int(seed) & 0x7fffffff, *what]).generate_state(1, np.uint64)[0]
    g = torch.Generator(device="cuda")
    g.manual_seed(int(x >> np.uint64(1)))
    return g


def _normal(g, shape, scale):
    return (torch.randn(shape, generator=g, device="cuda") * scale).to(torch.bfloat16)


def _tokens(g, shape):
    """Tokens a slot stands for: geometric with p = 1/2, the tail folded into MAX_TOKENS."""
    u = torch.rand(shape, generator=g, device="cuda")
    n = torch.ones(shape, dtype=torch.int32, device="cuda")
    for k in range(1, MAX_TOKENS):
        n += (u < 0.5 ** k).to(torch.int32)
    return n


def _layer_cache(c, seed, layer, slots):
    """One layer's stored keys (already turned) and values [B][Lmax][Hkv][d]."""
    shape = (c["batch"], int(slots.max()), c["kv_heads"], c["head_dim"])
    g = _gen(seed, 10, layer)
    return _normal(g, shape, c["scale"]), _normal(g, shape, c["scale"])


def _slot_tokens(c, seed, slots):
    t = _tokens(_gen(seed, 11), (c["batch"], max(1, int(slots.max()))))
    alive = torch.arange(t.shape[1], device="cuda")[None, :] < torch.from_numpy(slots).cuda()[:, None]
    return t * alive


def _decode_inputs(c, seed):
    B, Hkv, G, d, L, M = (c[k] for k in ("batch", "kv_heads", "group", "head_dim", "layers", "steps"))
    g = _gen(seed, 12)
    s = c["scale"]
    x = dict(ntok=_tokens(g, (M, B)))
    if c["path"] == "micro":
        x["ntok"] = torch.ones_like(x["ntok"])
    x["pos"] = torch.randint(0, 4 * c["hi"] + 4, (M, B), generator=g, device="cuda").to(torch.int32) \
        if c["pos"] == "given" else None
    if c["path"] == "front":
        H = c["hidden"]
        x["x"] = _normal(g, (M, L, B, H), 1.0)
        x["w"] = [_normal(g, ((G + 2) * Hkv * d, H), s ** 0.5 * H ** -0.5) for _ in range(L)]
    else:
        x["q"] = _normal(g, (M, L, B, Hkv * G, d), s)
        x["k"] = _normal(g, (M, L, B, Hkv, d), s)
        x["v"] = _normal(g, (M, L, B, Hkv, d), s)
    return x


def _prefill_inputs(c, seed):
    T = int(_rows(c).sum())
    Hkv, G, d, s = c["kv_heads"], c["group"], c["head_dim"], c["scale"]
    g = _gen(seed, 13)
    x = dict(q=_normal(g, (T, Hkv * G, d), s), k=_normal(g, (T, Hkv, d), s), v=_normal(g, (T, Hkv, d), s))
    x["ntok"] = _tokens(g, (T,)) if c["ntok"] else None
    x["pos"] = torch.randint(0, 4 * (c["hi"] + c["rows_hi"]), (T,), generator=g, device="cuda").to(
        torch.int32) if c["pos"] == "given" else None
    return x


def _embed_inputs(c, seed):
    H, g = c["hidden"], _gen(seed, 14)
    n = int(_patches(c).sum())
    x = {k: _normal(g, (H, H), H ** -0.5) for k in ("wq", "wk", "wv", "wo")}
    x["pos"] = _normal(g, (c["patch"], H), 1.0)
    if c["vocab"]:
        x["table"] = _normal(g, (c["vocab"], H), 1.0)
        x["ids"] = torch.randint(0, c["vocab"], (n,), generator=g, device="cuda").to(torch.int32)
    else:
        x["x"] = _normal(g, (n, H), 1.0)
    return x


# -------------------------------------------------------------------------------------------
# prepare and run
# -------------------------------------------------------------------------------------------
def _out_dtype(c):
    return torch.float32 if c["out"] == "f32" else torch.bfloat16


def _cache(c, seed, layers, room):
    """A cache of `layers` layers filled to the case's slot counts, with `room` slots to append."""
    slots = _slots(c)
    max_slots = int(slots.max()) + room
    pages = -(-max_slots // c["page_slots"])
    kv = ham.ham_kv_alloc(
        layers, c["batch"], c["kv_heads"] * c["group"], c["kv_heads"], c["head_dim"], c["page_slots"],
        max_slots, pos_mode=ham.HAM_POS_TOKEN if c["pos"] == "token" else ham.HAM_POS_SLOT,
        pool_pages=-(-5 * c["batch"] * pages // 4), rope_base=ROPE_BASE, page_seed=1 + seed % (1 << 30),
        kv_dtype=ham.HAM_KV_E4M3 if c.get("kv") == "fp8" else ham.HAM_KV_BF16)
    counts = torch.from_numpy(slots.astype(np.int32)).cuda()
    st = _slot_tokens(c, seed, slots)
    for layer in range(layers):
        if int(slots.max()) > 0:
            k, v = _layer_cache(c, seed, layer, slots)
            ham.ham_kv_fill(kv, layer, k, v, counts, ntok=st[:, :k.shape[1]].contiguous())
    return kv, counts, st.sum(1).to(torch.int64)


def prepare(case, seed):
    return {"decode": _prepare_decode, "prefill": _prepare_prefill, "embed": _prepare_embed}[case["kind"]](
        case, seed)


def _prepare_decode(c, seed):
    B, Hkv, G, d, L, M = (c[k] for k in ("batch", "kv_heads", "group", "head_dim", "layers", "steps"))
    x = _decode_inputs(c, seed)
    kv, counts, tokens = _cache(c, seed, L, M)
    heads = (M, L, B, Hkv * G, d)
    out = torch.zeros(heads, dtype=_out_dtype(c), device="cuda")
    q_rot = torch.zeros(heads, dtype=torch.bfloat16, device="cuda") \
        if c["q_rot"] or c["path"] == "front" else None
    calls = []
    for m in range(M):
        pos = None if x["pos"] is None else x["pos"][m]
        for l in range(L):
            if c["path"] == "front":
                ins = (x["x"][m, l], x["w"][l])
            else:
                ins = (x["q"][m, l], x["k"][m, l], x["v"][m, l])
            calls.append((l, ins, pos, x["ntok"][m], out[m, l], None if q_rot is None else q_rot[m, l]))
    results = dict(out=out)
    if c["path"] == "split":
        results["q"] = x["q"]
    elif q_rot is not None:
        results["q_rot"] = q_rot
    s = dict(kind="decode", path=c["path"], kv=kv, layers=L, counts=counts, tokens=tokens, calls=calls,
             results=results, read=c["read"], graph=None)
    if c["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode_calls(s)
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _decode_calls(s)
        s["graph"] = graph
    return s


def _decode_calls(s):
    kv = s["kv"]
    for l in range(s["layers"]):
        ham.ham_kv_set_lengths(kv, l, s["counts"], s["tokens"])
    path = s["path"]
    for l, ins, pos, ntok, out, q_rot in s["calls"]:
        if path == "step":
            ham.ham_decode_step(kv, l, *ins, pos, ntok, out, q_rot=q_rot)
        elif path == "micro":
            ham.ham_micro_step(kv, l, *ins, pos, ntok, out, q_rot=q_rot)
        elif path == "split":
            ham.ham_kv_append(kv, l, *ins, pos, ntok)
            ham.ham_decode_attn_ex(kv, l, ins[0], out)
        else:
            ham.ham_qkv_append(kv, l, *ins, ntok, q_rot, pos=pos)
            ham.ham_decode_attn_ex(kv, l, q_rot, out)


def _prepare_prefill(c, seed):
    rows = _rows(c)
    x = _prefill_inputs(c, seed)
    kv, counts, tokens = _cache(c, seed, 1, int(rows.max()))
    offsets = torch.from_numpy(np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)).cuda()
    out = torch.zeros(x["q"].shape, dtype=_out_dtype(c), device="cuda")
    return dict(kind="prefill", kv=kv, counts=counts, tokens=tokens, offsets=offsets, x=x, out=out)


def _prepare_embed(c, seed):
    x = _embed_inputs(c, seed)
    e = ham.ham_embedder_alloc(c["hidden"], c["heads"], c["batch"], c["patch"], x["wq"], x["wk"], x["wv"],
                               x["wo"], x["pos"])
    if c["vocab"]:
        ham.ham_embedder_set_vocab(e, x["table"])
    offsets = torch.from_numpy(np.concatenate([[0], np.cumsum(_patches(c))]).astype(np.int32)).cuda()
    out = torch.zeros((c["batch"], c["hidden"]), dtype=torch.bfloat16, device="cuda")
    return dict(kind="embed", e=e, x=x.get("x"), ids=x.get("ids"), offsets=offsets, out=out)


def run(state):
    s = state
    if s["kind"] == "decode":
        if s["graph"] is not None:
            s["graph"].replay()
        else:
            _decode_calls(s)
        if s["read"]:
            slots, tokens = ham.ham_slot_lengths(s["kv"])
            return dict(s["results"], slots=slots, tokens=tokens)
        return s["results"]
    if s["kind"] == "prefill":
        x = s["x"]
        ham.ham_kv_set_lengths(s["kv"], 0, s["counts"], s["tokens"])
        ham.ham_prefill(s["kv"], 0, x["q"], x["k"], x["v"], s["offsets"], s["out"], pos=x["pos"],
                        ntok=x["ntok"])
        return dict(out=s["out"], q=x["q"])
    if s["ids"] is not None:
        ham.ham_embed_tokens(s["e"], s["ids"], s["offsets"], s["out"])
    else:
        ham.ham_embed(s["e"], s["x"], s["offsets"], s["out"])
    return s["out"]


# -------------------------------------------------------------------------------------------
# the work of a pass and the error it may show
# -------------------------------------------------------------------------------------------
def work(case):
    c = case
    if c["kind"] == "embed":
        H, B, T = c["hidden"], c["batch"], int(_patches(c).sum())
        if c["vocab"]:     # tabulated projections: W_o, and each token's q, k and v rows
            return dict(bytes=2 * H * H + 12 * H * T + 2 * B * H, flops=2 * B * H * H)
        return dict(bytes=8 * H * H + 2 * T * H + 2 * B * H, flops=6 * T * H * H + 2 * B * H * H)
    Hkv, d = c["kv_heads"], c["head_dim"]
    Hq = Hkv * c["group"]
    row = d + 1 if c.get("kv") == "fp8" else 2 * d       # a stored key (or value) row of one head
    out = 4 if c["out"] == "f32" else 2
    n = _slots(c)
    if c["kind"] == "prefill":
        r = _rows(c)
        T = int(r.sum())
        pairs = int((r * n + r * (r + 1) // 2).sum())    # (row, attended slot)
        cached = int(n[r > 0].sum())
        return dict(bytes=T * Hq * d * (2 + 2 + out) + T * Hkv * d * 8 + cached * Hkv * 2 * row,
                    flops=4 * Hq * d * pairs)
    B, L, M = c["batch"], c["layers"], c["steps"]
    attended = L * (M * int(n.sum()) + B * M * (M + 1) // 2)
    stored = L * (M * int(n.sum()) + B * M * (M - 1) // 2)
    b = stored * Hkv * 2 * row + L * M * B * (Hkv * 2 * row + Hq * d * out)
    if c["path"] == "front":
        F, H = (Hq + 2 * Hkv) * d, c["hidden"]
        b += L * M * (2 * F * H + 2 * B * H + 2 * B * Hq * d)
        return dict(bytes=b, flops=4 * Hq * d * attended + 2 * L * M * B * F * H)
    b += L * M * B * (2 * Hq * d + 4 * Hkv * d + (2 * Hq * d if c["q_rot"] or c["path"] == "split" else 0))
    return dict(bytes=b, flops=4 * Hq * d * attended)


def tolerance(case):
    # Measured against 64 bits: attention 1.4e-3 to 2.4e-3 in the 2-norm (results rounded to bf16,
    # weights rounded to bf16 or to three e4m3 pieces for the tensor cores), the embedder and the
    # micro-step 1.2e-3 to 1.7e-3 (one rounding of the result).
    return dict(rel=7e-3 if case["kind"] == "embed" or case.get("path") == "micro" else 1e-2, max=8e-2)


# -------------------------------------------------------------------------------------------
# the same results in 64 bits
# -------------------------------------------------------------------------------------------
def _turn(x, p):
    """Rotate-half RoPE of x [..., heads, d] (float64) at positions p [...]."""
    d = x.shape[-1]
    f = ROPE_BASE ** (-torch.arange(0, d, 2, dtype=torch.float64, device=x.device) / d)
    a = p.double()[..., None, None] * f
    c, s = a.cos(), a.sin()
    x0, x1 = x[..., :d // 2], x[..., d // 2:]
    return torch.cat([x0 * c - x1 * s, x1 * c + x0 * s], -1)


def _stored(x, fp8):
    """What the cache holds of rows x (float64): bf16, or e4m3 codes times a power of two."""
    x = x.to(torch.bfloat16)
    if not fp8:
        return x.double()
    x = x.float()
    top = x.abs().amax(-1, keepdim=True)
    e = torch.where(top > 0, torch.frexp(top)[1] - 8, torch.zeros_like(top, dtype=torch.int32))
    e = e.clamp(-124, 119)
    return torch.ldexp(torch.ldexp(x, -e).to(torch.float8_e4m3fn).double(), e)


def exact(case, seed):
    return {"decode": _exact_decode, "prefill": _exact_prefill, "embed": _exact_embed}[case["kind"]](
        case, seed)


def _attend(q, k, v, seen, d):
    """q [R][G][d] of one KV head over k, v [N][d]; row r sees slots 0 .. seen[r] - 1."""
    R, G = q.shape[:2]
    s = (q.reshape(R * G, d) @ k.T).reshape(R, G, -1) * d ** -0.5
    hidden = torch.arange(k.shape[0], device=k.device)[None, :] >= seen[:, None]
    s.masked_fill_(hidden[:, None, :], -math.inf)
    s = torch.softmax(s, -1)
    return (s.reshape(R * G, -1) @ v).reshape(R, G, d)


def _exact_decode(c, seed):
    B, Hkv, G, d, L, M = (c[k] for k in ("batch", "kv_heads", "group", "head_dim", "layers", "steps"))
    fp8 = c["kv"] == "fp8"
    slots = _slots(c)
    x = _decode_inputs(c, seed)
    n0 = torch.from_numpy(slots).cuda()
    before = torch.cumsum(x["ntok"].long(), 0) - x["ntok"].long()          # [M][B]
    tokens = _slot_tokens(c, seed, slots).sum(1).long()
    if x["pos"] is not None:
        pos = x["pos"].long()
    elif c["pos"] == "token":
        pos = tokens[None, :] + before
    else:
        pos = n0[None, :] + torch.arange(M, device="cuda")[:, None]
    out = torch.empty((M, L, B, Hkv * G, d), dtype=torch.float64, device="cuda")
    q_rot = torch.empty_like(out)
    for l in range(L):
        if c["path"] == "front":
            y = (x["x"][:, l].double() @ x["w"][l].double().T).reshape(M, B, -1, d)
            q, k, v = y.split([Hkv * G, Hkv, Hkv], 2)
        else:
            q, k, v = (x[n][:, l].double() for n in ("q", "k", "v"))
        q_rot[:, l] = _turn(q, pos)
        q = q_rot[:, l].to(torch.bfloat16).double()
        k, v = _stored(_turn(k, pos), fp8), _stored(v, fp8)
        kc, vc = _layer_cache(c, seed, l, slots)
        for b in range(B):
            n = int(slots[b])
            seen = n + 1 + torch.arange(M, device="cuda")
            for g in range(Hkv):
                kk = torch.cat([_stored(kc[b, :n, g].double(), fp8), k[:, b, g]])
                vv = torch.cat([_stored(vc[b, :n, g].double(), fp8), v[:, b, g]])
                out[:, l, b, g * G:(g + 1) * G] = _attend(q[:, b, g * G:(g + 1) * G], kk, vv, seen, d)
    results = dict(out=out)
    if c["path"] == "split":
        results["q"] = q_rot
    elif c["q_rot"] or c["path"] == "front":
        results["q_rot"] = q_rot
    if c["read"]:
        results["slots"] = results["tokens"] = None
    return results


def _exact_prefill(c, seed):
    Hkv, G, d = c["kv_heads"], c["group"], c["head_dim"]
    slots, rows = _slots(c), _rows(c)
    x = _prefill_inputs(c, seed)
    tokens = _slot_tokens(c, seed, slots).sum(1).long()
    if int(slots.max()) > 0:
        kc, vc = _layer_cache(c, seed, 0, slots)
    out = torch.empty(x["q"].shape, dtype=torch.float64, device="cuda")
    q_all = torch.empty_like(out)
    a = 0
    for b in range(c["batch"]):
        n, r = int(slots[b]), int(rows[b])
        own = slice(a, a + r)
        a += r
        ar = torch.arange(r, device="cuda")
        if x["pos"] is not None:
            pos = x["pos"][own].long()
        elif c["pos"] == "token":
            t = x["ntok"][own].long() if x["ntok"] is not None else torch.ones_like(ar)
            pos = tokens[b] + torch.cumsum(t, 0) - t
        else:
            pos = n + ar
        q_all[own] = _turn(x["q"][own].double(), pos)
        q = q_all[own].to(torch.bfloat16).double()
        k, v = _stored(_turn(x["k"][own].double(), pos), False), x["v"][own].double()
        for g in range(Hkv):
            kk, vv = k[:, g], v[:, g]
            if n:
                kk = torch.cat([kc[b, :n, g].double(), kk])
                vv = torch.cat([vc[b, :n, g].double(), vv])
            for r0 in range(0, r, 1024):
                r1 = min(r, r0 + 1024)
                out[own][r0:r1, g * G:(g + 1) * G] = _attend(q[r0:r1, g * G:(g + 1) * G], kk[:n + r1],
                                                            vv[:n + r1], n + 1 + ar[r0:r1], d)
    return dict(out=out, q=q_all)


def _exact_embed(c, seed):
    H, nh = c["hidden"], c["heads"]
    x = _embed_inputs(c, seed)
    w = {k: x[k].double() for k in ("wq", "wk", "wv", "wo", "pos")}
    e = (x["table"][x["ids"].long()] if c["vocab"] else x["x"]).double()
    out = torch.empty((c["batch"], H), dtype=torch.float64, device="cuda")
    a = 0
    for b, n in enumerate(_patches(c)):
        xb = e[a:a + int(n)]
        a += int(n)
        if n == 1:
            out[b] = xb[0]
            continue
        y = xb + w["pos"][:int(n)]
        q = (w["wq"] @ xb.mean(0)).reshape(nh, -1)
        k, v = (y @ w["wk"].T).reshape(int(n), nh, -1), (y @ w["wv"].T).reshape(int(n), nh, -1)
        s = torch.softmax(torch.einsum("hd,nhd->hn", q, k) * q.shape[1] ** -0.5, -1)
        out[b] = w["wo"] @ torch.einsum("hn,nhd->hd", s, v).reshape(H)
    return out
