"""What is timed: the eviction step after a prefill, through the library's public entry points.

A case is one call (or one short sequence of calls) as a serving program makes it: the pseudo queries
and the K/V cache of one layer or of a whole model lie on the GPU (in pinned host memory for the
offloaded cache), the context exists, the output buffers exist; a pass scores, selects and compacts.

Inputs.  Keys and values are N(0, 1) at the shapes of the model; the pseudo queries of a KV head share a
common part (as the queries of neighbouring tokens do).  A share of the prompt - passages of some 16
tokens at positions drawn from the seed, and the attention sinks at its start - is relevant: the
component of those keys along the mean rotated query is large and spread, that of all others is
ordinary.  The budget K equals the number of relevant tokens, so that which tokens are kept does not
hang on the last bits of a score and the index lists and compacted rows can be compared exactly.
"""
from __future__ import annotations

import math

import torch

import paper_2603_11564_b200 as dq

D = 128
SINKS = 4           # relevant tokens at the start of every prompt
PASSAGE = 16        # length of a relevant passage


def _case(name, entry, layers, heads, kv_heads, window, lens, keep, dtype="bf16", pool=0, rope_base=5.0e5, rope="plain"):
    """lens: prompt lengths as text ("4096" or "900,130"); keep: rows kept per prompt, or "10%" of each."""
    return {"name": name, "entry": entry, "layers": layers, "heads": heads, "kv_heads": kv_heads, "window": window,
            "lens": lens, "keep": keep, "dtype": dtype, "pool": pool, "rope_base": rope_base, "rope": rope}


def listed():
    ragged = "14697,25058,8281,31072,12490,18803,25317,15085"
    return [
        # the smallest call: one layer of a small fp32 cache (the configuration of the smoke test)
        _case("fp32_2k", "evict", 1, 8, 2, 32, "2048", "128", dtype="f32", rope_base=1.0e4),
        # a layer at full precision, as one compares a bf16 deployment against
        _case("fp32_12k", "evict", 1, 32, 8, 32, "12345", "1024", dtype="f32"),
        # one layer's hook inside the prefill of an 8k prompt, the window and budget of the paper's throughput runs
        _case("8b_8k_layer", "evict", 1, 32, 8, 32, "8192", "256"),
        # a model without grouped queries: 32 query rows per KV head
        _case("mha_16k_layer", "evict", 1, 32, 32, 32, "16384", "512", rope_base=1.0e4),
        # every layer of a Llama-3-8B-shaped cache at 32k, 3 % kept
        _case("8b_32k", "layers", 32, 32, 8, 64, "32768", "983"),
        # every layer of a Qwen2.5-7B-shaped cache at 128k
        _case("qwen7b_128k", "layers", 28, 28, 4, 64, "131072", "4096", rope_base=1.0e6),
        # ragged serving batch on half of the layers (two pipeline stages), 10 % kept
        _case("8b_ragged8", "layers", 16, 32, 8, 32, ragged, "10%"),
        # the widest throughput run: many 8k prompts, budget 256
        _case("8b_8k_batch40", "layers", 2, 32, 8, 32, ",".join(["8192"] * 40), "256"),
        # the largest: a Llama-3-70B-shaped cache at 128k, one of four pipeline stages
        _case("70b_128k", "layers", 20, 64, 8, 128, "131072", "3932"),
        # odd lengths, Llama-3.1 frequencies, selection on max-pooled scores, scores handed out
        _case("8b_odd_pooled", "evict", 1, 32, 8, 32, "20011,777,5003", "12%", pool=7, rope="llama31"),
        # the steps one by one, with the log-sum-exp of the pseudo rows from the prefill attention
        _case("steps_64k_lse", "steps", 1, 32, 8, 64, "65537", "2048"),
        # a cache that lives in pinned host memory
        _case("8b_32k_host", "host", 4, 32, 8, 64, "32768", "983"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: entry point, head counts, window, lengths and budget at random."""
    kind = rng.choice(["layer", "layer", "model", "model", "batch", "batch", "fp32", "steps", "pooled", "mha", "host"])
    heads, kv = rng.choice([(32, 8), (32, 8), (28, 4), (64, 8), (40, 8), (16, 2)])
    window = rng.choice([32, 32, 48, 64, 100, 128])
    entry, layers, dtype, pool, rope = "evict", 1, "bf16", 0, rng.choice(["plain", "llama31"])
    if kind == "layer":
        lens = [_log_uniform(rng, 2048, 131072)]
    elif kind == "model":
        entry, layers = "layers", rng.randint(4, 12)
        lens = [_log_uniform(rng, 8192, 131072)]
    elif kind == "batch":
        entry, layers = "layers", rng.randint(2, 4)
        hi = _log_uniform(rng, 4096, 32768)
        lens = [rng.randint(hi // 8, hi) for _ in range(rng.randint(2, max(2, min(48, 400000 // hi))))]
    elif kind == "fp32":
        dtype, heads, kv, window = "f32", *rng.choice([(8, 2), (32, 8), (28, 4)]), rng.choice([16, 32, 64])
        lens = [_log_uniform(rng, 1024, 16384)]
    elif kind == "steps":
        entry = "steps"
        lens = [_log_uniform(rng, 4096, 131072)]
    elif kind == "pooled":
        pool = rng.choice([5, 7])
        lens = [_log_uniform(rng, 2048, 65536) for _ in range(rng.randint(1, 4))]
    elif kind == "mha":
        heads, kv, window = *rng.choice([(32, 32), (16, 16)]), rng.choice([16, 32, 48])
        lens = [_log_uniform(rng, 2048, 32768)]
    else:
        entry, layers = "host", 2
        lens = [_log_uniform(rng, 8192, 32768)]
    keep = "%d%%" % rng.randint(2, 12)
    if kind == "layer" and rng.random() < 0.5:
        keep = str(min(rng.choice([256, 512, 1024]), lens[0] // 4))
    c = _case("", entry, layers, heads, kv, window, ",".join(map(str, lens)), keep, dtype, pool,
              rng.choice([1.0e4, 5.0e5, 1.0e6]), rope)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------- inputs
def _sizes(case):
    lens = [int(x) for x in case["lens"].split(",")]
    k = case["keep"]
    least = SINKS + 4 * max(1, case["pool"])
    keep = [max(least, L * int(k[:-1]) // 100 if k.endswith("%") else int(k)) for L in lens]
    return lens, [min(a, L) for a, L in zip(keep, lens)]


def _relevant(L, keep, pool, kv_heads, g):
    """[kv_heads, L] bool: exactly the tokens whose (pooled) score will be large number `keep` per head.
    One slot of the prompt per passage, the passage at a random place of its slot."""
    r = pool // 2
    first = SINKS + r                                    # the sinks and what pooling adds to them
    rest = keep - first
    n = max(1, rest // (PASSAGE + 2 * r))
    size = [rest // n + (1 if i < rest % n else 0) for i in range(n)]
    slot = (L - first - r - 1) // n
    length = torch.tensor(size, device="cuda")
    room = slot - length - 2 * r - 1
    assert bool((room >= 0).all()), "budget too large for separate passages"
    at = (torch.rand((kv_heads, n), generator=g, device="cuda") * (room + 1)).long() + first + r + 1 + torch.arange(n, device="cuda") * slot
    edge = torch.zeros((kv_heads, L + 1), dtype=torch.int32, device="cuda")
    edge.scatter_add_(1, at + r, torch.ones_like(at, dtype=torch.int32))
    edge.scatter_add_(1, at + length - r, -torch.ones_like(at, dtype=torch.int32))
    mask = edge.cumsum(1)[:, :L] > 0
    mask[:, :SINKS] = True
    return mask


class _Context:
    """A library context that goes when the program drops it."""

    def __init__(self, **kw):
        self.handle = dq.dapq_create(**kw)

    def __del__(self):
        if getattr(self, "handle", None) is not None:
            dq.dapq_destroy(self.handle)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    lens, keep = _sizes(case)
    B, Hq, H, N, n = len(lens), case["heads"], case["kv_heads"], case["window"], case["layers"]
    G = Hq // H
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    cu_rows, cu_prompt = [0], [0]
    for L in lens:
        cu_rows.append(cu_rows[-1] + L + N)
        cu_prompt.append(cu_prompt[-1] + L)
    R, KT = cu_rows[-1], sum(keep)
    pool = dict(pool_mode=dq.DAPQ_POOL_MAX, pool_kernel=case["pool"]) if case["pool"] else {}
    freq = dict(inv_freq=dq.dapq_rope_inv_freq_llama3()) if case["rope"] == "llama31" else {}
    ctx = _Context(n_q_heads=Hq, n_kv_heads=H, n_pseudo=N, max_batch=B, max_total_rows=R,
                   dtype=dq.DAPQ_BF16 if case["dtype"] == "bf16" else dq.DAPQ_F32, rope_base=case["rope_base"], **pool, **freq)
    q = torch.empty((n, B, Hq, N, D), dtype=dt, device="cuda")
    k = torch.empty((n, H, R, D), dtype=dt, device="cuda")
    v = torch.empty((n, H, R, D), dtype=dt, device="cuda")
    q_rot = torch.empty((B, Hq, N, D), dtype=dt, device="cuda")
    for l in range(n):
        own = torch.randn((B, H, G, N, D), generator=g, device="cuda")
        common = torch.randn((1, H, 1, 1, D), generator=g, device="cuda")
        q[l] = (math.sqrt(0.5) * (own + common)).reshape(B, Hq, N, D).to(dt)
        dq.dapq_rope_pseudo_q(ctx.handle, q[l], lens, q_rot)
        u = q_rot.float().reshape(B, H, G * N, D).mean(2)
        u = u / u.norm(dim=2, keepdim=True)
        for b in range(B):
            lo, hi = cu_rows[b], cu_rows[b + 1]
            x = torch.randn((H, hi - lo, D), generator=g, device="cuda")
            along = torch.einsum("hrd,hd->hr", x, u[b])
            want = along.clamp(max=1.0)
            mask = _relevant(lens[b], keep[b], case["pool"], H, g)
            strong = 6.5 + torch.randn((H, lens[b]), generator=g, device="cuda").abs()
            strong[:, :SINKS] += 3.0
            want[:, :lens[b]] = torch.where(mask, strong, want[:, :lens[b]])
            x += (want - along)[:, :, None] * u[b][:, None, :]
            k[l, :, lo:hi] = x.to(dt)
        v[l].normal_(generator=g)
    s = {"case": case, "ctx": ctx, "cu_rows": cu_rows, "lens": lens, "keep": keep, "cu_prompt": cu_prompt}
    where = "cuda"
    if case["entry"] == "host":
        q, k, v = (t.cpu().pin_memory() for t in (q, k, v))
        where = "cpu"

    def out(*shape, dtype=dt):
        t = torch.zeros(shape, dtype=dtype, device=where)
        return t.pin_memory() if where == "cpu" else t

    s["k_out"], s["v_out"] = out(n, H, KT, D), out(n, H, KT, D)
    s["idx"] = out(n, H, KT, dtype=torch.int32)
    if case["entry"] == "evict":
        s["scores"] = out(H, sum(lens), dtype=torch.float32)
        s["q"], s["k"], s["v"] = q[0], k[0], v[0]
    elif case["entry"] == "steps":
        s["scores"] = out(H, sum(lens), dtype=torch.float32)
        s["q"], s["k"], s["v"], s["q_rot"] = q[0], k[0], v[0], torch.empty_like(q_rot)
        s["lse"] = torch.empty((B, Hq, N), dtype=torch.float32, device="cuda")
        # the prefill attention has these at hand; here the library's first sweep writes them once
        dq.dapq_score(ctx.handle, q_rot, s["k"], cu_rows, lens, s["scores"], lse_out=s["lse"])
    else:
        s["q"], s["k"], s["v"] = list(q.unbind(0)), list(k.unbind(0)), list(v.unbind(0))
        s["k_list"], s["v_list"], s["i_list"] = (list(s[x].unbind(0)) for x in ("k_out", "v_out", "idx"))
    dq.dapq_poll_status(ctx.handle)
    return s


# --------------------------------------------------------------------------------------------- pass
def run(s):
    h, cu, lens, keep = s["ctx"].handle, s["cu_rows"], s["lens"], s["keep"]
    entry = s["case"]["entry"]
    if entry == "evict":
        dq.dapq_evict(h, s["q"], s["k"], s["v"], cu, lens, keep, s["k_out"][0], s["v_out"][0], s["idx"][0], s["scores"])
    elif entry == "steps":
        dq.dapq_rope_pseudo_q(h, s["q"], lens, s["q_rot"])
        dq.dapq_score(h, s["q_rot"], s["k"], cu, lens, s["scores"], lse_in=s["lse"])
        dq.dapq_topk_select(h, s["scores"], s["cu_prompt"], keep, s["idx"][0])
        dq.dapq_compact_kv(h, s["k"], s["v"], cu, lens, s["idx"][0], keep, s["k_out"][0], s["v_out"][0])
    else:
        call = dq.dapq_evict_layers_host if entry == "host" else dq.dapq_evict_layers
        call(h, s["q"], s["k"], s["v"], cu, lens, keep, s["k_list"], s["v_list"], s["i_list"])
    out = {"k": s["k_out"], "v": s["v_out"], "idx": s["idx"]}
    if "scores" in s:
        out["scores"] = s["scores"]
    return out


def _rotate(q, lens, case):
    """Pseudo queries [B, Hq, N, d] at positions L_b + i, rotate-half pairs, in 64 bits."""
    c = torch.arange(D // 2, dtype=torch.float64, device="cuda")
    theta = case["rope_base"] ** (-2.0 * c / D) if case["rope"] == "plain" else None
    if theta is None:                                    # the Llama-3.1 frequencies: base 5e5, factor 8, 1 and 4, 8192
        theta = 5.0e5 ** (-2.0 * c / D)
        turns = 8192 * theta / (2.0 * math.pi)
        mix = (turns - 1.0) / 3.0
        theta = torch.where(turns > 4.0, theta, torch.where(turns < 1.0, theta / 8.0, (1.0 - mix) * theta / 8.0 + mix * theta))
    start = torch.tensor(lens, dtype=torch.float64, device="cuda")
    at = start[:, None] + torch.arange(q.shape[2], dtype=torch.float64, device="cuda")
    angle = (at[:, :, None] * theta)[:, None]
    cos, sin, (x, y) = angle.cos(), angle.sin(), q.double().split(D // 2, dim=3)
    return torch.cat([x * cos - y * sin, y * cos + x * sin], dim=3)


def exact(case, seed):
    """The same pass in 64 bits: softmax over the prompt and the synthetic keys that a pseudo query sees,
    summed per KV head; the best rows in ascending order."""
    s = prepare(case, seed)
    lens, keep, cu, H, N = s["lens"], s["keep"], s["cu_rows"], case["kv_heads"], case["window"]
    one = case["entry"] in ("evict", "steps")
    out = {"k": torch.zeros_like(s["k_out"]), "v": torch.zeros_like(s["v_out"]), "idx": torch.zeros_like(s["idx"])}
    if one:
        out["scores"] = torch.zeros((H, sum(lens)), dtype=torch.float64, device="cuda")
    for l, (q, k, v) in enumerate([(s["q"], s["k"], s["v"])] if one else zip(s["q"], s["k"], s["v"])):
        q, k, v = q.cuda(), k.cuda(), v.cuda()
        rot = _rotate(q, lens, case)
        if case["entry"] == "steps":
            rot = rot.to(q.dtype).double()               # the step between hands them on in the cache's type
        at, at_p = 0, 0
        for L, K, lo, qb in zip(lens, keep, cu, rot):
            for h in range(H):
                logits = qb.view(H, -1, D)[h] @ k[h, lo:lo + L + N].double().T / math.sqrt(D)
                unseen = torch.ones((N, N), dtype=torch.bool, device="cuda").triu(1)
                logits.view(-1, N, L + N)[:, :, L:].masked_fill_(unseen, -math.inf)
                score = logits.softmax(1)[:, :L].sum(0)
                chosen = score
                if case["pool"]:
                    chosen = torch.nn.functional.max_pool1d(score[None], case["pool"], 1, case["pool"] // 2)[0]
                idx = chosen.sort(descending=True, stable=True).indices[:K].sort().values
                out["idx"][l, h, at:at + K] = idx
                out["k"][l, h, at:at + K] = k[h, lo + idx]
                out["v"][l, h, at:at + K] = v[h, lo + idx]
                if one:
                    out["scores"][h, at_p:at_p + L] = score
            at, at_p = at + K, at_p + L
    return out


def work(case):
    """K once, the kept rows of K and V read and written, queries, indices, scores; one contraction of the
    pseudo queries with every key (the exponentials are not counted)."""
    lens, keep = _sizes(case)
    e = 2 if case["dtype"] == "bf16" else 4
    H, Hq, N, n = case["kv_heads"], case["heads"], case["window"], case["layers"]
    rows = sum(lens) + N * len(lens)
    per = H * rows * D * e + 4 * H * sum(keep) * D * e + len(lens) * Hq * N * D * e + 4 * H * sum(keep)
    if case["entry"] in ("evict", "steps"):
        per += 4 * H * sum(lens)
    return {"bytes": n * per, "flops": n * 2 * Hq * N * D * rows}


def tolerance(case):
    """Kept rows and indices do not depend on the rounding of the scores.  The scores themselves, about four
    times their distance from float64 on these inputs: 2.9e-5 (largest 1e-4) where the rotated queries are
    rounded to fp16; 3.6e-6 (1.5e-5) where the caller's bf16 queries enter the products exactly; 3.2e-7
    (2.3e-6) where queries, keys and sums are fp32 (fp32 caches, and fewer than 64 query rows per KV head)."""
    if case["entry"] in ("layers", "host"):
        return "exact"
    if case["dtype"] == "f32" or case["heads"] // case["kv_heads"] * case["window"] < 64:
        return {"rel": 1.3e-6, "max": 1e-5, "differ": 0.0}
    if case["entry"] == "steps":
        return {"rel": 1.5e-5, "max": 6e-5, "differ": 0.0}
    return {"rel": 1.2e-4, "max": 4e-4, "differ": 0.0}
