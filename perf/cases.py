"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values; `kind` says which path it takes:

  step         a trainer's attention step on a packed batch of compacted rollouts: mask metadata, forward,
               backward.  layout "split" takes q, k, v as tensors of their own, "packed" as the projection's
               output, "rope" rotates q and k first and rotates dq and dk back, "slots" sorts the keys by
               eviction step (token-level eviction) and brings k, v, dk, dv into and out of that order
  score        mask metadata and forward alone: log-probabilities of rollouts under the current policy
  dual         student and teacher forward of self-distillation
  decode       one decode step of the rollout engine over a fragmented paged cache
  turn         one generated turn: append and decode token by token, then the oldest turn leaves the cache
  host         the step from page-locked host buffers, results back on the host

Traces follow the repository's own retention rules (workloads.py): "summary", "last_k" (keep the last k turns),
"mixed" (either, trace by trace), "tokens" (token-level).  Trace and cache lengths are a function of the case;
turn boundaries, page tables and all values are drawn from the seed.
"""
import math

import numpy as np
import torch

from paper_2609_35750_b200 import binding as B
from paper_2609_35750_b200 import workloads as W

# (query heads, KV heads, head_dim) of the models that the configurations describe, and one small one
HEADS = ((4, 4, 64), (16, 4, 64), (16, 2, 128), (28, 4, 128), (32, 8, 128), (64, 8, 128))
MOST_FLOPS = 6e13               # a drawn step stays below the largest listed one


def listed():
    return [
        # one short tool-use rollout, the smallest configuration: latency and launches
        dict(name="step_tiny", kind="step", rule="summary", traces=1, shortest=1024, longest=1024, Hq=4, Hkv=4, d=64, grad="bf16", layout="split"),
        # a micro-batch of many short ragged rollouts packed back to back, fp32 gradients for accumulation
        dict(name="step_short_packed", kind="step", rule="mixed", traces=96, shortest=60, longest=900, Hq=16, Hkv=2, d=128, grad="fp32", layout="split"),
        # the 7B-class configuration: one summary-compacted rollout per micro-batch, odd GQA group, rotary embedding around it
        dict(name="step_7b_rope", kind="step", rule="summary", traces=1, shortest=32768, longest=32768, Hq=28, Hkv=4, d=128, grad="bf16", layout="rope"),
        # the headline configuration at full size: two long agentic rollouts that keep their last four turns
        dict(name="step_keep_last_4", kind="step", rule="last_k", traces=2, shortest=65536, longest=65536, Hq=32, Hkv=8, d=128, grad="bf16", layout="split"),
        # ragged rollouts of both retention rules on the projection's packed layout
        dict(name="step_varlen_packed", kind="step", rule="mixed", traces=12, shortest=1500, longest=12000, Hq=32, Hkv=8, d=128, grad="bf16", layout="packed"),
        # token-level eviction with sorted key slots, wide group
        dict(name="step_token_level", kind="step", rule="tokens", traces=1, shortest=24576, longest=24576, Hq=64, Hkv=8, d=128, grad="bf16", layout="slots"),
        # scoring one medium rollout: a forward that does not fill the chip many times over
        dict(name="score_medium", kind="score", rule="last_k", traces=1, shortest=7000, longest=7000, Hq=32, Hkv=8, d=128),
        # self-distillation forward
        dict(name="dual_distill", kind="dual", rule="mixed", traces=3, shortest=9000, longest=17000, Hq=32, Hkv=8, d=128),
        # a few sequences generating one tool-use turn: latency of append + decode, then the eviction of a turn
        dict(name="turn_few_seqs", kind="turn", seqs=4, shortest=1500, longest=5000, page=16, turn=16, Hq=32, Hkv=8, d=128),
        # a full rollout batch with ragged live caches in 16-token pages
        dict(name="decode_wide_ragged", kind="decode", seqs=48, shortest=1000, longest=16000, page=16, Hq=32, Hkv=8, d=128),
        # the engine with one-token pages on the 7B-class heads, every cache near its budget
        dict(name="decode_token_pages", kind="decode", seqs=64, shortest=6500, longest=7168, page=1, Hq=28, Hkv=4, d=128),
        # a trainer without device tensors: the whole step through host memory
        dict(name="host_varlen", kind="host", rule="mixed", traces=8, shortest=1500, longest=6000, Hq=32, Hkv=8, d=128, grad="bf16"),
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    kind = rng.choice(("step", "step", "step", "step", "score", "dual", "decode", "decode", "turn", "host"))
    Hq, Hkv, d = rng.choice(HEADS)
    if kind in ("decode", "turn"):
        longest = log(300, 24000 if kind == "decode" else 8000)
        case = dict(kind=kind, seqs=log(1, 64 if kind == "decode" else 8), shortest=max(1, int(longest * rng.uniform(0.1, 1.0))), longest=longest,
                    page=rng.choice((1, 16, 16, 16, 64)), Hq=Hq, Hkv=Hkv, d=d)
        if kind == "turn":
            case["turn"] = 16
            case["page"] = min(case["page"], 16)
        return case
    while True:
        longest = log(40, 65536)
        rule = rng.choice(("summary", "last_k", "mixed"))
        case = dict(kind=kind, rule=rule, traces=log(1, 128), shortest=max(1, int(longest * rng.uniform(0.1, 1.0))), longest=longest,
                    Hq=Hq, Hkv=Hkv, d=d)
        if kind in ("step", "host"):
            case["grad"] = rng.choice(("bf16", "bf16", "fp32"))
        if kind == "step":
            case["layout"] = rng.choice(("split", "packed", "rope", "slots"))
            if case["layout"] == "slots":
                case["rule"] = "tokens"
        total = int(lengths(case).sum())
        most = {"step": 131072, "host": 30000 * 32 // Hq}.get(kind, 40000)
        if total > most or work(case)["flops"] > MOST_FLOPS * (1.0 if kind == "step" else 0.2):
            continue
        return case


# ---- shapes and masks ------------------------------------------------------------------------------

def lengths(case):
    """Trace (or live cache) lengths: evenly spaced over the case's range, in a fixed shuffled order."""
    n = case["traces"] if "traces" in case else case["seqs"]
    x = np.linspace(case["shortest"], case["longest"], n + 2)[1:-1] if n > 1 else np.array([case["longest"]], dtype=float)
    return np.random.RandomState(n).permutation(np.maximum(1, np.rint(x)).astype(np.int64))


def eviction(case, seed):
    """evict_at of every trace, packed.  Prompt, turn and segment lengths scale with the trace like those of the
    configurations (a 64k trace has a 4k prompt and turns of 256 to 2048 tokens)."""
    r = np.random.default_rng([seed, 71])
    traces = []
    for b, T in enumerate(lengths(case)):
        T = int(T)
        rule = case["rule"]
        if rule == "mixed":
            rule = "summary" if b % 2 else "last_k"
        if rule == "tokens":
            ev = W.fine_grained_evict_at(T, max(1, T // 24), r, T / 16.0)
        elif rule == "summary":
            work, summary = max(1, T // 8), max(1, T // 64)
            ev = W.summary_evict_at(T, max(1, T // 16), r.integers(max(1, work // 2), work + 1, size=64), summary)
        else:
            longest = 2048 if T >= 32768 else max(8, T // 16)
            turns = r.integers(max(1, longest // 8), longest + 1, size=T // max(1, longest // 8) + 2)
            ev = W.keep_last_k_evict_at(T, T // 16, turns, 4)
        traces.append(ev)
    return np.concatenate(traces)


def pairs_of(case):
    """Unmasked (query, key) pairs under the mask, and under plain causal attention (one seed's mask: they differ little)."""
    lens, ev, at, kept = lengths(case), eviction(case, 0).astype(np.int64), 0, 0
    for T in lens:
        e = ev[at:at + T]
        kept += int((np.minimum(e, T) - np.arange(T)).sum())
        at += T
    return kept, int((lens * (lens + 1) // 2).sum())


# ---- what a user's program has in hand ---------------------------------------------------------------

def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    normal = lambda *shape: torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    s = dict(case)
    if case["kind"] in ("decode", "turn"):
        return prepare_cache(case, seed, s, normal)
    lens = lengths(case)
    Hq, Hkv, d = case["Hq"], case["Hkv"], case["d"]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    total, longest = int(cu[-1]), int(lens.max())
    evict = eviction(case, seed)
    s.update(batch=len(lens), longest=longest, scale=0.0)
    if case.get("layout") == "packed":
        s["qkv"] = normal(total, Hq + 2 * Hkv, d)
    else:
        s.update(q=normal(total, Hq, d), k=normal(total, Hkv, d), v=normal(total, Hkv, d))
    if case["kind"] in ("step", "host"):
        s["dout"] = normal(total, Hq, d)
        s["grad_dtype"] = B.GRAD_FP32 if case["grad"] == "fp32" else B.GRAD_BF16
    if case["kind"] == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        room = lambda *shape, dtype=torch.bfloat16: torch.empty(shape, dtype=dtype, pin_memory=True)  # noqa: E731
        gdt = torch.float32 if case["grad"] == "fp32" else torch.bfloat16
        for name in ("q", "k", "v", "dout"):
            s[name] = pin(s[name])
        s.update(evict=torch.from_numpy(evict).pin_memory(), cu=torch.from_numpy(cu), out=room(total, Hq, d),
                 lse=room(Hq, total, dtype=torch.float32), dq=room(total, Hq, d, dtype=gdt), dk=room(total, Hkv, d, dtype=gdt),
                 dv=room(total, Hkv, d, dtype=gdt))
        s["arena"] = torch.empty(B.kvs_host_arena_bytes(s["batch"], total, longest, Hq, Hkv, d, s["grad_dtype"]), dtype=torch.uint8, device="cuda")
        return s
    s.update(evict=torch.from_numpy(evict).cuda(), cu=torch.from_numpy(cu).cuda())
    s["meta"] = torch.empty(B.kvs_mask_meta_bytes(s["batch"], total, longest), dtype=torch.uint8, device="cuda")
    if case["kind"] == "dual":
        s["meta_evicted"] = torch.empty_like(s["meta"])
    if case["kind"] == "step":
        s["workspace"] = torch.empty(B.kvs_attn_bwd_workspace_bytes(total, Hq, Hkv, d, s["grad_dtype"]), dtype=torch.uint8, device="cuda")
    return s


def prepare_cache(case, seed, s, normal):
    """A paged cache as an engine has it after many evictions: the pages of every sequence scattered over the pool."""
    n, page, Hq, Hkv, d = lengths(case), case["page"], case["Hq"], case["Hkv"], case["d"]
    if case["kind"] == "turn":
        n = -(-n // page) * page                          # turns are padded to whole pages
    used = -(-n // page)
    spare = -(-case.get("turn", 0) // page) + 1
    max_pages = int(used.max()) + spare
    pool = int(used.sum()) + spare * len(n)
    cache = B.PagedCache(pool, page, len(n), max_pages, Hkv, d)
    cache.k_cache.copy_(normal(*cache.k_cache.shape))
    cache.v_cache.copy_(normal(*cache.v_cache.shape))
    order = np.random.default_rng([seed, 73]).permutation(pool).astype(np.int32)
    table, at = np.zeros((len(n), max_pages), dtype=np.int32), 0
    for i, u in enumerate(used):
        table[i, :u] = order[at:at + u]
        at += u
    free = np.concatenate([[pool - at, 0, 0, 0], order[at:], np.zeros(at, dtype=np.int32)]).astype(np.int32)
    cache.block_table.copy_(torch.from_numpy(table))
    cache.n_tokens.copy_(torch.from_numpy(n.astype(np.int32)))
    cache.free_list.copy_(torch.from_numpy(free))
    s.update(cache=cache, most=int(n.max()) + case.get("turn", 0))
    if case["kind"] == "decode":
        s["q"] = normal(len(n), Hq, d)
    else:
        s.update(q=normal(case["turn"], len(n), Hq, d), k=normal(case["turn"], len(n), Hkv, d), v=normal(case["turn"], len(n), Hkv, d))
        gone = [(i, 0, case["turn"] // page) for i in range(len(n))]
        s["gone"] = torch.tensor(gone, dtype=torch.int32, device="cuda")
    return s


# ---- one pass ------------------------------------------------------------------------------------------

def run(s):
    return {"step": run_step, "score": run_score, "dual": run_dual, "decode": run_decode, "turn": run_turn, "host": run_host}[s["kind"]](s)


def run_step(s):
    batch, longest, grad = s["batch"], s["longest"], s["grad_dtype"]
    if s["layout"] == "packed":
        meta = B.kvs_mask_meta(s["evict"], s["cu"], longest, s["meta"])
        out, lse = B.kvs_attn_fwd_packed(s["qkv"], meta, batch, longest, s["Hq"], s["Hkv"], s["scale"])
        dqkv = B.kvs_attn_bwd_packed(s["dout"], s["qkv"], out, lse, meta, batch, longest, s["Hq"], s["Hkv"], s["scale"], grad, workspace=s["workspace"])
        return out, lse, dqkv
    q, k, v = s["q"], s["k"], s["v"]
    if s["layout"] == "slots":
        perm, first, evict = B.kvs_reorder_keys(s["evict"], s["cu"], longest, min(4096, longest))
        meta = B.kvs_mask_meta_keys(first, evict, s["cu"], longest, s["meta"])
        k, v = B.kvs_permute_rows(k, perm), B.kvs_permute_rows(v, perm)
    else:
        meta = B.kvs_mask_meta(s["evict"], s["cu"], longest, s["meta"])
        if s["layout"] == "rope":
            q, k = B.kvs_rope_qk(q, k, s["cu"])
    out, lse = B.kvs_attn_fwd(q, k, v, meta, batch, longest, s["scale"])
    dq, dk, dv = B.kvs_attn_bwd(s["dout"], q, k, v, out, lse, meta, batch, longest, s["scale"], grad, workspace=s["workspace"])
    if s["layout"] == "rope":
        dq, dk = B.kvs_rope_qk(dq, dk, s["cu"], inverse=True, q_out=dq, k_out=dk)
    if s["layout"] == "slots":
        dk, dv = B.kvs_permute_rows(dk, perm, inverse=True), B.kvs_permute_rows(dv, perm, inverse=True)
    return out, lse, dq, dk, dv


def run_score(s):
    meta = B.kvs_mask_meta(s["evict"], s["cu"], s["longest"], s["meta"])
    return B.kvs_attn_fwd(s["q"], s["k"], s["v"], meta, s["batch"], s["longest"], s["scale"])


def run_dual(s):
    student = B.kvs_mask_meta(s["evict"], s["cu"], s["longest"], s["meta"])
    evicted = B.kvs_mask_meta_evicted(s["evict"], s["cu"], s["longest"], s["meta_evicted"])
    return B.kvs_attn_fwd_dual(s["q"], s["k"], s["v"], student, evicted, s["batch"], s["longest"], s["scale"])


def run_decode(s):
    return s["cache"].decode(s["q"], max_tokens=s["most"])


def run_turn(s):
    """Every sequence generates `turn` tokens; then its oldest pages, as many as the turn filled, are evicted.  The cache
    is as long afterwards as before.  Which page a token went to depends on the order in which the sequences took theirs,
    so the outputs are what the caller sees: the attention of every token and the live lengths."""
    cache, got = s["cache"], []
    for t in range(s["turn"]):
        cache.append(s["k"][t], s["v"][t])
        got.append(cache.decode(s["q"][t], max_tokens=s["most"]))
    cache.evict(s["gone"])
    return got, cache.n_tokens


def run_host(s):
    B.kvs_attn_fwd_bwd_host(s["evict"], s["cu"], s["q"], s["k"], s["v"], s["dout"], s["longest"], s["scale"], s["grad_dtype"],
                            s["out"], s["lse"], s["dq"], s["dk"], s["dv"], s["arena"])
    return s["out"], s["lse"], s["dq"], s["dk"], s["dv"]


# ---- what a pass cannot do without -----------------------------------------------------------------------

def work(case):
    Hq, Hkv, d = case["Hq"], case["Hkv"], case["d"]
    n = lengths(case)
    if case["kind"] in ("decode", "turn"):
        steps = case.get("turn", 1)
        if case["kind"] == "turn":
            n = -(-n // case["page"]) * case["page"]
        live = int(n.sum()) * steps + (len(n) * steps * (steps + 1) // 2 if case["kind"] == "turn" else 0)
        rows = len(n) * steps
        return {"bytes": 4 * d * Hkv * live + rows * Hq * (4 * d + 4) + (8 * d * Hkv * rows if case["kind"] == "turn" else 0), "flops": 4 * d * Hq * live}
    total = int(n.sum())
    kept, causal = pairs_of(case)
    per_q, per_kv = total * Hq * d, total * Hkv * d
    io = 4 * total + 2 * (per_q + 2 * per_kv) + 2 * per_q + 4 * total * Hq           # mask, q, k, v, out, lse
    if case["kind"] == "score":
        return {"bytes": io, "flops": 4 * d * Hq * kept}
    if case["kind"] == "dual":
        return {"bytes": io + 2 * per_q + 4 * total * Hq, "flops": 4 * d * Hq * causal}      # the student's pairs are among the teacher's
    size = 4 if case["grad"] == "fp32" else 2
    return {"bytes": io + 2 * per_q + size * (per_q + 2 * per_kv), "flops": 14 * d * Hq * kept}


def tolerance(case):
    """bf16 operands and results with fp32 sums.  Against 64-bit sums out, dq, dk, dv are off by 1.6e-3 to 2.1e-3 in the
    2-norm (rounding of the probabilities, the score gradients and the output to 8 bits); two such results differ by
    up to 3e-3 from one another.  Single elements reach about six standard deviations, more on the first keys of a trace."""
    if case["kind"] in ("decode", "turn"):
        return {"rel": 8e-3, "max": 0.1}
    return {"rel": 8e-3, "max": 0.3}


# ---- the same outputs in 64 bits --------------------------------------------------------------------------

def exact(case, seed):
    """What run() returns, as dense attention over the visible keys gives it in float64 (torch on the GPU)."""
    s = prepare(case, seed)
    wide = lambda t: t.cuda().double()  # noqa: E731
    scale = case["d"] ** -0.5
    if case["kind"] in ("decode", "turn"):
        return exact_cache(case, s, wide, scale)
    evict, cu = s["evict"].cuda(), s["cu"].tolist()
    if case.get("layout") == "packed":
        q, k, v = wide(s["qkv"]).split((case["Hq"], case["Hkv"], case["Hkv"]), dim=1)
    else:
        q, k, v = wide(s["q"]), wide(s["k"]), wide(s["v"])
    if case.get("layout") == "rope":
        q, k = rotated(q, cu, 1), rotated(k, cu, 1)
    if case["kind"] in ("score", "dual"):
        got = attention64(q, k, v, evict, cu, scale)[:2]
        return got if case["kind"] == "score" else got + attention64(q, k, v, torch.full_like(evict, 2 ** 31 - 1), cu, scale)[:2]
    out, lse, dq, dk, dv = attention64(q, k, v, evict, cu, scale, s["dout"].cuda())
    if case.get("layout") == "packed":
        return out, lse, torch.cat((dq, dk, dv), dim=1)
    if case.get("layout") == "rope":
        dq, dk = rotated(dq, cu, -1), rotated(dk, cu, -1)
    return out, lse, dq, dk, dv


def attention64(q, k, v, evict, cu, scale, dout=None, rows=1024):
    (total, Hq, d), Hkv = q.shape, k.shape[1]
    G = Hq // Hkv
    out, lse = torch.empty_like(q), q.new_empty(Hq, total)
    dq, dk, dv = (None, None, None) if dout is None else (torch.zeros_like(q), torch.zeros_like(k), torch.zeros_like(v))
    for a, z in zip(cu[:-1], cu[1:]):
        for i0 in range(a, z, rows):
            i1 = min(z, i0 + rows)
            keys = a + torch.nonzero(evict[a:i1] > i0 - a).squeeze(1)          # any of these queries may see them
            i = torch.arange(i0, i1, device=q.device)
            hidden = (keys > i[:, None]) | (evict[keys] <= i[:, None] - a)
            for g in range(Hkv):
                h = slice(g * G, (g + 1) * G)
                qq, kk, vv = q[i0:i1, h].transpose(0, 1).reshape(-1, d), k[keys, g], v[keys, g]
                s = (qq @ kk.T).mul_(scale).view(G, i1 - i0, -1).masked_fill_(hidden, -math.inf)
                top = torch.logsumexp(s, dim=2)
                p = s.sub_(top[..., None]).exp_().view(len(qq), -1)
                o = p @ vv
                lse[h, i0:i1] = top
                out[i0:i1, h] = o.view(G, -1, d).transpose(0, 1)
                if dout is not None:
                    do = dout[i0:i1, h].double().transpose(0, 1).reshape(-1, d)
                    dv[:, g].index_add_(0, keys, p.T @ do)
                    ds = (do @ vv.T).sub_((do * o).sum(1, keepdim=True)).mul_(p).mul_(scale)
                    dq[i0:i1, h] = (ds @ kk).view(G, -1, d).transpose(0, 1)
                    dk[:, g].index_add_(0, keys, ds.T @ qq)
    return out, lse, dq, dk, dv


def rotated(x, cu, sign):
    """Rotary embedding with the position in the trace, halves of the head paired (sign -1: its transpose)."""
    half = x.shape[-1] // 2
    at = torch.cat([torch.arange(z - a, device=x.device) for a, z in zip(cu[:-1], cu[1:])]).double()
    angle = at[:, None] * 10000.0 ** (-torch.arange(half, device=x.device).double() / half)
    c, n = angle.cos()[:, None], sign * angle.sin()[:, None]
    lo, hi = x[..., :half], x[..., half:]
    return torch.cat((lo * c - hi * n, hi * c + lo * n), dim=-1)


def exact_cache(case, s, wide, scale):
    cache, Hkv, d = s["cache"], case["Hkv"], case["d"]
    steps = case.get("turn", 1)
    q = wide(s["q"]).view(steps, -1, Hkv, case["Hq"] // Hkv, d)
    out, lse = torch.empty_like(q), q.new_empty(q.shape[:-1])
    for b, n in enumerate(cache.n_tokens.tolist()):
        pages = cache.block_table[b, :-(-n // case["page"])].long()
        k, v = (wide(c[pages]).reshape(-1, Hkv, d)[:n].transpose(0, 1) for c in (cache.k_cache, cache.v_cache))
        for t in range(steps):
            if case["kind"] == "turn":
                k, v = torch.cat((k, wide(s["k"][t, b])[:, None]), dim=1), torch.cat((v, wide(s["v"][t, b])[:, None]), dim=1)
            score = q[t, b] @ k.transpose(1, 2) * scale
            lse[t, b] = torch.logsumexp(score, dim=2)
            out[t, b] = torch.softmax(score, dim=2) @ v
    got = [(o.flatten(1, 2), m.flatten(1, 2)) for o, m in zip(out, lse)]
    return got[0] if case["kind"] == "decode" else (got, cache.n_tokens)
