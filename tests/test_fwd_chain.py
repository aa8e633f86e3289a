"""The forward that goes on from item to item in one CTA (needs a B200): large packed batches of short ragged traces.

Single heads of odd groups among pairs (their two streams are merged through the memory of the K/V ring while the next item's
loads wait for it), rows without keys between others, key slots with their own intervals, empty traces.  Compared with the
definition in fp64 (roundings: those of the other forward tests, 2e-2 and 5e-3), and bit for bit with the traces on their own, which
take a CTA per item: a row's arithmetic does not depend on its neighbours.
"""
import numpy as np
import pytest
import torch

from paper_2609_35750_b200 import binding as B
from paper_2609_35750_b200 import workloads as W

pytestmark = pytest.mark.gpu
INF = 2 ** 31 - 1
LENS = [int(x) for x in np.random.default_rng(1).permutation(np.concatenate([np.linspace(1, 900, 90).astype(int), [0, 0, 1, 128, 129, 1024]]))]


def _chained(lens, Hq, Hkv):
    """The condition of the dispatch: traces of 2048 tokens or less on average and more than two waves of CTAs, or 4096 and six."""
    ctas = (sum(lens) // 128 + len(lens)) * Hkv * ((Hq // Hkv + 1) // 2)
    mean = sum(lens) // len(lens)
    return (mean <= 2048 and ctas > 2 * 148) or (mean <= 4096 and ctas > 6 * 148)


def _evict(lens, rule, seed):
    r = np.random.default_rng(seed)
    out = []
    for b, T in enumerate(lens):
        if T == 0:
            continue
        kind = ("summary", "turns")[b % 2] if rule == "mixed" else rule
        if kind == "tokens":
            out.append(W.fine_grained_evict_at(T, max(1, T // 24), r, T / 16.0))
        elif kind == "summary":
            out.append(W.summary_evict_at(T, max(1, T // 16), r.integers(max(1, T // 16), max(2, T // 8 + 1), size=64), max(1, T // 64)))
        else:
            out.append(W.keep_last_k_evict_at(T, max(1, T // 16), r.integers(2, max(3, T // 16 + 2), size=T), 4))
    return np.concatenate(out).astype(np.int32)


def _inputs(lens, Hq, Hkv, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda h: torch.randn((sum(lens), h, d), generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    return rnd(Hq), rnd(Hkv), rnd(Hkv)


def _definition(q, k, v, first, evict):
    """One trace: query i sees slot j iff first[j] <= i < evict[j]."""
    G = q.shape[1] // k.shape[1]
    i = torch.arange(q.shape[0], device="cuda")[:, None]
    seen = (first[None] <= i) & (i < evict[None])
    s = torch.einsum("ihd,jhd->hij", q.double(), k.double().repeat_interleave(G, 1)) * q.shape[2] ** -0.5
    s = s.masked_fill(~seen, -float("inf"))
    lse = torch.logsumexp(s, 2)
    p = torch.exp(s - lse[..., None]).nan_to_num(0.0)                    # a row that sees nothing
    return torch.einsum("hij,jhd->ihd", p, v.double().repeat_interleave(G, 1)), lse


def _compare(lens, cu, out, lse, ref_of):
    err = size = 0.0
    for b, T in enumerate(lens):
        if T == 0:
            continue
        a = int(cu[b])
        ro, rl = ref_of(b, slice(a, a + T))
        got, gl = out[a:a + T].double(), lse[:, a:a + T].double()
        assert torch.isfinite(got).all() and (got - ro).abs().max() <= 2e-2, (b, T)
        none = rl == -float("inf")
        assert torch.equal(none, gl == -float("inf")) and ((gl - rl)[~none].abs() <= 1e-3).all(), (b, T)
        err += float((got - ro).pow(2).sum())
        size += float(ro.pow(2).sum())
    assert err <= (5e-3) ** 2 * size


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("Hq,Hkv,rule", [(4, 4, "mixed"), (6, 2, "tokens"), (7, 1, "mixed"), (14, 2, "mixed"), (8, 2, "tokens")])
def test_chained_forward(Hq, Hkv, rule, d):
    assert _chained(LENS, Hq, Hkv)
    ev = torch.from_numpy(_evict(LENS, rule, Hq)).cuda()
    cu = np.concatenate([[0], np.cumsum(LENS)]).astype(np.int32)
    q, k, v = _inputs(LENS, Hq, Hkv, d, Hq + d)
    meta = B.kvs_mask_meta(ev, torch.from_numpy(cu).cuda(), max(LENS))
    out, lse = B.kvs_attn_fwd(q, k, v, meta, len(LENS), max(LENS))
    assert B.kvs_device_status(meta) == B.KVS_OK
    j = torch.arange(max(LENS), device="cuda")
    _compare(LENS, cu, out, lse, lambda b, z: _definition(q[z], k[z], v[z], j[:LENS[b]], ev[z]))
    for b in range(0, len(LENS), 7):
        T, z = LENS[b], slice(int(cu[b]), int(cu[b]) + LENS[b])
        if T == 0:
            continue
        assert not _chained([T], Hq, Hkv)
        one = B.kvs_mask_meta(ev[z].contiguous(), torch.tensor([0, T], dtype=torch.int32, device="cuda"), T)
        o, m = B.kvs_attn_fwd(q[z].contiguous(), k[z].contiguous(), v[z].contiguous(), one, 1, T)
        assert torch.equal(o, out[z]) and torch.equal(m, lse[:, z]), (b, T)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("Hq,Hkv", [(4, 4), (7, 1), (8, 2)])
def test_chained_rows_without_keys(Hq, Hkv, d):
    # the evicted keys alone: the first rows of every trace, and whole traces, see nothing
    assert _chained(LENS, Hq, Hkv)
    ev = torch.from_numpy(_evict(LENS, "mixed", 5)).cuda()
    cu = np.concatenate([[0], np.cumsum(LENS)]).astype(np.int32)
    q, k, v = _inputs(LENS, Hq, Hkv, d, d)
    cud, longest = torch.from_numpy(cu).cuda(), max(LENS)
    student, evicted = B.kvs_mask_meta(ev, cud, longest), B.kvs_mask_meta_evicted(ev, cud, longest)
    out, lse = B.kvs_attn_fwd(q, k, v, evicted, len(LENS), longest)
    never = torch.full((longest,), INF, device="cuda")
    _compare(LENS, cu, out, lse, lambda b, z: _definition(q[z], k[z], v[z], ev[z], never[:LENS[b]]))
    _, _, out_t, lse_t = B.kvs_attn_fwd_dual(q, k, v, student, evicted, len(LENS), longest)
    j = torch.arange(longest, device="cuda")
    _compare(LENS, cu, out_t, lse_t, lambda b, z: _definition(q[z], k[z], v[z], j[:LENS[b]], never[:LENS[b]]))


@pytest.mark.parametrize("Hq,Hkv,d", [(7, 1, 128), (4, 4, 64)])
def test_chained_key_slots(Hq, Hkv, d):
    assert _chained(LENS, Hq, Hkv)
    ev = torch.from_numpy(_evict(LENS, "tokens", 9)).cuda()
    cu = np.concatenate([[0], np.cumsum(LENS)]).astype(np.int32)
    q, k, v = _inputs(LENS, Hq, Hkv, d, 2)
    cud, longest = torch.from_numpy(cu).cuda(), max(LENS)
    perm, first, evict = B.kvs_reorder_keys(ev, cud, longest, 300)
    meta = B.kvs_mask_meta_keys(first, evict, cud, longest)
    out, lse = B.kvs_attn_fwd(q, B.kvs_permute_rows(k, perm), B.kvs_permute_rows(v, perm), meta, len(LENS), longest)
    j = torch.arange(longest, device="cuda")
    _compare(LENS, cu, out, lse, lambda b, z: _definition(q[z], k[z], v[z], j[:LENS[b]], ev[z]))


def test_chained_longer_traces():
    Hq, Hkv, d, lens = 9, 3, 128, [4096, 2111, 4095, 3000, 4001, 4000, 3999, 3500, 2900]      # pairs and single heads
    assert _chained(lens, Hq, Hkv) and sum(lens) // len(lens) > 2048
    ev = torch.from_numpy(_evict(lens, "mixed", 3)).cuda()
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    q, k, v = _inputs(lens, Hq, Hkv, d, 4)
    meta = B.kvs_mask_meta(ev, torch.from_numpy(cu).cuda(), max(lens))
    out, lse = B.kvs_attn_fwd(q, k, v, meta, len(lens), max(lens))
    assert B.kvs_device_status(meta) == B.KVS_OK
    for b, T in enumerate(lens):
        z = slice(int(cu[b]), int(cu[b]) + T)
        assert not _chained([T], Hq, Hkv)
        one = B.kvs_mask_meta(ev[z].contiguous(), torch.tensor([0, T], dtype=torch.int32, device="cuda"), T)
        o, m = B.kvs_attn_fwd(q[z].contiguous(), k[z].contiguous(), v[z].contiguous(), one, 1, T)
        assert torch.equal(o, out[z]) and torch.equal(m, lse[:, z]), (b, T)
