"""Metadata of small batches by one CTA, units and items that are chained in a CTA (needs a B200).

Up to 64 blocks and 5120 tokens the metadata is one kernel, above it is two: a batch at the line gives the same results, bit for bit, as the same
traces with one-token traces behind them.  Rows and whole key blocks (a workspace of the base size) are summed in the same order
on both sides, so out, lse, dk and dv are equal; dq is added in the order of arrival, fp32, each term at most 2^-24 off."""
import numpy as np
import pytest
import torch

from paper_2609_35750_b200 import binding as B
from paper_2609_35750_b200 import workloads as W

from .test_bwd_units import _backward, _base_bytes, _inputs, _same

pytestmark = pytest.mark.gpu


def _pass(ev, cu, longest, ts, Hq, general=None):
    q, k, v, do = ts
    batch = len(cu) - 1
    cud = torch.from_numpy(cu).cuda()
    meta = B.kvs_mask_meta_keys(*general, cud, longest) if general else B.kvs_mask_meta(ev, cud, longest)
    out, lse = B.kvs_attn_fwd(q, k, v, meta, batch, longest)
    ws = torch.empty(-(-(256 + 4 * q.shape[0] * Hq) // 256) * 256, dtype=torch.uint8, device="cuda")
    grads = B.kvs_attn_bwd(do, q, k, v, out, lse, meta, batch, longest, 0.0, B.GRAD_FP32, workspace=ws)
    assert B.kvs_device_status(meta) == B.KVS_OK and B.kvs_device_status(ws) == B.KVS_OK
    cls = B.kvs_mask_meta_export(meta, cu, q.shape[0], longest)
    return (out, lse) + grads, cls


@pytest.mark.parametrize("lens", [[5120], [5121], [4993], [1], [80] * 64, [80] * 63 + [81], [127, 0, 129, 0, 0, 385, 1], [1024, 1025, 1, 3000], [1] * 62 + [129]])
def test_one_cta_equals_two_kernels(lens):
    Hq, Hkv, d = 2, 1, 64
    r = np.random.default_rng(len(lens))
    ev = np.concatenate([W.keep_last_k_evict_at(T, max(1, T // 16), r.integers(8, max(9, T // 8), size=T), 4) for T in lens if T])
    more = lens + [1] * 65
    total, all_tokens = sum(lens), sum(more)
    ev = torch.from_numpy(np.concatenate([ev, np.full(65, 2 ** 31 - 1, dtype=np.int32)]).astype(np.int32)).cuda()
    g = torch.Generator(device="cuda").manual_seed(total)
    ts = [torch.randn((all_tokens, h, d), generator=g, device="cuda", dtype=torch.bfloat16) for h in (Hq, Hkv, Hkv, Hq)]
    cu = np.concatenate([[0], np.cumsum(more)]).astype(np.int32)
    small, cls = _pass(ev[:total].clone(), cu[:len(lens) + 1].copy(), max(lens), [t[:total].clone() for t in ts], Hq)
    large, cls_l = _pass(ev, cu, max(lens), ts, Hq)
    for a, b in zip(cls, cls_l):
        assert np.array_equal(a, b[:len(a)])
    for name, a, b in zip(("out", "lse", "dq", "dk", "dv"), small, large):
        b = b[:, :total] if name == "lse" else b[:total]
        if name == "dq":
            assert (a - b).norm() <= 2.0 ** -24 * -(-max(lens) // 128) * max(1.0, b.norm().item()) * 4
        else:
            assert torch.equal(a, b), name


@pytest.mark.parametrize("Hq,Hkv,d", [(4, 4, 64), (4, 2, 128)])
def test_chained_units_with_key_blocks_that_nobody_sees(Hq, Hkv, d):
    # 300 traces of 300: several units a CTA; every third key block is seen by no query (no tiles, zero gradients), single keys
    # of others neither
    T, n = 300, 300
    r = np.random.default_rng(d)
    first = np.tile(np.arange(T, dtype=np.int32), n)
    evict = np.full(T * n, 2 ** 31 - 1, dtype=np.int32)
    block = (np.arange(T * n) % T) // 128 + 3 * (np.arange(T * n) // T)
    evict[(block % 3 == 1) & (r.random(3 * n) < 0.5)[block]] = 0
    evict[(first % 128 != 0) & (r.random(T * n) < 0.1)] = 0
    g = torch.Generator(device="cuda").manual_seed(d)
    ts = [torch.randn((T * n, h, d), generator=g, device="cuda", dtype=torch.bfloat16) for h in (Hq, Hkv, Hkv, Hq)]
    cu = np.arange(0, T * n + 1, T).astype(np.int32)
    fd, ed = torch.from_numpy(first).cuda(), torch.from_numpy(evict).cuda()
    (out, lse, dq, dk, dv), _ = _pass(None, cu, T, ts, Hq, (fd, ed))
    gone = ed == 0
    assert not dk[gone].any() and not dv[gone].any()
    q, k, v, do = (t.double().view(n, T, -1, d) for t in ts)
    i = torch.arange(T, device="cuda")
    seen = (i[None, None] <= i[None, :, None]) & ~gone.view(n, 1, T)
    k, v = k.repeat_interleave(Hq // Hkv, 2), v.repeat_interleave(Hq // Hkv, 2)
    s = (torch.einsum("bihd,bjhd->bhij", q, k) * d ** -0.5).masked_fill(~seen[:, None], -float("inf"))
    p = torch.softmax(s, 3)
    o = torch.einsum("bhij,bjhd->bihd", p, v)
    ds = p * (torch.einsum("bihd,bjhd->bhij", do, v) - (do * o).sum(3).transpose(1, 2)[..., None]) * d ** -0.5
    fold = lambda t: t.view(n, T, Hkv, -1, d).sum(3)  # noqa: E731
    want = (o, torch.einsum("bhij,bjhd->bihd", ds, k), fold(torch.einsum("bhij,bihd->bjhd", ds, q)), fold(torch.einsum("bhij,bihd->bjhd", p, do)))
    for name, a, b in zip(("out", "dq", "dk", "dv"), (out, dq, dk, dv), want):
        b = b.reshape(a.shape)
        assert ((a - b).norm() / b.norm()) <= 5e-3, name          # bf16 operands: probabilities and score gradients to 8 bits


@pytest.mark.parametrize("lens,Hq,Hkv,d", [([1], 2, 1, 64), ([300] * 80, 8, 2, 128), ([300] * 80, 6, 2, 64), ([2000, 130], 7, 1, 128)])
def test_teacher_rows_are_merged_as_they_are_written(lens, Hq, Hkv, d):
    # rows without an evicted key are the student's; against plain causal attention of the same kernel.  The student's part comes
    # as bf16 (half a unit in the last place, 2^-9), the result is rounded once more.
    r = np.random.default_rng(d)
    ev = np.concatenate([W.keep_last_k_evict_at(T, max(1, T // 16), r.integers(8, max(9, T // 8), size=T), 4) for T in lens])
    cu = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda()
    g = torch.Generator(device="cuda").manual_seed(d)
    q, k, v = (torch.randn((sum(lens), h, d), generator=g, device="cuda", dtype=torch.bfloat16) for h in (Hq, Hkv, Hkv))
    evd = torch.from_numpy(ev).cuda()
    ms, me = B.kvs_mask_meta(evd, cu, max(lens)), B.kvs_mask_meta_evicted(evd, cu, max(lens))
    os, ls, ot, lt = B.kvs_attn_fwd_dual(q, k, v, ms, me, len(lens), max(lens))
    full = B.kvs_mask_meta(torch.full_like(evd, 2 ** 31 - 1), cu, max(lens))
    want, lse = B.kvs_attn_fwd(q, k, v, full, len(lens), max(lens))
    plain, _ = B.kvs_attn_fwd(q, k, v, ms, len(lens), max(lens))
    assert torch.equal(os, plain)
    assert (lt - lse).abs().max() <= 2e-3
    assert ((ot.float() - want.float()).norm() / want.float().norm()) <= 2.0 ** -8
    at = np.concatenate([np.arange(T) for T in lens])
    nothing = np.concatenate([np.arange(T) < e.min() for T, e in zip(lens, np.split(ev, np.cumsum(lens)[:-1]))])
    rows = torch.from_numpy(np.nonzero(nothing)[0]).cuda()
    assert len(at) == len(nothing) and torch.equal(ot[rows], os[rows])


@pytest.mark.parametrize("lens,Hq,Hkv,d,rule", [
    ([300] * 90, 8, 2, 128, "turns"), ([300, 129, 0, 1, 700] * 40, 4, 4, 128, "tokens"), ([2200] * 9, 12, 2, 64, "causal"), ([4000] + [333] * 40, 16, 1, 64, "turns"),
])
def test_units_listed_by_trace_equal_whole_items(lens, Hq, Hkv, d, rule):
    # batches whose Q, dO and dQ do not fit in L2: most traces in the order of the batch, the others last.  Against whole items in
    # the metadata's order; the bound is that of test_bwd_units
    assert sum(lens) * Hq * d * 8 > 96 << 20
    x = _inputs(lens, Hq, Hkv, d, rule)
    out, lse, ref = _backward(x, lens, True)
    _, _, got = _backward(x, lens, False, out, lse)
    _same(got, ref, max(lens), Hq // Hkv)


@pytest.mark.parametrize("at", [0, 5, 150])
def test_one_long_trace_among_short_ones(at):
    # listed by trace: no units of all heads first, and some of them last.  The long trace at a place where it comes last, in the
    # order of the batch, and at its end
    Hq, Hkv, d = 32, 8, 128
    lens = [200] * at + [2000] + [200] * (150 - at)
    x = _inputs(lens, Hq, Hkv, d, "causal")
    out, lse, ref = _backward(x, lens, True)
    ev, cu, q, k, v, do = x
    meta = B.kvs_mask_meta(ev, cu, max(lens))
    ws = torch.zeros(B.kvs_attn_bwd_workspace_bytes(sum(lens), Hq, Hkv, d, B.GRAD_FP32), dtype=torch.uint8, device="cuda")
    got = B.kvs_attn_bwd(do, q, k, v, out, lse, meta, len(lens), max(lens), 0.0, B.GRAD_FP32, workspace=ws)
    assert B.kvs_device_status(ws) == B.KVS_OK
    units, _, first, apart = ws[_base_bytes(sum(lens), Hq):][:16].view(torch.int32).tolist()          # the plan's header
    assert first == 0 and 0 < apart < units
    _same(got, ref, max(lens), Hq // Hkv)


def test_a_short_range_of_a_host_batch_by_pairs():
    # two ranges of one trace each; the second one's metadata is made by one CTA, and with a mean of 17000 tokens its keys are
    # taken by CTA pairs, which go by the tables of pairs of key blocks
    lens, Hq, Hkv, d = [30000, 4000], 8, 4, 128
    ev, cu, q, k, v, do = x = _inputs(lens, Hq, Hkv, d, "turns")
    assert B.kvs_host_chunk_plan(cu.cpu(), max(lens), Hkv) == [(0, 1), (1, 2)]
    out, lse, ref = _backward(x, lens, False)
    pin = lambda t: t.cpu().pin_memory()  # noqa: E731
    room = lambda t, dtype: torch.full(t.shape, float("nan"), dtype=dtype).pin_memory()  # noqa: E731
    o = [room(out, out.dtype), room(lse, lse.dtype)] + [room(t, torch.float32) for t in (q, k, v)]
    arena = torch.empty(B.kvs_host_arena_bytes(2, sum(lens), max(lens), Hq, Hkv, d, B.GRAD_FP32), dtype=torch.uint8, device="cuda")
    B.kvs_attn_fwd_bwd_host(pin(ev), pin(cu), pin(q), pin(k), pin(v), pin(do), max(lens), 0.0, B.GRAD_FP32, *o, arena)
    assert torch.equal(o[0], out.cpu()) and torch.equal(o[1], lse.cpu())
    assert torch.equal(o[3], ref[1].cpu()) and torch.equal(o[4], ref[2].cpu())
    _same([t.cuda() for t in o[2:]], ref, max(lens), Hq // Hkv)


@pytest.mark.parametrize("lens", [[1000, 1, 300], [300] * 40])
def test_a_buffer_without_room_for_the_entries_of_the_blocks(lens):
    # 16 bytes a block less, each array in whole 256 bytes: the same results by the tables of the traces; one byte less is refused
    Hq, Hkv, d, total = 2, 1, 64, sum(lens)
    ev, cu, q, k, v, do = _inputs(lens, Hq, Hkv, d, "turns")
    blocks = min(len(lens) * -(-max(lens) // 128), total // 128 + len(lens))
    least = B.kvs_mask_meta_bytes(len(lens), total, max(lens)) - -(-16 * blocks // 256) * 256
    small = B.kvs_mask_meta(ev, cu, max(lens), torch.empty(least, dtype=torch.uint8, device="cuda"))
    full = B.kvs_mask_meta(ev, cu, max(lens))
    got = []
    for meta in (small, full):
        out, lse = B.kvs_attn_fwd(q, k, v, meta, len(lens), max(lens))
        ws = torch.empty(-(-(256 + 4 * total * Hq) // 256) * 256, dtype=torch.uint8, device="cuda")
        got.append((out, lse) + B.kvs_attn_bwd(do, q, k, v, out, lse, meta, len(lens), max(lens), 0.0, B.GRAD_FP32, workspace=ws))
        assert B.kvs_device_status(meta) == B.KVS_OK
    assert all(torch.equal(a, b) for i, (a, b) in enumerate(zip(*got)) if i != 2)           # dq is added in the order of arrival
    with pytest.raises(B.KvsError):
        B.kvs_mask_meta(ev, cu, max(lens), torch.empty(least - 1, dtype=torch.uint8, device="cuda"))
