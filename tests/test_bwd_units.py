"""Backward: items cut into units, and the kernel of CTA pairs, against the whole-item single-CTA path (needs a B200).

The single-CTA path with whole items is compared with the oracle in test_gpu_parity; a workspace of the base size selects it.
Both sides form the same products from the same bf16 operands and add them in fp32 in another order.  The tensor core does
not round its running sum but cuts it off, an error of at most 2^-23 of the sum per 16-wide step and always towards zero, so
a sum of n steps that grows evenly ends up to n 2^-24 low, and two orders differ by at most that: n = 8 steps a tile times the
tiles of the longest key block (heads of the group times query blocks).  1e-5 covers the fp32 additions of short sums.
"""
import numpy as np
import pytest
import torch

from paper_2609_35750_b200 import binding as B
from paper_2609_35750_b200 import workloads as W

pytestmark = pytest.mark.gpu


def _inputs(lens, Hq, Hkv, d, rule, seed=0):
    r = np.random.default_rng(seed)
    ev = []
    for T in lens:
        if rule == "causal":
            ev.append(np.full(T, 2 ** 31 - 1, dtype=np.int32))
        elif rule == "turns":
            ev.append(W.keep_last_k_evict_at(T, max(1, T // 16), r.integers(16, max(17, T // 8), size=T), 4))
        else:
            ev.append(W.fine_grained_evict_at(T, max(1, T // 24), r, T / 16.0))
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda h: torch.randn((sum(lens), h, d), generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    ev = torch.from_numpy(np.concatenate(ev)).cuda()
    cu = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda()
    return ev, cu, rnd(Hq), rnd(Hkv), rnd(Hkv), rnd(Hq)


def _base_bytes(total, Hq):
    up = lambda x: -(-x // 256) * 256  # noqa: E731
    return up(256 + 4 * total * Hq)                       # fp32 gradients: header and row sums


def _backward(x, lens, whole, out=None, lse=None):
    ev, cu, q, k, v, do = x
    meta = B.kvs_mask_meta(ev, cu, max(lens))
    out, lse = B.kvs_attn_fwd(q, k, v, meta, len(lens), max(lens)) if out is None else (out, lse)
    need = B.kvs_attn_bwd_workspace_bytes(q.shape[0], q.shape[1], k.shape[1], q.shape[2], B.GRAD_FP32)
    ws = torch.empty(_base_bytes(q.shape[0], q.shape[1]) if whole else need, dtype=torch.uint8, device="cuda")
    g = B.kvs_attn_bwd(do, q, k, v, out, lse, meta, len(lens), max(lens), 0.0, B.GRAD_FP32, workspace=ws)
    assert B.kvs_device_status(meta) == B.KVS_OK and B.kvs_device_status(ws) == B.KVS_OK
    return out, lse, g


def _same(a, b, longest, G):
    bound = max(1e-5, 8 * G * -(-longest // 128) * 2.0 ** -24)
    for name, x, y in zip(("dq", "dk", "dv"), a, b):
        assert torch.isfinite(x).all(), name
        off, size = (x - y).norm().item(), y.norm().item()        # a single token has no dq and no dk
        assert off <= bound * size, (name, off, size)


@pytest.mark.parametrize("lens,Hq,Hkv,d,rule", [
    ([1], 1, 1, 64, "causal"), ([129], 8, 1, 128, "causal"), ([1024], 4, 4, 64, "turns"), ([1000], 16, 2, 128, "turns"),
    ([4097], 28, 4, 128, "causal"), ([2500, 1, 0, 77], 7, 1, 64, "tokens"), ([8192], 8, 1, 128, "tokens"), ([300] * 40, 16, 4, 64, "turns"),
])
def test_cut_items_equal_whole_items(lens, Hq, Hkv, d, rule):
    x = _inputs(lens, Hq, Hkv, d, rule)
    out, lse, ref = _backward(x, lens, True)
    _, _, got = _backward(x, lens, False, out, lse)
    _, _, again = _backward(x, lens, False, out, lse)
    _same(got, ref, max(lens), Hq // Hkv)
    assert torch.equal(got[1], again[1]) and torch.equal(got[2], again[2])        # the slots are added in a fixed order


@pytest.mark.parametrize("T,rule", [(24000, "turns"), (24064, "tokens"), (24193, "turns"), (24321, "causal"), (16000, "tokens"), (16129, "turns")])
def test_pairs_equal_single_ctas(T, rule):
    # a long trace alone is taken by CTA pairs; with a one-token trace behind it the mean length is below their line and
    # single CTAs take the same keys.  Block counts: 188 (even, last block half full), 188 (full), 190, 191 (odd, one row), 125, 127
    Hq, Hkv, d = 4, 2, 128
    x = _inputs([T], Hq, Hkv, d, rule)
    out, lse, got = _backward(x, [T], False)
    _, _, whole = _backward(x, [T], True, out, lse)
    ev, cu, *ts = x
    y = (torch.cat([ev, ev.new_full((1,), 2 ** 31 - 1)]), torch.tensor([0, T, T + 1], dtype=torch.int32, device="cuda"),
         *(torch.cat([t, t[:1]]) for t in ts))
    _, _, ref = _backward(y, [T, 1], True)
    _same(got, [t[:T] for t in ref], T, Hq // Hkv)
    _same(whole, [t[:T] for t in ref], T, Hq // Hkv)


@pytest.mark.parametrize("tiles,went_on", [(0, 0), (8, 128)])
def test_warps_of_a_group_go_on_together_after_a_wait(tiles, went_on):
    # Two of four warps are through their wait at once, the others after 3 steps: with the limit of 9 steps all go on, with that of
    # one step (0.01 s) the wait runs out and none does, although two had seen no reason to stop.
    status = B.KVS_OK if went_on else B.KVS_ERR_TIMEOUT
    assert B.kvs_selftest_group_wait(tiles, 20_000_000) == (status, went_on)
    with pytest.raises(B.KvsError):
        B.kvs_selftest_group_wait(17, 1000)


@pytest.mark.parametrize("T,Hq,Hkv,d,longest", [(600, 16, 2, 128, 4), (1000, 16, 2, 128, 4), (384, 16, 4, 64, 3), (1024, 4, 4, 64, 2), (300, 2, 2, 128, 3)])
def test_short_items_are_cut_into_few_units(T, Hq, Hkv, d, longest):
    # an item's last unit adds up the slots of all of them: units of fewer than four tiles only where four of them are an item
    x = _inputs([T], Hq, Hkv, d, "causal")
    out, lse, ref = _backward(x, [T], True)
    ev, cu, q, k, v, do = x
    meta = B.kvs_mask_meta(ev, cu, T)
    ws = torch.zeros(B.kvs_attn_bwd_workspace_bytes(T, Hq, Hkv, d, B.GRAD_FP32), dtype=torch.uint8, device="cuda")
    got = B.kvs_attn_bwd(do, q, k, v, out, lse, meta, 1, T, 0.0, B.GRAD_FP32, workspace=ws)
    _same(got, ref, T, Hq // Hkv)
    plan = ws[_base_bytes(T, Hq):]
    units = plan[256:][:16 * plan[:4].view(torch.int32).item()].view(torch.int32).view(-1, 4)          # key block, first tile, end, slots
    assert (units[:, 2] - units[:, 1]).max().item() == longest
