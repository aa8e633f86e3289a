"""Backward workspaces and host arenas with fewer slots than kvs_attn_bwd_workspace_bytes and kvs_host_arena_bytes ask for (needs
a B200).  Units of four tiles at least ask for the sizes below; a buffer of such a size is accepted and its key blocks are still cut."""
import numpy as np
import pytest
import torch

from paper_2609_35750_b200 import binding as B

from .test_bwd_units import _backward, _base_bytes, _inputs, _same

pytestmark = pytest.mark.gpu

# tokens, query heads, KV heads, head_dim: workspace (fp32 gradients), arena (one trace, fp32 gradients), of units of four tiles
SIZES = [
    (1024, 4, 4, 64, 4753920, 9105664),
    (600, 16, 2, 128, 15780096, 29963008),
    (130, 3, 1, 64, 267008, 625920),
    (1, 1, 1, 64, 1024, 9472),
    (4000, 32, 8, 128, 39381248, 119182080),       # all the slots there are, with either unit
]


@pytest.mark.parametrize("T,Hq,Hkv,d,size,arena", SIZES)
def test_a_workspace_with_fewer_slots(T, Hq, Hkv, d, size, arena):
    x = _inputs([T], Hq, Hkv, d, "causal")
    ev, cu, q, k, v, do = x
    out, lse, ref = _backward(x, [T], True)
    meta = B.kvs_mask_meta(ev, cu, T)
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    got = B.kvs_attn_bwd(do, q, k, v, out, lse, meta, 1, T, 0.0, B.GRAD_FP32, workspace=ws)
    assert B.kvs_device_status(ws) == B.KVS_OK
    _same(got, ref, T, Hq // Hkv)
    plan = ws[_base_bytes(T, Hq):][:4].view(torch.int32).item()          # the plan's first word: units of a KV head
    blocks = -(-T // 128)
    assert plan > blocks if T >= 600 else plan == blocks                 # the two shortest have nothing to gain from a cut


@pytest.mark.parametrize("T,Hq,Hkv,d,size,arena", SIZES)
def test_an_arena_with_fewer_slots(T, Hq, Hkv, d, size, arena):
    x = _inputs([T], Hq, Hkv, d, "causal")
    ev, cu, q, k, v, do = x
    out, lse, ref = _backward(x, [T], True)
    pin = lambda t: t.cpu().pin_memory()  # noqa: E731
    room = lambda t, dtype: torch.full(t.shape, float("nan"), dtype=dtype).pin_memory()  # noqa: E731
    o = [room(q, torch.bfloat16), torch.full((Hq, T), float("nan")).pin_memory()] + [room(t, torch.float32) for t in (q, k, v)]
    call = lambda n: B.kvs_attn_fwd_bwd_host(pin(ev), pin(cu), pin(q), pin(k), pin(v), pin(do), T, 0.0, B.GRAD_FP32, *o,  # noqa: E731
                                             torch.empty(n, dtype=torch.uint8, device="cuda"))
    call(arena)
    assert torch.equal(o[0], out.cpu()) and torch.equal(o[1], lse.cpu())
    _same([t.cuda() for t in o[2:]], ref, T, Hq // Hkv)
    with pytest.raises(B.KvsError) as e:
        call(arena - 1)
    assert e.value.code == B.KVS_ERR_WORKSPACE


def test_sizes_asked_for_are_no_smaller():
    for T, Hq, Hkv, d, size, arena in SIZES:
        assert B.kvs_attn_bwd_workspace_bytes(T, Hq, Hkv, d, B.GRAD_FP32) >= size
        assert B.kvs_host_arena_bytes(1, T, T, Hq, Hkv, d, B.GRAD_FP32) >= arena
        assert np.all([size % 256 == 0, arena % 256 == 0])
