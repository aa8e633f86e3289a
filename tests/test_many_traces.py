"""Batches of very many short traces (needs a B200): more blocks than the launch orders keep in shared memory, sorted by eight warps;
more key blocks than the backward's plan has room for, so that they stay whole; runs of the sort with a remainder.  Traces of one
token have a known result (out = v, dv = dout, no other gradient), the others are compared with the definition in fp64."""
import numpy as np
import pytest
import torch

from paper_2609_35750_b200 import binding as B

pytestmark = pytest.mark.gpu


def _definition(q, k, v, do, evict):
    T, Hq, d = q.shape
    G = Hq // k.shape[1]
    i = torch.arange(T, device="cuda")
    seen = (i[None] <= i[:, None]) & (i[:, None] < evict[None])
    q, k, v, do = q.double(), k.double().repeat_interleave(G, 1), v.double().repeat_interleave(G, 1), do.double()
    s = (torch.einsum("ihd,jhd->hij", q, k) * d ** -0.5).masked_fill(~seen, -float("inf"))
    p, lse = torch.softmax(s, 2), torch.logsumexp(s, 2)
    out = torch.einsum("hij,jhd->ihd", p, v)
    ds = p * (torch.einsum("ihd,jhd->hij", do, v) - (do * out).sum(2).T[..., None]) * d ** -0.5
    fold = lambda t: t.view(T, -1, G, d).sum(2)  # noqa: E731
    return out, lse, torch.einsum("hij,jhd->ihd", ds, k), fold(torch.einsum("hij,ihd->jhd", ds, q)), fold(torch.einsum("hij,ihd->jhd", p, do))


@pytest.mark.parametrize("ones,others", [
    (13001, [129] * 3 + [700, 128, 257]),                # exact order; 13014 blocks, the last run of the sort is short
    (6000, [129, 3000, 640]),                            # coarse order
    (64, [64]), (63, [1]),                               # around the smallest batch that is sorted by eight warps
])
def test_many_short_traces(ones, others):
    Hq, Hkv, d = 2, 1, 64
    r = np.random.default_rng(ones)
    lens = r.permutation(np.array([1] * ones + others + [0] * 5))
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    total, longest = int(cu[-1]), int(lens.max())
    ev = np.concatenate([np.minimum(np.arange(T) + r.integers(1, 400, size=T), 2 ** 31 - 1) for T in lens]).astype(np.int32)
    g = torch.Generator(device="cuda").manual_seed(ones)
    rnd = lambda h: torch.randn((total, h, d), generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, k, v, do = rnd(Hq), rnd(Hkv), rnd(Hkv), rnd(Hq)
    evd = torch.from_numpy(ev).cuda()
    meta = B.kvs_mask_meta(evd, torch.from_numpy(cu).cuda(), longest)
    out, lse = B.kvs_attn_fwd(q, k, v, meta, len(lens), longest)
    dq, dk, dv = B.kvs_attn_bwd(do, q, k, v, out, lse, meta, len(lens), longest, 0.0, B.GRAD_FP32)
    assert B.kvs_device_status(meta) == B.KVS_OK
    one = torch.from_numpy(cu[:-1][lens == 1]).cuda().long()
    assert torch.equal(out[one], v[one].expand(-1, Hq, -1))
    # the tensor core cuts the smaller of two terms off at the last bit of the larger one (2^-23 of it)
    assert ((dv[one, 0] - do[one].float().sum(1)).abs() <= 2.0 ** -22 * do[one].float().abs().sum(1)).all()
    # dS = P (dP - D): the two are the same dot product of bf16 numbers, formed in two orders in fp32
    assert dq[one].abs().max() <= 1e-4 and dk[one].abs().max() <= 1e-4
    for b in np.nonzero(lens > 1)[0]:
        z = slice(int(cu[b]), int(cu[b + 1]))
        for name, got, ref in zip(("out", "lse", "dq", "dk", "dv"), (out[z], lse[:, z], dq[z], dk[z], dv[z]),
                                  _definition(q[z], k[z], v[z], do[z], evd[z])):
            assert ((got - ref).norm() / ref.norm()) <= 5e-3, (name, int(lens[b]))
