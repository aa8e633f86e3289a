"""The longest trace that the metadata takes, 65535 blocks of 128 tokens (needs a B200).

Masks whose definition can be evaluated for 8 million rows: every query sees itself and token 0, whose key block is then seen by
all 65535 query blocks (the longest column); or the last query sees every key and the others none (the longest row).  Outputs are
compared with fp64 sums over the same bf16 inputs: probabilities, score gradients and outputs are rounded to bf16 (a relative
2^-9 each at most), so a result is off by at most three such parts in the 2-norm.
"""
import pytest
import torch

from paper_2609_35750_b200 import binding as B

pytestmark = pytest.mark.gpu
T, D = 65535 * 128, 64
INF = 2 ** 31 - 1


def _inputs():
    g = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda: torch.randn((T, 1, D), generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    return rnd(), rnd(), rnd(), rnd(), torch.tensor([0, T], dtype=torch.int32, device="cuda")


def _two_keys(q, k, v, do, rows):
    """Attention of the rows over themselves and key 0, in fp64: out, lse, p0 and the rows' score gradients."""
    a, b, x, y = (t[rows, 0].double() for t in (q, k, v, do))
    scale = D ** -0.5
    s = torch.stack((a @ k[0, 0].double(), (a * b).sum(1)), dim=1) * scale
    s[rows == 0, 0] = -float("inf")                                   # token 0 sees itself once
    lse = torch.logsumexp(s, dim=1)
    p = torch.exp(s - lse[:, None])
    out = p[:, :1] * v[0, 0].double() + p[:, 1:] * x
    dp = torch.stack((y @ v[0, 0].double(), (y * x).sum(1)), dim=1)
    ds = p * (dp - (y * out).sum(1, keepdim=True)) * scale
    return out, lse, p, ds, dp


def test_longest_column():
    q, k, v, do, cu = _inputs()
    evict = torch.arange(1, T + 1, dtype=torch.int32, device="cuda")
    evict[0] = INF
    meta = B.kvs_mask_meta(evict, cu, T)
    out, lse = B.kvs_attn_fwd(q, k, v, meta, 1, T)
    dq, dk, dv = B.kvs_attn_bwd(do, q, k, v, out, lse, meta, 1, T, 0.0, B.GRAD_FP32)
    assert B.kvs_device_status(meta) == B.KVS_OK
    dk0, dv0 = torch.zeros(D, dtype=torch.float64, device="cuda"), torch.zeros(D, dtype=torch.float64, device="cuda")
    for i0 in range(0, T, 1 << 20):
        rows = torch.arange(i0, min(T, i0 + (1 << 20)), device="cuda")
        ro, rl, p, ds, dp = _two_keys(q, k, v, do, rows)
        assert (lse[0, rows] - rl).abs().max() <= 1e-4, i0
        assert ((out[rows, 0] - ro).norm() / ro.norm()) <= 5e-3, i0
        k0, v0 = k[0, 0].double(), v[0, 0].double()
        rdq = ds[:, :1] * k0 + ds[:, 1:] * k[rows, 0].double()
        assert ((dq[rows, 0] - rdq).norm() / rdq.norm()) <= 5e-3, i0
        a, y = q[rows, 0].double(), do[rows, 0].double()
        dk0 += (ds[:, :1] * a).sum(0)
        dv0 += (p[:, :1] * y).sum(0)
        own = rows != 0
        rdk, rdv = (ds[:, 1:] * a)[own], (p[:, 1:] * y)[own]
        assert ((dk[rows[own], 0] - rdk).norm() / rdk.norm()) <= 5e-3, i0
        assert ((dv[rows[own], 0] - rdv).norm() / rdv.norm()) <= 5e-3, i0
        if i0 == 0:
            dk0 += ds[0, 1] * a[0]
            dv0 += p[0, 1] * y[0]
    # 8 million terms of either sign: their rounding errors add up like their square root, and so does the sum itself
    assert (dk[0, 0] - dk0).norm() <= 2e-2 * dk0.norm()
    assert (dv[0, 0] - dv0).norm() <= 2e-2 * dv0.norm()


def test_longest_row():
    q, k, v, _, cu = _inputs()
    first = torch.full((T,), T - 1, dtype=torch.int32, device="cuda")          # every key for the last query alone
    meta = B.kvs_mask_meta_keys(first, torch.full_like(first, INF), cu, T)
    out, lse = B.kvs_attn_fwd(q, k, v, meta, 1, T)
    assert B.kvs_device_status(meta) == B.KVS_OK
    assert (lse[0, :-1] == -float("inf")).all() and (out[:-1] == 0).all()
    s = (k[:, 0].double() @ q[-1, 0].double()) * D ** -0.5
    ref = torch.softmax(s, 0) @ v[:, 0].double()
    assert abs(float(lse[0, -1]) - float(torch.logsumexp(s, 0))) <= 1e-4
    # beside the roundings: the tensor core cuts its running sum off, by up to 2^-24 on average in each of 8 steps a tile
    assert (out[-1, 0] - ref).norm() <= (5e-3 + 8 * 65535 * 2.0 ** -24) * ref.norm()
