"""The merge of the splits of decode attention (needs a B200): grids below and above one wave, one split, more splits than a warp
has lanes and than there are tiles, sequences without a token; against the definition in fp64, and a workspace that still holds
another call's results.  Bounds: weights and outputs are rounded to bf16 (2^-9 relative each), and |out| is below 4 on these
inputs, so 2e-2 as in the other decode tests."""
import numpy as np
import pytest
import torch

from paper_2609_35750_b200 import binding as B

pytestmark = pytest.mark.gpu


def _cache(lens, page, Hkv, d, seed):
    """Scattered pages; rows that hold no token are NaN.  Returns the cache and the live K, V of every sequence."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    pages = [-(-n // page) for n in lens]
    cache = B.PagedCache(sum(pages) + 3, page, len(lens), max(pages) + 1, Hkv, d)
    order = torch.from_numpy(np.random.default_rng(seed).permutation(sum(pages) + 3)).cuda()
    cache.k_cache.fill_(float("nan"))
    cache.v_cache.fill_(float("nan"))
    live, at = [], 0
    for s, (n, p) in enumerate(zip(lens, pages)):
        mine = order[at:at + p]
        at += p
        cache.block_table[s, :p] = mine.int()
        kv = torch.randn((2, n, Hkv, d), generator=g, device="cuda", dtype=torch.bfloat16)
        slot = torch.arange(n, device="cuda")
        rows = mine[slot // page] * page + slot % page
        cache.k_cache.view(-1, Hkv, d)[rows] = kv[0]
        cache.v_cache.view(-1, Hkv, d)[rows] = kv[1]
        live.append(kv)
    cache.n_tokens.copy_(torch.tensor(lens, dtype=torch.int32))
    return cache, live


def _bytes(S, Hq, d, splits):
    least = 256 + -(-4 * S * Hq * splits * (d + 2) // 256) * 256
    assert int(B.load().kvs_decode_workspace_bytes(S, Hq, d, splits)) == least
    return least


@pytest.mark.parametrize("S,lens,page,Hkv,G,d,splits", [
    (48, (0, 1, 700), 16, 8, 4, 128, 3),        # 1152 CTAs
    (112, (0, 5, 300), 1, 8, 2, 128, 1),        # a single split
    (64, (0, 3, 400), 4, 4, 7, 128, 4),         # the most splits that are merged 4 at a time
    (64, (0, 3, 900), 4, 4, 1, 128, 5),         # ... 16 at a time
    (120, (0, 1, 257), 16, 4, 2, 64, 2),
    (2, (5000, 1), 1, 2, 7, 128, 40),           # more splits than a warp has lanes
    (3, (4000, 0, 33), 16, 2, 8, 128, 64),      # ... and more than there are tiles
    (2, (3000, 10), 16, 3, 1, 64, 33),
    (5, (2100, 0), 16, 2, 4, 64, 17),
])
def test_merge_gives_the_definition(S, lens, page, Hkv, G, d, splits):
    lens = [lens[s % len(lens)] for s in range(S)]
    cache, live = _cache(lens, page, Hkv, d, S + splits)
    q = torch.randn((S, Hkv * G, d), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda", dtype=torch.bfloat16)
    ws = torch.full((_bytes(S, Hkv * G, d, splits),), 0xff, dtype=torch.uint8, device="cuda")      # NaN in every partial result
    out, lse = cache.decode(q, num_splits=splits, workspace=ws)
    assert B.kvs_device_status(ws) == B.KVS_OK
    again = cache.decode(q, num_splits=splits, workspace=ws)
    assert torch.equal(out, again[0]) and torch.equal(lse, again[1])
    for s, n in enumerate(lens):
        if n == 0:
            assert (out[s] == 0).all() and (lse[s] == -float("inf")).all()
            continue
        k, v = (x.double().repeat_interleave(G, dim=1) for x in live[s])
        score = torch.einsum("hd,nhd->hn", q[s].double(), k) * d ** -0.5
        ref = torch.einsum("hn,nhd->hd", torch.softmax(score, 1), v)
        assert (out[s] - ref).abs().max() <= 2e-2 and (lse[s] - torch.logsumexp(score, 1)).abs().max() <= 2e-3, s


def test_workspace_limits():
    cache, _ = _cache([300], 16, 2, 128, 0)
    q = torch.randn((1, 8, 128), device="cuda", dtype=torch.bfloat16)
    least = _bytes(1, 8, 128, 2)
    with pytest.raises(B.KvsError) as e:
        cache.decode(q, num_splits=2, workspace=torch.empty(least - 1, dtype=torch.uint8, device="cuda"))
    assert e.value.code == B.KVS_ERR_WORKSPACE
    cache.decode(q, num_splits=2, workspace=torch.empty(least, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("page,G,d", [(16, 4, 128), (1, 7, 128), (1, 1, 128), (16, 2, 64)])
@pytest.mark.parametrize("splits", [1, 5, 40])
def test_bad_page_is_reported_and_the_next_call_is_clean(page, G, d, splits):
    # page ids outside the cache are not followed (page 0 is read instead); the status comes with the partial results
    cache, _ = _cache([2000, 700, 0], page, 2, d, splits)
    q = torch.randn((3, 2 * G, d), device="cuda", dtype=torch.bfloat16)
    ws = torch.full((_bytes(3, 2 * G, d, splits),), 0xff, dtype=torch.uint8, device="cuda")
    last = (2000 - 1) // page
    good = int(cache.block_table[0, last])
    for bad in (-1, cache.num_pages, 2 ** 31 - 1):
        cache.block_table[0, last] = bad
        cache.decode(q, num_splits=splits, workspace=ws)
        assert B.kvs_device_status(ws) == B.KVS_ERR_INVALID_ARG
        out, lse = cache.decode(q, num_splits=splits, workspace=ws)
        assert torch.isfinite(out).all() and torch.isfinite(lse[:2]).all()
        cache.block_table[0, last] = good
        cache.decode(q, num_splits=splits, workspace=ws)
        assert B.kvs_device_status(ws) == B.KVS_OK
