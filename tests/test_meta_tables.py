"""The tables inside a metadata buffer, of the one-CTA kernel and of the two kernels, against a NumPy restatement of their
definitions (csrc/kvs_common.cuh: MetaView, meta_layout) (needs a B200).  The attention's results do not depend on the launch
orders and the sums of lengths, so nothing else sees a wrong one."""
import numpy as np
import pytest
import torch

from paper_2609_35750_b200 import binding as B
from paper_2609_35750_b200 import workloads as W

TILE = 128
HEADER = ("magic status batch total_tokens max_seqlen nblk_total ncls_total general npair_total rows_done blk_most pair_most blk_tiles pair_tiles "
          "has_info").split()


def layout(batch, total, longest):
    """Name -> (byte offset, dtype, entries)."""
    up = lambda x: -(-x // 256) * 256  # noqa: E731
    longest = min(longest, total)
    nbmax = -(-longest // TILE)
    cap = max(1, min(batch * nbmax, total // TILE + batch))
    tiles = max(1, cap * nbmax)
    at, L = up(4 * len(HEADER)), {}
    for name, n in [("blk_off", batch + 1), ("cls_off", batch + 1), ("seq_start", batch + 1)] + [(x, cap) for x in (
            "blk_trace", "kmin", "kmax", "fmin", "fmax", "col_first", "col_last", "row_cnt", "fwd_order", "bwd_order", "pair_order", "bwd_len",
            "pair_len")] + [("evict", max(total, 1)), ("kfirst", max(total, 1))]:
        L[name] = (at, np.int32, n)
        at = up(at + 4 * n)
    L["tile_class"] = (at, np.uint8, tiles)
    at = up(at + tiles)
    L["row_list"] = (at, np.uint16, tiles)
    at = up(at + 2 * tiles)
    L["info"] = (at, np.int32, 4 * cap)
    return L, up(at + 16 * cap)


def restated(first, evict, lens, longest, general):
    """first, evict: per key slot, trace-local."""
    t = {k: [] for k in "blk_off cls_off seq_start blk_trace kmin kmax fmin fmax col_first col_last row_cnt tile_class row_list info pair".split()}
    tok = 0
    for b, T in enumerate(lens):
        nb, base, cls0 = -(-T // TILE), len(t["kmin"]), len(t["tile_class"])
        t["blk_off"].append(base)
        t["cls_off"].append(cls0)
        t["seq_start"].append(tok)
        for n in range(nb):
            s = slice(tok + n * TILE, min(tok + (n + 1) * TILE, tok + T))
            f, e = first[s].astype(np.int64), evict[s].astype(np.int64)
            last = min((e.max() - 1) // TILE, nb - 1)
            if not general:
                last = max(last, n)
            for name, x in (("blk_trace", b), ("kmin", e.min()), ("kmax", e.max()), ("fmin", f.min()), ("fmax", f.max()),
                            ("col_first", min(f.min() // TILE, nb)), ("col_last", -1 if e.max() <= 0 else last)):
                t[name].append(x)
            t["info"] += [tok, T, n, cls0 + n * nb]
        block = lambda name: np.array(t[name][base:])  # noqa: E731
        for m in range(nb):
            q0, q1 = m * TILE, min(m * TILE + TILE, T) - 1
            empty = (block("fmin") > q1) | (block("kmax") <= q0)
            full = ~empty & (block("fmax") <= q0) & (block("kmin") > q1)
            t["tile_class"] += np.where(empty, B.CLASS_EMPTY, np.where(full, B.CLASS_FULL, B.CLASS_PARTIAL)).tolist()
            seen = np.nonzero(~empty)[0].tolist()
            t["row_cnt"].append(len(seen))
            t["row_list"] += seen + [-1] * (nb - len(seen))            # -1: nothing is written there
        for n in range(0, nb, 2):
            spans = [(t["col_first"][base + i], t["col_last"][base + i]) for i in range(n, min(n + 2, nb))]
            live = [s for s in spans if s[1] >= s[0]]
            t["pair"].append((base + n, max(s[1] for s in live) - min(s[0] for s in live) + 1 if live else 0))
        tok += T
    t["blk_off"].append(len(t["kmin"]))
    t["cls_off"].append(len(t["tile_class"]))
    t["seq_start"].append(tok)
    bins = min(longest, tok) // TILE // 16 + 2
    bucket = lambda n: n if min(longest, tok) <= 16 * TILE else min(n // 16, bins - 1)  # noqa: E731
    order = lambda items: sorted(items, key=lambda x: (-bucket(x[1]), x[0]))  # noqa: E731
    cols = [(i, max(z - a + 1, 0)) for i, (a, z) in enumerate(zip(t["col_first"], t["col_last"]))]
    t["fwd_order"] = [i for i, _ in order(enumerate(t["row_cnt"]))]
    t["bwd_order"], t["bwd_len"] = (list(x) for x in zip(*order(cols))) if cols else ([], [])
    t["pair_order"], t["pair_len"] = (list(x) for x in zip(*order(t["pair"]))) if cols else ([], [])
    head = dict(status=0, batch=len(lens), total_tokens=tok, max_seqlen=min(longest, tok), nblk_total=len(cols), ncls_total=len(t["tile_class"]),
                general=int(general), npair_total=len(t["pair"]), blk_most=max([n for _, n in cols], default=0), has_info=1,
                pair_most=max([n for _, n in t["pair"]], default=0), blk_tiles=sum(n for _, n in cols), pair_tiles=sum(n for _, n in t["pair"]))
    del t["pair"]
    return t, head


def masks(lens, kind, seed):
    r = np.random.default_rng(seed)
    evict = np.concatenate([W.keep_last_k_evict_at(T, max(1, T // 16), r.integers(8, max(9, T // 8), size=T), 4) for T in lens if T] or [[]]).astype(np.int32)
    first = np.concatenate([np.arange(T) for T in lens]).astype(np.int32)
    if kind == "keys":              # slots in another order, some of them never seen, and whole blocks that nobody sees
        at = 0
        for T in lens:
            p = at + r.permutation(T)
            first[at:at + T], evict[at:at + T] = first[p], evict[p]
            at += T
        evict[r.random(len(evict)) < 0.1] = 0
        evict[(np.arange(len(evict)) // 100) % 5 == 3] = 0
    return first, evict


# up to 64 blocks and 5120 tokens: one CTA; the others: two kernels
@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["plain", "keys", "evicted"])
@pytest.mark.parametrize("lens,slack", [
    ([1], 0), ([5120], 0), ([4993, 0, 127], 0), ([80] * 64, 0), ([127, 0, 129, 0, 0, 385, 1], 300), ([1024, 1025, 1, 3000], 0), ([1] * 62 + [129], 0), ([2048, 2049], 0),
    ([5121], 0), ([80] * 65, 0), ([300, 8000, 0, 129] + [300] * 30, 100), ([20000], 0),
])
def test_tables(lens, slack, kind):
    first, evict = masks(lens, kind, len(lens))
    total, longest = sum(lens), max(lens) + slack
    L, size = layout(len(lens), total, longest)
    assert B.kvs_mask_meta_bytes(len(lens), total, longest) == size
    cu = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda()
    buf = torch.full((size,), 0xEE, dtype=torch.uint8, device="cuda")
    dev = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    if kind == "plain":
        B.kvs_mask_meta(dev(evict), cu, longest, buf)
    elif kind == "keys":
        B.kvs_mask_meta_keys(dev(first), dev(evict), cu, longest, buf)
    else:
        B.kvs_mask_meta_evicted(dev(evict), cu, longest, buf)
        first, evict = evict, np.full_like(evict, 2 ** 31 - 1)
    got = buf.cpu().numpy()
    want, head = restated(first, evict, lens, longest, kind != "plain")
    words = dict(zip(HEADER, got[:4 * len(HEADER)].view(np.int32).tolist()))
    assert {k: words[k] for k in head} == head
    table = lambda name: got[L[name][0]:][:L[name][2] * np.dtype(L[name][1]).itemsize].view(L[name][1])  # noqa: E731
    for name, x in want.items():
        x = np.array(x, dtype=np.int64)
        y = table(name)[:len(x)].astype(np.int64)
        at = x >= 0 if name == "row_list" else np.ones(len(x), dtype=bool)
        assert np.array_equal(y[at], x[at]), name
    assert np.array_equal(table("evict")[:total], evict)
    if kind != "plain":
        assert np.array_equal(table("kfirst")[:total], first)
