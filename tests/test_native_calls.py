"""The native calls of the binding refuse what the path does not take, as Python errors (no GPU needed)."""
import threading
import time

import pytest
import torch

from paper_2609_35750_b200 import binding as B
from paper_2609_35750_b200 import build

CPU = {"evict": torch.ones(4, dtype=torch.int32), "cu": torch.tensor([0, 4], dtype=torch.int32), "q": torch.zeros((4, 2, 64), dtype=torch.bfloat16)}


def test_host_tensors_are_refused():
    meta = torch.zeros(1 << 16, dtype=torch.uint8)
    with pytest.raises(ValueError, match="CUDA"):
        B.kvs_mask_meta(CPU["evict"], CPU["cu"], 4, meta)
    with pytest.raises(ValueError, match="CUDA"):
        B.kvs_attn_fwd(CPU["q"], CPU["q"], CPU["q"], meta, 1, 4)
    with pytest.raises(ValueError, match="CUDA"):
        B.kvs_permute_rows(CPU["q"], CPU["cu"])
    with pytest.raises(ValueError, match="CUDA"):
        B.kvs_rope_qk(CPU["q"], None, CPU["cu"])


def test_wrong_arguments_are_python_errors():
    with pytest.raises(TypeError):
        B.kvs_attn_fwd(None, CPU["q"], CPU["q"], CPU["q"], 1, 4)
    with pytest.raises(TypeError):
        B.kvs_mask_meta(CPU["evict"], CPU["cu"], "4")
    with pytest.raises(ValueError):
        B.kvs_attn_fwd(CPU["q"][0], CPU["q"], CPU["q"], CPU["q"], 1, 4)              # two dimensions
    with pytest.raises(ValueError, match="heads"):
        B.kvs_attn_fwd_packed(CPU["q"], CPU["q"], 1, 4, 2, 1)
    with pytest.raises(IndexError):
        B.kvs_permute_rows(torch.zeros(()), CPU["cu"])


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.int64, torch.float16, torch.float64, torch.bool, torch.uint8])
def test_a_wrong_dtype_is_named_as_torch_names_it(dtype):
    cu = CPU["cu"].cuda()
    with pytest.raises(ValueError, match=f"^evict_at must be torch.int32, got {dtype}$"):
        B.kvs_mask_meta(torch.ones(4, dtype=dtype, device="cuda"), cu, 4)
    q = torch.zeros((4, 2, 64), dtype=dtype, device="cuda")
    with pytest.raises(ValueError, match=f"^q must be torch.bfloat16, got {dtype}$"):
        B.kvs_attn_fwd(q, q, q, torch.zeros(1 << 16, dtype=torch.uint8, device="cuda"), 1, 4)


def test_other_threads_run_while_outputs_are_allocated():
    # An allocation may wait (for the device, or as here for 800 MB to be filled); it is refused afterwards for being on the host
    total = 1 << 21
    evict = torch.ones(total, dtype=torch.int32)
    cu = torch.tensor([0, total], dtype=torch.int32)
    ticks, stop = [0], threading.Event()

    def tick():
        while not stop.is_set():
            ticks[0] += 1
            time.sleep(1e-3)

    B.load()
    thread = threading.Thread(target=tick)
    before = torch.are_deterministic_algorithms_enabled()
    torch.use_deterministic_algorithms(True)                  # new tensors are filled
    thread.start()
    try:
        t0, n0 = time.perf_counter(), ticks[0]
        with pytest.raises(ValueError, match="CUDA"):
            B.kvs_mask_meta(evict, cu, total)
        took, n = time.perf_counter() - t0, ticks[0] - n0
    finally:
        torch.use_deterministic_algorithms(before)
        stop.set()
        thread.join()
    assert n >= took / 0.02, (took, n)        # a tick takes a millisecond; held up, there are two at most (of 0.1 s)


def test_host_only_functions_do_without_the_native_calls(monkeypatch):
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "_native", None)
    monkeypatch.setattr(B, "native_path", lambda: "/nowhere/_kvs_native.so")
    assert B.kvs_mask_meta_bytes(1, 1024, 1024) > 0 and B.strerror(0) == "ok"
    assert B.kvs_attn_bwd_workspace_bytes(1024, 4, 4, 64, B.GRAD_BF16) > 0 and B.kvs_host_arena_bytes(1, 1024, 1024, 4, 4, 64, B.GRAD_BF16) > 0
    assert B.kvs_host_chunk_plan([0, 5, 9], 5, 1) == [(0, 1), (1, 2)]
    with pytest.raises(FileNotFoundError):
        B.kvs_mask_meta(CPU["evict"], CPU["cu"], 4)


def test_a_module_built_against_another_torch_is_not_used(monkeypatch):
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    monkeypatch.setattr(B, "_native", None)
    assert build.needs_build()
    with pytest.raises(FileNotFoundError, match="0.0.1"):
        B.kvs_mask_meta(CPU["evict"], CPU["cu"], 4)


@pytest.mark.parametrize("dtype", [torch.float16, torch.float64, torch.int32])
def test_rope_refuses_what_it_does_not_rotate(dtype):
    # found before the device is asked for; halves used to be rotated as if their bits were bfloat16
    x = torch.zeros((4, 2, 64), dtype=dtype)
    with pytest.raises(ValueError, match=f"^q must be torch.bfloat16 or torch.float32, got {dtype}$"):
        B.kvs_rope_qk(x, None, CPU["cu"])
    with pytest.raises(ValueError, match=f"^k must be torch.bfloat16 or torch.float32, got {dtype}$"):
        B.kvs_rope_qk(None, x, CPU["cu"])


@pytest.mark.gpu
def test_calls_go_to_the_stream_that_is_given():
    # the current stream is busy for a second meanwhile; results of the given one are there before that, and equal
    Hq, Hkv, d, T = 4, 2, 64, 300
    g = torch.Generator(device="cuda").manual_seed(0)
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, k, v, do, qkv = rnd(T, Hq, d), rnd(T, Hkv, d), rnd(T, Hkv, d), rnd(T, Hq, d), rnd(T, Hq + 2 * Hkv, d)
    ev = (torch.arange(T, device="cuda") + 100).int()
    first, perm, cu = torch.arange(T, device="cuda").int(), torch.arange(T - 1, -1, -1, device="cuda").int(), torch.tensor([0, T], device="cuda").int()
    kn, vn, qn = rnd(2, Hkv, d), rnd(2, Hkv, d), rnd(2, Hq, d)
    size = B.kvs_mask_meta_bytes(1, T, T)
    workspace = torch.zeros(B.kvs_attn_bwd_workspace_bytes(T, Hq, Hkv, d, B.GRAD_FP32), dtype=torch.uint8, device="cuda")
    scratch = torch.zeros(1 << 22, dtype=torch.uint8, device="cuda")
    caches = [B.PagedCache(4, 16, 2, 2, Hkv, d) for _ in range(2)]

    def buffers():
        new = lambda like, dtype=None: torch.full_like(like, -1, dtype=dtype)  # noqa: E731
        lse = lambda: torch.full((Hq, T), -1.0, device="cuda")  # noqa: E731
        return dict(meta=[torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in range(3)], fwd=[new(q), lse()], packed=[new(q), lse()],
                    dual=[new(q), lse(), new(q), lse()], bwd=[new(t, torch.float32) for t in (q, k, v)], dqkv=[new(qkv, torch.float32)],
                    rows=[new(k)], rope=[new(q), new(k)], decode=[new(qn), torch.full((2, Hq), -1.0, device="cuda")])

    def calls(b, cache, stream):
        m = b["meta"]
        B.kvs_mask_meta(ev, cu, T, m[0], stream=stream)
        B.kvs_mask_meta_evicted(ev, cu, T, m[1], stream=stream)
        B.kvs_mask_meta_keys(first, ev, cu, T, m[2], stream=stream)
        B.kvs_attn_fwd(q, k, v, m[2], 1, T, 0.0, *b["fwd"], stream=stream)
        B.kvs_attn_fwd_packed(qkv, m[0], 1, T, Hq, Hkv, 0.0, *b["packed"], stream=stream)
        B.kvs_attn_fwd_dual(q, k, v, m[0], m[1], 1, T, 0.0, *b["dual"], stream=stream)
        B.kvs_attn_bwd(do, q, k, v, *b["fwd"], m[2], 1, T, 0.0, B.GRAD_FP32, *b["bwd"], workspace, stream=stream)
        B.kvs_attn_bwd_packed(do, qkv, *b["packed"], m[0], 1, T, Hq, Hkv, 0.0, B.GRAD_FP32, *b["dqkv"], workspace, stream=stream)
        B.kvs_permute_rows(k, perm, b["rows"][0], True, stream=stream)
        B.kvs_rope_qk(q, k, cu, q_out=b["rope"][0], k_out=b["rope"][1], stream=stream)
        cache.append(kn, vn, stream=stream)
        cache.decode(qn, 0.0, 1, *b["decode"], scratch, stream=stream)

    want, got, side = buffers(), buffers(), torch.cuda.Stream()
    calls(want, caches[0], None)
    torch.cuda.synchronize()
    torch.cuda._sleep(1 << 31)
    busy = torch.cuda.Event()
    busy.record()
    calls(got, caches[1], side)
    with torch.cuda.stream(side):
        copies = {n: [t.cpu() for t in x] for n, x in got.items() if n != "meta"}
    assert not busy.query()
    torch.cuda.synchronize()
    for n, x in copies.items():
        for a, b in zip(x, want[n]):
            # dq: two key blocks and more are added in the order of arrival, in fp32
            assert torch.allclose(a.float(), b.cpu().float(), rtol=0, atol=1e-5 if n in ("bwd", "dqkv") else 0), n
