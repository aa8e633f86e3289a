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
    # An allocation may wait (for the device, or as here for 500 MB to be filled); it is refused afterwards for being on the host
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
    assert took > 0.02 and n >= took / 0.02, (took, n)        # a tick takes a millisecond; held up, there are at most two


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
