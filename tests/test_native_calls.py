"""The native calls of the binding refuse what the path does not take, as Python errors (no GPU needed)."""
import pytest
import torch

from paper_2609_35750_b200 import binding as B

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
