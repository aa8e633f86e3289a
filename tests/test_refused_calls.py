"""A call that the CUDA runtime refuses leaves nothing behind (needs a B200).

The refusal is made on the host, before anything reaches the GPU: a launch into the legacy stream while a stream that
synchronises with it is being captured."""
import pytest
import torch
from cuda.bindings import driver

from paper_2609_35750_b200 import binding as B

pytestmark = pytest.mark.gpu


def _next_call_is_fine(cu):
    # this entry point checks its launches by the runtime's last error
    ev = B.kvs_evict_at_from_events(torch.tensor([[0, 7, 1, 3]], dtype=torch.int32, device="cuda"), cu, 4)
    assert ev.tolist() == [2 ** 31 - 1, 7, 7, 2 ** 31 - 1]


def _ok(result):
    assert result[0] == driver.CUresult.CUDA_SUCCESS, result[0]
    return result[1] if len(result) > 1 else None


def test_refused_launch():
    cache = B.PagedCache(4, 16, 1, 4, 2, 64)
    new = torch.ones((1, 2, 64), dtype=torch.bfloat16, device="cuda")
    cu = torch.tensor([0, 4], dtype=torch.int32, device="cuda")
    _next_call_is_fine(cu)
    torch.cuda.synchronize()
    blocking = _ok(driver.cuStreamCreate(driver.CUstream_flags.CU_STREAM_DEFAULT))
    _ok(driver.cuStreamBeginCapture(blocking, driver.CUstreamCaptureMode.CU_STREAM_CAPTURE_MODE_RELAXED))
    with pytest.raises(B.KvsError) as refused:
        cache.append(new, new)                              # legacy stream: would have to wait for the captured one
    driver.cuStreamEndCapture(blocking)                     # the capture is void by now
    _ok(driver.cuStreamDestroy(blocking))
    assert refused.value.code == B.KVS_ERR_CUDA
    _next_call_is_fine(cu)
    cache.append(new, new)
    assert cache.n_tokens.tolist() == [1] and cache.status() == (B.KVS_OK, 3)
