"""Calls go to the current stream of the current device."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_stream_handle_follows_the_current_stream():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_01580_gb300 import qmlr as q
    assert (q._stream().value or 0) == torch.cuda.default_stream().cuda_stream
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert q._stream().value == s.cuda_stream
        # work queued behind the stream's own: the grouping sees the elements that the copy before it writes
        elem = torch.zeros(5000, dtype=torch.int32, device="cuda")
        torch.cuda._sleep(2_000_000)
        elem.copy_(torch.arange(5000, dtype=torch.int32, device="cuda") % 5)
        perm, offs = q.group_by_element(elem, 5)
    s.synchronize()
    assert offs.tolist() == [0, 1000, 2000, 3000, 4000, 5000]
    assert torch.equal(perm[:3].cpu(), torch.tensor([0, 5, 10], dtype=torch.int32))
    assert (q._stream().value or 0) == torch.cuda.default_stream().cuda_stream
