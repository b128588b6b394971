"""Scratch of a call is asked for, and given back, on the call's own stream: a block that is free on the
stream the handle was made on may still be in use there."""
import pytest
import torch

from paper_2308_00106_gb300 import maxe
from tests.test_gpu_order_scratch import CountingAllocator, _handle

pytestmark = pytest.mark.gpu


class StreamAllocator(CountingAllocator):
    def __init__(self):
        self.streams = []
        super().__init__()

    def _alloc(self, nbytes, ctx, stream):
        self.streams.append(stream or 0)
        return super()._alloc(nbytes, ctx, stream)

    def _free(self, p, ctx, stream):
        self.streams.append(stream or 0)
        super()._free(p, ctx, stream)


@pytest.mark.parametrize("call", ["power", "spmm", "tune"])
def test_scratch_is_on_the_stream_of_the_call(call):
    al = StreamAllocator()
    h, _, _ = _handle(5003, "f32", al)
    made_on = torch.cuda.current_stream().cuda_stream
    assert set(al.streams) == {made_on}
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    al.streams.clear()
    if call == "power":
        maxe.maxe_power_iteration(h, torch.ones(h.cols, device="cuda"), 3, stream=s)
    elif call == "spmm":
        maxe.maxe_spmm(h, torch.ones(h.cols, 9, device="cuda"), stream=s)
    else:
        maxe.maxe_batch_tune(h, 4, stream=s)
    assert al.streams and set(al.streams) == {s.cuda_stream}
    torch.cuda.synchronize()
    h.close()
    assert not al.live
