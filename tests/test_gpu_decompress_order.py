"""decompress on a stream of the caller's choice reads the header in that stream's order: buffers that hold
an older stream when the call is made, and get the new one from work still in flight on the stream itself, on
another stream it waits for, or on the current stream.  Values bit for bit (tolerance 0)."""
import numpy as np
import pytest
import torch

from paper_2511_04140_gb300 import synth

pytestmark = pytest.mark.gpu

SOME_MS = 20_000_000                              # clock cycles of a waiting kernel


@pytest.fixture(scope="module")
def F():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2511_04140_gb300 import build
    build.build()
    from paper_2511_04140_gb300 import falcon
    return falcon


@pytest.mark.parametrize("old_n,new_n", [(1000, 1020), (1020, 1000), (1000, 5000), (5000, 1000)])
@pytest.mark.parametrize("producer", ["same", "joined", "current"])
@pytest.mark.parametrize("given", [True, False])
def test_buffer_written_again(F, old_n, new_n, producer, given):
    old = torch.from_numpy(synth.random_walk(old_n, seed=1)).cuda()
    new = torch.from_numpy(synth.random_walk(new_n, seed=2)).cuda()
    most = max(old_n, new_n)
    buf = torch.zeros(F.bound(most, F.F64), dtype=torch.uint8, device="cuda")
    ws = torch.empty(F.workspace_bytes(8), dtype=torch.uint8, device="cuda")
    res = torch.zeros(2, dtype=torch.int64, device="cuda")
    out = torch.zeros(most, dtype=torch.float64, device="cuda")
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    writer = {"same": side, "joined": other, "current": torch.cuda.current_stream()}[producer]
    for st in (side, other):                      # the kernels are loaded before the ordering matters
        F.decompress(F.compress(new, stream=st), stream=st)
    F.compress_async(old, 1024, buf, ws, res)
    torch.cuda.synchronize()
    with torch.cuda.stream(writer):
        torch.cuda._sleep(SOME_MS)
    F.compress_async(new, 1024, buf, ws, res, stream=writer)
    if producer == "joined":
        side.wait_stream(other)
    y = F.decompress(buf, out=out if given else None, stream=side)
    assert y.numel() == new_n
    assert np.array_equal(y.cpu().numpy().view(np.uint64), new.cpu().numpy().view(np.uint64))
