"""decompress of tensors that are no plain run of bytes: a strided view whose bytes start no stream is a
corrupt stream, whatever lies in memory at its first byte; views that do start one decode bit for bit."""
import numpy as np
import pytest
import torch

from paper_2511_04140_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2511_04140_gb300 import build
    build.build()
    from paper_2511_04140_gb300 import falcon
    return falcon


@pytest.fixture(scope="module")
def stream(oracle):
    vals = synth.random_walk(3000, seed=4)
    return vals, torch.frombuffer(bytearray(oracle.compress(vals, 1024)), dtype=torch.uint8).cuda()


@pytest.mark.parametrize("step", [2, 3, 4, 7, 16])
def test_strided_view_over_a_stream(F, stream, step):
    _, s = stream
    room = torch.zeros(step * s.numel(), dtype=torch.uint8, device="cuda")
    room[:s.numel()] = s                         # a whole stream at the view's first byte
    with pytest.raises(F.FalconError) as e:
        F.decompress(room[::step])
    assert e.value.status == F.ERR_CORRUPT


def test_views_that_start_a_stream(F, stream):
    vals, s = stream
    rows = torch.zeros((4, s.numel() + 64), dtype=torch.uint8, device="cuda")
    rows[0, :s.numel()] = s
    for view in (s.view(1, -1), rows[0, :s.numel()], rows[:, :s.numel()]):
        y = F.decompress(view)
        assert np.array_equal(y.cpu().numpy().view(np.uint64), vals.view(np.uint64))
