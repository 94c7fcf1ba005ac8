"""Streams of the oracle's own encoder with every row sparse, every row dense and mixed, in every dtype and
at block sizes from one row word up, tails included: decoded bit for bit, and the library's streams of the
same variant byte for byte (tolerance 0)."""
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


@pytest.mark.parametrize("variant", ["VARIANT_SPARSE", "VARIANT_DENSE", "VARIANT_FALCON"])
@pytest.mark.parametrize("block", [2, 65, 129, 1000, 1024, 1025])
@pytest.mark.parametrize("dtype", [np.float64, np.float32, np.float16])
def test_rows(F, oracle, dtype, block, variant):
    n = 3 * block + 7
    rng = np.random.default_rng(block)
    segments = synth.segments_f16(n, seed=2) if dtype == np.float16 else synth.segments(n, seed=2, dtype=dtype)
    for vals in (synth.random_walk(n, seed=1, places=1).astype(dtype), rng.standard_normal(n).astype(dtype), segments,
                 np.zeros(n, dtype)):
        s = oracle.compress(vals, block, getattr(F, variant))
        y = F.decompress(torch.frombuffer(bytearray(s), dtype=torch.uint8).cuda())
        assert y.cpu().numpy().tobytes() == vals.tobytes()
        got = F.compress_variant(torch.from_numpy(vals).cuda(), block, getattr(F, variant))
        assert got.cpu().numpy().tobytes() == s
