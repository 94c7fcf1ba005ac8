"""Job tables around the chunk lookup's steps of 32 jobs, empty series and all dtypes in turn: each
stream against the oracle byte for byte, each decoded series bit for bit (tolerance 0).  And single streams
around the count of chunks up to which the emit adds record sizes up itself."""
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


@pytest.mark.parametrize("count", [1, 31, 32, 33, 64, 1023, 1024, 1025, 1057])
def test_tables(F, oracle, count):
    rng = np.random.default_rng(count)
    series = []
    for i in range(count):
        n = int(rng.choice([0, 0, 1, 30, 64, 65, 130]))
        make = (synth.random_walk, lambda n, seed: synth.random_walk(n, seed=seed, dtype=np.float32), synth.segments_f16)
        series.append(make[i % 3](n, seed=i) if n else np.zeros(0, (np.float64, np.float32, np.float16)[i % 3]))
    block = 64
    b = F.Batch(F.COMPRESS, [torch.from_numpy(np.ascontiguousarray(s)).cuda() for s in series], block=block)
    b.launch()
    torch.cuda.synchronize()
    streams = b.streams()
    for s, (nb, st), out in zip(series, b.results(), streams):
        assert st == 0
        assert out.cpu().numpy().tobytes() == oracle.compress(s, block)
    dec = F.Batch(F.DECOMPRESS, [(o, o.numel(), o[:32].cpu().numpy().tobytes()) for o in streams])
    dec.launch()
    torch.cuda.synchronize()
    for s, (nv, st), y in zip(series, dec.results(), dec.outputs):
        assert st == 0 and nv == len(s)
        assert y[:len(s)].cpu().numpy().tobytes() == s.tobytes()
    b.close()
    dec.close()


@pytest.mark.parametrize("chunks", [1, 2, 31, 33, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("tail", [0, 1])
def test_chunk_counts(F, oracle, chunks, tail):
    vals = synth.segments(8 * chunks - 7 * tail, seed=chunks, dtype=np.float32)
    out = F.compress(torch.from_numpy(vals).cuda(), 8)
    assert out.cpu().numpy().tobytes() == oracle.compress(vals, 8)
    assert F.decompress(out).cpu().numpy().tobytes() == vals.tobytes()
