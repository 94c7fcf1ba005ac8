"""Record positions of job tables: counts of jobs at which the jobs per CTA change (one, two, 32), and jobs
of the chunk counts at which a warp's work passes to its CTA (32 chunks for each job of the CTA), empty ones
among them, in both directions.  Streams against the oracle byte for byte, values bit for bit (tolerance 0)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2511_04140_gb300 import build
    build.build()
    from paper_2511_04140_gb300 import falcon
    return falcon


@pytest.mark.parametrize("jobs,edge", [(304, 32), (305, 64), (608, 64), (609, 96), (9700, 1024), (9729, 1024), (9999, 1024)])
def test_job_and_chunk_counts(F, oracle, jobs, edge):
    rng = np.random.default_rng(jobs)
    block = 2
    lens = rng.integers(0, 9, jobs)
    special = [edge * block, edge * block - 1, edge * block + 1, 33 * block, 32 * block, 1025 * block, 2500 * block, 0]
    at = rng.choice(jobs, 4 * len(special), replace=False)
    lens[at] = special * 4
    lens[-1] = edge * block + 1                   # the last CTA has fewer jobs
    series = [np.round(rng.standard_normal(n), 1).astype((np.float64, np.float32, np.float16)[i % 3]) for i, n in enumerate(lens)]
    want = [oracle.compress(s, block) for s in series]
    room = [torch.empty(max(32, F.bound(len(s), i % 3, block)), dtype=torch.uint8, device="cuda") for i, s in enumerate(series)]
    b = F.Batch(F.COMPRESS, [torch.from_numpy(s).cuda() for s in series], block=block, outputs=room)
    for _ in range(2):
        b.launch()
    torch.cuda.synchronize()
    assert b.results() == [(len(w), 0) for w in want]
    streams = b.streams()
    got = torch.cat(streams).cpu().numpy().tobytes()
    assert got == b"".join(want)
    dec = F.Batch(F.DECOMPRESS, [(o, o.numel(), w[:32]) for o, w in zip(streams, want)])
    for _ in range(2):
        dec.launch()
    torch.cuda.synchronize()
    assert dec.results() == [(len(s), 0) for s in series]
    for s, y in zip(series, dec.outputs):
        assert y[:len(s)].cpu().numpy().tobytes() == s.tobytes()
    b.close()
    dec.close()
