"""Job tables whose warps meet chunks of all three dtypes one after the other, with records longer than
a narrower kind's whole buffer (full-precision values): one warp on each SM and several chunks per warp,
so that every warp draws tickets, reuses its buffers and changes dtype.  Each stream against the oracle
byte for byte, each decoded series bit for bit (tolerance 0), over repeated launches."""
import numpy as np
import pytest
import torch

from paper_2511_04140_gb300 import synth

pytestmark = pytest.mark.gpu

DTYPES = (np.float64, np.float32, np.float16)


@pytest.fixture(scope="module")
def F():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2511_04140_gb300 import build
    build.build()
    from paper_2511_04140_gb300 import falcon
    falcon.set_cta_warps(1, 1)
    falcon.set_launch_config(1, 1)
    yield falcon
    falcon.set_cta_warps(4, 4)
    falcon.set_launch_config(0, 0)


def full_precision(n, dtype, seed):
    """Every bit of the significand in use: Case 2, nearly every row dense."""
    return np.random.default_rng(seed).standard_normal(n).astype(dtype)


def run(F, oracle, series, block, launches=10):
    want = [oracle.compress(s, block) for s in series]
    b = F.Batch(F.COMPRESS, [torch.from_numpy(s).cuda() for s in series], block=block)
    for _ in range(launches):
        for o in b.outputs:
            o.zero_()
        b.launch()
        torch.cuda.synchronize()
        assert [(len(w), 0) for w in want] == b.results()
        for w, s in zip(want, b.streams()):
            assert s.cpu().numpy().tobytes() == w
    dec = F.Batch(F.DECOMPRESS, [(o, o.numel(), w[:32]) for o, w in zip(b.streams(), want)])
    for _ in range(launches):
        for o in dec.outputs:
            o.zero_()
        dec.launch()
        torch.cuda.synchronize()
        for s, (nv, st), y in zip(series, dec.results(), dec.outputs):
            assert st == 0 and nv == len(s) and y[:len(s)].cpu().numpy().tobytes() == s.tobytes()
    b.close()
    dec.close()


@pytest.mark.parametrize("block", [1024, 1025])
@pytest.mark.parametrize("kinds", [(0, 1, 2), (0, 1), (0, 2), (1, 2)])
def test_dtypes_change_within_a_warp(F, oracle, kinds, block):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # as many chunks of each kind as warps, in series of one to three chunks: the table is in dtype order,
    # so nearly every warp goes from each kind to the next
    series = []
    for k in kinds:
        left = sms
        while left > 0:
            c = min(left, 1 + len(series) % 3)
            series.append(full_precision(c * block - len(series) % 2, DTYPES[k], 100 * k + len(series)))
            left -= c
    run(F, oracle, series, block)


def test_many_chunks_per_warp(F, oracle):
    series = []
    for i in range(40):
        n = 5 * 1024 * (1 + i % 7) + i
        series.append(full_precision(n, DTYPES[i % 3], i) if i % 2 else
                      (synth.random_walk(n, seed=i) if i % 3 == 0 else
                       synth.segments(n, seed=i, dtype=np.float32) if i % 3 == 1 else synth.segments_f16(n, seed=i)))
    run(F, oracle, series, 1024, launches=3)


def test_server_tables_in_request_order(F, oracle):
    """The server's tables stay in request order, so the kinds alternate there."""
    from paper_2511_04140_gb300.serve import Server
    payloads = [full_precision(1024 * (1 + i % 2), DTYPES[i % 3], i) for i in range(600)]
    host = [torch.from_numpy(p).pin_memory() for p in payloads]
    with Server(budget_bytes=256 << 20, host_budget_bytes=128 << 20) as srv:
        futs = [srv.submit("compress", h) for h in host]
        outs = [f.result(timeout=120).numpy().tobytes() for f in futs]
        assert srv.stats["multi_request_batches"] >= 1
    for p, o in zip(payloads, outs):
        assert o == oracle.compress(p, 1024)
