"""The decoder's paths by alignment and magnitude, each against the oracle bit for bit (tolerance 0):
whole-sector stores of 32-byte aligned FP64 chunks, staged 16-byte units, single values elsewhere;
records whose rows are all sparse, all dense or mixed; Case-1 chunks whose integers all fit 32 bits
(the 96-bit reciprocal) next to chunks one step beyond; record positions over several CTAs' shares."""
import numpy as np
import pytest
import torch

from paper_2511_04140_gb300 import synth
from test_gpu_case1_decode import stream_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2511_04140_gb300 import build
    build.build()
    from paper_2511_04140_gb300 import falcon
    return falcon


def _u(a):
    return a.view({8: np.uint64, 4: np.uint32, 2: np.uint16}[a.dtype.itemsize])


@pytest.mark.parametrize("shift", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("n,block", [(3 * 1024, 1024), (3 * 1025 + 40, 1025), (2 * 1000 + 1, 1000), (2048 + 33, 1024)])
def test_output_alignment(F, oracle, shift, n, block):
    for vals in (synth.segments(n, seed=5), synth.segments(n, seed=6, dtype=np.float32), synth.segments_f16(n, seed=7)):
        s = torch.frombuffer(bytearray(oracle.compress(vals, block)), dtype=torch.uint8).cuda()
        room = torch.zeros(n + 64, dtype=torch.from_numpy(vals[:1]).dtype, device="cuda")
        y = F.decompress(s, out=room[shift:shift + n])
        assert np.array_equal(_u(y.cpu().numpy()), _u(vals))
        assert not room[:shift].any() and not room[shift + n:].any()          # nothing outside


@pytest.mark.parametrize("variant", ["VARIANT_SPARSE", "VARIANT_DENSE", "VARIANT_FALCON"])
@pytest.mark.parametrize("block", [65, 129, 1000, 1024, 1025])
def test_row_mixes(F, variant, block):
    rng = np.random.default_rng(block)
    for vals in (synth.random_walk(3 * block + 7, seed=1), rng.standard_normal(3 * block + 7),
                 synth.segments(3 * block + 7, seed=2, dtype=np.float32), synth.segments_f16(3 * block + 7, seed=3)):
        s = F.compress_variant(torch.from_numpy(vals).cuda(), block, getattr(F, variant))
        assert np.array_equal(_u(F.decompress(s).cpu().numpy()), _u(vals))


@pytest.mark.parametrize("alpha", range(23))
def test_case1_32_bit_boundary(F, oracle, alpha):
    rng = np.random.default_rng(alpha)
    lim = 1 << 31
    g = [0, 1, -1, lim - 1, -lim, -(lim - 1), lim // 2, 10 ** 9]
    g += [k * 5 ** alpha + d for k in (1, 2, 3, 7) for d in (-2, -1, 0, 1, 2) if k * 5 ** alpha + 2 < lim]
    g += list(rng.integers(-lim, lim, 1024 - len(g)))                          # one chunk within 32 bits
    wide = list(rng.integers(-lim, lim, 1024))
    wide[int(rng.integers(0, 1024))] = lim                                     # one step beyond
    gs = np.array(g + wide + [-lim - 1, 5], dtype=np.int64)
    s = stream_of(oracle, gs, alpha, 15, 0, 1024)
    got = F.decompress(torch.frombuffer(bytearray(s), dtype=torch.uint8).cuda()).cpu().numpy()
    assert np.array_equal(got.view(np.uint64), oracle.decompress(s).view(np.uint64))


@pytest.mark.parametrize("chunks", [1023, 1024, 1025, 5000, 152 * 1024 + 1])
def test_record_positions_over_shares(F, oracle, chunks):
    vals = synth.random_walk(2 * chunks - 1, seed=chunks % 11, dtype=np.float32)
    s = torch.frombuffer(bytearray(oracle.compress(vals, 2)), dtype=torch.uint8).cuda()
    assert np.array_equal(_u(F.decompress(s).cpu().numpy()), _u(vals))


def test_synchronous_calls_on_other_streams_and_many_threads(F, oracle):
    """The synchronous calls on streams of their own, from several threads at once: every result is the
    one-thread result."""
    import threading
    vals = synth.random_walk(3000, seed=1)
    want = oracle.compress(vals, 1024)
    x = torch.from_numpy(vals).cuda()
    y = F.decompress(F.compress(x, 1024, stream=torch.cuda.Stream()), stream=torch.cuda.Stream())
    assert np.array_equal(_u(y.cpu().numpy()), _u(vals))
    torch.cuda.synchronize()
    bad = []

    streams = {s.cuda_stream: s for s in (torch.cuda.Stream() for _ in range(24))}    # distinct ones

    def work(st):
        with torch.cuda.stream(st):
            for _ in range(10):
                s = F.compress(x, 1024)
                if s.cpu().numpy().tobytes() != want or not torch.equal(F.decompress(s), x):
                    bad.append(1)

    threads = [threading.Thread(target=work, args=(st,)) for st in streams.values()]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    s = torch.frombuffer(bytearray(want[:20]), dtype=torch.uint8).cuda()
    with pytest.raises(F.FalconError) as e:
        F.decompress(s)
    assert e.value.status == F.ERR_CORRUPT
