"""Early stops of Alg. 2 (FP32 values of seven digits, FP16 values of three) by place: none, or one value that
stops early among values that do not, at the first and last place of lanes, 16-byte units and tails, as its
lane's largest value or below it.  Streams against the oracle byte for byte (tolerance 0)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DIGITS = {np.float32: 7, np.float16: 3}
SENTINEL = {np.float32: 11, np.float16: 5}         # alpha byte of a Case-2 record


@pytest.fixture(scope="module")
def F():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2511_04140_gb300 import build
    build.build()
    from paper_2511_04140_gb300 import falcon
    return falcon


@pytest.fixture(scope="module")
def decimals(oracle):
    """dtype -> (values that are Case 1 by themselves, values that stop early), of the most digits."""
    out = {}
    for dtype, p in DIGITS.items():
        k = np.random.default_rng(p).permutation(np.arange(10 ** (p - 1), 10 ** p, 1 if p < 4 else 97))[:20000]
        v = np.unique((k / 10.0 ** p).astype(dtype))
        s = oracle.compress(np.repeat(v, 2), 2)    # a chunk for each value
        sizes = np.frombuffer(s[32:32 + 4 * len(v)], np.uint32)
        at = 32 + 4 * len(v) + np.cumsum(sizes, dtype=np.int64) - sizes
        stops = np.frombuffer(s, np.uint8)[at] == SENTINEL[dtype]
        out[dtype] = v[~stops], v[stops]
        assert len(out[dtype][0]) > 100 and len(out[dtype][1]) > 5
    return out


def check(F, oracle, vals, block):
    got = F.compress(torch.from_numpy(vals).cuda(), block).cpu().numpy().tobytes()
    assert got == oracle.compress(vals, block)
    return got


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("n,block", [(1, 1024), (2, 1024), (3, 2), (31, 1024), (33, 1024), (500, 64), (1023, 1024), (1024, 1024),
                                     (1025, 1025), (1025, 1024), (1057, 1024), (2047, 1024), (4000, 1000)])
def test_places(F, oracle, decimals, dtype, n, block):
    good, stop = decimals[dtype]
    rng = np.random.default_rng(n)
    few = good[rng.integers(0, len(good), 8)]      # chunks of few values, so that many are Case 1
    for base in (rng.choice(few, n), np.sort(rng.choice(good, n)), np.full(n, good[0], dtype), np.full(n, good[-1], dtype)):
        base = base.astype(dtype)
        check(F, oracle, base, block)
        for place in {0, 1, 3, 4, 7, 8, 31, 32, 63, 991, 992, 1022, 1023, 1024, n - 2, n - 1, n // 2}:
            if 0 <= place < n:
                for v in (stop.min(), stop.max(), -stop[len(stop) // 2]):
                    vals = base.copy()
                    vals[place] = v
                    check(F, oracle, vals, block)


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
def test_only_early_stops(F, oracle, decimals, dtype):
    _, stop = decimals[dtype]
    for n in (1, 2, 30, 1023, 1025, 5000):
        check(F, oracle, np.resize(stop, n), 1024)


def test_some_chunks_are_case_1(F, oracle, decimals):
    for dtype in (np.float32, np.float16):
        got = check(F, oracle, np.full(1024, decimals[dtype][0][-1], dtype), 1024)
        assert got[36] != SENTINEL[dtype]
