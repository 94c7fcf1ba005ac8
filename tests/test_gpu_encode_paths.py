"""The encoder's paths by alignment, tail and row mix, each stream against the oracle byte for byte
(tolerance 0): value loads at every alignment (whole sectors, 16-byte units, the 8-modulo-16 window at
both ends of the input, single values), tail chunks of every phase, chunks whose largest value lies at
a power of ten, and chunks from a few to all rows sparse (groups of four sparse rows, filled up)."""
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


def check(F, oracle, vals, block, shift=0):
    room = np.concatenate([np.zeros(shift, vals.dtype), vals])
    x = torch.from_numpy(room).cuda()[shift:]
    assert F.compress(x, block).cpu().numpy().tobytes() == oracle.compress(vals, block)


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 4, 7])
@pytest.mark.parametrize("n,block", [(1024, 1024), (1025, 1025), (2 * 1024, 1024), (3 * 1025, 1025), (3 * 1025 + 1, 1025),
                                     (2 * 1000 + 1, 1000), (4 * 1024 + 1, 1024), (2 * 1025 + 1024, 1025)])
def test_value_alignment(F, oracle, shift, n, block):
    for vals in (synth.segments(n, seed=5), synth.random_walk(n, seed=2, places=3),
                 synth.segments(n, seed=6, dtype=np.float32), synth.segments_f16(n, seed=7)):
        check(F, oracle, vals, block, shift)


@pytest.mark.parametrize("tail", [1, 2, 3, 31, 32, 33, 63, 64, 65, 66, 511, 992, 993, 1022, 1023])
def test_tails(F, oracle, tail):
    for vals in (synth.random_walk(1024 + tail, seed=tail, places=2), synth.segments(1024 + tail, seed=tail),
                 synth.random_walk(1024 + tail, seed=tail, places=1, dtype=np.float32),
                 synth.segments_f16(1024 + tail, seed=tail)):
        check(F, oracle, vals, 1024)


@pytest.mark.parametrize("k", range(-4, 15))
def test_largest_value_at_a_power_of_ten(F, oracle, k):
    """Two largest values on both sides of 10^k that agree in their upper bits, in either order."""
    rng = np.random.default_rng(k + 50)
    for places in (0, 3, max(0, 14 - k), max(0, 15 - k)):
        unit = 10 ** max(0, k + places)
        if k + places < 0 or unit >= 1 << 52:
            continue
        for below, above in ((unit - 1, unit), (unit - 1, unit + 1), (unit, unit - 1), (unit - 2, unit - 1)):
            d = rng.integers(-unit // 2, unit // 2 + 1, 1024)
            d[100], d[900] = below, above
            check(F, oracle, synth.decimal_to_f64(d, min(places, 22)), 1024)


@pytest.mark.parametrize("dtype,digits", [(np.float64, 8), (np.float64, 9), (np.float64, 14), (np.float32, 6), (np.float32, 7)])
@pytest.mark.parametrize("places", [0, 1, 2, 3, 4, 6, 9, 13, 14])
def test_decimals_of_every_size(F, oracle, dtype, digits, places):
    """Decimals of 0 to `digits` digits in one chunk (zeros, the smallest, both sides of the 32-bit
    arithmetic's limit), then chunks with one value an ulp beside its decimal."""
    rng = np.random.default_rng(places + 100 * digits)
    d = np.trunc(rng.choice([-1.0, 1.0], 4 * 1025) * 10.0 ** rng.uniform(-0.5, digits, 4 * 1025)).astype(np.int64)
    vals = (d.astype(np.float64) / 10.0 ** places).astype(dtype) + dtype(0)         # no -0
    for i, at in ((1, 5), (2, 1024), (3, 700)):
        vals[1025 * i + at] = np.nextafter(vals[1025 * i + at], dtype(np.inf if i == 1 else -np.inf))
    vals += dtype(0)
    check(F, oracle, vals, 1025)


@pytest.mark.parametrize("dtype", [np.float64, np.float32, np.float16])
@pytest.mark.parametrize("block", [64, 65, 1000, 1024, 1025])
def test_row_mixes(F, oracle, dtype, block):
    rng = np.random.default_rng(block)
    bits = {8: np.uint64, 4: np.uint32, 2: np.uint16}[np.dtype(dtype).itemsize]
    top = 8 * np.dtype(dtype).itemsize
    chunks = []
    for i in range(70):
        v = np.zeros(block, bits)
        cnt = min(block, 1 << rng.integers(0, 11))
        pos = rng.choice(block, cnt, replace=False)
        width = int(rng.integers(1, top + 1))                   # rows 1 .. width in use
        v[pos] = rng.integers(0, 1 << 62, cnt, dtype=np.uint64).astype(bits) >> bits(top - width)
        chunks.append(np.cumsum(v, dtype=bits) if i % 3 == 0 else v)
    check(F, oracle, np.concatenate(chunks).view(dtype), block)


def test_all_variants_of_mixed_rows(F, oracle):
    vals = synth.segments(5 * 1025 + 3, seed=3)
    for dtype in (np.float64, np.float32):
        v = vals.astype(dtype)
        for variant in (F.VARIANT_SPARSE, F.VARIANT_DENSE, F.VARIANT_ELF):
            s = F.compress_variant(torch.from_numpy(v).cuda(), 1025, variant)
            assert s.cpu().numpy().tobytes() == oracle.compress(v, 1025, variant)
