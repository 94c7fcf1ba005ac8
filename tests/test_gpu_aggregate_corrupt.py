"""The asynchronous aggregate of a stream with rejected records, whatever the workspace held before: the
status says so, and the other chunks' values alone make count, min, max and sum (whole numbers, so that
every order of additions gives the same sum; tolerance 0)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

W = {np.float64: 64, np.float32: 32, np.float16: 16}


@pytest.fixture(scope="module")
def F():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2511_04140_gb300 import build
    build.build()
    from paper_2511_04140_gb300 import falcon
    return falcon


@pytest.mark.parametrize("fill", [0x00, 0xFF, 0x40])
@pytest.mark.parametrize("how", ["size", "width", "flags"])
@pytest.mark.parametrize("dtype", [np.float64, np.float32, np.float16])
def test_rejected_chunks_add_nothing(F, oracle, dtype, how, fill):
    block, chunks = 64, 200
    vals = np.random.default_rng(3).integers(-500, 500, block * chunks).astype(dtype)
    s = bytearray(oracle.compress(vals, block))
    sizes = np.frombuffer(bytes(s[32:32 + 4 * chunks]), np.uint32).copy()
    starts = 32 + 4 * chunks + np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(int)
    width_at = 2 + W[dtype] // 8
    kept = np.ones(chunks, bool)
    for c in ([chunks - 1] if how == "size" else [0, 7, 8, 150, chunks - 1]):
        at = int(starts[c])
        if how == "size":                         # the last chunk's: no other record moves
            s[32 + 4 * c:36 + 4 * c] = (5).to_bytes(4, "little")
        elif how == "width":
            s[at + width_at] = 200
        else:
            assert s[at + width_at] > 0
            s[at + width_at + (s[at + width_at] + 7) // 8] ^= 1           # plane 0 in the other form
        kept[c] = False
    rest = vals.reshape(chunks, block)[kept].astype(np.float64)
    d = torch.frombuffer(s, dtype=torch.uint8).cuda()
    ws = torch.full((F.workspace_bytes(chunks),), fill, dtype=torch.uint8, device="cuda")
    st = torch.zeros(F.STATS_BYTES, dtype=torch.uint8, device="cuda")
    F.aggregate_async(d, d.numel(), bytes(s[:32]), ws, st)
    got = F.stats_of(st)
    assert got["status"] == F.ERR_CORRUPT
    assert got["count"] == len(vals) and got["nan_count"] == 0
    assert (got["min"], got["max"], got["sum"]) == (rest.min(), rest.max(), rest.sum())
