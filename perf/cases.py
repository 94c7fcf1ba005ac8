"""What a user of libfalcon has it do, as measurable cases.

A case is one call, or a compress call and the decompress call of its result, through the
public binding (``paper_2511_04140_gb300.falcon``) on inputs made on the GPU from a seed alone.

  op        "compress" / "decompress": the asynchronous entry points with the caller's buffers and
            workspace, as a resident program or a captured graph calls them;
            "roundtrip": both, one after the other on the same stream;
            "sync": falcon.compress (into the caller's buffer) then falcon.decompress, which wait;
            "aggregate": count, NaN count, min, max and sum from a stream, without its values;
            "batch": many series of both wide dtypes and uneven lengths, one planned launch per direction;
            "pipeline": page-locked host values through the device in frames, and back.
  kind      "walk": random walk with steps N(0, 0.5) rounded to `places` decimals; "outliers": the same
            with 0.5 % full-precision outliers (nearly every 1024-value chunk holds one);
            "segments": 4096-value segments, 0..6 decimal places each, sinusoid plus AR(1) noise, 1 %
            outliers and 0.01 % NaN / infinities / subnormals / -0; "decimal": segments without
            outliers and specials.  FP16 segments have amplitude 10^U(-1,1), 0..2 places, 0.01 % outliers.
  dtype     "f64", "f32" or "f16"; n: values; block: values per chunk (1024 is the binding's default,
            1025 the paper's chunk, whose chunk starts are not 16-byte aligned).

Values come back as their bit patterns: the codec is lossless, so every bit counts.
"""
from __future__ import annotations

import torch

from paper_2511_04140_gb300 import falcon

_DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}
_BITS = {"f64": torch.int64, "f32": torch.int32, "f16": torch.int16}
_SIZE = {"f64": 8, "f32": 4, "f16": 2}
_CODE = {"f64": falcon.F64, "f32": falcon.F32, "f16": falcon.F16}

# stream bytes / value bytes of the generators, for work()
_RATIO = {("walk", "f64"): 0.13, ("outliers", "f64"): 0.77, ("segments", "f64"): 0.78, ("decimal", "f64"): 0.20,
          ("walk", "f32"): 0.26, ("outliers", "f32"): 0.68, ("segments", "f32"): 0.70, ("decimal", "f32"): 0.40,
          ("segments", "f16"): 0.29}


def _case(name, op, kind, dtype, n, block=1024, **more):
    return dict(name=name, op=op, kind=kind, dtype=dtype, n=n, block=block, **more)


def listed():
    return [
        # one sensor's short series through the synchronous calls: latency and launches
        _case("sync_f64_1k", "sync", "walk", "f64", 1000),
        # the paper-shaped 2^20-value random walk (2 places): an ordinary column
        _case("roundtrip_walk_f64_1m", "roundtrip", "walk", "f64", 1 << 20),
        # the throughput workload, each direction and both wide dtypes: outliers make the chunks Case 2
        _case("compress_segments_f64_64m", "compress", "segments", "f64", 1 << 26),
        _case("decompress_segments_f64_64m", "decompress", "segments", "f64", 1 << 26),
        _case("compress_segments_f32_64m", "compress", "segments", "f32", 1 << 26),
        _case("decompress_segments_f32_64m", "decompress", "segments", "f32", 1 << 26),
        # clean decimal measurements (Case 1 chunks) in the paper's 1025-value chunks, odd length:
        # chunk starts off 16 bytes, a ragged tail
        _case("compress_decimal_f64_40m_b1025", "compress", "decimal", "f64", 40_000_003, 1025),
        _case("decompress_decimal_f64_40m_b1025", "decompress", "decimal", "f64", 40_000_003, 1025),
        # half-precision readings, both directions
        _case("roundtrip_segments_f16_16m", "roundtrip", "segments", "f16", (1 << 24) + 5),
        # a table of uneven series, FP64 and FP32, one planned launch per direction
        _case("batch_mixed_256", "batch", "outliers", "mixed", 0, series=256, max_len=1 << 20),
        # a query over a compressed column
        _case("aggregate_outliers_f64_16m", "aggregate", "outliers", "f64", 1 << 24),
        # host data in frames through the device and back
        _case("pipeline_outliers_f64_16m", "pipeline", "outliers", "f64", (1 << 24) + 1, frame=1 << 21),
    ]


def draw(rng):
    op = rng.choice(["compress", "decompress", "compress", "decompress", "roundtrip", "sync", "aggregate", "batch",
                     "pipeline"])
    block = rng.choice([1024, 1024, 1025, 512, 1000])
    if op == "batch":
        return dict(op=op, kind=rng.choice(["walk", "outliers"]), dtype="mixed", n=0, block=block,
                    series=int(2 ** rng.uniform(3, 8)), max_len=int(2 ** rng.uniform(12, 20)))
    dtype = rng.choice(["f64", "f64", "f32", "f32", "f16"])
    kind = "segments" if dtype == "f16" else rng.choice(["walk", "outliers", "segments", "decimal"])
    top = {"sync": 22, "pipeline": 24, "aggregate": 24, "roundtrip": 24}.get(op, 26)
    low = {"sync": 6, "pipeline": 18}.get(op, 10)
    n = int(2 ** rng.uniform(low, top))
    if op == "aggregate" and kind == "segments":
        kind, dtype = "outliers", "f64"           # infinities of both signs would leave no sum to compare
    case = dict(op=op, kind=kind, dtype=dtype, n=n, block=block)
    if op == "pipeline":
        case["frame"] = int(2 ** rng.uniform(17, 22))
    return case


def _specials(bits, pos, kind, payload, wide):
    """Puts NaNs with payloads, infinities, subnormals and -0 at pos of an integer view of the values."""
    sign, inf, quiet, mant = ((-1 << 63, 0x7FF0 << 48, 1 << 51, (1 << 51) - 1) if wide
                              else (-1 << 31, 0x7F80 << 16, 1 << 22, (1 << 22) - 1))
    payload = (payload & mant) | 1
    table = torch.stack([inf | quiet | payload, inf | payload, torch.full_like(payload, inf),
                         torch.full_like(payload, sign | inf), payload, torch.full_like(payload, sign)])
    bits[pos] = table.gather(0, kind[None])[0].to(bits.dtype)


def _walk(n, g, places, dtype, outlier_rate):
    steps = torch.round(torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * (0.5 * 10 ** places))
    k = torch.cumsum(steps.to(torch.int64), 0) + 20 * 10 ** places
    x = k.to(torch.float64) / 10.0 ** places                     # exact operands: the nearest FP64
    v = x.to(_DTYPE[dtype])
    if outlier_rate:
        pos = torch.randint(0, n, (int(n * outlier_rate),), generator=g, device="cuda").unique()
        u = torch.rand(pos.numel(), generator=g, device="cuda", dtype=torch.float64) * 5 + 3
        v[pos] = ((x[pos] + 0.123) * torch.pow(10.0, u)).to(v.dtype)
    return v


def _segments(n, g, dtype, outlier_rate, special_rate):
    seg = 4096
    rows = (n + seg - 1) // seg

    def u(lo, hi):
        return torch.rand(rows, 1, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo

    half = dtype == "f16"
    places = torch.floor(u(0, 3 if half else 7))
    amp = torch.pow(10.0, u(-1, 1) if half else u(0, 4))
    period, phase = u(64, 4096), u(0, 6.283185307179586)
    ar = torch.randn(rows, seg, generator=g, device="cuda", dtype=torch.float64)
    for s in (1, 2, 4, 8, 16, 32, 64, 128):                      # AR(1), phi = 0.95, by doubling
        ar = torch.cat([ar[:, :s], ar[:, s:] + 0.95 ** s * ar[:, :-s]], 1)
    t = torch.arange(seg, device="cuda", dtype=torch.float64)[None]
    x = torch.sin(t * (6.283185307179586 / period) + phase).add_(ar, alpha=0.01).mul_(amp)
    del ar
    scale = torch.pow(10.0, places).round()
    x = x.view(-1)[:n]
    v = (torch.round(x * scale.expand(rows, seg).reshape(-1)[:n]) / scale.expand(rows, seg).reshape(-1)[:n])
    v = v.to(_DTYPE[dtype])
    for rate, what in ((outlier_rate, "outlier"), (special_rate, "special")):
        cnt = int(n * rate)
        if not cnt:
            continue
        pos = torch.randint(0, n, (cnt,), generator=g, device="cuda").unique()
        if what == "outlier":
            up = torch.rand(pos.numel(), generator=g, device="cuda", dtype=torch.float64) * 5 + 3
            v[pos] = (x[pos] * (3.141592653589793 if half else torch.pow(10.0, up))).to(v.dtype)
        elif half:
            table = torch.tensor([float("nan"), float("inf"), float("-inf"), -0.0, 6e-8], dtype=v.dtype, device="cuda")
            v[pos] = table[torch.randint(0, 5, (pos.numel(),), generator=g, device="cuda")]
        else:
            kind = torch.randint(0, 6, (pos.numel(),), generator=g, device="cuda")
            payload = torch.randint(0, 1 << 62, (pos.numel(),), generator=g, device="cuda")
            _specials(v.view(_BITS[dtype]), pos, kind, payload, dtype == "f64")
    return v.contiguous()


def _values(kind, dtype, n, g, places=2):
    if kind == "walk":
        return _walk(n, g, places, dtype, 0.0)
    if kind == "outliers":
        return _walk(n, g, 3, dtype, 0.005)
    if dtype == "f16":
        return _segments(n, g, dtype, 1e-4, 1e-5)
    return _segments(n, g, dtype, 0.01 if kind == "segments" else 0.0, 1e-4 if kind == "segments" else 0.0)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _inputs(case, seed):
    return _values(case["kind"], case["dtype"], case["n"], _generator(seed))


def _lengths(case):
    """(length, dtype) of a batch's series: log-uniform from 1024 to max_len, 70 % FP64."""
    top = max(case["max_len"], 1025) / 1024.0
    return [(int(1024 * top ** ((i * 0.6180339887498949) % 1.0)), "f64" if (i * 7) % 10 < 7 else "f32")
            for i in range(case["series"])]


def _batch_inputs(case, seed):
    g = _generator(seed)
    return [_values(case["kind"], dt, n, g, places=i % 7) for i, (n, dt) in enumerate(_lengths(case))]


def _chunks(case):
    return (case["n"] + case["block"] - 1) // case["block"]


def _prepare_batch(case, seed):
    xs = _batch_inputs(case, seed)
    code = {torch.float64: falcon.F64, torch.float32: falcon.F32}
    room = [(falcon.bound(x.numel(), code[x.dtype], case["block"]) + 15) // 16 * 16 for x in xs]
    streams = torch.zeros(sum(room), dtype=torch.uint8, device="cuda")
    sizes = [(x.numel() * x.element_size() + 15) // 16 * 16 for x in xs]
    values = torch.zeros(sum(sizes), dtype=torch.uint8, device="cuda")
    outs, back, a, b = [], [], 0, 0
    for x, r, s in zip(xs, room, sizes):
        outs.append(streams[a:a + r])
        back.append(values[b:b + x.numel() * x.element_size()].view(x.dtype))
        a, b = a + r, b + s
    comp = falcon.Batch(falcon.COMPRESS, xs, block=case["block"], outputs=outs)
    comp.launch()
    torch.cuda.synchronize()
    made = [(o, nb) for o, (nb, _) in zip(outs, comp.results())]
    heads = torch.stack([o[:32] for o in outs]).cpu().numpy()
    dec = falcon.Batch(falcon.DECOMPRESS, [(o[:nb], nb, h.tobytes()) for (o, nb), h in zip(made, heads)], outputs=back)
    return dict(op="batch", comp=comp, dec=dec, xs=xs, outs=outs, back=back,
                ret={"streams": streams, "values": values, "comp": comp.results_dev, "dec": dec.results_dev})


def prepare(case, seed):
    op, block = case["op"], case["block"]
    if op == "batch":
        return _prepare_batch(case, seed)
    x = _inputs(case, seed)
    st = dict(op=op, x=x, block=block, bits=_BITS[case["dtype"]])
    if op == "pipeline":
        st["x"] = torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)
        frames = (case["n"] + case["frame"] - 1) // case["frame"]
        st["frame"] = case["frame"]
        st["out"] = torch.zeros(frames * falcon.bound(case["frame"], _CODE[case["dtype"]], block), dtype=torch.uint8,
                                pin_memory=True)
        st["back"] = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
        return st
    if op in ("compress", "roundtrip", "sync"):
        st["stream"] = torch.zeros(falcon.bound(case["n"], _CODE[case["dtype"]], block), dtype=torch.uint8, device="cuda")
    if op == "sync":
        return st
    ws = falcon.workspace_bytes(_chunks(case))
    if op in ("compress", "roundtrip"):
        st["ws"] = torch.empty(ws, dtype=torch.uint8, device="cuda")
        st["res"] = torch.zeros(2, dtype=torch.int64, device="cuda")
        if op == "compress":
            return st
    made = falcon.compress(x, block)
    st["header"] = made[:falcon.HEADER_BYTES].cpu().numpy().tobytes()
    st["nbytes"] = made.numel()
    if op != "roundtrip":
        st["stream"] = made.clone()
    st["ws2"] = torch.empty(ws, dtype=torch.uint8, device="cuda")
    if op == "aggregate":
        st["stats"] = torch.zeros(falcon.STATS_BYTES, dtype=torch.uint8, device="cuda")
        ints, floats = st["stats"].view(torch.int64), st["stats"].view(torch.float64)
        st["ret"] = {"counts": ints[0:2], "range_sum": floats[2:5], "status": ints[5:6]}
        del st["x"]
        return st
    st["res2"] = torch.zeros(2, dtype=torch.int64, device="cuda")
    st["back"] = torch.zeros_like(x)
    st["back_bits"] = st["back"].view(st["bits"])
    if op == "decompress":
        del st["x"]
    return st


def run(st):
    op = st["op"]
    if op == "compress":
        falcon.compress_async(st["x"], st["block"], st["stream"], st["ws"], st["res"])
        return {"stream": st["stream"], "result": st["res"]}
    if op == "decompress":
        falcon.decompress_async(st["stream"], st["nbytes"], st["header"], st["back"], st["ws2"], st["res2"])
        return {"values": st["back_bits"], "result": st["res2"]}
    if op == "roundtrip":
        falcon.compress_async(st["x"], st["block"], st["stream"], st["ws"], st["res"])
        falcon.decompress_async(st["stream"], st["nbytes"], st["header"], st["back"], st["ws2"], st["res2"])
        return {"stream": st["stream"], "result": st["res"], "values": st["back_bits"], "back": st["res2"]}
    if op == "sync":
        s = falcon.compress(st["x"], st["block"], out=st["stream"])
        y = falcon.decompress(s)
        return {"stream": st["stream"], "values": y.view(st["bits"])}
    if op == "aggregate":
        falcon.aggregate_async(st["stream"], st["nbytes"], st["header"], st["ws2"], st["stats"])
        return st["ret"]
    if op == "batch":
        st["comp"].launch()
        st["dec"].launch()
        return st["ret"]
    s, frames = falcon.pipeline_compress(st["x"], st["block"], st["frame"], out=st["out"])
    y = falcon.pipeline_decompress(s, frames, out=st["back"])
    return {"stream": st["out"], "values": y.view(st["bits"])}


def work(case):
    """Each value and each stream byte once per direction (compressed sizes as the generators give them)."""
    def one(n, dtype):
        return n * _SIZE[dtype] * (1.0 + _RATIO[(case["kind"], dtype)])
    both = 2 if case["op"] in ("roundtrip", "sync", "batch", "pipeline") else 1
    if case["op"] == "batch":
        return {"bytes": both * sum(one(n, dt) for n, dt in _lengths(case)), "flops": 0}
    if case["op"] == "aggregate":
        return {"bytes": case["n"] * _SIZE[case["dtype"]] * _RATIO[(case["kind"], case["dtype"])], "flops": 0}
    return {"bytes": both * one(case["n"], case["dtype"]), "flops": 0}


def exact(case, seed):
    """Decompression gives the inputs back bit for bit; the aggregate in plain FP64.  A stream's
    bytes have no value but the format's own."""
    op = case["op"]
    if op == "compress":
        return None
    if op == "batch":
        parts = []
        for x in _batch_inputs(case, seed):
            raw = x.view(torch.uint8)
            parts.append(torch.nn.functional.pad(raw, (0, -raw.numel() % 16)))
        return {"streams": None, "values": torch.cat(parts), "comp": None, "dec": None}
    x = _inputs(case, seed)
    if op == "aggregate":
        v = x.to(torch.float64)
        nan = torch.isnan(v)
        v = v[~nan]
        return {"counts": torch.stack([torch.tensor(case["n"], device="cuda"), nan.sum()]),
                "range_sum": torch.stack([v.min(), v.max(), v.sum()]), "status": None}
    bits = x.view(_BITS[case["dtype"]])
    if op == "decompress":
        return {"values": bits, "result": None}
    if op == "roundtrip":
        return {"stream": None, "result": None, "values": bits, "back": None}
    return {"stream": None, "values": bits}
