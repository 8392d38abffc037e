"""What the performance of this library is measured on: encodes, scans, batches and serving.

Each case is one pass through the public entry points (paper_2306_15374_gb300.leco) on seeded
synthetic columns of the shapes the benchmark and the tests use (workloads.py), made on the GPU:
near-linear values with bounded noise, sorted normal and lognormal samples, piecewise-linear series,
wrapping 32-bit timestamps and a sine mixture.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_15374_gb300 import leco

MODELS = {"constant": leco.LECO_MODEL_CONSTANT, "linear": leco.LECO_MODEL_LINEAR, "poly": leco.LECO_MODEL_POLY}
TAU = 0.03  # split threshold of the benchmark's variable-partition columns


def listed() -> list[dict]:
    return [
        # a small table segment written and read back once: launches and the host path count
        dict(name="encode-fixed-100k-u64", op="encode", dist="linear", bits=64, n=100_003, policy="fixed", L=1024,
             model="linear"),
        # bulk load of a large sorted column, fixed partitions (the benchmark's 200M-value columns)
        dict(name="encode-fixed-200m-u64", op="encode", dist="normal", bits=64, n=200_000_000, policy="fixed", L=4096,
             model="linear"),
        # bulk load of a 32-bit column into buffers the caller owns, ragged partitions, FOR
        dict(name="encode-noalloc-20m-u32", op="noalloc", dist="linear", bits=32, n=20_000_003, policy="fixed", L=1000,
             model="constant"),
        # variable partitions of a series with slope changes (the benchmark's piecewise column, half size)
        dict(name="encode-var-100m-u64", op="encode", dist="piecewise", bits=64, n=100_000_000, policy="var", L=0,
             model="linear"),
        # variable partitions of jumping timestamps (the benchmark's 32-bit column, half size)
        dict(name="encode-var-250m-u32", op="encode", dist="timestamps", bits=32, n=250_000_000, policy="var", L=0,
             model="linear"),
        # a sensor-like column under the polynomial model
        dict(name="encode-poly-50m-u64", op="encode", dist="sine", bits=64, n=50_000_000, policy="fixed", L=4096,
             model="poly"),
        # a dashboard query on a small resident column: a range, some points, a selective sum
        dict(name="scan-fixed-1m-u64", op="scan", dist="linear", bits=64, n=1_000_000, policy="fixed", L=1024,
             model="linear", count=65_537, k=4_096),
        # the benchmark's step on one of its columns: full decode, 10M lookups, filter + sum
        dict(name="scan-fixed-200m-u64", op="scan", dist="lognormal", bits=64, n=200_000_000, policy="fixed", L=4096,
             model="linear", count=200_000_000, k=10_000_000),
        # the same over variable partitions of 32-bit timestamps
        dict(name="scan-var-100m-u32", op="scan", dist="timestamps", bits=32, n=100_000_007, policy="var", L=0,
             model="linear", count=100_000_007, k=5_000_000),
        # the same over polynomial partitions
        dict(name="scan-poly-50m-u64", op="scan", dist="sine", bits=64, n=50_000_000, policy="fixed", L=4096,
             model="poly", count=50_000_000, k=2_500_000),
        # a compaction job: many columns of mixed length, model and partition size re-encoded, then read
        dict(name="batch-96-u64", op="batch", dist="mixed", bits=64, n=200_000_000, cols=96),
        # a burst of requests against resident columns: lookups and range decodes to host memory
        dict(name="serve-64", op="serve", dist="mixed", bits=64, n=60_000_000, cols=24, requests=64),
    ]


def _size(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    op = rng.choice(["encode", "encode", "encode", "scan", "scan", "scan", "noalloc", "batch", "serve"])
    if op == "batch":
        return dict(op=op, dist="mixed", bits=64, n=_size(rng, 2_000_000, 200_000_000), cols=rng.randint(8, 96))
    if op == "serve":
        return dict(op=op, dist="mixed", bits=64, n=_size(rng, 5_000_000, 60_000_000), cols=rng.randint(4, 24),
                    requests=rng.randint(1, 64))
    if op == "noalloc":
        bits = rng.choice([32, 64])
        return dict(op=op, dist=rng.choice(["linear", "timestamps"] if bits == 32 else ["linear", "normal", "lognormal"]),
                    bits=bits, n=_size(rng, 20_000, 20_000_000), policy="fixed", L=rng.choice([256, 1000, 1024, 2047, 4096]),
                    model=rng.choice(["constant", "linear"]))
    kind = rng.choice(["fixed", "fixed", "var", "var", "poly", "auto" if op == "encode" else "fixed"])
    if kind == "var":
        bits = rng.choice([32, 64])
        c = dict(op=op, dist="timestamps" if bits == 32 else rng.choice(["piecewise", "normal"]), bits=bits,
                 n=_size(rng, 20_000, 100_000_000), policy=rng.choice(["var", "var", "var", "seeded"]), L=0,
                 model="linear")
    elif kind == "poly":
        c = dict(op=op, dist="sine", bits=64, n=_size(rng, 20_000, 50_000_000), policy="fixed",
                 L=rng.choice([1024, 1500, 4096]), model="poly")
    else:
        c = dict(op=op, dist=rng.choice(["linear", "normal", "lognormal", "timestamps"]), bits=64,
                 n=_size(rng, 20_000, 200_000_000), policy=kind, L=rng.choice([256, 1000, 1024, 2047, 4096, 10_000]),
                 model=rng.choice(["constant", "linear", "linear"]))
        if c["dist"] == "timestamps" or (c["dist"] == "linear" and rng.random() < 0.5):
            c["bits"] = 32
        if kind == "auto":
            c["L"] = 0
    if op == "scan":
        c["count"] = c["n"] if rng.random() < 0.6 else _size(rng, 1_000, c["n"])
        c["k"] = _size(rng, 100, max(200, min(10_000_000, c["n"] // 10)))
    return c


# ------------------------------------------------------------------------------------ values


def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _values(dist: str, n: int, bits: int, seed: int) -> torch.Tensor:
    """n values on the GPU as int64 / int32 bit patterns; the same for the same arguments."""
    g, h = _gen(seed), np.random.default_rng(seed)
    dev = "cuda"
    if dist == "linear":  # base + slope i + U{-a..a}
        a = int(2 ** h.integers(9, 13))
        v = torch.randint(-a, a + 1, (n,), generator=g, device=dev)
        v += torch.arange(n, device=dev) * int(h.integers(11, 60)) + (1 << 20)
    elif dist in ("normal", "lognormal"):
        z = torch.randn(n, generator=g, device=dev, dtype=torch.float64).sort().values
        z = z * float(1 << 36) + float(1 << 40) if dist == "normal" else (z * 2.0).exp_() * 1e9
        v = z.round_().clamp_(0, 9e18).to(torch.int64)
    elif dist == "piecewise":  # continuous, slope changes every ~200K values, noise 2^0 .. 2^20 per segment
        s = max(1, n // 200_000)
        edges = np.sort(h.integers(0, n, size=s - 1)) if s > 1 else np.zeros(0, np.int64)
        lens = np.diff(np.concatenate([[0], edges, [n]])).astype(np.int64)
        slopes = h.uniform(1.0, 1e4, size=s)
        rise = np.floor(slopes * lens).astype(np.int64)
        first = torch.from_numpy((1 << 22) + np.concatenate([[0], np.cumsum(rise)[:-1]])).to(dev)
        offs = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)[:-1]])).to(dev)
        amp = torch.from_numpy(np.int64(1) << h.integers(0, 21, size=s)).to(dev)
        seg = torch.repeat_interleave(torch.arange(s, device=dev), torch.from_numpy(lens).to(dev), output_size=n)
        j = torch.arange(n, device=dev) - offs[seg]
        v = first[seg] + (j.to(torch.float64) * torch.from_numpy(slopes).to(dev)[seg]).floor_().to(torch.int64)
        u = torch.randint(0, 1 << 40, (n,), generator=g, device=dev)
        v += u % (2 * amp + 1)[seg] - amp[seg]
    elif dist == "timestamps":  # 1000 i + a daily swing + rare jumps, wrapping at 2^32
        i = torch.arange(n, device=dev)
        table = np.rint(300 * np.sin(2 * np.pi * np.arange(86400) / 86400)).astype(np.int64)
        jump = torch.rand(n, generator=g, device=dev) < 0.001
        v = torch.cumsum(torch.randint(1, 1_000_001, (n,), generator=g, device=dev) * jump, 0)
        v += i * 1000 + torch.from_numpy(table).to(dev)[i % 86400] + 300
    elif dist == "sine":  # two superposed sines and uniform noise
        i = torch.arange(n, device=dev, dtype=torch.float64)
        s = (i * (2 * math.pi / 1e6)).sin_() * 1e9 + (i * (2 * math.pi / 4e4)).sin_() * 1e7
        v = s.floor_().to(torch.int64) + (1 << 40) + torch.randint(-128, 129, (n,), generator=g, device=dev)
    else:
        raise ValueError(dist)
    return v.to(torch.int32) if bits == 32 else v


def _policy(case: dict) -> leco.PartitionPolicy:
    kind = case["policy"]
    if kind == "fixed":
        return leco.fixed(case["L"])
    if kind == "auto":
        return leco.auto()
    return leco.variable(TAU, seeded=kind == "seeded")


def _unsigned(x: torch.Tensor) -> int:
    return int(x.item()) & (0xFFFFFFFF if x.dtype == torch.int32 else (1 << 64) - 1)


def _queries(case: dict, v: torch.Tensor, seed: int):
    """(begin of the decoded range, lookup positions, filter bounds that select about 1 % of a sorted column)."""
    n = case["n"]
    begin = int(np.random.default_rng(seed + 1).integers(0, n - case["count"] + 1))
    idx = torch.randint(0, n, (case["k"],), generator=_gen(seed + 2), device="cuda")
    a, b = _unsigned(v[int(0.495 * n)]), _unsigned(v[int(0.505 * n)])
    return begin, idx, min(a, b), max(a, b)


def _lens(case: dict, lo: int) -> np.ndarray:
    """Column lengths spread over their logarithm, about case["n"] values in all (the case's own, for every seed)."""
    w = np.exp(np.random.default_rng(case["n"]).uniform(0.0, math.log(1e3), size=case["cols"]))
    return np.maximum(lo, np.rint(w * (case["n"] / w.sum()))).astype(np.int64)


def _batch(case: dict, seed: int):
    h = np.random.default_rng(seed)
    lens = [int(x) for x in _lens(case, 1000)]
    vals = [_values(("linear", "normal", "lognormal")[int(h.integers(0, 3))], n, 64, seed + 31 * c)
            for c, n in enumerate(lens)]
    models = [int(x) for x in h.integers(0, 2, size=len(lens))]
    sizes = [int(x) for x in h.choice([256, 1024, 4096], size=len(lens))]
    return lens, vals, models, sizes


def _serve_columns(case: dict, seed: int):
    lens = [int(x) for x in _lens(case, 100_000)]
    return lens, [_values("piecewise" if c % 2 else "linear", n, 64, seed + 31 * c) for c, n in enumerate(lens)]


def _requests(case: dict, lens, seed: int):
    """(column, positions) for a lookup, (column, begin, count) for a range decode, in submission order. Columns and
    sizes are the case's own, for every seed; the positions are the seed's."""
    mix, h = np.random.default_rng(case["n"] + 1), np.random.default_rng(seed + 3)
    reqs = []
    for _ in range(case["requests"]):
        c = int(mix.integers(0, len(lens)))
        if mix.random() < 0.5:
            k = int(np.exp(mix.uniform(0.0, math.log(4096))))
            reqs.append((c, h.integers(0, lens[c], size=k, dtype=np.uint64)))
        else:
            k = min(lens[c], int(np.exp(mix.uniform(math.log(1e3), math.log(1e6)))))
            reqs.append((c, int(h.integers(0, lens[c] - k + 1)), k))
    return reqs


# ------------------------------------------------------------------------------------ the passes


def prepare(case: dict, seed: int) -> dict:
    op = case["op"]
    if op == "batch":
        lens, vals, models, sizes = _batch(case, seed)
        flat = torch.empty(sum(lens), dtype=torch.int64, device="cuda")
        return dict(op=op, vals=vals, models=models, sizes=sizes, flat=flat, outs=list(flat.split(lens)))
    if op == "serve":
        lens, vals = _serve_columns(case, seed)
        cols = [leco.leco_encode(v, leco.variable(TAU) if c % 2 else leco.fixed(4096)) for c, v in enumerate(vals)]
        server = leco.leco_server_create(8 << 30)
        ids = [leco.leco_server_admit(server, c) for c in cols]
        reqs = _requests(case, lens, seed)
        flat = np.zeros(sum(r[2] if len(r) == 3 else r[1].size for r in reqs), dtype=np.uint64)
        outs = np.split(flat, np.cumsum([r[2] if len(r) == 3 else r[1].size for r in reqs])[:-1])
        return dict(op=op, server=server, ids=ids, reqs=reqs, flat=flat, outs=outs)
    v = _values(case["dist"], case["n"], case["bits"], seed)
    if op == "noalloc":
        m = -(-case["n"] // case["L"])
        rec = torch.zeros(4 * m, dtype=torch.int64, device="cuda")
        words = torch.zeros(case["n"] * (case["bits"] + 2) // 64 + 64, dtype=torch.int64, device="cuda")
        return dict(op=op, v=v, L=case["L"], model=MODELS[case["model"]], rec=rec, words=words)
    if op == "encode":
        return dict(op=op, v=v, policy=_policy(case), model=MODELS[case["model"]], out=torch.empty_like(v))
    begin, idx, lo, hi = _queries(case, v, seed)
    col = leco.leco_encode(v, _policy(case), MODELS[case["model"]])
    return dict(op=op, col=col, n=case["n"], begin=begin, count=case["count"], idx=idx, lo=lo, hi=hi,
                out=torch.empty(case["count"], dtype=v.dtype, device="cuda"),
                vals=torch.empty(case["k"], dtype=v.dtype, device="cuda"),
                res=torch.zeros(3, dtype=torch.int64, device="cuda"))


def run(s: dict):
    op = s["op"]
    if op == "encode":  # write a column, read it back
        col = leco.leco_encode(s["v"], s["policy"], s["model"])
        leco.leco_decode_all(col, s["out"])
        st = col.stats()
        col.free_async()
        return {"values": s["out"], "sizes": [st["partitions"], st["residual_bits"], st["total_bytes"], st["part_size"]]}
    if op == "noalloc":
        nw = leco.leco_encode_fixed_noalloc(s["v"], s["L"], s["rec"], s["words"], s["model"])
        return {"records": s["rec"], "words": s["words"], "count": nw}
    if op == "scan":
        if s["count"] == s["n"]:
            leco.leco_decode_all(s["col"], s["out"])
        else:
            leco.leco_decode_range(s["col"], s["begin"], s["count"], s["out"])
        leco.leco_random_access(s["col"], s["idx"], s["vals"])
        leco.leco_filter_sum(s["col"], s["lo"], s["hi"], s["res"])
        return {"range": s["out"], "points": s["vals"], "sum": s["res"]}
    if op == "batch":
        cols = leco.leco_batch_encode(s["vals"], s["models"], s["sizes"])
        leco.leco_batch_decode(cols, s["outs"])
        sizes = np.array([c.stats()["residual_bits"] for c in cols], dtype=np.int64)
        for c in cols:
            c.free_async()
        return {"values": s["flat"], "sizes": sizes}
    server, tickets = s["server"], []
    for r, out in zip(s["reqs"], s["outs"]):
        if len(r) == 3:
            tickets.append(leco.leco_server_submit_range(server, s["ids"][r[0]], r[1], r[2], out))
        else:
            tickets.append(leco.leco_server_submit_lookup(server, s["ids"][r[0]], r[1], out))
    status = [leco.leco_server_wait(server, t) for t in tickets]
    return {"values": s["flat"].view(np.int64), "status": np.array(status, dtype=np.int64)}


# ------------------------------------------------------------------------------------ what a pass needs

# bits per value of the stored residuals, about (by distribution; L sets how much of a sorted sample
# or a constant model's slope a partition spans)
def _bits(case: dict) -> float:
    d, n, L = case["dist"], case["n"], max(256, case.get("L") or 2048)
    if d in ("linear", "mixed"):
        return 12.0 if case.get("model") != "constant" else max(12.0, math.log2(35 * L))
    if d == "timestamps":
        return 3.0 if case["policy"] in ("var", "seeded") else 20.0
    if d == "piecewise":
        return 12.0
    if d == "sine":
        return 9.5
    slope = (float(1 << 36) if d == "normal" else 4e9) / n  # a sorted sample's step near its median
    return math.log2(2 + slope * (math.sqrt(L) if case.get("model") != "constant" else L))


def work(case: dict) -> dict:
    op, n, vb = case["op"], case["n"], case["bits"] // 8
    stored = n * _bits(case) / 8
    if op == "serve":  # range values and points, decoded and copied to the host
        values = case["requests"] * (0.5 * 1.45e5 + 0.5 * 490)
        return {"bytes": values * (12 / 8 + 2 * 8), "flops": 8.0 * values}
    if op == "noalloc":
        return {"bytes": n * vb + stored, "flops": 10.0 * n}
    if op in ("encode", "batch"):  # values in, stream out; stream in, values out
        return {"bytes": 2 * (n * vb + stored), "flops": 15.0 * n}
    part = case["count"] / n
    return {"bytes": stored * (1 + part) + case["count"] * vb + case["k"] * (8 + vb + 32),
            "flops": 5.0 * (n + case["count"] + case["k"])}


def exact(case: dict, seed: int):
    """Decoded values are the inputs; sizes, records and words have no value without an encoder."""
    op = case["op"]
    if op == "noalloc":
        return None
    if op == "batch":
        return {"values": torch.cat(_batch(case, seed)[1]), "sizes": None}
    if op == "serve":
        lens, vals = _serve_columns(case, seed)
        got = [vals[r[0]][r[1]:r[1] + r[2]].cpu() if len(r) == 3 else vals[r[0]].cpu()[torch.from_numpy(r[1].astype(np.int64))]
               for r in _requests(case, lens, seed)]
        return {"values": torch.cat(got).numpy(), "status": np.zeros(case["requests"], dtype=np.int64)}
    v = _values(case["dist"], case["n"], case["bits"], seed)
    if op == "encode":
        return {"values": v, "sizes": [None] * 4}
    begin, idx, lo, hi = _queries(case, v, seed)
    u = (v.to(torch.int64) & 0xFFFFFFFF) if case["bits"] == 32 else v  # every 64-bit value here is below 2^63
    sel = u[(u >= lo) & (u <= hi)]
    total = (int((sel >> 32).sum().item()) << 32) + int((sel & 0xFFFFFFFF).sum().item())
    words = np.array([sel.numel(), total & ((1 << 64) - 1), total >> 64], dtype=np.uint64).view(np.int64)
    return {"range": v[begin:begin + case["count"]], "points": v[idx], "sum": torch.from_numpy(words)}
