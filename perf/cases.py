"""The selections that programs make through this package, as timed cases.

A case is one call of a public entry point with the few torch operations that
a program puts behind it.  The library writes a selected set in no particular
order, so a program puts it where it belongs itself:

  threshold : topk_select_kth, the rank-k pair alone (a quantile, a median, a
              cut-off that the program then compares against);
  select    : topk_select, then the selected keys written at their positions in
              an array of the program's (everything not selected keeps the
              value it had there: a sparsified copy, a mask, an update);
  runs      : topk_select_sorted_runs, the split positions and the rank-k object;
  pop       : topk_runs_delete_min from given cursors, the cursors it leaves
              and the largest object deleted;
  batched   : topk_select_batched over rows of uneven length and k, then the
              selected keys of every row written at their positions;
  frequent  : topk_frequent (Algorithm EC), the objects ordered by count.

A program keeps one context for all its calls (scratch memory and device
status); outputs are buffers of its own, and it reads the latched status when
it next waits for its stream, not after every call.  Keys are returned as the
integers of the same bits: a selection moves keys, it computes none.

Requests through topk_serve_* run the same kernels (a batch of small ones, one
selection for a large one) behind a host thread; their time is the thread's.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1502_03942_gb300 as tk
from paper_1502_03942_gb300 import workloads as wl

WIDTH = {"u32": 4, "i32": 4, "f32": 4, "bf16": 2, "u64": 8}
BITS = {"u32": torch.int32, "i32": torch.int32, "f32": torch.int32, "bf16": torch.int16, "u64": torch.int64}
KEY = {"u32": torch.uint32, "i32": torch.int32, "f32": torch.float32, "bf16": torch.bfloat16, "u64": torch.uint64}
UNSET = -1  # what the program's array holds where nothing was selected


def listed():
    return [
        # one short row: the cut-off of the 50 largest of 1000 scores (one block)
        {"name": "threshold_tiny", "op": "threshold", "dtype": "f32", "dist": "normal", "n": 1000, "k": 50,
         "largest": True},
        # a short list, ragged, near the upper end of what one block finishes
        {"name": "select_small", "op": "select", "dtype": "u32", "dist": "uniform", "n": 12345, "k": 100},
        # the plain selection of the benchmark: 2^20 u32 keys, k = 1000, 64 partitions
        {"name": "select_plain", "op": "select", "dtype": "u32", "dist": "uniform", "n": 1 << 20, "k": 1000,
         "partitions": 64},
        # a low quantile of 16-bit keys with heavy ties, ragged length
        {"name": "threshold_bf16", "op": "threshold", "dtype": "bf16", "dist": "zipf", "n": 5000011, "k": 50000},
        # 64-bit keys inside a larger array (not 16-byte aligned), a third of them selected
        {"name": "select_u64", "op": "select", "dtype": "u64", "dist": "uniform", "n": 3000001, "k": 1000000,
         "offset": 1},
        # the smaller half of 2^25 signed keys (half of the input goes to the output)
        {"name": "select_half", "op": "select", "dtype": "i32", "dist": "uniform", "n": 1 << 25, "k": 1 << 24},
        # the large selections of the benchmark: 2^28 f32 keys, few, many and half of them
        {"name": "select_few", "op": "select", "dtype": "f32", "dist": "normal", "n": 1 << 28, "k": 1024},
        {"name": "select_many", "op": "select", "dtype": "f32", "dist": "zipf", "n": 1 << 28, "k": 1 << 20},
        {"name": "median", "op": "threshold", "dtype": "f32", "dist": "uniform", "n": 1 << 28, "k": 1 << 27},
        # 1024 sorted runs of 2^U(10, 20) 64-bit keys, the smaller half of all objects split off
        {"name": "runs_half", "op": "runs", "runs": 1024, "lo": 10, "hi": 20, "part": 0.5},
        # 4096 rows of 2^U(10, 18) keys, k from 1 to 1024, the library's own settings
        {"name": "batched", "op": "batched", "dtype": "f32", "rows": 4096, "lo": 10, "hi": 18, "kmax": 1024},
        # the 32 most frequent of 2^28 Zipf objects at the paper's accuracy
        {"name": "frequent", "op": "frequent", "n": 1 << 28, "k": 32, "epsilon": 3e-4, "delta": 1e-4},
    ]


def _spread(rng, lo, hi):
    """A whole number from lo to hi, evenly over its logarithm."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    op = rng.choice(["threshold"] * 5 + ["select"] * 8 + ["batched"] * 3 + ["runs", "pop", "frequent"])
    if op in ("runs", "pop"):
        lo = rng.randint(6, 14)
        return {"op": op, "runs": _spread(rng, 16, 1024), "lo": lo, "hi": lo + rng.randint(1, 6),
                "part": rng.choice([rng.uniform(0.001, 0.02), rng.uniform(0.1, 0.9)])}
    if op == "batched":
        lo = rng.randint(8, 13)
        return {"op": op, "dtype": rng.choice(["f32", "f32", "u32", "i32", "bf16", "u64"]),
                "rows": _spread(rng, 64, 4096), "lo": lo, "hi": lo + rng.randint(1, 4), "kmax": _spread(rng, 16, 1024)}
    if op == "frequent":
        return {"op": op, "n": _spread(rng, 1 << 20, 1 << 27), "k": rng.randint(8, 64), "epsilon": 1e-3, "delta": 1e-4}
    dtype = rng.choice(["f32", "f32", "f32", "u32", "i32", "bf16", "u64"])
    n = _spread(rng, 1000, 1 << 27 if dtype != "u64" else 1 << 26)
    few, many = max(2, min(n // 4, _spread(rng, 4, 1 << 20))), max(2, int(n * rng.uniform(0.02, 0.98)))
    k = rng.choice([few, many] if op == "threshold" else [few, few, many])
    case = {"op": op, "dtype": dtype, "dist": rng.choice({"f32": ["uniform", "normal", "zipf"], "u32": ["uniform", "zipf"],
                                                            "i32": ["uniform"], "bf16": ["normal", "zipf"],
                                                            "u64": ["uniform"]}[dtype]), "n": n, "k": k}
    if rng.random() < 0.3:
        case["largest"] = True
    if rng.random() < 0.2:
        case["offset"] = rng.randint(1, 3)
    return case


# ------------------------------------------------------------------ inputs

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = tk.Context(torch.cuda.current_device())
    return _ctx


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _random_i32(n, g):
    return torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device="cuda", dtype=torch.int32)


def _random_i64(n, g):
    return (_random_i32(n, g).to(torch.int64) << 32) ^ (_random_i32(n, g).to(torch.int64) & 0xFFFFFFFF)


def _keys(dtype, dist, n, seed):
    """n keys as their bits (BITS[dtype])."""
    if dist == "zipf":
        r = wl.device_f32_dataset("zipf", n, seed)
        if dtype == "f32":
            return r.view(torch.int32)
        return (r.to(torch.int32) + 0x3F80).to(torch.int16) if dtype == "bf16" else r.to(torch.int32)
    if dtype == "f32":
        return wl.device_f32_dataset(dist, n, seed).view(torch.int32)
    g = _generator(seed)
    if dtype == "bf16":
        return torch.randn(n, generator=g, device="cuda").to(torch.bfloat16).view(torch.int16)
    return _random_i64(n, g) if dtype == "u64" else _random_i32(n, g)


def _batch_keys(case, n, seed):
    if case["dtype"] == "f32":
        return (torch.randn(n, generator=_generator(seed), device="cuda") * 3.0).view(torch.int32)
    return _keys(case["dtype"], "normal" if case["dtype"] == "bf16" else "uniform", n, seed)


def _rows(case):
    """Row lengths, row offsets and ranks of a batched case (host): part of the case, as a program's layout is."""
    g = wl.rng(case["rows"] * 64 + case["hi"])
    lens = np.floor(2.0 ** g.uniform(case["lo"], case["hi"], size=case["rows"])).astype(np.int64)
    off = np.zeros(case["rows"] + 1, np.int64)
    off[1:] = np.cumsum(lens)
    ks = np.minimum(g.integers(1, case["kmax"], size=case["rows"], endpoint=True), lens).astype(np.int64)
    return lens, off, ks


def _sorted_runs(case, seed):
    """(keys as int64 bits, offsets on the host, run of every key): every run sorted as unsigned."""
    g = wl.rng(seed)
    lens = np.floor(2.0 ** g.uniform(case["lo"], case["hi"], size=case["runs"])).astype(np.int64)
    off = np.zeros(case["runs"] + 1, np.int64)
    off[1:] = np.cumsum(lens)
    run = torch.repeat_interleave(torch.arange(case["runs"], dtype=torch.int16, device="cuda"),
                                  torch.from_numpy(lens).cuda())
    x = _random_i64(int(off[-1]), _generator(seed)).sort().values  # in the order of the signed image
    # deal the sorted values out to the runs at random, keeping their order in each run
    perm = run[torch.randperm(run.numel(), generator=_generator(seed + 1), device="cuda")]
    x = x[perm.sort(stable=True).indices] ^ (-(1 << 63))
    return x, off, run


def _buffers(n, m, dtype):
    return (torch.empty(n, dtype=KEY[dtype], device="cuda"), torch.empty(n, dtype=torch.uint32, device="cuda"),
            torch.empty(m, dtype=KEY[dtype], device="cuda"), torch.empty(m, dtype=torch.uint32, device="cuda"))


def prepare(case, seed):
    op, s = case["op"], {"op": case["op"], "ctx": _context()}
    if op in ("threshold", "select"):
        n, k, dtype, skip = case["n"], case["k"], case["dtype"], case.get("offset", 0)
        out = _buffers(k if op == "select" else 0, 1, dtype)
        s.update(keys=_keys(dtype, case["dist"], n + skip, seed)[skip:].view(KEY[dtype]), k=k, bits=BITS[dtype],
                 params=tk.make_params(partitions=case.get("partitions", 0),
                                       flags=tk.TOPK_FLAG_LARGEST if case.get("largest") else 0),
                 out=out if op == "select" else out[2:])
        if op == "select":
            s["placed"] = torch.full((n,), UNSET, dtype=BITS[dtype], device="cuda")
    elif op in ("runs", "pop"):
        x, off, _ = _sorted_runs(case, seed)
        s.update(keys=x.view(torch.uint64), off=torch.from_numpy(off).cuda().view(torch.uint64),
                 k=max(1, int(off[-1] * case["part"])))
        if op == "pop":  # a queue some way into its life: a tenth of every run already deleted
            s["from"] = torch.from_numpy(np.diff(off) // 10).cuda()
            s["cursor"] = s["from"].clone()
            s["k"] = max(1, int((off[-1] - (np.diff(off) // 10).sum()) * case["part"]))
    elif op == "batched":
        _, off, ks = _rows(case)
        dtype = case["dtype"]
        oo = np.zeros(case["rows"] + 1, np.int64)
        oo[1:] = np.cumsum(ks)
        s.update(keys=_batch_keys(case, int(off[-1]), seed).view(KEY[dtype]), bits=BITS[dtype],
                 off=torch.from_numpy(off).cuda().view(torch.uint64),
                 ks=torch.from_numpy(ks.astype(np.int32)).cuda().view(torch.uint32),
                 out_off=torch.from_numpy(oo).cuda().view(torch.uint64),
                 base=torch.from_numpy(np.repeat(off[:-1], ks)).cuda(),
                 out=_buffers(int(oo[-1]), case["rows"], dtype),
                 placed=torch.full((int(off[-1]),), UNSET, dtype=BITS[dtype], device="cuda"))
    elif op == "frequent":
        s.update(objects=wl.device_zipf_objects(case["n"], seed),
                 params=tk.make_freq_params(case["k"], tk.TOPK_FREQ_EC, case["epsilon"], case["delta"]))
    return s


# ------------------------------------------------------------------ passes

def run(s):
    op, ctx = s["op"], s["ctx"]
    if op == "threshold":
        kk, ki = tk.topk_select_kth(ctx, s["keys"], s["k"], params=s["params"], out=s["out"], check=False)
        return {"key": kk.view(s["bits"]), "pos": ki.view(torch.int32)}
    if op == "select":
        ok, oi, kk, ki = tk.topk_select(ctx, s["keys"], s["k"], params=s["params"], out=s["out"], check=False)
        placed = s["placed"].scatter_(0, oi.view(torch.int32).long(), ok.view(s["bits"]))
        return {"placed": placed, "key": kk.view(s["bits"]), "pos": ki.view(torch.int32)}
    if op == "runs":
        split, kk, kr, kp = tk.topk_select_sorted_runs(ctx, s["keys"], s["off"], s["k"], check=False)
        return [split.view(torch.int64), kk.view(torch.int64), kr.view(torch.int32), kp.view(torch.int64)]
    if op == "pop":
        cursor = s["cursor"].copy_(s["from"])
        kk, kr, kp = tk.topk_runs_delete_min(ctx, s["keys"], s["off"], cursor.view(torch.uint64), s["k"], check=False)
        return [cursor, kk.view(torch.int64), kr.view(torch.int32), kp.view(torch.int64)]
    if op == "batched":
        ok, oi, kk, ki, _ = tk.topk_select_batched(ctx, s["keys"], s["off"], s["ks"], out=s["out"],
                                                   out_off=s["out_off"], check=False)
        placed = s["placed"].scatter_(0, s["base"] + oi.view(torch.int32), ok.view(s["bits"]))
        return {"placed": placed, "key": kk.view(s["bits"]), "pos": ki.view(torch.int32)}
    objects, counts, size = tk.topk_frequent(ctx, s["objects"], s["params"], check=False)
    word = (counts.view(torch.int64) << 32) | (objects.view(torch.int32).long() & 0xFFFFFFFF)
    return {"counts_objects": word.sort().values, "sample": size.view(torch.int64)}


def work(case):
    op = case["op"]
    if op in ("threshold", "select"):
        n, k, w = case["n"], case["k"], WIDTH[case["dtype"]]
        return {"bytes": n * w + (1 if op == "threshold" else k + 1) * (w + 4), "flops": 0}
    if op in ("runs", "pop"):  # a binary search in every run, the offsets, and the splits
        return {"bytes": case["runs"] * (8 * (case["hi"] + 1) + 8 + (16 if op == "pop" else 8)), "flops": 0}
    if op == "batched":
        w = WIDTH[case["dtype"]]
        mean = (2.0 ** case["hi"] - 2.0 ** case["lo"]) / (math.log(2.0) * (case["hi"] - case["lo"]))
        return {"bytes": case["rows"] * (mean * w + case["kmax"] / 2 * (w + 4) + 20 + w + 4), "flops": 0}
    return {"bytes": case["n"] * 4 + case["k"] * 8 + 8, "flops": 0}


# --------------------------------------------------------- plain references

def _image(bits, dtype, largest=False):
    """An int64 whose order is the order of the keys (ties left to a stable sort)."""
    if dtype in ("f32", "bf16"):
        b = bits.to(torch.int64)
        x = torch.where(b < 0, ~(b & (0x7FFFFFFF if dtype == "f32" else 0x7FFF)), b)
    elif dtype == "u32":
        x = bits.to(torch.int64) & 0xFFFFFFFF
    elif dtype == "u64":
        x = bits ^ (-(1 << 63))
    else:
        x = bits.to(torch.int64)
    return ~x if largest else x


def exact(case, seed):
    op = case["op"]
    if op == "frequent":
        return None  # whole numbers that follow from the sample drawn
    if op in ("threshold", "select"):
        n, k, dtype, skip = case["n"], case["k"], case["dtype"], case.get("offset", 0)
        keys = _keys(dtype, case["dist"], n + skip, seed)[skip:]
        first = _image(keys, dtype, case.get("largest", False)).sort(stable=True).indices[:k].clone()
        last = first[k - 1:]
        if op == "threshold":
            return {"key": keys[last], "pos": last}
        placed = torch.full((n,), UNSET, dtype=keys.dtype, device="cuda").scatter_(0, first, keys[first])
        return {"placed": placed, "key": keys[last], "pos": last}
    if op in ("runs", "pop"):
        x, off, run_of = _sorted_runs(case, seed)
        start = np.zeros(case["runs"], np.int64)
        k = max(1, int(off[-1] * case["part"]))
        alive = torch.arange(x.numel(), device="cuda")
        if op == "pop":
            start = np.diff(off) // 10
            k = max(1, int((off[-1] - start.sum()) * case["part"]))
            at = torch.from_numpy(off[:-1] + start).cuda()
            alive = alive[alive >= at[run_of.long()]]
        taken = alive[(x[alive] ^ (-(1 << 63))).sort(stable=True).indices[:k]]
        split = torch.bincount(run_of[taken].long(), minlength=case["runs"]) + torch.from_numpy(start).cuda()
        last = taken[k - 1:]
        r = run_of[last].long()
        return [split, x[last], r, last - torch.from_numpy(off).cuda()[r]]
    lens, off, ks = _rows(case)
    keys = _batch_keys(case, int(off[-1]), seed)
    row = torch.repeat_interleave(torch.arange(case["rows"], dtype=torch.int16, device="cuda"),
                                  torch.from_numpy(lens).cuda())
    by_key = _image(keys, case["dtype"]).sort(stable=True).indices
    order = by_key[row[by_key].sort(stable=True).indices]
    start, k = torch.from_numpy(off[:-1]).cuda(), torch.from_numpy(ks).cuda()
    last = order[start + k - 1]
    first = order[torch.arange(order.numel(), device="cuda") - start[row.long()] < k[row.long()]]
    placed = torch.full_like(keys, UNSET).scatter_(0, first, keys[first])
    return {"placed": placed, "key": keys[last], "pos": last - start}
