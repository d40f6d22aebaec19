"""Rows of small k in one read: lengths around the list and the warps' steps, k
around the largest that is taken, unaligned rows, ties on the bound, rows whose
list has to be cut back, and rows left to the general path among them."""
import numpy as np
import pytest

import oracle
from paper_1502_03942_gb300 import workloads as wl

from _gpu import to_device
from test_batched_gpu import check_rows, rows_for, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tk():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_03942_gb300 as tk
    return tk


@pytest.fixture(scope="module")
def ctx(tk):
    c = tk.Context(0)
    yield c
    c.close()


def bits(name, n, seed, alphabet):
    g = np.random.Generator(np.random.Philox(seed))
    if alphabet:
        v = g.integers(0, alphabet, size=n)
        return (v * 97).astype({"bf16": np.uint16, "u64": np.uint64}.get(name, np.uint32))
    if name == "u64":
        return wl.uniform_u64(n, seed)
    if name == "f32":
        return wl.normal_f32(n, seed).view(np.uint32)
    return wl.uniform_u32(n, seed).astype(np.uint16 if name == "bf16" else np.uint32)


@pytest.mark.parametrize("name", ["u32", "i32", "f32", "bf16", "u64"])
@pytest.mark.parametrize("alphabet", [None, 5])
def test_edges(tk, ctx, name, alphabet):
    cap = 2048 if name == "u64" else 4096
    lens = [1, 2, 511, 512, 513, 1023, cap - 1, cap, cap + 1, cap + 513, 3 * cap + 7, 70001]
    shapes = [(n, k) for n in lens for k in sorted({1, 2, 31, cap // 2, cap // 2 + 1, n // 2, n - 1, n}) if 1 <= k <= n]
    off = np.zeros(len(shapes) + 1, np.uint64)
    off[1:] = np.cumsum([n for n, _ in shapes])
    ks = np.array([k for _, k in shapes], np.uint32)
    keys = bits(name, int(off[-1]), 91, alphabet)
    res = run(tk, ctx, keys, off, ks, name)
    check_rows(keys, off, ks, name, res, range(len(shapes)))


def test_list_cut_back(tk, ctx):
    """Rows whose sample misleads: every 64th key is large, so a bound drawn too
    high floods the list, and descending rows, which refill it."""
    n = 60000
    rows = []
    for r in range(6):
        x = wl.uniform_u32(n, 100 + r)
        x = np.sort(x)[::-1].copy() if r % 2 else np.where(np.arange(n) % 64 < 40, x | np.uint32(0x80000000), x >> np.uint32(12))
        rows.append(x.astype(np.uint32))
    keys = np.concatenate(rows)
    off = (np.arange(7) * n).astype(np.uint64)
    ks = np.array([2048, 2048, 2000, 1, 1500, 2047], np.uint32)
    check_rows(keys, off, ks, "u32", run(tk, ctx, keys, off, ks, "u32"), range(6))


def test_more_rows_than_blocks(tk, ctx):
    """Enough rows for the queue, with rows of large k and long rows left over;
    twice, so that the counters are left as they were found."""
    keys, off, ks = rows_for("f32", 700, 0, 11, 300, seed=77)
    lens = np.diff(off).astype(np.int64)
    big = np.concatenate([keys, bits("f32", 600000, 5, None)])
    off = np.append(off, np.uint64(off[-1] + 600000))
    ks = np.append(ks, np.uint32(3000))
    ks[::9] = np.maximum(1, lens[::9]).astype(np.uint32)[: ks[::9].size]
    for _ in range(2):
        check_rows(big, off, ks, "f32", run(tk, ctx, big, off, ks, "f32"), list(range(0, 700, 3)) + [700])
