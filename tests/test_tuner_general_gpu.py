"""The batched tuner times its settings on the path that they set: every row by
the general path, in every timed run and in the one that leaves the outputs,
also for rows that a call without settings reads once (k_rows).  Then rows that
only the general path takes, with the settings it chose."""
import numpy as np
import pytest

from _gpu import to_device
from test_batched_gpu import check_rows, rows_for

pytestmark = pytest.mark.gpu


def test_tuner_runs_the_general_path():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_03942_gb300 as tk
    rows = 500  # (more than start at once, so that k_rows would have a launch of its own)
    keys, off, ks = rows_for("f32", rows, 8, 13, 256, seed=52)
    d_keys, d_off, d_k = to_device(keys, "f32"), to_device(off, "u64"), to_device(ks, "u32")
    c = tk.Context(0)
    ok, oi, kk, ki, out_off = tk.topk_select_batched(c, d_keys, d_off, d_k)
    out = (torch.empty_like(ok), torch.empty_like(oi), torch.empty_like(kk), torch.empty_like(ki))
    c.profile(True)
    c.profile_read(reset=True)
    best = tk.topk_tune_batched(c, d_keys, d_off, d_k, out, out_off)
    launches = c.profile_read(reset=True)["launches"]
    c.profile(False)
    check_rows(keys, off, ks, "f32", (*out, out_off), range(rows))
    # four runs of each setting and split length: order, the wide rows' two, the rows
    assert launches == 4 * (24 * 4 + 3 * 4 + 2) + (2 if best.split_rows == tk.TOPK_SPLIT_NONE else 4)

    keys, off, ks = rows_for("f32", 100, 13, 16, 10, seed=53)
    ks = np.minimum(np.diff(off).astype(np.int64) // 2, 3000 + ks).astype(np.uint32)
    d_keys, d_off, d_k = to_device(keys, "f32"), to_device(off, "u64"), to_device(ks, "u32")
    for params in (best, None):
        res = tk.topk_select_batched(c, d_keys, d_off, d_k, params=params)
        check_rows(keys, off, ks, "f32", res, range(0, 100, 3))
    c.close()
