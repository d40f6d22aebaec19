"""Rounds of the exact selection over sorted runs, one warp per run: numbers of
runs around a block's warps and around the limits for the shared prefix and for
the pivots per round, numbers of pivots around a lane's share, ties, empty runs."""
import numpy as np
import pytest

import oracle

from _gpu import bits_of, to_device
from test_runs_gpu import make_runs, run_and_check

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


@pytest.mark.parametrize("p,maxlen", [(1, 40000), (7, 9000), (8, 9000), (9, 9000), (1000, 300), (4096, 30), (4097, 30),
                                      (8193, 20)])
@pytest.mark.parametrize("alphabet", [None, 3])
def test_rounds_by_runs(tk, ctx, p, maxlen, alphabet):
    keys, off = make_runs(p, maxlen, seed=p + maxlen, alphabet=alphabet)
    total = int(off[-1])
    for k in sorted({1, total // 3 + 1, total - 1} - {0}):
        run_and_check(tk, ctx, keys, off, k)


@pytest.mark.parametrize("d", [1, 31, 32, 33, 64, 65, 128, 129, 255])
def test_rounds_by_pivots(tk, ctx, d):
    keys, off = make_runs(300, 900, seed=d, alphabet=None if d % 2 else 1000)
    run_and_check(tk, ctx, keys, off, int(off[-1]) // 2, params=tk.make_params(sample_size=d))
