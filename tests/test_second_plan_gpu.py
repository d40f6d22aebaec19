"""Selections whose candidates sit on a few values: from 2^20 expected candidates
on, a level by sampling follows the bins.  Every k class on both sides of that
line, selected sets checked whole, and the rank-k pair alone."""
import numpy as np
import pytest

import oracle

from _gpu import bits_of, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tk():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_03942_gb300 as tk
    return tk


@pytest.mark.parametrize("values,n", [(3, 1 << 25), (200, (1 << 25) + 11), (200, 1 << 22)])
def test_ties_in_the_bracket(tk, values, n):
    ctx, orc = tk.Context(0), oracle.default()
    g = np.random.Generator(np.random.Philox(values + n))
    at = (2.0 ** np.linspace(-100, 100, values)).astype(np.float32)
    keys = at[g.integers(0, values, size=n)].view(np.uint32)
    d = to_device(keys, "f32")
    for k in (n // 3, n // 2, int(n * 0.9)):
        ok, oi, kk, ki = tk.topk_select(ctx, d, k)
        assert orc.check_selection(keys, "f32", k, bits_of(oi), int(bits_of(ki)[0]), out_keys=bits_of(ok),
                                   kth_key=bits_of(kk)) == 0
        k2, i2 = tk.topk_select_kth(ctx, d, k)
        assert int(bits_of(k2)[0]) == int(bits_of(kk)[0]) and int(bits_of(i2)[0]) == int(bits_of(ki)[0])
    ctx.close()
