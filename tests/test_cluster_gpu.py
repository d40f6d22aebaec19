"""The pivots and the finish of a selection, each run by a cluster of blocks, at
the sizes and inputs where their windows go wrong first: one block and several,
a list that just fits, candidates that sit on a few distant values (so that the
bins of the bracket resolve nothing and the finish streams its source), brackets
open at an end of the keys, and the second pass over the candidates."""
import numpy as np
import pytest

import oracle

from _gpu import bits_of, check_against_oracle, to_device
from test_select_gpu import keys_for

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


@pytest.fixture(scope="module")
def orc():
    return oracle.default()


@pytest.mark.parametrize("name", ["u32", "i32", "f32", "bf16", "u64"])
@pytest.mark.parametrize("kind", ["uniform", "ties"])
@pytest.mark.parametrize("n", [2, 33, 1025, 4096, 4097, 8192, 8193, 16384])
def test_finish_alone(tk, ctx, orc, name, kind, n):
    keys = keys_for(name, n, seed=n + 1, kind=kind)
    d = to_device(keys, name)
    for k in sorted({2, n // 3 + 1, n - 1} & set(range(1, n + 1))):
        check_against_oracle(keys, name, k, tk.topk_select(ctx, d, k), orc)


@pytest.mark.parametrize("n", [1 << 18, (1 << 21) + 5])
@pytest.mark.parametrize("values", [2, 40])
def test_candidates_on_few_values(tk, ctx, orc, n, values):
    """Keys on distant values, rank k near the edge between two of them."""
    g = np.random.Generator(np.random.Philox(n + values))
    at = (2.0 ** np.linspace(-60, 60, values)).astype(np.float32)
    keys = at[g.integers(0, values, size=n)].view(np.uint32)
    d = to_device(keys, "f32")
    edge = int((keys <= at.view(np.uint32)[values // 2 - 1]).sum())
    for k in (edge - 1, edge, edge + 1):
        check_against_oracle(keys, "f32", k, tk.topk_select(ctx, d, k), orc)
        kk, ki = tk.topk_select_kth(ctx, d, k)
        _, want = orc.select(keys, "f32", k)
        assert int(bits_of(ki)[0]) == want and int(bits_of(kk)[0]) == int(keys[want])


@pytest.mark.parametrize("name", ["u32", "f32", "bf16", "u64"])
def test_open_brackets_and_second_pass(tk, ctx, orc, name):
    """k at both ends and in the middle of enough keys for a second pass."""
    n = (1 << 21) + 7
    keys = keys_for(name, n, seed=23)
    d = to_device(keys, name)
    for k in (2, 37, n // 2, n - 40, n - 1):
        check_against_oracle(keys, name, k, tk.topk_select(ctx, d, k), orc)
