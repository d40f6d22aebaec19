"""topk_select_kth with many elements below rank k: the first pass counts them
and writes none.  Sizes around the pass's tiles of 4096 keys, every key type,
both orders, aligned and unaligned input, ties on the pivots; the rank-k pair
has to be the oracle's, bit for bit."""
import pytest

import oracle

from _gpu import bits_of, to_device
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
@pytest.mark.parametrize("n", [16385, 5 * 4096, 5 * 4096 + 1, 70001, 1 << 19])
@pytest.mark.parametrize("kind", ["uniform", "ties"])
def test_kth_counts_a(tk, ctx, orc, name, n, kind):
    if kind == "ties" and name == "u64":
        pytest.skip("no tied 64-bit inputs")
    keys = keys_for(name, n, seed=n + 3, kind=kind)
    d = to_device(keys, name)
    for k in (n // 8, n // 2 + 1, n - 2):
        kk, ki = tk.topk_select_kth(ctx, d, k)
        _, want = orc.select(keys, name, k)
        assert int(bits_of(ki)[0]) == want and int(bits_of(kk)[0]) == int(keys[want])
        kk, ki = tk.topk_select_kth(ctx, d, k, params=tk.make_params(flags=tk.TOPK_FLAG_LARGEST))
        _, want = orc.select_largest(keys, name, k)
        assert int(bits_of(ki)[0]) == want and int(bits_of(kk)[0]) == int(keys[want])
    rest = keys[1:].copy()
    kk, ki = tk.topk_select_kth(ctx, d[1:], n // 3)
    _, want = orc.select(rest, name, n // 3)
    assert int(bits_of(ki)[0]) == want and int(bits_of(kk)[0]) == int(rest[want])
