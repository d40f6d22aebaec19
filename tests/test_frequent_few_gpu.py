"""The exact recount of few candidates (EC): one to 33 of them (33 take the
general recount), aligned and unaligned inputs, ragged tails, objects whose
values are structured, among them 0, 1 and 0xFFFFFFFF."""
import numpy as np
import pytest

from _gpu import bits_of, to_device

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


@pytest.mark.parametrize("k", [1, 2, 31, 32, 33])
@pytest.mark.parametrize("shape", ["small", "shift27", "shift24", "multiples", "ends"])
@pytest.mark.parametrize("n,skip", [(8192 * 3, 0), (100_003, 0), (100_001, 1)])
def test_recount(tk, ctx, k, shape, n, skip):
    g = np.random.Generator(np.random.Philox(k * 31 + n))
    kinds = 32 if shape == "shift27" else 60
    if k > kinds:
        pytest.skip("fewer distinct objects than asked for")
    v = np.arange(kinds, dtype=np.uint64)
    objects = {"small": v, "shift27": v << np.uint64(27), "shift24": v << np.uint64(24),
               "multiples": v * np.uint64(0x10001), "ends": np.where(v % 2, v // 2, 0xFFFFFFFF - v // 2)}[shape]
    p = 1.0 / (1.0 + np.arange(kinds)) ** 0.3
    draw = g.choice(kinds, size=n + skip, p=p / p.sum())
    x = objects.astype(np.uint32)[draw]
    d = to_device(x, "u32")[skip:]
    fp = tk.make_freq_params(k, tk.TOPK_FREQ_EC, rho=1.0, kstar=k)
    obj, cnt, size = tk.topk_frequent(ctx, d, fp)
    want, times = np.unique(x[skip:], return_counts=True)
    order = np.lexsort((want, -times))[:k]
    got = dict(zip(bits_of(obj).tolist(), bits_of(cnt).tolist()))
    assert got == {int(want[i]): int(times[i]) for i in order}
    assert int(bits_of(size)[0]) == n
