"""Which rows a default batched call reads once (k_rows) and which it leaves to the
general path: few long rows, long rows among many short ones, rows of large k,
with and without the kernel that orders them, each twice, so that the queues are
left as they were found.  And rows whose sampled bound is too low, which go to the
general path after they were read."""
import numpy as np
import pytest

from _gpu import to_device
from test_batched_gpu import check_rows, run
from test_batched_rows_gpu import bits

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


# (length, k, rows) groups of one batch
BATCHES = {
    "few long rows": [(300_000, 100, 3)],
    "longest row and one more": [(1 << 19, 50, 1), ((1 << 19) + 1, 50, 1)],
    "long rows and short ones": [(200_001, 7, 4), (2000, 100, 60)],
    "rows just below the split length too": [(200_001, 7, 4), (20_000, 100, 20)],
    "large k only": [(9000, 3000, 20), (40_000, 3000, 3)],
    "large k among small": [(9000, 3000, 5), (20_000, 30, 10), (500, 500, 10)],
    "queue: long rows and short ones": [(250_000, 7, 3), (1500, 20, 700)],
    "queue: some left": [(600_000, 5, 1), (30_000, 2500, 9), (700, 60, 600)],
    "queue: none taken": [(5000, 4900, 500)],
}


@pytest.mark.parametrize("name", ["f32", "u64", "bf16"])
@pytest.mark.parametrize("batch", BATCHES)
def test_routes(tk, ctx, name, batch):
    g = np.random.Generator(np.random.Philox(len(batch)))
    rows = np.array([(n, k) for n, k, r in BATCHES[batch] for _ in range(r)])[:, :]
    rows = rows[g.permutation(len(rows))]
    off = np.zeros(len(rows) + 1, np.uint64)
    off[1:] = np.cumsum(rows[:, 0])
    ks = rows[:, 1].astype(np.uint32)
    keys = bits(name, int(off[-1]), 17, None)
    for _ in range(2):
        res = run(tk, ctx, keys, off, ks, name)
        check_rows(keys, off, ks, name, res, range(0, len(rows), 1 + len(rows) // 60))


@pytest.mark.parametrize("rows", [3, 500])
def test_bad_row_on_either_route(tk, ctx, rows):
    for n in (40_000, 300_000 if rows < 10 else 3000):
        off = (np.arange(rows + 1) * n).astype(np.uint64)
        keys = bits("u32", int(off[-1]), 3, None)
        for k in (50, 2500):
            ks = np.full(rows, k, np.uint32)
            ks[rows // 2] = 0
            with pytest.raises(tk.TopkError) as e:
                run(tk, ctx, keys, off, ks, "u32")
            assert e.value.status == tk.TOPK_EINVAL
            ks[rows // 2] = 1
            check_rows(keys, off, ks, "u32", run(tk, ctx, keys, off, ks, "u32"), [0, rows // 2, rows - 1])


@pytest.mark.parametrize("name", ["f32", "u64"])
@pytest.mark.parametrize("rows", [40, 600])
def test_bound_too_low(tk, ctx, name, rows):
    """A margin of a hundredth of a standard deviation: many bounds miss low."""
    g = np.random.Generator(np.random.Philox(rows))
    lens = g.integers(5000, 20000, size=rows)
    off = np.zeros(rows + 1, np.uint64)
    off[1:] = np.cumsum(lens)
    ks = g.integers(300, 1000, size=rows).astype(np.uint32)
    keys = bits(name, int(off[-1]), 29, None)
    d = to_device(keys, name), to_device(off, "u64"), to_device(ks, "u32")
    for seed in (1, 2, 3):
        res = tk.topk_select_batched(ctx, *d, params=tk.make_params(delta_factor=0.01, seed=seed))
        check_rows(keys, off, ks, name, res, range(0, rows, 1 + rows // 60))
