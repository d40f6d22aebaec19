"""Orderings inside a kernel that no run can be relied on to show when they are
broken (the latencies of the other work hide them), read off the source on the
CPU: what has to lie before or after which barrier.  The GPU test repeats the
call whose result depended on them.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1502_03942_gb300", "csrc")


def body_of(path, kernel):
    """The body of a __global__ function, without comments."""
    with open(os.path.join(CSRC, path)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = re.search(r"__global__ void [^;{]*\b" + kernel + r"\(", text).start()
    at = text.index("{", start)
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
        i += 1


def test_plan_clears_before_the_cluster_barrier():
    """k_plan: the words that other blocks reduce into are cleared before this
    block arrives at the barrier that lets them, and no block leaves after a
    failed selection while the others still read its bins."""
    body = body_of("select_cluster.cuh", "k_plan")
    first = {what: body.index(what) for what in ("cl_clear(", "cl_arrive(", "cl_wait(", "cl_range(", "cl_select<")}
    assert first["cl_clear("] < first["cl_arrive("] < first["cl_wait("] < first["cl_range("] < first["cl_select<"]
    assert body.count("cl_clear(") == 1
    after = body[first["cl_select<"]:]
    assert 0 <= after.find("if (!ok) cl_sync();") < after.index("return")


def test_rows_queue_word_is_written_at_the_top_only():
    """k_rows: the word that hands out a row is read by every thread after the
    loop's barrier, the last time without another barrier behind it, so it is
    written at the top of the loop and nowhere else."""
    body = body_of("batched.cu", "k_rows")
    writes = [m.start() for m in re.finditer(r"\bsm\.row\s*=(?!=)", body)]
    loop = body.index("while (true)")
    assert len(writes) == 1 and loop < writes[0] < body.index("__syncthreads()", loop)


@pytest.mark.gpu
@pytest.mark.parametrize("n,k", [(20000, 7000), (1 << 21, 1 << 20)])
def test_plan_repeats(n, k):
    """The pivots follow from the seed: the same call counts the same candidates
    every time, beside another context's calls on a second stream."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_03942_gb300 as tk
    from paper_1502_03942_gb300 import workloads as wl
    from _gpu import to_device
    d = to_device(wl.uniform_u32(n, 3), "u32")
    c, other, beside = tk.Context(0), tk.Context(0), torch.cuda.Stream()
    beside.wait_stream(torch.cuda.current_stream())
    seen = set()
    for _ in range(200):
        with torch.cuda.stream(beside):
            tk.topk_select_kth(other, d, k, check=False)
        kk, ki = tk.topk_select_kth(c, d, k)
        seen.add((c.last_stats()["first_candidates"], int(ki.view(torch.int32))))
    beside.synchronize()
    c.close()
    other.close()
    assert len(seen) == 1
