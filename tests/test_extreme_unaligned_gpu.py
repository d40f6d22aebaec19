"""k = 1 and k = n (one reduction kernel) on inputs that start inside a 16-byte
segment, at lengths around its tiles of 4096 keys: the last keys then lie in a
tile that the length alone does not reach.  The extreme key is put there."""
import numpy as np
import pytest

import oracle

from _gpu import NP_BITS, bits_of, check_against_oracle, to_device
from test_select_gpu import keys_for

pytestmark = pytest.mark.gpu

LOWEST = {"u32": 0, "i32": 0x80000000, "f32": 0xFF800000, "bf16": 0xFF80, "u64": 0}
HIGHEST = {"u32": 0xFFFFFFFF, "i32": 0x7FFFFFFF, "f32": 0x7F800000, "bf16": 0x7F80, "u64": 0xFFFFFFFFFFFFFFFF}


@pytest.mark.parametrize("name", ["u32", "i32", "f32", "bf16", "u64"])
@pytest.mark.parametrize("n", [4095, 4096, 4097, 3 * 4096 - 1, 3 * 4096, 1 << 18])
def test_extreme_at_the_end(name, n):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_03942_gb300 as tk
    ctx, orc = tk.Context(0), oracle.default()
    largest = tk.make_params(flags=tk.TOPK_FLAG_LARGEST)
    for skip in range(16 // np.dtype(NP_BITS[name]).itemsize):
        for end in (LOWEST, HIGHEST):
            keys = keys_for(name, n + skip, seed=n + skip)
            keys[-1] = end[name]
            part, d = keys[skip:].copy(), to_device(keys, name)[skip:]
            for k in (1, n):
                check_against_oracle(part, name, k, tk.topk_select(ctx, d, k), orc)
                check_against_oracle(part, name, k, tk.topk_select_noalloc(d, k), orc)
                kk, ki = tk.topk_select_kth(ctx, d, k)
                want = orc.select(part, name, k)[1]
                assert int(bits_of(ki)[0]) == want and int(bits_of(kk)[0]) == int(part[want])
                kk, ki = tk.topk_select_kth(ctx, d, k, params=largest)
                want = orc.select_largest(part, name, k)[1]
                assert int(bits_of(ki)[0]) == want and int(bits_of(kk)[0]) == int(part[want])
    ctx.close()
