"""Misaligned inputs with many selected keys (the dense register pass, which also
counts its candidates over bins): lengths around its tiles of 4096 keys, every
start inside 16 bytes, every key type, and ties that make a whole tile candidates."""
import numpy as np
import pytest

import oracle

from _gpu import NP_BITS, bits_of, to_device
from test_select_gpu import keys_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["u32", "i32", "f32", "bf16", "u64"])
@pytest.mark.parametrize("kind", ["uniform", "ties"])
def test_unaligned_dense(name, kind):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_03942_gb300 as tk
    ctx, orc = tk.Context(0), oracle.default()
    for n in (5 * 4096 - 1, 5 * 4096, 100003, 1 << 20):
        for skip in range(1, 16 // np.dtype(NP_BITS[name]).itemsize):
            keys = keys_for(name, n + skip, seed=n + skip, kind=kind)
            part, d = keys[skip:].copy(), to_device(keys, name)[skip:]
            for k in (n // 10, n // 2, n - n // 10):
                ok, oi, kk, ki = tk.topk_select(ctx, d, k)
                assert orc.check_selection(part, name, k, bits_of(oi), int(bits_of(ki)[0]), out_keys=bits_of(ok),
                                           kth_key=bits_of(kk)) == 0
    ctx.close()
