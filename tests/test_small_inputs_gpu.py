"""Inputs that one block selects in one launch (k_small): the sizes around its
limit of 8192 keys and the smallest, both forms of the call and both orders,
every key type, ties, and an input that is not 16-byte aligned."""
import pytest

import oracle

from _gpu import bits_of, check_against_oracle, to_device
from test_select_gpu import keys_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["u32", "i32", "f32", "bf16", "u64"])
@pytest.mark.parametrize("kind", ["uniform", "ties"])
def test_small_inputs(name, kind):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_03942_gb300 as tk
    ctx, orc = tk.Context(0), oracle.default()
    ctx.profile(True)
    largest = tk.make_params(flags=tk.TOPK_FLAG_LARGEST)
    for n in (2, 3, 31, 1024, 8191, 8192, 8193):
        keys = keys_for(name, n + 1, seed=n + 5, kind=kind)
        whole = to_device(keys, name)
        for skip in (0, 1):
            part, d = keys[skip:n + skip].copy(), whole[skip:n + skip]
            for k in sorted({1, 2, n // 2, n - 1, n} - {0}):
                ctx.profile_read(reset=True)
                out = tk.topk_select(ctx, d, k)
                launches = 4 if n > 8192 and name == "u64" and 1 < k < n else 1
                assert ctx.profile_read(reset=True)["launches"] == launches
                check_against_oracle(part, name, k, out, orc)
                kk, ki = tk.topk_select_kth(ctx, d, k)
                assert int(bits_of(kk)[0]) == int(bits_of(out[2])[0]) and int(bits_of(ki)[0]) == int(bits_of(out[3])[0])
                kk, ki = tk.topk_select_kth(ctx, d, k, params=largest)
                _, want = orc.select_largest(part, name, k)
                assert int(bits_of(ki)[0]) == want and int(bits_of(kk)[0]) == int(part[want])
                got = bits_of(tk.topk_select(ctx, d, k, params=largest)[1])
                assert sorted(got.tolist()) == sorted(orc.select_largest(part, name, k)[0].tolist())
    ctx.close()
