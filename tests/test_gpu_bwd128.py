"""The head_dim 128 backward of self-contained blocks at the sizes where it can go wrong: row blocks of 1, 15, 16, 17, 127
and 128 rows, one item a CTA and several (an odd and an even number: its accumulators take turns in tensor
memory), dO . O computed inside and by a pass of its own."""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import check_close, dev_struct, dev_tensor, host

pytestmark = pytest.mark.gpu

CASES = {      # documents (sentence lengths of their sections), heads
    "one_row_blocks": ([[[1], [127]], [[126], [1, 127, 127]]], 3),
    "edges": ([[[14], [15, 127]], [[16, 127, 13, 127, 125]], [[0, 0, 127, 126, 14]]], 2),
    "two_items": ([[[60, 50, 70, 40, 90, 30] * 2]], 40),
    "several_items": ([[[33, 5, 60, 17, 127, 44, 9] * 4], [[20] * 25]], 48),
}


@pytest.mark.parametrize("separate_delta", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_bwd128(name, separate_delta):
    import paper_2407_08330_b200 as P
    docs, H = CASES[name]
    b = gen.pack([gen.layout(s) for s in docs])
    t = gen.make_tensors(11, b.total_tokens, H, 128, "bf16")
    q, k, v, do = (dev_tensor(t[n], "bf16") for n in ("q", "k", "v", "do"))
    P.hdt_set_option("no_fused_delta", separate_delta)
    try:
        idx = P.hdt_build_index(*dev_struct(b))
        o, lse = P.hdt_attn_fwd(idx, q, k, v)
        g = P.hdt_attn_bwd(idx, q, k, v, o, lse, do)
        P.hdt_device_status()
    finally:
        P.hdt_set_option("no_fused_delta", 0)
    want = oracle.backward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"], t["do"])
    # (the bounds of the random batches: the stated tolerance, and the rounding of a stored result beyond 4)
    for x, r, what in zip(g, want, ("dQ", "dK", "dV")):
        check_close(host(x), r, "bf16", f"{what} {name}", out_rounding=True)
