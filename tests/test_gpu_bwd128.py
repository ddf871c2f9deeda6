"""The head_dim 128 backward of self-contained blocks at the sizes where it can go wrong: row blocks of 2, 15, 16, 17, 127 and
128 rows, one item a CTA and several (an odd and an even number: its accumulators take turns in tensor memory), beside
EMPTY blocks and without them; dO . O computed inside, where there are none, and by a pass of its own."""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import check_close, dev_struct, dev_tensor, host
from oracle import index_oracle as ix

pytestmark = pytest.mark.gpu

DOC = gen.layout
EDGES = (2, 15, 16, 17, 127, 128)
ROOTS = [gen.layout_tree([[]] * (n - 1)) for n in EDGES]      # a family each, the root its head: a block of n rows
CASES = {      # sequences, heads, whether dO . O can be computed inside (no EMPTY block)
    "one_item": (ROOTS, 3, True),
    "two_or_three_items": (ROOTS, 60, True),
    "edges_and_documents": (ROOTS + [DOC([[60, 50, 70, 40, 90, 30]]), DOC([[20, 100], [7] * 30])], 25, True),
    "short_documents": ([DOC([[1], [127]]), DOC([[126], [1, 127, 127]])], 3, False),
    "beside_empty": ([DOC([[14], [15, 127]]), DOC([[16, 127, 13, 127, 125]]), DOC([[0, 0, 127, 126, 14]])], 2, False),
    "two_items": ([DOC([[60, 50, 70, 40, 90, 30] * 2])], 40, True),
    "several_items": ([DOC([[33, 5, 60, 17, 127, 44, 9] * 4]), DOC([[20] * 25])], 48, True),
}


@pytest.mark.parametrize("separate_delta", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_bwd128(name, separate_delta):
    import paper_2407_08330_b200 as P
    seqs, H, inside = CASES[name]
    b = gen.pack(seqs)
    index = ix.build(b.level, b.parent, b.cu_seqlens)
    s0 = index.stages[0]
    assert (s0.n_fused == len(s0.blocks)) == inside and index.nnz > 10 * b.total_tokens
    if seqs[0] is ROOTS[0]:
        assert set(EDGES) <= set((s0.blocks[:, 1] - s0.blocks[:, 0]).tolist())
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
