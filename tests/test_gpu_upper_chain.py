"""The stages above 0 as programmatic dependents of stage 0 on the caller's stream, the merge behind them, against the oracle: two
and three stages, stage 1 of more self-contained blocks than it completes by itself and of families longer than a block,
head_dim 64 and 128, behind a waiting build and behind a deferred one whose counts the host does not have yet.  Calls back to
back that share a workspace give what calls with workspaces of their own give."""
import numpy as np
import pytest
import torch

import gen
import oracle
from gpu_util import check_close, dev_struct, dev_tensor, host
from oracle import index_oracle as ix

pytestmark = pytest.mark.gpu

DOC, TREE = gen.layout, gen.layout_tree
# sequences, heads at head_dim 64 and 128, whether the forward takes the chain too (else stage 1 completes its elements itself)
CASES = {
    "three_stages": ([DOC([[7, 30, 12, 5] * 12] * 3), DOC([[20] * 90])], (64, 32), False),
    "one_section_longer": ([DOC([[40] * 3, [9] * 60, [], [3]])], (96, 48), False),
    "many_short": ([DOC([[1] * 60] * 6), DOC([[25] * 40] * 2)], (24, 16), False),
    "many_blocks": ([DOC([[1] * 60] * 6), DOC([[25] * 40] * 2)], (80, 80), True),
    "long_section": ([DOC([[2, 9] * 100, [3] * 30, [14] * 128]), DOC([[5] * 150])], (24, 12), True),
    "two_stages": ([TREE([[[]] * 12] * 150), TREE([[[]] * 20] * 127)], (16, 8), True),
}


def assert_route(b, n_stages, H, d, forward):
    """What sends the backward (and the forward) to the chain, from the oracle's index: full tensor-core stage 0, too many pairs above it for the
    row-wise kernel, and a stage 1 that the forward does not let complete its elements by itself."""
    index = ix.build(b.level, b.parent, b.cu_seqlens)
    s0, s1 = index.stages[:2]
    pairs = [int((s.rng[:, 1] - s.rng[:, 0]).sum()) for s in index.stages]
    assert len(index.stages) == n_stages
    assert s0.n_fused == len(s0.blocks) and index.nnz > 10 * b.total_tokens and sum(pairs[1:]) * H * (d // 64) > 300000
    whole = all(f & (ix.F_SELF | ix.F_EMPTY) for f in s1.blocks[:, 4])
    assert forward == (not whole or len(s1.blocks) * H > 2 * torch.cuda.get_device_properties(0).multi_processor_count)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("name", sorted(CASES))
def test_upper_chain(name, d):
    import paper_2407_08330_b200 as P
    seqs, heads, forward = CASES[name]
    H, n_stages = heads[d == 128], 2 if name == "two_stages" else 3
    b = gen.pack(seqs)
    assert_route(b, n_stages, H, d, forward)
    idx = P.hdt_build_index(*dev_struct(b))
    ws = [[torch.empty(P.hdt_attn_workspace_bytes(idx, H, d, torch.bfloat16, w), dtype=torch.uint8, device="cuda") for w in (0, 1)] for _ in range(2)]
    sets = []
    for seed in (1, 2):
        t = gen.make_tensors(seed, b.total_tokens, H, d, "bf16")
        sets.append((t, [dev_tensor(t[n], "bf16") for n in ("q", "k", "v", "do")]))

    def run(index, x, w):
        q, k, v, do = x
        o, lse = P.hdt_attn_fwd(index, q, k, v, workspace=w[0])
        return (o, lse) + tuple(P.hdt_attn_bwd(index, q, k, v, o, lse, do, workspace=w[1]))

    launches = P.hdt_launch_count()
    got = [run(idx, x, ws[0]) for _, x in sets]          # (queued without a wait between them)
    assert P.hdt_launch_count() - launches == 2 * (2 * n_stages + 1 + forward)      # a kernel a stage, and the merges
    P.hdt_device_status()
    for (_, x), g in zip(sets, got):
        # (the size query would wait for the counts: the workspaces are there before)
        deferred = P.hdt_build_index(*dev_struct(b), deferred=True)
        for a, c in zip(g, run(deferred, x, ws[1])):
            assert torch.equal(a, c)
    t, g = sets[1][0], got[1]
    o_r, lse_r = oracle.forward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"])
    g_r = oracle.backward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"], t["do"])
    for x, r, what in zip(g, (o_r, lse_r) + tuple(g_r), ("O", "LSE", "dQ", "dK", "dV")):
        check_close(host(x), r, "bf16", f"{what} {name}", out_rounding=True)
