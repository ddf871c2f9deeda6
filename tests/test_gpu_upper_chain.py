"""The stages above 0 as programmatic dependents of stage 0 on the caller's stream, behind waiting and deferred builds, against the
oracle: two and three stages, documents without sections, head_dim 64 and 128.  Calls back to back that share a workspace
give what calls with workspaces of their own give."""
import numpy as np
import pytest
import torch

import gen
import oracle
from gpu_util import check_close, dev_struct, dev_tensor, host

pytestmark = pytest.mark.gpu

CASES = {      # documents, heads: enough pairs above stage 0 that their kernels, not the row-wise ones, take them
    "three_stages": ([[[7, 30, 12, 5] * 12] * 3, [[20] * 90]], {64: 64, 128: 32}),
    "two_stages": ([[[40] * 3, [9] * 60, [], [3]]], {64: 96, 128: 48}),
    "many_blocks": ([[[1] * 60] * 6, [[25] * 40] * 2], {64: 24, 128: 16}),
}


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("name", sorted(CASES))
def test_upper_chain(name, d):
    import paper_2407_08330_b200 as P
    docs, heads = CASES[name]
    H = heads[d]
    b = gen.pack([gen.layout(s) for s in docs])
    idx = [P.hdt_build_index(*dev_struct(b), deferred=x) for x in (False, True)]
    ws = [torch.empty(max(256, P.hdt_attn_workspace_bytes(idx[0], H, d, torch.bfloat16, w)), dtype=torch.uint8, device="cuda") for w in (0, 1)]
    sets = []
    for seed in (1, 2):
        t = gen.make_tensors(seed, b.total_tokens, H, d, "bf16")
        x = [dev_tensor(t[n], "bf16") for n in ("q", "k", "v", "do")]
        sets.append((t, x))
    got = []
    for _, (q, k, v, do) in sets:          # (queued without a wait between them)
        o, lse = P.hdt_attn_fwd(idx[0], q, k, v, workspace=ws[0])
        got.append((o, lse) + tuple(P.hdt_attn_bwd(idx[0], q, k, v, o, lse, do, workspace=ws[1])))
    P.hdt_device_status()
    for (t, (q, k, v, do)), g in zip(sets, got):
        o, lse = P.hdt_attn_fwd(idx[1], q, k, v)
        for x, y in zip(g, (o, lse) + tuple(P.hdt_attn_bwd(idx[1], q, k, v, o, lse, do))):
            assert torch.equal(x, y)
    t, g = sets[1][0], got[1]
    o_r, lse_r = oracle.forward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"])
    g_r = oracle.backward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"], t["do"])
    for x, r, what in zip(g, (o_r, lse_r) + tuple(g_r), ("O", "LSE", "dQ", "dK", "dV")):
        check_close(host(x), r, "bf16", f"{what} {name}", out_rounding=True)
