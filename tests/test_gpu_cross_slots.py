"""Cross-attention backward (bf16) around the ends of its block slots and of the zeroing kernel's pieces: encoders of 31 to 4097
tokens, subsets that fill a block exactly, leave the last slots unused or take every token, documents without decoder
rows before and behind those that have some.  Rows that no decoder row attends to are exact zeros."""
import numpy as np
import pytest
import torch

import gen
from oracle import cross_oracle as co
from gpu_util import check_close, dev_tensor, host

pytestmark = pytest.mark.gpu

CASES = {      # sequences (sentence lengths of their sections), decoder rows of each, level mask, heads, head_dim
    "one_warp": ([[[28]]], [5], 8, 1, 64),
    "piece_edges": ([[[29]], [[12, 15]], [[61]]], [0, 9, 130], 12, 2, 64),
    "block_filled": ([[[0] * 127], [[3] * 128], [[1] * 129]], [128, 1, 17], 4, 3, 64),
    "many_unused": ([[[60] * 33], [[60] * 30]], [40, 30], 2, 2, 128),
    "every_token": ([[[60] * 33, [50] * 10], [[7] * 3]], [20, 0], 15, 1, 64),
    "long": ([[[31] * 64, [31] * 63]], [33], 6, 1, 64),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_cross_slots(name):
    import paper_2407_08330_b200 as P
    docs, nq, mask, H, d = CASES[name]
    b = gen.pack([gen.layout(s) for s in docs])
    rng = np.random.default_rng(3)
    cu_q = np.concatenate([[0], np.cumsum(nq)]).astype(np.int32)
    q, do = (gen.round_bf16(rng.standard_normal((int(cu_q[-1]), H, d)).astype(np.float32)) for _ in range(2))
    k, v = (gen.round_bf16(rng.standard_normal((b.total_tokens, H, d)).astype(np.float32)) for _ in range(2))
    lv, cuk, cuq = (torch.from_numpy(x).cuda() for x in (b.level, b.cu_seqlens, cu_q))
    tq, tk, tv, tdo = (dev_tensor(x, "bf16") for x in (q, k, v, do))
    o, lse = P.hdt_cross_attn_fwd(lv, cuk, cuq, mask, tq, tk, tv)
    g = [torch.full_like(x, float("nan")) for x in (tq, tk, tv)]
    P.hdt_cross_attn_bwd(lv, cuk, cuq, mask, tq, tk, tv, o, lse, tdo, dq=g[0], dk=g[1], dv=g[2])
    P.hdt_device_status()
    want = co.backward(b.level, b.cu_seqlens, mask, cu_q, q, k, v, do)
    # (a chosen row collects gradient from every decoder row: the bounds of the other cross-attention tests)
    for x, r, what in zip(g, want, ("dQ", "dK", "dV")):
        check_close(host(x), r, "bf16", f"{what} {name}", out_rounding=True)
    doc = np.repeat(np.arange(b.batch), np.diff(b.cu_seqlens))
    rest = torch.from_numpy(~(((mask >> np.maximum(b.level, 0)) & 1).astype(bool) & (b.level >= 0) & (np.asarray(nq)[doc] > 0))).cuda()
    assert (g[1][rest] == 0).all() and (g[2][rest] == 0).all()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("docs,nq,mask,H,d", [
    ([[[3]]], [1], 15, 1, 64),                              # one piece
    ([[[31] * 4], [[0] * 3], [[60] * 2]], [1, 1, 1], 15, 12, 64),      # a piece of 32 tokens and more, two CTAs an SM
    ([[[60] * 40]], [1], 15, 16, 128),                      # four CTAs an SM
    ([[[60] * 40], [[9] * 7]], [2, 1], 6, 40, 128),         # more heads than a CTA takes, anchors alone
    ([[[50] * 160]], [3], 8, 3, 64),                        # the longest pieces, a document with every row
])
def test_decode_pieces(docs, nq, mask, H, d, dtype):
    import paper_2407_08330_b200 as P
    b = gen.pack([gen.layout(s) for s in docs])
    rng = np.random.default_rng(4)
    f = gen.round_bf16 if dtype == "bf16" else (lambda x: x)
    cu_q = np.concatenate([[0], np.cumsum(nq)]).astype(np.int32)
    q = f(rng.standard_normal((int(cu_q[-1]), H, d)).astype(np.float32))
    k, v = (f(rng.standard_normal((b.total_tokens, H, d)).astype(np.float32)) for _ in range(2))
    lv, cuk, cuq = (torch.from_numpy(x).cuda() for x in (b.level, b.cu_seqlens, cu_q))
    o, lse = P.hdt_cross_attn_fwd(lv, cuk, cuq, mask, *(dev_tensor(x, dtype) for x in (q, k, v)))
    P.hdt_device_status()
    o_r, lse_r = co.forward(b.level, b.cu_seqlens, mask, cu_q, q, k, v)
    check_close(host(o), o_r, dtype, "O")
    check_close(host(lse), lse_r, "f32" if dtype == "f32" else "bf16", "LSE")


@pytest.mark.parametrize("T", [591, 592, 593, 1184, 1185, 18943, 18945, 20001])
def test_zero_rows(T):
    """Around the sizes where a warp of the zeroing kernel takes one token more, and where it comes back for others."""
    import paper_2407_08330_b200 as P
    level = np.full(T, 3, np.int8)
    level[[0, 5, T // 2, T - 2]] = [0, 2, 2, 2]
    lv, cuk, cuq = (torch.from_numpy(np.asarray(x)).cuda() for x in (level, np.array([0, T], np.int32), np.array([0, 3], np.int32)))
    rng = np.random.default_rng(5)
    q, do = (gen.round_bf16(rng.standard_normal((3, 1, 64)).astype(np.float32)) for _ in range(2))
    k, v = (gen.round_bf16(rng.standard_normal((T, 1, 64)).astype(np.float32)) for _ in range(2))
    tq, tk, tv, tdo = (dev_tensor(x, "bf16") for x in (q, k, v, do))
    o, lse = P.hdt_cross_attn_fwd(lv, cuk, cuq, 4, tq, tk, tv)
    g = [torch.full_like(x, float("nan")) for x in (tq, tk, tv)]
    P.hdt_cross_attn_bwd(lv, cuk, cuq, 4, tq, tk, tv, o, lse, tdo, dq=g[0], dk=g[1], dv=g[2])
    P.hdt_device_status()
    for x, r, what in zip(g, co.backward(level, np.array([0, T], np.int32), 4, np.array([0, 3], np.int32), q, k, v, do), ("dQ", "dK", "dV")):
        check_close(host(x), r, "bf16", what, out_rounding=True)
    rest = torch.from_numpy(level != 2).cuda()
    assert (g[1][rest] == 0).all() and (g[2][rest] == 0).all()
