"""Split key lists and the decoding kernel of the cross-attention, the streaming positional encoding: the sizes where
their splits change, against the oracles."""
import numpy as np
import pytest

import gen
from oracle import cross_oracle, hpe_oracle
from tests.gpu_util import check_close, dev_struct, dev_tensor, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("bf16", 128), ("f32", 64)])
@pytest.mark.parametrize("lengths,rows,mask", [
    ([40], [1], 15), ([700, 33], [4, 4], 15), ([700, 33, 1], [1, 0, 1], 6), ([60], [4], 2),      # decoding: one and several splits, no key
    ([1500, 90], [130, 5], 15), ([600], [20], 15), ([2100], [7], 15),                            # tiles with split key lists
])
def test_cross_splits(dtype, d, lengths, rows, mask):
    import torch
    import paper_2407_08330_b200 as P
    rng = np.random.default_rng(11)
    b = gen.pack([gen.gen_fill(rng, n, (2, 6), (2, 8), (3, 20))[:2] for n in lengths])
    H, T, Tq = 3, b.total_tokens, sum(rows)
    cu_q = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    t = gen.make_tensors(3, T, H, d, dtype, names=("k", "v"))
    tq = gen.make_tensors(4, Tq, H, d, dtype, names=("q", "do"))
    level, _, cu = dev_struct(b)
    q, do, k, v = (dev_tensor(x, dtype) for x in (tq["q"], tq["do"], t["k"], t["v"]))
    cq = torch.from_numpy(cu_q).cuda()
    o, lse = P.hdt_cross_attn_fwd(level, cu, cq, mask, q, k, v)
    g = P.hdt_cross_attn_bwd(level, cu, cq, mask, q, k, v, o, lse, do)
    torch.cuda.synchronize()
    P.hdt_device_status()
    o_r, lse_r = cross_oracle.forward(b.level, b.cu_seqlens, mask, cu_q, tq["q"], t["k"], t["v"])
    g_r = cross_oracle.backward(b.level, b.cu_seqlens, mask, cu_q, tq["q"], t["k"], t["v"], tq["do"])
    check_close(host(o), o_r, dtype, "O", out_rounding=True)
    check_close(lse.cpu().numpy(), lse_r, dtype, "LSE")
    for x, r, what in zip(g, g_r, ("dQ", "dK", "dV")):
        check_close(host(x), r, dtype, what, out_rounding=True, row_rel=2.0 ** -8)


@pytest.mark.parametrize("n,longest", [(40, 1500), (1100, 260)])        # (the scan takes 1024 documents at a time)
def test_cross_index_counted(n, longest):
    """More documents times tokens than every block of the index kernel counts itself, at odd places in the arrays."""
    import torch
    import paper_2407_08330_b200 as P
    rng = np.random.default_rng(n)
    docs = [gen.gen_fill(rng, int(k), (2, 6), (2, 8), (3, 20))[:2] for k in rng.integers(1, longest, n)]
    docs[n // 2] = (np.zeros(0, np.int8), np.zeros(0, np.int32))
    b = gen.pack(docs)
    rows = rng.integers(0, 12, n)
    rows[n // 3] = 150
    H, d, T, Tq = 2, 64, b.total_tokens, int(rows.sum())
    assert n * T > 200000 and Tq > 4 * n
    cu_q = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    t = gen.make_tensors(3, T, H, d, "bf16", names=("k", "v"))
    tq = gen.make_tensors(4, Tq, H, d, "bf16", names=("q", "do"))
    _, _, cu = dev_struct(b)
    level = torch.empty(T + 1, dtype=torch.int8, device="cuda")
    q, do, k, v = (dev_tensor(x, "bf16") for x in (tq["q"], tq["do"], t["k"], t["v"]))
    cq = torch.from_numpy(cu_q).cuda()
    for mask, shift in ((6, 0), (15, 0), (6, 1)):          # (levels at an odd address: no wide loads)
        lv = level[shift:shift + T]
        lv.copy_(torch.from_numpy(b.level))
        o, lse = P.hdt_cross_attn_fwd(lv, cu, cq, mask, q, k, v)
        g = P.hdt_cross_attn_bwd(lv, cu, cq, mask, q, k, v, o, lse, do)
        torch.cuda.synchronize()
        P.hdt_device_status()
        o_r, lse_r = cross_oracle.forward(b.level, b.cu_seqlens, mask, cu_q, tq["q"], t["k"], t["v"])
        g_r = cross_oracle.backward(b.level, b.cu_seqlens, mask, cu_q, tq["q"], t["k"], t["v"], tq["do"])
        check_close(host(o), o_r, "bf16", "O", out_rounding=True)
        check_close(lse.cpu().numpy(), lse_r, "bf16", "LSE")
        for x, r, what in zip(g, g_r, ("dQ", "dK", "dV")):
            check_close(host(x), r, "bf16", what, out_rounding=True, row_rel=2.0 ** -8)


@pytest.mark.parametrize("rows", [[0] * 9 + [57] + [0] * 5 + [1], [17] + [0] * 8, [1] * 12 + [33, 0, 18, 1] + [0] * 3, [16] * 2 + [0] * 10 + [20, 1]])
def test_cross_decode_uneven(rows):
    """Few decoder rows a document on average, most of them in one: its rows beyond those that one block walks."""
    import torch
    import paper_2407_08330_b200 as P
    assert sum(rows) <= 4 * len(rows)
    rng = np.random.default_rng(len(rows))
    b = gen.pack([gen.gen_fill(rng, int(k), (2, 6), (2, 8), (3, 20))[:2] for k in rng.integers(1, 700, len(rows))])
    H, d, T, Tq = 3, 64, b.total_tokens, sum(rows)
    cu_q = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    t = gen.make_tensors(3, T, H, d, "f32", names=("k", "v"))
    q = gen.make_tensors(4, Tq, H, d, "f32", names=("q",))["q"]
    level, _, cu = dev_struct(b)
    o, lse = P.hdt_cross_attn_fwd(level, cu, torch.from_numpy(cu_q).cuda(), 15, *(dev_tensor(x, "f32") for x in (q, t["k"], t["v"])))
    torch.cuda.synchronize()
    P.hdt_device_status()
    o_r, lse_r = cross_oracle.forward(b.level, b.cu_seqlens, 15, cu_q, q, t["k"], t["v"])
    check_close(host(o), o_r, "f32", "O")
    check_close(host(lse), lse_r, "f32", "LSE")


def test_cross_decode_many_documents():
    """A decoding step for more documents than a grid has rows: one token and one decoder row each, so O is V and the
    log-sum-exp the one score."""
    import torch
    import paper_2407_08330_b200 as P
    B, H, d = 65537, 2, 64
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v = (torch.randn(B, H, d, generator=g, device="cuda") for _ in range(3))
    cu = torch.arange(B + 1, dtype=torch.int32, device="cuda")
    o, lse = P.hdt_cross_attn_fwd(torch.zeros(B, dtype=torch.int8, device="cuda"), cu, cu, 1, q, k, v)
    torch.cuda.synchronize()
    P.hdt_device_status()
    check_close(host(o), host(v), "f32", "O")
    check_close(host(lse), host((q.double() * k.double()).sum(-1).T / d ** 0.5), "f32", "LSE")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("accumulate", [True, False])
@pytest.mark.parametrize("T,d_model", [(1, 8), (31, 1024), (33, 256), (9473, 64), (9999, 264)])
def test_hpe_stream(T, d_model, dtype, accumulate):
    import torch
    import paper_2407_08330_b200 as P
    rng = np.random.default_rng(T)
    n = max(1, T - T // 10)
    lv, pa = gen.gen_fill(rng, n, (4, 24), (3, 20), (5, 60))[:2]
    b = gen.pack([gen.fit(lv, pa, T, pad=True)])
    level, parent, cu = dev_struct(b)
    idx = P.hdt_build_index(level, parent, cu)
    x0 = gen.make_tensors(1, T, 1, d_model, dtype, names=("x",))["x"][:, 0]
    x = dev_tensor(x0, dtype)
    P.hdt_hpe(idx, level, parent, cu, d_model, x=x, accumulate=accumulate)
    torch.cuda.synchronize()
    P.hdt_device_status()
    want = hpe_oracle.hpe(b.level, b.parent, b.cu_seqlens, d_model, 3)
    if accumulate:
        want = want + x0
    check_close(host(x), want, dtype, "x", out_rounding=True)
