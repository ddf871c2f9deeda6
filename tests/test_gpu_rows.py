"""The row-wise kernels and the fp32 stage-0 kernels against the oracle, at the sizes where their splits
change: rows shared by several groups of lanes or not, ragged last rows and key chunks, families longer
than a piece of shared memory, one row, PAD, direction bits."""
import numpy as np
import pytest

import gen
import oracle
from tests.gpu_util import check_close, dev_struct, dev_tensor, host

pytestmark = pytest.mark.gpu


def _doc(*sections):
    return gen.layout([list(s) for s in sections])


def _trees(n, seed):
    rng = np.random.default_rng(seed)
    return [gen.layout_tree(gen.listops_tree(rng, 20, 5, 300, 0.45)) for _ in range(n)]


def _pad(seq, n):
    return gen.fit(seq[0], seq[1], n, pad=True)


CASES = {
    "root": (lambda: [(np.array([0], np.int8), np.array([-1], np.int32))], 3, 0),
    "few_rows": (lambda: [_doc([8, 8, 8], [8, 8, 8])], 1, 0),
    "chunk_edges": (lambda: [_doc([n for n in range(0, 20)], [1], [])], 2, 0),
    "long_upper": (lambda: [_doc([1] * 150, *[[2]] * 70)], 3, 0),
    "long_family": (lambda: [_doc([95, 96, 97, 47, 48, 49, 200], [130])], 2, 0),
    "pad": (lambda: [_pad(_doc([5, 30], [12]), 77), _pad(_doc([3]), 64)], 5, 0),
    "trees": (lambda: _trees(6, 1), 2, 24),
    "trees_many_rows": (lambda: _trees(40, 2), 16, 24),
}


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 128)])
@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("directions", [7, 4])
def test_rows(name, dtype, d, directions):
    import torch
    import paper_2407_08330_b200 as P
    make, H, stages = CASES[name]
    if name == "trees_many_rows" and (directions != 7 or d == 128):
        pytest.skip("one setting is enough for the many rows")
    b = gen.pack(make())
    t = gen.make_tensors(5, b.total_tokens, H, d, dtype)
    idx = P.hdt_build_index(*dev_struct(b), max_stages=stages, directions=directions)
    q, k, v, do = (dev_tensor(t[n], dtype) for n in ("q", "k", "v", "do"))
    o, lse = P.hdt_attn_fwd(idx, q, k, v)
    g = P.hdt_attn_bwd(idx, q, k, v, o, lse, do)
    torch.cuda.synchronize()
    P.hdt_device_status()
    o_r, lse_r = oracle.forward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"], directions=directions)
    g_r = oracle.backward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"], t["do"], directions=directions)
    check_close(host(o), o_r, dtype, "O", out_rounding=True)
    check_close(lse.cpu().numpy(), lse_r, dtype, "LSE")
    for x, r, what in zip(g, g_r, ("dQ", "dK", "dV")):
        check_close(host(x), r, dtype, what, out_rounding=True, row_rel=2.0 ** -8)


@pytest.mark.parametrize("length", [2000, 4000])
def test_f32_tile_kernels(length):
    """fp32 calls with more rows than the row-wise kernels take in a wave."""
    import torch
    import paper_2407_08330_b200 as P
    rng = np.random.default_rng(length)
    H, d = 12, 64
    b = gen.pack([gen.gen_fill(rng, length, (4, 24), (3, 20), (5, 60)), gen.gen_pseudo(rng, length // 2 + 1, (5, 150))])
    t = gen.make_tensors(6, b.total_tokens, H, d, "f32")
    idx = P.hdt_build_index(*dev_struct(b))
    q, k, v, do = (dev_tensor(t[n], "f32") for n in ("q", "k", "v", "do"))
    o, lse = P.hdt_attn_fwd(idx, q, k, v)
    g = P.hdt_attn_bwd(idx, q, k, v, o, lse, do)
    torch.cuda.synchronize()
    o_r, lse_r = oracle.forward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"])
    g_r = oracle.backward(b.level, b.parent, b.cu_seqlens, t["q"], t["k"], t["v"], t["do"])
    check_close(host(o), o_r, "f32", "O")
    check_close(lse.cpu().numpy(), lse_r, "f32", "LSE")
    for x, r, what in zip(g, g_r, ("dQ", "dK", "dV")):
        check_close(host(x), r, "f32", what)
