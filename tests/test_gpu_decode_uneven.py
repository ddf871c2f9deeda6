"""Decoding on documents of different lengths (forward of the cross-attention with few decoder rows a document): pieces dealt by
length, at the lengths where a document gets one more, with documents without tokens or rows, fewer and more documents than
a warp sees at once, documents of more than eight rows; against the oracle."""
import numpy as np
import pytest
import torch

from oracle import cross_oracle as co
from gpu_util import check_close, dev_tensor, host

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 31, 32, 33, 63, 64, 65, 95, 96, 0]
CASES = {      # tokens and decoder rows of each document, level mask, heads, head_dim
    "edges": (EDGES, [1] * 11, 15, 3, 64),
    "edges_some_rows": (EDGES, [0, 1, 2, 8, 1, 0, 3, 0, 2, 1, 1], 6, 2, 128),
    "one_long": ([4000] + [40] * 30, [1] * 31, 15, 12, 64),
    "long_last": ([70] * 31 + [9000], [1] * 32, 15, 12, 64),            # pieces of more than 32 tokens
    "many": ([300, 0, 5] * 20 + [2000] + [33] * 40, [1, 2, 0] * 20 + [30] + [1] * 40, 15, 4, 64),
    "rows_on_one": ([900] + [10] * 9, [20] + [1] * 9, 15, 2, 64),       # a document of more than eight rows
    "rows_on_some": ([100, 300, 50, 7, 900, 40] + [20] * 8, [3, 9, 11, 8, 9, 2] + [1] * 8, 15, 2, 128),      # two of them in eight rows of all
    "rows_on_many": ([64, 200, 5, 31] * 10, [9, 0, 1, 5] * 10, 15, 12, 64),
    "few_parts": ([120, 250, 500, 1000], [2, 1, 8, 1], 15, 20, 64),     # a warp and a CTA of the merge a head
    "many_rows": ([3] * 350 + [5000] + [40] * 350, [1] * 701, 15, 3, 64),      # several heads to a CTA of the merge
    "no_pieces": ([20], [1], 15, 2, 64),
    "long_pieces": ([700, 1, 40000], [1, 1, 1], 15, 33, 128),           # two groups of heads
}


def _inputs(lengths, rows, H, d, dtype, seed=3):
    rng = np.random.default_rng(seed)
    cu = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    cq = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    level = rng.integers(0, 4, cu[-1]).astype(np.int8)
    x = [torch.from_numpy(rng.standard_normal((n, H, d)).astype(np.float32)) for n in (cq[-1], cu[-1], cu[-1])]
    x = [(y.bfloat16().float() if dtype == "bf16" else y).numpy() for y in x]
    return level, cu, cq, x


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_decode_uneven(name, dtype):
    import paper_2407_08330_b200 as P
    lengths, rows, mask, H, d = CASES[name]
    level, cu, cq, x = _inputs(lengths, rows, H, d, dtype)
    assert cq[-1] <= 4 * len(lengths)          # (more rows: the tile kernels)
    lv, cuk, cuq = (torch.from_numpy(a).cuda() for a in (level, cu, cq))
    q, k, v = (dev_tensor(a, dtype) for a in x)
    o, lse = torch.full_like(q, float("nan")), torch.full((H, q.shape[0]), float("nan"), device="cuda")
    P.hdt_cross_attn_fwd(lv, cuk, cuq, mask, q, k, v, out=o, lse=lse)
    P.hdt_device_status()
    o_r, lse_r = co.forward(level, cu, mask, cq, *x)
    check_close(host(o), o_r, dtype, "O")
    check_close(host(lse), lse_r, "f32" if dtype == "f32" else "bf16", "LSE")


def test_one_long_document_costs_what_its_tokens_cost():
    """A long document among short ones is shared by as many CTAs as its tokens are of the batch's: the call takes about what
    an even batch of as many tokens takes (1.0 to 1.5 times, measured on several batches; ten times where every document has
    an equal share of the CTAs)."""
    import paper_2407_08330_b200 as P
    H, d = 12, 64

    def time(lengths):
        level, cu, cq, x = _inputs(lengths, [1] * len(lengths), H, d, "bf16")
        lv, cuk, cuq = (torch.from_numpy(a).cuda() for a in (level, cu, cq))
        q, k, v = (dev_tensor(a, "bf16") for a in x)
        o, lse = torch.empty_like(q), torch.empty((H, q.shape[0]), device="cuda")
        ws = torch.empty(P.hdt_cross_workspace_bytes(len(lengths), len(level), len(lengths), H, d, torch.bfloat16, 0), dtype=torch.uint8, device="cuda")
        us = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(50):
                P.hdt_cross_attn_fwd(lv, cuk, cuq, 15, q, k, v, out=o, lse=lse, workspace=ws)
            b.record()
            b.synchronize()
            us.append(a.elapsed_time(b) * 20)
        return sorted(us)[4]
    assert time([8192] + [256] * 63) < 3 * time([380] * 64)
