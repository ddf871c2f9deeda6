"""When a build may be relied on: a waiting build has read the structure arrays when it returns, so that another stream may
change them; every call on another stream than the build's waits for its end, of a deferred build too; a destroyed
index's workspace is free; several threads may make the first use of one index."""
import threading

import numpy as np
import pytest
import torch

import gen
from oracle import index_oracle as ix
from gpu_util import dev_struct, dev_tensor

pytestmark = pytest.mark.gpu


def many():
    """Sequences of several lengths, long ones among them: the kernels that finish the build run for a while."""
    rng = np.random.default_rng(5)
    return gen.pack([gen.gen_fill(rng, int(n), (2, 8), (2, 12), (5, 40))[:2] for n in rng.integers(1, 900, 300)] +
                    [gen.gen_fill(rng, 20000, (4, 24), (3, 20), (5, 60))[:2]])


def same(idx, want):
    for s, st in enumerate(want.stages):
        got = idx.export(s)
        for key in ("tok", "par", "rng", "up", "blocks", "queue"):
            assert np.array_equal(got[key], getattr(st, key)), (s, key)


@pytest.mark.parametrize("deferred", [False, True])
def test_other_stream_reads_the_index(deferred):
    import paper_2407_08330_b200 as P
    b = many()
    H, d = 2, 64
    t = gen.make_tensors(1, b.total_tokens, H, d, "bf16")
    q, k, v, do = (dev_tensor(t[n], "bf16") for n in ("q", "k", "v", "do"))
    st = dev_struct(b)
    idx = P.hdt_build_index(*st)
    o0, lse0 = P.hdt_attn_fwd(idx, q, k, v)
    g0 = P.hdt_attn_bwd(idx, q, k, v, o0, lse0, do)
    want = ix.build(b.level, b.parent, b.cu_seqlens)
    build, use = torch.cuda.Stream(), torch.cuda.Stream()
    ws = torch.zeros(P.hdt_index_workspace_bytes(b.batch, b.total_tokens), dtype=torch.uint8, device="cuda")
    ws_f = torch.empty(P.hdt_attn_workspace_bytes(idx, H, d, q.dtype, 0), dtype=torch.uint8, device="cuda")
    for _ in range(4):
        ws.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(build):
            idx = P.hdt_build_index(*st, workspace=ws, deferred=deferred)
        with torch.cuda.stream(use):
            o, lse = P.hdt_attn_fwd(idx, q, k, v, workspace=ws_f)
            g = P.hdt_attn_bwd(idx, q, k, v, o, lse, do)
            same(idx, want)
        torch.cuda.synchronize()
        assert torch.equal(o, o0) and torch.equal(lse, lse0)
        assert all(torch.equal(x, y) for x, y in zip(g, g0))
    P.hdt_device_status()


def test_structure_arrays_may_change_behind_the_wait():
    import paper_2407_08330_b200 as P
    b = many()
    want = ix.build(b.level, b.parent, b.cu_seqlens)
    build, use = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(4):
        st = dev_struct(b)
        torch.cuda.synchronize()
        with torch.cuda.stream(build):
            idx = P.hdt_build_index(*st)
        with torch.cuda.stream(use):
            for x in st:
                x.fill_(-1)
        torch.cuda.synchronize()
        same(idx, want)


def test_workspace_is_free_behind_destroy():
    """A build into a workspace that the build before it, on another stream, has just left."""
    import paper_2407_08330_b200 as P
    b = many()
    want = ix.build(b.level, b.parent, b.cu_seqlens)
    st = dev_struct(b)
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    ws = torch.empty(P.hdt_index_workspace_bytes(b.batch, b.total_tokens), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for _ in range(4):
        with torch.cuda.stream(first):
            P.hdt_build_index(*st, workspace=ws).close()
        with torch.cuda.stream(second):
            ws.zero_()
            idx = P.hdt_build_index(*st, workspace=ws)
            same(idx, want)
            idx.close()


@pytest.mark.parametrize("deferred", [False, True])
def test_nothing_to_build(deferred):
    import paper_2407_08330_b200 as P
    e = torch.zeros(0, dtype=torch.int8, device="cuda")
    idx = P.hdt_build_index(e, e.to(torch.int32), torch.zeros(1, dtype=torch.int32, device="cuda"), deferred=deferred)
    assert idx.nnz == 0 and idx.n_stages == 1
    idx.close()


def test_threads_share_an_index():
    import paper_2407_08330_b200 as P
    b = many()
    want = ix.build(b.level, b.parent, b.cu_seqlens)
    st = dev_struct(b)
    for _ in range(10):
        idx = P.hdt_build_index(*st, deferred=True)
        got, gate = [], threading.Barrier(4)

        def first_use():
            gate.wait()
            got.append(int(P.lib().hdt_attn_workspace_bytes(idx.handle, 2, 64, P.binding.HDT_BF16, 1)))
        ts = [threading.Thread(target=first_use) for _ in range(4)]
        for x in ts:
            x.start()
        for x in ts:
            x.join()
        assert len(set(got)) == 1 and got[0] > 0
    same(idx, want)


@pytest.mark.parametrize("own", [False, True])
def test_counted_index_under_capture(own):
    """A deferred index whose counts are on the host serves a graph captured on another stream, or on its own."""
    import paper_2407_08330_b200 as P
    b = gen.small_random_batch(210, n_seqs=4, max_len=500, K=(0, 40))
    H, d = 2, 64
    t = gen.make_tensors(1, b.total_tokens, H, d, "bf16")
    q, k, v = (dev_tensor(t[n], "bf16") for n in ("q", "k", "v"))
    st = dev_struct(b)
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    build, use = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(build):
        idx = P.hdt_build_index(*st, deferred=True)
        o0, lse0 = P.hdt_attn_fwd(idx, q, k, v, workspace=ws)
        o, lse = torch.zeros_like(o0), torch.zeros_like(lse0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=build if own else use):
        P.hdt_attn_fwd(idx, q, k, v, out=o, lse=lse, workspace=ws)
        assert idx.n_stages == 3 and idx.nnz > 0
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(o, o0) and torch.equal(lse, lse0)
    graph.reset()
