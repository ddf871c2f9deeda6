"""Index build at the edges of what its kernels hold in shared memory, against the sequential definition."""
import numpy as np
import pytest

import gen
from tests.test_gpu_parity import assert_index_equal

pytestmark = pytest.mark.gpu


def _chain(n):
    """A path: every token the only child of the one before it, for at most 20 levels, repeated under the root."""
    lv, pa = [0], [-1]
    while len(lv) < n:
        p = 0
        for d in range(1, 20):
            if len(lv) == n:
                break
            pa.append(p)
            p = len(lv)
            lv.append(d)
    return np.array(lv, np.int8), np.array(pa, np.int32)


def _doc(n, seed=0, words=(5, 60)):
    return gen.gen_fill(np.random.default_rng(seed), n, (4, 24), (3, 20), words)[:2]


CASES = {
    # lengths around one CTA's and a cluster's slices, the 16-bit limit, and beyond it
    "one_769": lambda: [_doc(769)],
    "one_8191": lambda: [_doc(8191)],
    "one_32768": lambda: [_doc(32768)],
    "one_32769": lambda: [_doc(32769)],
    # a sequence far longer than the mean works in the workspace
    "uneven": lambda: [_doc(9000)] + [_doc(20 + i, i) for i in range(40)],
    # many sequences: offsets and ranks in several rounds
    "many_300": lambda: [_doc(10 + i % 37, i, (1, 6)) for i in range(300)],
    # many blocks: offsets from a scan, ranks from sorted runs, also where every block costs the same
    "many_1500": lambda: [_doc(i % 23, i, (1, 6)) if i % 23 else (np.zeros(0, np.int8), np.zeros(0, np.int32)) for i in range(1500)],
    "same_1300": lambda: [_doc(9, 1, (1, 3))] * 1300,
    "long_150000": lambda: [_doc(150000, 5)],
    "uneven_1200": lambda: [_chain(900)] + [_doc(3 + i % 50, i, (1, 6)) for i in range(1200)] + [_doc(3000, 8)],
    # upper stages too large for their arrays in shared memory, with and without the maps of all stages
    "deep_small": lambda: [_chain(600) for _ in range(3)],
    "deep_2000": lambda: [_chain(2000)],
    "deep_6000": lambda: [_chain(6000)],
    # one family longer than any block list, one-word sentences
    "short_sentences": lambda: [_doc(6000, 3, (0, 1))],
}


@pytest.mark.parametrize("block", [128, 3])
@pytest.mark.parametrize("name", sorted(CASES))
def test_index_edges(name, block):
    import paper_2407_08330_b200 as P
    assert_index_equal(P, gen.pack(CASES[name]()), block, max_stages=24, block_m_upper=block)


def test_error_in_a_large_batch():
    import torch
    import paper_2407_08330_b200 as P
    b = gen.pack([_doc(12, i, (1, 6)) for i in range(1500)])
    parent = b.parent.copy()
    parent[b.cu_seqlens[1234] + 5] = 9                     # a parent behind its token
    level, _, cu = (torch.from_numpy(x).cuda() for x in (b.level, b.parent, b.cu_seqlens))
    for deferred in (False, True):
        with pytest.raises(P.HdtError) as e:
            P.hdt_build_index(level, torch.from_numpy(parent).cuda(), cu, deferred=deferred).nnz
        assert e.value.code == -2
    P.hdt_device_status()
