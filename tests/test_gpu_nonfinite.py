"""fp32 calls: an infinite row reaches the rows of its own family and nothing else.  The rows of a warp walk their keys in
step, so a row without keys where another has some (a [DOC] or [SEC] row, a row whose family lies in another piece of
shared memory, PAD) is handed keys of a family it does not belong to, at weight 0; 0 x inf would be NaN.  Every other row has to
be what it is without the infinite one, bit for bit."""
import numpy as np
import pytest
import torch

import gen
from gpu_util import dev_struct, dev_tensor

pytestmark = pytest.mark.gpu


def _batch():
    # families shorter and longer than a piece, sections of one sentence, anchors without children, PAD behind both documents
    seqs = [gen.layout([[7, 30, 12, 5], [1], [95, 96, 0, 200], []]), gen.layout([[20] * 9, [3, 60]])]
    return gen.pack([gen.fit(*s, len(s[0]) + n, pad=True) for s, n in zip(seqs, (37, 5))])


def _family(b, w):
    """Rows that attend to token w, which are the rows it attends to."""
    seq = np.repeat(np.arange(b.batch), np.diff(b.cu_seqlens))
    par = np.where(b.parent >= 0, b.parent + b.cu_seqlens[seq], -1)
    near = (par == w) | ((par == par[w]) & (par >= 0))
    near[w] = True
    if par[w] >= 0:
        near[par[w]] = True
    return near


@pytest.mark.parametrize("d,H", [(64, 64), (128, 32)])
@pytest.mark.parametrize("no_rows", [0, 1])      # the kernels with keys in shared memory; those that walk a whole block's span
def test_infinite_row_stays_in_its_family(d, H, no_rows):
    import paper_2407_08330_b200 as P
    b = _batch()
    T = b.total_tokens
    assert T * H * (d // 64) > 40000             # (fewer: all rows on the row-wise kernels, which end row by row)
    t = gen.make_tensors(7, T, H, d, "f32")
    x = {n: dev_tensor(t[n], "f32") for n in ("q", "k", "v", "do")}
    idx = P.hdt_build_index(*dev_struct(b))
    real = np.flatnonzero(b.level >= 0)
    tokens = np.unique(np.concatenate([real[:6], np.flatnonzero(b.level == 2)[::3], np.random.default_rng(1).choice(real, 10, replace=False)]))
    P.hdt_set_option("no_rows", no_rows)
    try:
        def run(y, o=None, lse=None):
            if o is None:
                return P.hdt_attn_fwd(idx, y["q"], y["k"], y["v"])
            return P.hdt_attn_bwd(idx, y["q"], y["k"], y["v"], o, lse, y["do"])

        o, lse = run(x)
        g = run(x, o, lse)
        for w in tokens:
            rest = torch.from_numpy(~_family(b, int(w))).cuda()
            for n in x:
                y = dict(x)
                y[n] = x[n].clone()
                y[n][int(w)] = float("inf")
                got = (run(y) if n != "do" else ()) + tuple(run(y, o, lse))
                for a, c, what in zip(got, ((o, lse) if n != "do" else ()) + tuple(g), ("O", "LSE", "dQ", "dK", "dV")[5 - len(got):]):
                    if what == "LSE":
                        a, c = a.T, c.T
                    assert torch.equal(a[rest], c[rest]), f"{n} of token {w}: {what}"
        # a PAD row's own values are multiplied by nothing at all
        pad = torch.from_numpy(b.level < 0).cuda()
        y = {n: v.clone() for n, v in x.items()}
        for v in y.values():
            v[pad] = float("inf")
        for a, c in zip(tuple(run(y)) + tuple(run(y, o, lse)), (o, lse) + tuple(g)):
            assert torch.equal(a, c)
        assert all((a[pad] == 0).all() for a in (o,) + tuple(g)) and torch.isneginf(lse[:, pad]).all()
    finally:
        P.hdt_set_option("no_rows", 0)
    P.hdt_device_status()
