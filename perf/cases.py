"""The work a user of this library has it do, as a list of cases that can be timed.

A case is a dict of plain values.  Three kinds:

  attn   one batch of documents (or expression trees): hdt_build_index, then hdt_attn_fwd for every
         layer, then hdt_attn_bwd for every layer in reverse where gradients are wanted.  The index
         belongs to the batch and serves all layers, so a pass holds one build.
           plain = True : the calls of the README (waiting build, results and workspaces allocated
                          by the binding);
           plain = False: a training or serving loop that keeps its buffers (deferred build, outputs
                          and workspaces passed in).
  hpe    hdt_hpe on an index that the batch already has: the positional encoding at the encoder input.
  cross  hdt_cross_attn_fwd / _bwd: decoder rows attend to a subset of the encoder levels; one decoder
         row per document is a step of autoregressive decoding.

Hierarchies come from the generators of `gen` (documents with uniform sections, sentences and words,
padded, filled or packed; flat text in pseudo-sections; skewed documents; ListOps-shaped trees);
tensors are N(0,1), drawn on the device.
"""
import math

import numpy as np
import torch

import gen
import paper_2407_08330_b200 as P

# sections per document, sentences per section, words per sentence
SHORT = ((2, 8), (2, 12), (5, 40))
LONG = ((4, 24), (3, 20), (5, 60))


def _attn(docs, batch, length, heads, head_dim, dtype, backward, layers=1, plain=False, directions=7):
    return dict(kind="attn", docs=docs, batch=batch, length=length, heads=heads, head_dim=head_dim, dtype=dtype,
                backward=backward, layers=layers, plain=plain, directions=directions)


def _hpe(docs, batch, length, d_model, dtype, accumulate):
    return dict(kind="hpe", docs=docs, batch=batch, length=length, d_model=d_model, dtype=dtype, accumulate=accumulate)


def _cross(batch, length, rows, level_mask, heads, head_dim, dtype, backward, plain=False):
    return dict(kind="cross", docs="fill", batch=batch, length=length, rows=rows, level_mask=level_mask, heads=heads,
                head_dim=head_dim, dtype=dtype, backward=backward, plain=plain)


def listed():
    return [
        # configuration 1: the smallest call there is, an index and a forward pass over 57 tokens in fp32
        dict(name="tiny_57_f32_fwd", **_attn("tiny", 1, 57, 1, 64, "f32", False, plain=True)),
        # inference of a 12-layer encoder on one document of 4096 tokens (the paper's complexity table)
        dict(name="infer_1x4096_12layers", **_attn("fill", 1, 4096, 12, 64, "bf16", False, layers=12, plain=True)),
        # configuration 2: a padded batch, forward only
        dict(name="pad_8x2048_fwd", **_attn("pad", 8, 2048, 12, 64, "bf16", False)),
        # configuration 3: the training shape of the paper's single-layer protocol
        dict(name="train_4x8192", **_attn("fill", 4, 8192, 12, 64, "bf16", True)),
        # configuration 4: documents of very different lengths packed without padding, head_dim 128
        dict(name="varlen_16_d128", **_attn("varlen", 16, 16384, 16, 128, "bf16", True)),
        # configuration 5: long skewed documents, families far longer than a tile
        dict(name="skew_2x32768", **_attn("skew", 2, 32768, 12, 64, "bf16", True)),
        # fine-tuning on flat text in pseudo-sections, an odd length, two layers, the README's calls
        dict(name="pseudo_3x3001_2layers", **_attn("pseudo", 3, 3001, 12, 64, "bf16", True, layers=2, plain=True)),
        # configuration 7 with the directed mask of the ListOps experiment: deep trees, few children
        dict(name="trees_200_directed", **_attn("tree", 200, 512, 2, 64, "bf16", True, directions=6)),
        # training in fp32
        dict(name="train_f32_2x2048", **_attn("fill", 2, 2048, 12, 64, "f32", True)),
        # positional encoding added to the embeddings of configuration 3's batch
        dict(name="hpe_4x8192_d768", **_hpe("fill", 4, 8192, 768, "bf16", True)),
        # a training step of decoder cross-attention to [SEC] and [SENT] anchors, 256 decoder rows a document
        dict(name="cross_train_4x8192_r256", **_cross(4, 8192, 256, 6, 12, 64, "bf16", True)),
        # one step of autoregressive decoding over all encoder tokens
        dict(name="cross_decode_4x8192_r1", **_cross(4, 8192, 1, 15, 12, 64, "bf16", False, plain=True)),
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread evenly over its logarithm."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    what = rng.choice(["fill", "pad", "varlen", "pseudo", "skew", "tree", "f32", "infer", "hpe", "cross", "decode"])
    heads, d = rng.choice([(12, 64), (12, 64), (8, 64), (16, 128), (6, 128), (3, 64)])
    plain = rng.random() < 0.4
    if what in ("fill", "pad", "varlen", "pseudo"):
        length = _log(rng, 200, 16384)
        batch = _log(rng, 1, max(1, min(16, 131072 // length)))
        return _attn(what, batch, length, heads, d, "bf16", rng.random() < 0.75, rng.choice([1, 1, 2]) if batch * length <= 40000 else 1, plain)
    if what == "skew":
        return _attn(what, rng.randint(1, 2), _log(rng, 4000, 32768), 12, 64, "bf16", rng.random() < 0.75, 1, plain)
    if what == "tree":
        return _attn(what, _log(rng, 1, 200), 512, rng.choice([2, 4]), 64, "bf16", rng.random() < 0.75, 1, plain, rng.choice([7, 6, 4]))
    if what == "f32":
        length = _log(rng, 57, 4096)
        return _attn("fill", rng.randint(1, max(1, min(4, 4096 // length))), length, rng.choice([1, 4, 12]), rng.choice([64, 64, 128]), "f32", rng.random() < 0.6, 1, plain)
    if what == "infer":
        return _attn("fill", rng.randint(1, 2), _log(rng, 200, 4096), 12, 64, "bf16", False, rng.choice([6, 12]), plain)
    if what == "hpe":
        length = _log(rng, 200, 16384)
        return _hpe("fill", _log(rng, 1, max(1, min(8, 65536 // length))), length, rng.choice([256, 512, 768, 1024]),
                    rng.choice(["bf16", "bf16", "f32"]), rng.random() < 0.75)
    length = _log(rng, 300, 8192)
    batch = rng.randint(1, 8)
    if what == "cross":
        return _cross(batch, length, _log(rng, 16, 256), rng.choice([2, 6, 15]) if batch <= 4 else rng.choice([2, 6]), heads, d, "bf16", rng.random() < 0.75, plain)
    return _cross(batch, length, 1, rng.choice([2, 6, 15]), heads, d, "bf16", False, plain)


# ---- inputs -------------------------------------------------------------------------------------
def _structure(case, seed):
    rng = np.random.default_rng(seed)
    docs, n, L = case["docs"], case["batch"], case["length"]
    if docs == "tiny":
        return gen.pack([gen.layout([[8, 8, 8], [8, 8, 8]])])
    if docs == "pad":
        return gen.pack([gen.gen_pad(rng, L, *SHORT) for _ in range(n)])
    if docs == "fill":
        return gen.pack([gen.gen_fill(rng, L, *LONG) for _ in range(n)])
    if docs == "varlen":  # the lengths belong to the case, their order and the hierarchies to the seed
        lengths = np.random.default_rng(n + L).integers(max(1, L // 32), L + 1, n)
        return gen.pack([gen.gen_fill(rng, int(k), *LONG) for k in rng.permutation(lengths)])
    if docs == "pseudo":
        return gen.pack([gen.gen_pseudo(rng, L, LONG[2]) for _ in range(n)])
    if docs == "skew":
        return gen.pack([gen.gen_skew(rng, L) for _ in range(n)])
    if docs == "tree":    # the trees belong to the case (their sizes differ), their order to the seed
        pool = np.random.default_rng(n + L)
        trees = [gen.layout_tree(gen.listops_tree(pool, 20, 5, L, 0.45)) for _ in range(n)]
        return gen.pack([trees[i] for i in rng.permutation(n)])
    raise KeyError(docs)


DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def prepare(case, seed):
    b = _structure(case, seed)
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    dt = DTYPES[case["dtype"]]

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=dev, dtype=torch.float32).to(dt)

    level, parent, cu = (torch.from_numpy(x).to(dev) for x in (b.level, b.parent, b.cu_seqlens))
    s = dict(case=case, level=level, parent=parent, cu=cu)
    T = b.total_tokens
    if case["kind"] == "hpe":
        s["index"] = P.hdt_build_index(level, parent, cu)
        s["x"] = normal(T, case["d_model"])
        s["ws"] = torch.empty(max(256, P.hdt_hpe_workspace_bytes(s["index"], 3)), dtype=torch.uint8, device=dev)
        return s
    H, d = case["heads"], case["head_dim"]
    if case["kind"] == "cross":
        n, rows = case["batch"], case["rows"]
        s["cu_q"] = torch.arange(0, (n + 1) * rows, rows, dtype=torch.int32, device=dev)
        s["q"], s["do"] = normal(n * rows, H, d), normal(n * rows, H, d)
        s["k"], s["v"] = normal(T, H, d), normal(T, H, d)
        if not case["plain"]:
            s["o"], s["dq"], s["dk"], s["dv"] = (torch.empty_like(s[k]) for k in ("q", "q", "k", "v"))
            s["lse"] = torch.empty((H, n * rows), dtype=torch.float32, device=dev)
            s["ws"] = torch.empty(max(P.hdt_cross_workspace_bytes(n, T, n * rows, H, d, dt, w) for w in (0, 1)),
                                  dtype=torch.uint8, device=dev)
        return s
    s["stages"] = 24 if case["docs"] == "tree" else 0
    names = ("q", "k", "v", "do") if case["backward"] else ("q", "k", "v")
    s["layers"] = [{k: normal(T, H, d) for k in names} for _ in range(case["layers"])]
    if not case["plain"]:
        s["ws_index"] = torch.empty(P.hdt_index_workspace_bytes(b.batch, T, 0, s["stages"]), dtype=torch.uint8, device=dev)
        idx = P.hdt_build_index(level, parent, cu, max_stages=s["stages"], workspace=s["ws_index"], directions=case["directions"])
        for w in (0, 1) if case["backward"] else (0,):
            s["ws%d" % w] = torch.empty(max(256, P.hdt_attn_workspace_bytes(idx, H, d, dt, w)), dtype=torch.uint8, device=dev)
        for t in s["layers"]:
            t["o"], t["lse"] = torch.empty_like(t["q"]), torch.empty((H, T), dtype=torch.float32, device=dev)
            if case["backward"]:
                t["dq"], t["dk"], t["dv"] = (torch.empty_like(t["q"]) for _ in range(3))
    return s


# ---- one pass -----------------------------------------------------------------------------------
def _run_attn(s):
    c = s["case"]
    idx = P.hdt_build_index(s["level"], s["parent"], s["cu"], max_stages=s["stages"], workspace=s.get("ws_index"),
                            directions=c["directions"], deferred=not c["plain"])
    outs = []
    for t in s["layers"]:
        outs.append(P.hdt_attn_fwd(idx, t["q"], t["k"], t["v"], out=t.get("o"), lse=t.get("lse"), workspace=s.get("ws0")))
    if c["backward"]:
        for t, (o, lse) in zip(reversed(s["layers"]), reversed(outs[:c["layers"]])):
            outs.append(P.hdt_attn_bwd(idx, t["q"], t["k"], t["v"], o, lse, t["do"], dq=t.get("dq"), dk=t.get("dk"),
                                       dv=t.get("dv"), workspace=s.get("ws1")))
    return outs


def _run_cross(s):
    c = s["case"]
    a = (s["level"], s["cu"], s["cu_q"], c["level_mask"], s["q"], s["k"], s["v"])
    o, lse = P.hdt_cross_attn_fwd(*a, out=s.get("o"), lse=s.get("lse"), workspace=s.get("ws"))
    if not c["backward"]:
        return o, lse
    return (o, lse) + tuple(P.hdt_cross_attn_bwd(*a, o, lse, s["do"], dq=s.get("dq"), dk=s.get("dk"), dv=s.get("dv"), workspace=s.get("ws")))


def run(s):
    c = s["case"]
    if c["kind"] == "attn":
        return _run_attn(s)
    if c["kind"] == "cross":
        return _run_cross(s)
    return P.hdt_hpe(s["index"], s["level"], s["parent"], s["cu"], c["d_model"], n_levels=3, x=s["x"],
                     accumulate=c["accumulate"], workspace=s["ws"])


# ---- what a pass cannot do without ----------------------------------------------------------------
def _pairs(b, directions):
    """Unmasked (query, key) pairs of a batch: self, parent, siblings, children."""
    seq = np.repeat(np.arange(b.batch), np.diff(b.cu_seqlens))
    par = np.where(b.parent >= 0, b.parent + b.cu_seqlens[seq], -1)
    kids = np.bincount(par[par >= 0], minlength=b.total_tokens).astype(np.int64)
    edges = int(kids.sum())
    siblings = int((kids * (kids - 1)).sum())
    return int((b.level >= 0).sum()) + (edges if directions & 1 else 0) + (siblings if directions & 2 else 0) + (edges if directions & 4 else 0)


def work(case):
    """Counted on the hierarchy of seed 0: those of other seeds are of the same size within a few percent."""
    b = _structure(case, 0)
    T, real = b.total_tokens, int((b.level >= 0).sum())
    esz = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "hpe":
        d = case["d_model"]
        return {"bytes": T * (d * esz * (2 if case["accumulate"] else 1) + 5), "flops": real * d * 3}
    H, d = case["heads"], case["head_dim"]
    row = H * d * esz
    if case["kind"] == "cross":
        keys = int(sum(((b.level == l).sum() for l in range(4) if case["level_mask"] >> l & 1)))
        Tq = case["batch"] * case["rows"]
        pairs = keys * case["rows"]
        byt = 2 * Tq * row + 2 * keys * row + 4 * H * Tq + T
        if case["backward"]:
            byt += 4 * Tq * row + 2 * keys * row + 2 * T * row + 4 * H * Tq
        return {"bytes": byt, "flops": (14 if case["backward"] else 4) * d * pairs * H}
    byt = 3 * real * row + T * row + 4 * H * T
    if case["backward"]:
        byt += 5 * real * row + 3 * T * row + 4 * H * T
    pairs = _pairs(b, case["directions"])
    return {"bytes": case["layers"] * byt + 5 * T, "flops": case["layers"] * (14 if case["backward"] else 4) * d * pairs * H}


def tolerance(case):
    # bf16: rounding of P, dS and of the stored results; fp32: sums of a few hundred products
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 1e-5}
