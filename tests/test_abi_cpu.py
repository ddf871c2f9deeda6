"""CPU-side checks of the C-ABI library: it loads and exports every function the header declares
(no compute calls here), workspace sizing is host arithmetic, and the oracle and the CUDA sources
are independent of each other."""
import os
import re

import paper_2407_08330_b200 as P
from paper_2407_08330_b200 import binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_exports_every_declared_symbol():
    declared, missing = P.exported_symbols()
    assert {"hdt_build_index", "hdt_attn_fwd", "hdt_attn_bwd"} <= set(declared)
    assert missing == []


def test_workspace_bytes_host_arithmetic():
    assert P.hdt_index_workspace_bytes(4, 32768) > 0
    assert P.hdt_index_workspace_bytes(4, 32768, block_m=256) == 0      # invalid block_m
    assert P.hdt_index_workspace_bytes(-1, 10) == 0
    a = P.hdt_index_workspace_bytes(4, 1000)
    b = P.hdt_index_workspace_bytes(4, 2000)
    assert b > a


def test_oracle_and_cuda_path_share_nothing():
    for dirpath, _, files in os.walk(os.path.join(ROOT, "paper_2407_08330_b200")):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                txt = open(os.path.join(dirpath, f)).read()
                assert not re.search(r"^\s*(from|import)\s+oracle\b", txt, re.M), f
                assert "hdt_oracle" not in txt, f
    for f in os.listdir(os.path.join(ROOT, "oracle")):
        if f.endswith((".py", ".c")):
            txt = open(os.path.join(ROOT, "oracle", f)).read()
            assert "paper_2407_08330_b200" not in txt and "libhdt.so" not in txt, f


def test_cross_workspace_holds_either_path():
    """A bf16 call runs on 128-row blocks or, with option force_simt, on 32-row blocks, whose records take more room."""
    import torch
    al = lambda n: (n + 255) // 256 * 256
    for B, T, Tq, H in ((1, 1 << 20, 1, 1), (3, 50000, 7, 1), (1, 100, 4000, 2), (70, 9000, 0, 1)):
        blocks = Tq // 32 + T // 32 + 2 * (B + 1)
        for bwd in (0, 1):
            need = al(20 * blocks) + 12 * (T + Tq) + 4 * blocks + (4 * H * Tq if bwd else 0)
            assert P.hdt_cross_workspace_bytes(B, T, Tq, H, 64, torch.bfloat16, bwd) >= need, (B, T, Tq, H, bwd)
