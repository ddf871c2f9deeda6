"""Positional encoding at the row widths where the streaming kernel's tile size changes (fp32 rows of which three tiles
of 32 tokens, or two, no longer fit in shared memory), with a ragged last tile."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_model", [536, 544, 640, 824, 832, 1024])
def test_hpe_wide_rows(d_model):
    import paper_2407_08330_b200 as P
    from test_gpu_hpe import run
    b = gen.pack([gen.gen_fill(np.random.default_rng(d_model), n, (4, 24), (3, 20), (5, 60)) for n in (9001, 1203)])
    run(P, b, d_model, 3, torch.float32, max_stages=4)
