"""Edges of the paired-SM GEMM through the FFN site: rows of consecutive anchors tiled as one run,
a pair whose second row tile is empty, row tiles that end inside an anchor, both tile widths, both
output types and no bias, against the CPU oracle (bound of the other GEMM tests)."""
import numpy as np
import pytest
import torch

import oracle.cast_oracle as O
from synthetic import generators as G
from tests.gpu_util import ATTN_REL_MAX, to_dev, to_host

pytestmark = pytest.mark.gpu

CASES = [
    # F, grid, D, D_ff, anchors, r dtype, bias
    (1, (5, 13), 72, 136, (0,), "bf16", True),            # one ragged row tile, its pair empty
    (4, (9, 19), 136, 712, (1, 2), "f32", True),          # consecutive anchors: one run of rows
    (5, (9, 19), 136, 712, (0, 2, 4), "bf16", False),     # three runs of two row tiles
    (4, (40, 33), 264, 2056, (0, 1, 2, 3), "bf16", True),  # 42 row tiles, 256-column tiles
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"F{c[0]}S{c[1][0] * c[1][1]}D{c[2]}_{c[5]}")
def test_ffn_anchor_rows(lib, case):
    F, grid, D, Dff, anchors, rdt, bias = case
    S = grid[0] * grid[1]
    parts = np.random.SeedSequence(90 + S + D).spawn(5)
    x = G.round_bf16(G.normal(parts[0], (F, S, D)))
    w1 = G.round_bf16(G.normal(parts[1], (Dff, D), D ** -0.5))
    w2 = G.round_bf16(G.normal(parts[2], (D, Dff), Dff ** -0.5))
    b1 = G.round_bf16(G.normal(parts[3], (Dff,), 0.1)) if bias else None
    b2 = G.round_bf16(G.normal(parts[4], (D,), 0.1)) if bias else None
    r_out = torch.full((F, S, D), 7.0, dtype=torch.float32 if rdt == "f32" else torch.bfloat16, device="cuda")
    lib.cast_ffn_step(to_dev(x, "bf16"), list(anchors), to_dev(w1, "bf16"), to_dev(b1, "bf16") if bias else None,
                      to_dev(w2, "bf16"), to_dev(b2, rdt) if bias else None, grid, r_out)
    lib.cast_check_device()
    zero = (np.zeros(Dff, np.float32), np.zeros(D, np.float32))
    ref = O.anchor_ffn(x, list(anchors), w1, b1 if bias else zero[0], w2, b2 if bias else zero[1])
    r = to_host(r_out)
    for i, a in enumerate(anchors):
        assert np.max(np.abs(r[a] - ref[i])) / np.max(np.abs(ref[i])) <= ATTN_REL_MAX
