"""The paired-SM GEMM with tiles of 256 columns (tests/test_gpu_dense_pairs.py stays below the size
that gets them): a ragged last column tile and the f32 and bf16 epilogues through the FFN site,
against the CPU oracle; the width is asked of the kernel's own rule."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

import oracle.cast_oracle as O
from synthetic import generators as G
from tests.gpu_util import ATTN_REL_MAX, to_dev, to_host

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34144_gb300", "csrc")
CASES = [
    # F, grid, D, D_ff, anchors, r dtype, bias
    (4, (40, 33), 1032, 2056, (0, 1, 2, 3), "f32", True),     # one run of rows, 41.25 row tiles
    (6, (40, 33), 1032, 2056, (0, 2, 4, 5), "bf16", False),   # four runs of 10.3
]


@pytest.fixture(scope="module")
def columns(tmp_path_factory):
    """columns(rows of each run, N, K, pairs of SMs): what tile_columns gives the GEMM."""
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("dense")
    (d / "c.cpp").write_text('#include <cstdio>\n#include <cstdlib>\n#include "dense_plan.h"\n'
                             "int main(int, char** v) {\n  int a[4];\n  for (int i = 0; i < 4; ++i) a[i] = std::atoi(v[i + 1]);\n"
                             '  std::printf("%d", cast::tile_columns(a[0], a[1], a[2], a[3]));\n}\n')
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "c.cpp"), "-o", str(d / "c")], check=True, capture_output=True)

    def ask(runs, N, K, pairs):
        row_pairs = (sum(-(-r // 128) for r in runs) + 1) // 2
        out = subprocess.run([str(d / "c"), *map(str, (row_pairs, N, -(-K // 64), pairs))], check=True, capture_output=True)
        return int(out.stdout)
    return ask


def _widths(columns, case, pairs):
    F, grid, D, Dff, anchors, _, _ = case
    S, n = grid[0] * grid[1], len(anchors)
    one = all(b == a + 1 for a, b in zip(anchors, anchors[1:]))
    # the hidden activations of every anchor lie one after another: always one run
    return columns([n * S] if one else [S] * n, Dff, D, pairs), columns([n * S], D, Dff, pairs)


def test_rule_on_152_sms(columns):
    for case in CASES:
        assert _widths(columns, case, 76) == (256, 256)
    # a Matrix-Game-shaped FFN site, and one that 256 columns would leave without work for every SM
    assert columns([1560] * 4, 6144, 1536, 76) == 256
    assert columns([1320 * 4], 2056, 264, 76) == 128


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[5]}_{len(c[4])}of{c[0]}")
def test_ffn_in_256_columns(lib, columns, case):
    F, grid, D, Dff, anchors, rdt, bias = case
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    assert _widths(columns, case, pairs) == (256, 256)
    S = grid[0] * grid[1]
    parts = np.random.SeedSequence(190 + F).spawn(5)
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
