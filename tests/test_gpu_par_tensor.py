"""bf16 PAR (transforms and blend on the tensor cores) at its edges: tile sides that are not powers
of two, truncated tiles in both directions, channel counts around the 64- and 128-channel boxes,
groups of one and two targets, channel weights, and a NaN that stays inside its own tile."""
import numpy as np
import pytest

import oracle.cast_oracle as O
from synthetic import generators as G
from synthetic import workloads as W
from tests.gpu_util import par_check
from tests.test_gpu_par import _ambiguous_tiles, _oracle, _run

pytestmark = pytest.mark.gpu

CASES = [
    # F, Hg, Wg, C, anchors, weights, extra
    (4, 8, 8, 8, (0, 3), False, {}),                          # one tile, one chunk of 8 channels
    (7, 15, 21, 72, (0, 6), True, {}),                        # h = 7, w = 5; five targets of one pair
    (6, 13, 11, 136, (1, 2, 5), False, {}),                   # a pair without targets; h = 5, w = 3
    (5, 17, 9, 392, (0, 2, 4), True, {"band_radius": 2.0}),          # h = 1, w = 1; four chunks, the last of 8
    (4, 14, 20, 64, (0, 3), False, {"tile": (7, 5)}),         # smaller tiles, loaded row by row
    (4, 11, 13, 200, (0, 2), True, {"tile": (3, 8)}),         # ... truncated in both directions
    (5, 9, 16, 128, (0, 4), False, {"tile": (8, 6)}),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[1]}x{c[2]}_C{c[3]}_{c[6]}")
def test_par_bf16_edges(lib, case):
    F, Hg, Wg, C, anchors, weights, extra = case
    R, _ = G.grf_sequence(np.random.SeedSequence([F, Hg, Wg, C]), F, Hg, Wg, C, ell=3.0)
    R += 0.1 * np.random.default_rng(1).standard_normal(R.shape).astype(np.float32)
    mask = W.anchor_mask(F, anchors)
    wch = np.random.default_rng(2).uniform(0, 1, C).astype(np.float32) if weights else None
    gpu = _run(lib, R, mask, "bf16", wch, **extra)
    ref, info, p = _oracle(R, mask, "bf16", wch, **extra)
    tiles = O.tiles_of(Hg, Wg, p.tile_h, p.tile_w)
    amb = _ambiguous_tiles(info, tiles)
    assert len(amb) <= max(1, len(tiles) // 100)
    par_check(gpu, ref, [t for t in range(F) if not mask[t]], "bf16", excluded_tiles=amb, th=p.tile_h, tw=p.tile_w)
    for a in anchors:
        assert np.array_equal(gpu[a], G.round_bf16(R[a]).astype(np.float64))


@pytest.mark.parametrize("tile", [(8, 8), (5, 6)])
def test_par_bf16_nan_stays_in_its_tile(lib, tile):
    F, Hg, Wg, C = 3, 16, 18, 72
    R, _ = G.grf_sequence(np.random.SeedSequence(5), F, Hg, Wg, C, ell=3.0)
    mask = [1, 0, 1]
    clean = _run(lib, R, mask, "bf16", None, tile=tile)
    R[2, 9, 7, 3] = np.nan
    got = _run(lib, R, mask, "bf16", None, tile=tile)
    y0, x0 = 9 // tile[0] * tile[0], 7 // tile[1] * tile[1]
    inside = np.zeros((Hg, Wg), bool)
    inside[y0:y0 + tile[0], x0:x0 + tile[1]] = True
    assert np.isnan(got[1][inside][:, 3]).all()
    assert np.array_equal(got[1][~inside], clean[1][~inside])
