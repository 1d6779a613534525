"""bf16 PAR with tile sides other than 8: complete tiles (one box each way), the truncated last column
(row by row), fewer columns than a tile has, the last rows of a tile that are not four, and a NaN
that stays inside its tile on every side."""
import numpy as np
import pytest

import oracle.cast_oracle as O
from synthetic import generators as G
from synthetic import workloads as W
from tests.gpu_util import par_check
from tests.test_gpu_par import _ambiguous_tiles, _oracle, _run

pytestmark = pytest.mark.gpu

CASES = [
    # grid, tile, C
    ((12, 20), (4, 4), 72),     # complete tiles only, one group of four rows each
    ((13, 21), (4, 4), 136),    # ... and truncated both ways
    ((16, 14), (8, 7), 64),     # two groups of four rows, complete columns
    ((11, 15), (7, 7), 200),    # four rows and three
    ((9, 24), (3, 8), 64),      # eight columns, rows by ones
    ((10, 17), (5, 8), 72),     # ... truncated
    ((9, 5), (6, 7), 72),       # no complete column
    ((5, 9), (1, 1), 64),       # single tokens
    ((8, 6), (8, 1), 64),       # columns
    ((7, 16), (1, 8), 64),      # rows
]


@pytest.mark.parametrize("grid,tile,C", CASES)
def test_tile_sides(lib, grid, tile, C):
    F, (Hg, Wg) = 6, grid
    mask = W.anchor_mask(F, (0, 3, 5))
    R, _ = G.grf_sequence(np.random.SeedSequence([Hg, Wg, C]), F, Hg, Wg, C, ell=3.0)
    R += 0.1 * np.random.default_rng(1).standard_normal(R.shape).astype(np.float32)
    got = _run(lib, R, mask, "bf16", None, tile=tile)
    ref, info, _ = _oracle(R, mask, "bf16", None, tile=tile)
    assert not _ambiguous_tiles(info, O.tiles_of(Hg, Wg, *tile))
    par_check(got, ref, [1, 2, 4], "bf16")
    for a in (0, 3, 5):
        assert np.array_equal(got[a], G.round_bf16(R[a]).astype(np.float64))


@pytest.mark.parametrize("tile", [(4, 4), (7, 5), (3, 8), (8, 6)])
def test_nan_stays_in_its_tile(lib, tile):
    F, Hg, Wg, C = 3, 17, 19, 72
    R, _ = G.grf_sequence(np.random.SeedSequence(5), F, Hg, Wg, C, ell=3.0)
    clean = _run(lib, R, [1, 0, 1], "bf16", None, tile=tile)
    for y, x in ((9, 7), (9, 18), (16, 3), (0, 0)):
        S = R.copy()
        S[2, y, x, 3] = np.nan
        got = _run(lib, S, [1, 0, 1], "bf16", None, tile=tile)
        y0, x0 = y // tile[0] * tile[0], x // tile[1] * tile[1]
        inside = np.zeros((Hg, Wg), bool)
        inside[y0:y0 + tile[0], x0:x0 + tile[1]] = True
        assert np.isnan(got[1][inside][:, 3]).all()
        assert np.array_equal(got[1][~inside], clean[1][~inside])
