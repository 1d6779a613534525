"""bf16 PAR where a CTA of the statistics goes through full, right-edge, corner and bottom-edge tiles
and every unit is a single channel chunk, so that only one of its two issuers takes part in a unit."""
import numpy as np
import pytest

import oracle.cast_oracle as O
from synthetic import generators as G
from synthetic import workloads as W
from tests.gpu_util import par_check
from tests.test_gpu_par import _ambiguous_tiles, _oracle, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,tile", [(64, (8, 8)), (128, (8, 8)), (8, (5, 6))])
def test_single_chunk_units_across_tile_shapes(lib, C, tile):
    F, Hg, Wg = 65, 12, 84
    anchors = tuple(range(0, F, 2))
    R, _ = G.grf_sequence(np.random.SeedSequence([C, tile[0]]), F, Hg, Wg, C, ell=3.0)
    R += 0.1 * np.random.default_rng(1).standard_normal(R.shape).astype(np.float32)
    mask = W.anchor_mask(F, anchors)
    got = _run(lib, R, mask, "bf16", None, tile=tile)
    ref, info, _ = _oracle(R, mask, "bf16", None, tile=tile)
    assert not _ambiguous_tiles(info, O.tiles_of(Hg, Wg, *tile))
    par_check(got, ref, [t for t in range(F) if not mask[t]], "bf16")
