"""Channel weights far from one: the reconstruction does not depend on a common factor of the weights
(with eps = eta_abs = 0), as long as the pooled spectra themselves stay within the range of a float."""
import numpy as np
import pytest

from synthetic import generators as G
from tests.gpu_util import par_check
from tests.test_gpu_par import _run

pytestmark = pytest.mark.gpu


# the products of two spectra are about 64 here: w |F_a| |F_b| of 3e19 and 1e-20, whose squares a
# float does not hold; pooled over the channels and normalised both are in range
@pytest.mark.parametrize("C,factor", [(8, 2.0 ** 59), (4096, 2.0 ** -72)])
@pytest.mark.parametrize("tile", [(8, 8), (6, 5)])
def test_common_factor_of_the_weights(lib, C, factor, tile):
    rng = np.random.default_rng(C)
    h, w = tile
    R = np.zeros((4, h, w, C), np.float32)
    R[0] = rng.standard_normal((h, w, C))
    R[3] = np.roll(R[0], (1, 2), (0, 1)) + 0.2 * rng.standard_normal((h, w, C))   # moved within the tile
    R = G.round_bf16(R)
    wch = rng.uniform(0.5, 1.0, C).astype(np.float32)
    kw = dict(tile=tile, eps=0.0, eta_abs=0.0)
    want = _run(lib, R, [1, 0, 0, 1], "bf16", wch, **kw)
    got = _run(lib, R, [1, 0, 0, 1], "bf16", wch * np.float32(factor), **kw)
    still = _run(lib, R, [1, 0, 0, 1], "bf16", wch, gate="zero", **kw)
    assert np.abs(want[1] - still[1]).max() > 0.1      # the phases matter in this field
    par_check(got, want, [1, 2], "bf16")
