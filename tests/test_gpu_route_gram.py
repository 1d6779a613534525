"""Gram matrices that do not start on a 16-byte boundary (views into a packed buffer): the same
scores and blocks, bit for bit, as from an aligned copy."""
import numpy as np
import pytest
import torch

from tests.gpu_util import to_dev
from tests.test_gpu_route import _inputs

pytestmark = pytest.mark.gpu


def _gram_at(offset, H, d):
    """f32 [H, d, d] Gram matrices that start `offset` floats behind a 16-byte boundary."""
    P = np.random.default_rng(7).standard_normal((H, d, d)) / np.sqrt(d)
    g = torch.from_numpy(np.einsum("hod,hoe->hde", P, P).astype(np.float32)).cuda()
    view = torch.zeros(g.numel() + 8, device="cuda")[offset:offset + g.numel()].view_as(g)
    view.copy_(g)
    assert view.data_ptr() % 16 == 4 * offset % 16
    return view


# one CTA per head with 9 and 130 (anchor, block) pairs (below and across the 64 of a round), and
# the clustered kernel with an uneven last CTA
@pytest.mark.parametrize("d,M,anchors", [(64, 9, [1]), (128, 65, [0, 1]), (128, 700, [0, 1]), (64, 1030, [0, 1])])
def test_scores_of_an_unaligned_gram(lib, d, M, anchors):
    H, K = 3, 5
    q, k, v = (to_dev(x, "bf16") for x in _inputs(60 + M, 2, 40, H, d, M, 6, "bf16"))
    want_idx, want_u = lib.cast_route_topk(q, anchors, k, v, K, gram=_gram_at(0, H, d), want_u=True)
    for offset in (1, 2, 3):
        idx, u = lib.cast_route_topk(q, anchors, k, v, K, gram=_gram_at(offset, H, d), want_u=True)
        assert torch.equal(u, want_u) and torch.equal(idx, want_idx)
    lib.cast_check_device()


def test_block_step_with_an_unaligned_gram(lib):
    N, H, d, M, K, grid = 4, 2, 128, 12, 3, (5, 8)
    q, k, v = (to_dev(x, "bf16") for x in _inputs(70, N, grid[0] * grid[1], H, d, M, 24, "bf16"))
    got = []
    for offset in (0, 1):
        r = torch.zeros((N, grid[0] * grid[1], H * d), device="cuda")
        idx = torch.full((2, H, K), -1, dtype=torch.int32, device="cuda")
        lib.cast_block_step(q, q.clone(), q.clone(), [0, 3], k, v, K, grid, r, idx_out=idx, gram=_gram_at(offset, H, d))
        got.append((r, idx))
    torch.cuda.synchronize()
    lib.cast_check_device()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
