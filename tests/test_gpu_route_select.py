"""TopK and refinement of the clustered per-head kernel on both sides of the 1,024 blocks whose
keys its threads hold in registers, with candidate sets and with blocks of equal score."""
import numpy as np
import pytest
import torch

from tests.gpu_util import to_dev, to_host
from tests.test_gpu_refine import PAPER, check_refined
from tests.test_gpu_route import _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,equal", [(300, 60, 0), (480, 479, 3), (512, 100, 0), (513, 1, 0), (513, 513, 0),
                                       (1023, 300, 7), (1024, 205, 1024), (1025, 205, 5), (1025, 206, 0)])
@pytest.mark.parametrize("restricted", [False, True])
def test_wide_selection(lib, M, K, equal, restricted):
    """TopK: exactly the stable descending order of the returned scores, equal ones to the lower
    block (`equal` > 0: the blocks repeat with that period; M: all alike).  Refined masks: the
    oracle's on the same scores."""
    H, S, d, Bv, anchors, N = 4, 40, 128, 4, [0, 2, 5], 7
    q, k, v = _inputs(900 + M, N, S, H, d, M, Bv, "bf16")
    if equal:
        period = 1 if equal == M else equal
        k, v = k[np.arange(M) % period], v[np.arange(M) % period]
    cand = None
    if restricted:
        rng = np.random.default_rng(M + K)
        Mc = max(K, M // 2)
        cand = np.stack([[rng.permutation(M)[:Mc] for _ in range(H)] for _ in anchors]).astype(np.int32)
    kw = {} if cand is None else {"candidates": torch.from_numpy(cand).cuda()}
    dev = [to_dev(q, "bf16"), anchors, to_dev(k, "bf16"), to_dev(v, "bf16"), K]
    idx, u = lib.cast_route_topk(*dev, want_u=True, **kw)
    torch.cuda.synchronize()
    lib.cast_check_device()
    g, ug = idx.cpu().numpy(), to_host(u)
    for i in range(len(anchors)):
        for h in range(H):
            s = ug[i, h].astype(np.float64)
            if cand is not None:
                out = np.ones(M, bool)
                out[cand[i, h]] = False
                s[out] = -np.inf
            want = np.sort(np.argsort(-s, kind="stable")[:K])
            np.testing.assert_array_equal(g[i, h], want)
    if not equal and 1 < K < M:
        idx, u = lib.cast_route_topk(*dev, want_u=True, refine=PAPER, **kw)
        torch.cuda.synchronize()
        changed, amb = check_refined(idx.cpu().numpy(), to_host(u), anchors, N, K, PAPER, candidates=cand)
        assert amb < H
