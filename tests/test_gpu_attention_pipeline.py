"""Edges of the attention kernel's K/V pipeline: one, two and three K/V tiles with one and two
query tiles (the S buffer's hand-over, the last PV), both head dims, and units split along K/V
(the parts' merge), against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle.cast_oracle as O
from synthetic import generators as G
from tests.gpu_util import ATTN_REL_MAX, to_dev, to_host

pytestmark = pytest.mark.gpu

CASES = [
    # N, S, H, M, Bv, K, anchors
    (1, 100, 2, 0, 1, 0, (0,)),        # one K/V tile, one query tile
    (1, 129, 1, 0, 1, 0, (0,)),        # two K/V tiles, the second holds one key; two query tiles
    (1, 256, 1, 2, 1, 1, (0,)),        # a history block of one token
    (2, 130, 1, 3, 40, 2, (1,)),       # five K/V tiles, three of them ragged
    (4, 300, 1, 4, 300, 4, (0, 3)),    # units split along K/V, a pair and a single query tile
]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"N{c[0]}S{c[1]}Bv{c[4]}K{c[5]}")
def test_attention_pipeline_edges(lib, case, d):
    N, S, H, M, Bv, K, anchors = case
    parts = np.random.SeedSequence(50 + S + d).spawn(5)
    q, kc, vc = (G.round_bf16(G.tokens_with_offsets(p, N, S, H, d, 0.5)) for p in parts[:3])
    kh, vh = (G.round_bf16(G.tokens_with_offsets(p, max(M, 1), Bv, H, d, 0.5)) for p in parts[3:])
    rng = np.random.default_rng(S)
    idx = np.stack([[rng.permutation(M)[:K] for _ in range(H)] for _ in anchors]).astype(np.int32) if M else None
    dev = (lambda x: to_dev(x, "bf16"))
    o, lse = lib.cast_anchor_attention(dev(q), dev(kc), dev(vc), list(anchors), dev(kh) if M else None,
                                       dev(vh) if M else None, torch.from_numpy(idx).cuda() if M else None,
                                       out_dtype=torch.float32, want_lse=True)
    lib.cast_check_device()
    ref, lse_ref = O.routed_attention(q, kc, vc, kh, vh, list(anchors), idx, with_lse=True)
    ref = ref.reshape(len(anchors), S, H * d)
    assert np.max(np.abs(to_host(o) - ref)) / np.max(np.abs(ref)) <= ATTN_REL_MAX
    np.testing.assert_allclose(to_host(lse), lse_ref, atol=2e-2)
