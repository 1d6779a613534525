"""PAR's workspace by residual type (no GPU needed): bf16 keeps theta and g on the SM."""
import ctypes as C

import pytest

from tests.test_abi import _fake, _par, lib  # noqa: F401


@pytest.mark.parametrize("ch", [64, 512, 3072])
def test_bf16_workspace_size(lib, ch):  # noqa: F811
    so = lib.library()
    want = (4 * 2 * -(-ch // 128) * 120 * 4 + 255) // 256 * 256      # 4 tiles, 2 anchors
    a = _par(lib, [1, 0, 1], C=ch, dtype=lib.BF16)
    assert so.cast_par_workspace_size(C.byref(a)) == want
    assert so.cast_par_reconstruct(C.byref(a), _fake(0x100000), want - 1, None) == 1
    assert so.cast_par_workspace_size(C.byref(_par(lib, [1, 0, 1], C=ch))) > want    # f32
