"""Where a Gram tensor may start: validated on the host before any launch (no GPU needed)."""
import ctypes as C

import pytest

from tests.test_abi import _block, _fake, _route, lib  # noqa: F401


@pytest.mark.parametrize("addr,mode,ok", [(0x50000, 0, True), (0x50004, 0, True), (0x50008, 0, True), (0x50002, 0, False),
                                          (0x50002, 1, True)])     # by similarity: never read
def test_gram_alignment_validation(lib, addr, mode, ok):  # noqa: F811
    """Any float boundary is taken (the call only fails later, for the missing workspace)."""
    so = lib.library()
    assert so.cast_route_topk(C.byref(_route(lib, gram=_fake(addr), mode=mode)), None, 0, None) == 1
    assert (b"workspace" if ok else b"gram") in so.cast_last_error_detail()
    assert so.cast_block_step(C.byref(_block(lib, gram=_fake(addr), route_mode=mode)), None, 0, None) == 1
    assert (b"workspace" if ok else b"gram") in so.cast_last_error_detail()
