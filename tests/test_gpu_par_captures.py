"""More open captures of f32 PAR (full and truncated tiles) than there are side streams: the calls that
find none run both tile kinds on their own stream, and every graph gives a lone call's result."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu

F, HG, WG, CH, MASK = 3, 12, 13, 40, [1, 0, 1]
RELAXED = 2


def _runtime():
    for name in (f"libcudart.so.{torch.version.cuda.split('.')[0]}", "libcudart.so"):
        try:
            return C.CDLL(name)
        except OSError:
            pass
    pytest.skip("no shared CUDA runtime")


def test_more_captures_than_side_streams(lib):
    rt = _runtime()
    n = 18
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    src = [torch.randn((F, HG, WG, CH), generator=g, device="cuda") for _ in range(n)]
    want = [lib.cast_par_reconstruct(x.clone(), MASK) for x in src]
    got = [x.clone() for x in src]
    ws = [torch.empty(lib.par_workspace_size(src[0], MASK), dtype=torch.uint8, device="cuda") for _ in range(n)]
    streams = [torch.cuda.Stream() for _ in range(n)]
    torch.cuda.synchronize()
    graphs = [C.c_void_p() for _ in range(n)]
    for s in streams:
        assert rt.cudaStreamBeginCapture(C.c_void_p(s.cuda_stream), RELAXED) == 0
    try:
        for r, w, s in zip(got, ws, streams):
            lib.cast_par_reconstruct(r, MASK, workspace=w, stream=s)
    finally:
        ended = [rt.cudaStreamEndCapture(C.c_void_p(s.cuda_stream), C.byref(gr)) for s, gr in zip(streams, graphs)]
    assert ended == [0] * n
    for s, gr in zip(streams, graphs):
        ex = C.c_void_p()
        assert rt.cudaGraphInstantiate(C.byref(ex), gr, C.c_ulonglong(0)) == 0
        assert rt.cudaGraphLaunch(ex, C.c_void_p(s.cuda_stream)) == 0
    torch.cuda.synchronize()
    lib.cast_check_device()
    for r, t in zip(got, want):
        assert torch.equal(r, t)
    # with the captures closed the side streams are free again
    assert torch.equal(lib.cast_par_reconstruct(src[0].clone(), MASK), want[0])
