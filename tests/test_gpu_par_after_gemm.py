"""bf16 PAR on the stream directly behind a library GEMM that writes the anchors it reads (the
statistics start while the kernel before them ends)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [(16, 16), (30, 52)])
def test_par_behind_a_gemm(lib, rows):
    F, C, K, mask = 4, 256, 512, [1, 0, 0, 1]
    Hg, Wg = rows
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    w = (torch.randn((K, C), generator=g, device="cuda") / K ** 0.5).to(torch.bfloat16)
    xs = [torch.randn((F * Hg * Wg, K), generator=g, device="cuda").to(torch.bfloat16) for _ in range(6)]
    r = torch.empty((F, Hg, Wg, C), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(lib.par_workspace_size(r, mask), dtype=torch.uint8, device="cuda")
    want = []
    for x in xs:
        torch.mm(x, w, out=r.view(-1, C))
        torch.cuda.synchronize()
        want.append(lib.cast_par_reconstruct(r, mask, workspace=ws).clone())
    torch.cuda.synchronize()
    got = [torch.empty_like(r) for _ in xs]
    for x, o in zip(xs, got):
        torch.mm(x, w, out=r.view(-1, C))
        lib.cast_par_reconstruct(r, mask, workspace=ws)
        o.copy_(r)
    torch.cuda.synchronize()
    lib.cast_check_device()
    for o, t in zip(got, want):
        assert torch.equal(o, t)
