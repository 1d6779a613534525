"""Concurrent callers of f32 PAR with full and truncated tiles: host threads on streams of their own
and a capture that is open while another thread calls, each with the results of a lone call."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

F, HG, WG, C, MASK = 5, 20, 21, 264, [1, 0, 1, 0, 1]


class _Caller:
    def __init__(self, lib, seed):
        self.lib, self.stream = lib, torch.cuda.Stream()
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        self.src = torch.randn((F, HG, WG, C), generator=g, device="cuda")
        self.r = torch.zeros_like(self.src)
        self.ws = torch.empty(lib.par_workspace_size(self.r, MASK), dtype=torch.uint8, device="cuda")
        self.error = None
        self.step()
        torch.cuda.synchronize()
        self.want = self.r.clone()

    def step(self):
        """New anchors, then their reconstruction, both on this caller's stream."""
        with torch.cuda.stream(self.stream):
            self.r.zero_()
            self.r.copy_(self.src)
            self.lib.cast_par_reconstruct(self.r, MASK, workspace=self.ws, stream=self.stream)

    def loop(self, n):
        try:
            for _ in range(n):
                self.step()
        except Exception as e:   # noqa: BLE001  (reported by the test)
            self.error = e


def _check(lib, callers):
    torch.cuda.synchronize()
    lib.cast_check_device()
    for c in callers:
        assert c.error is None, c.error
        assert torch.equal(c.r, c.want)


def test_threads_on_their_own_streams(lib):
    callers = [_Caller(lib, s) for s in range(4)]
    for _ in range(5):
        threads = [threading.Thread(target=c.loop, args=(20,)) for c in callers]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        _check(lib, callers)


def test_call_while_another_thread_captures(lib):
    a, b = _Caller(lib, 10), _Caller(lib, 11)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=a.stream, capture_error_mode="thread_local"):
        a.step()
        other = threading.Thread(target=b.loop, args=(2,))
        other.start()
        other.join()
    _check(lib, [b])
    for _ in range(2):
        a.r.zero_()
        torch.cuda.synchronize()
        graph.replay()
        _check(lib, [a])
