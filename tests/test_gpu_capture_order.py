"""Forward calls behind an expansion inside a stream capture and around one: on the expansion's stream, on a stream that has joined
behind it, on a stream that joins it to its own work, and behind a replay.  The expansion's last kernel lets what follows it by a
programmatic edge start before its codes are written, so no such edge may leave it."""
import ctypes

import pytest
import torch

from paper_2311_15806_b200 import binding as B
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    H.ensure_built()


class Edge(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte), ("reserved", ctypes.c_ubyte * 5)]


def edges_of(graph):
    """[(from, to, type)] of a captured graph; type 0 is an ordinary edge, 1 a programmatic one."""
    rt = ctypes.CDLL("libcudart.so.12")
    handle, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert rt.cudaGraphGetEdges_v2(handle, None, None, None, ctypes.byref(n)) == 0
    fr, to, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (Edge * n.value)()
    assert rt.cudaGraphGetEdges_v2(handle, fr, to, data, ctypes.byref(n)) == 0
    return [(fr[i], to[i], data[i].type) for i in range(n.value)]


class Case:
    def __init__(self, T, K):
        self.T, self.O, self.I = T, 1024, 1024
        gen = torch.Generator(device="cuda")
        gen.manual_seed(T)
        # (one order: the expansion ends with the kernel that writes the codes, or with its tables)
        self.d = B.make_desc(self.O, self.I, 4, K, 8, 64, 1)
        lay = B.pipe_layout(self.d)
        self.blob, self.ws = B.alloc_bytes(lay.blob_bytes), B.alloc_bytes(lay.expand_ws_bytes)
        self.base = torch.empty(self.O, self.I, device="cuda").normal_(generator=gen) * 0.02
        self.W = self.base.clone()
        self.xq = torch.randint(-127, 128, (T, self.I), dtype=torch.int8, device="cuda", generator=gen)
        self.sx = torch.tensor([0.01], device="cuda")
        self.y = torch.zeros(T, self.O, device="cuda")
        self.other = torch.zeros(4096, device="cuda")
        self.expand(None)
        self.forward(None)
        torch.cuda.synchronize()

    def expand(self, s):
        B.pipe_expand_weights(self.d, self.W, self.blob, self.ws, s)

    def forward(self, s):
        B.pipe_expanded_linear(self.d, self.blob, self.xq, self.sx, self.y, None, None, s)

    def want(self, r):
        self.W.copy_(self.base * (1.0 + r))
        torch.cuda.synchronize()
        self.expand(None)
        torch.cuda.synchronize()
        self.forward(None)
        torch.cuda.synchronize()
        return self.y.clone()


@pytest.mark.parametrize("K", [1, 3])
@pytest.mark.parametrize("T", [1, 48, 200])
@pytest.mark.parametrize("form", ["same", "cross", "join"])
def test_no_forward_starts_on_an_expansions_release(form, T, K):
    c = Case(T, K)
    want = [c.want(r) for r in range(4)]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    launches = B.pipe_launch_count()
    with torch.cuda.graph(graph, stream=s1):
        if form == "same":
            c.expand(s1)
            c.forward(s1)
        elif form == "cross":
            c.expand(s1)
            s2.wait_stream(s1)
            c.forward(s2)
            s1.wait_stream(s2)
        else:
            s2.wait_stream(s1)
            c.expand(s2)
            c.other.add_(1)
            s1.wait_stream(s2)
            c.forward(s1)
    launches = B.pipe_launch_count() - launches
    edges = edges_of(graph)
    last = {to for _, to, _ in edges} - {fr for fr, _, _ in edges}
    assert len(last) == 1                                    # the forward's kernel
    into = [(fr, kind) for fr, to, kind in edges if to in last]
    # what the expansion queued: the nodes from which the forward is reached without c.other's kernel, which has no edge into it
    before = {to for _, to, _ in edges}
    for fr, kind in into:
        if fr in before:
            assert kind == 0, "a programmatic edge leaves the expansion"
    assert launches >= 2
    graph.instantiate()
    for r in (1, 2, 3, 0, 2):
        c.W.copy_(c.base * (1.0 + r))
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(c.y.view(torch.int32), want[r].view(torch.int32))


@pytest.mark.parametrize("T", [1, 48, 200])
def test_a_forward_behind_a_replayed_expansion(T):
    c = Case(T, 3)
    want = [c.want(r) for r in range(4)]
    graph = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        with torch.cuda.graph(graph, stream=s):
            c.expand(s)
        got = []
        for r in (1, 2, 3, 0, 2, 1):
            torch.mul(c.base, 1.0 + r, out=c.W)
            graph.replay()
            c.forward(s)
            got.append((r, c.y.clone()))
    torch.cuda.synchronize()
    for r, y in got:
        assert torch.equal(y.view(torch.int32), want[r].view(torch.int32))


@pytest.mark.parametrize("T", [1, 48, 200])
def test_a_forward_behind_an_expansion_and_a_capture(T):
    """A forward captured on the expansion's stream has not run there: the next one on the stream still stands directly behind the
    expansion."""
    c = Case(T, 3)
    want = [c.want(r) for r in range(4)]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    got, graphs = [], []
    with torch.cuda.stream(s):
        for r in (1, 2, 3, 0):
            torch.mul(c.base, 1.0 + r, out=c.W)
            c.expand(s)
            graph = torch.cuda.CUDAGraph()
            graph.capture_begin()
            c.forward(s)
            graph.capture_end()
            c.forward(s)
            got.append((r, c.y.clone()))
            graphs.append(graph)
    torch.cuda.synchronize()
    for r, y in got:
        assert torch.equal(y.view(torch.int32), want[r].view(torch.int32))
    for r in (2, 1):
        c.W.copy_(c.base * (1.0 + r))
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            c.expand(s)
            graphs[r].replay()   # behind the expansion, as a graph
            y = c.y.clone()
        torch.cuda.synchronize()
        assert torch.equal(y.view(torch.int32), want[r].view(torch.int32))
