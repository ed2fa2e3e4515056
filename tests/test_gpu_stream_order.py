"""A call's place in its stream, read off a captured graph.  The kernels of one
call overlap: the edges between them are programmatic.  The edges into a call's
first kernel and out of its last one are full ones, whatever the caller's
kernels are.  The captured graph then replays the call on other inputs."""

import ctypes

import pytest
import torch

from paper_2606_14782_gb300 import bacon, build, workloads

pytestmark = pytest.mark.gpu

KERNEL, MEMCPY = 0, 1      # CUgraphNodeType
FULL, PROGRAMMATIC = 0, 1  # CUgraphDependencyType
vp = ctypes.c_void_p


class EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte),
                ("type", ctypes.c_ubyte), ("reserved", ctypes.c_ubyte * 5)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    bacon.load()


class Captured:
    """The work that `body` puts on a stream, as a graph."""

    def __init__(self, body):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.stream = torch.cuda.Stream()
        self.graph, self.exec = vp(), vp()
        torch.cuda.synchronize()
        with torch.cuda.stream(self.stream):
            body()  # scratch, allocator blocks and kernels are there before the capture
            self.stream.synchronize()
            self.do("cuStreamBeginCapture_v2", vp(self.stream.cuda_stream), ctypes.c_int(2))
            try:
                self.result = body()
            finally:
                self.do("cuStreamEndCapture", vp(self.stream.cuda_stream),
                        ctypes.byref(self.graph))
        self.do("cuGraphInstantiateWithFlags", ctypes.byref(self.exec), self.graph,
                ctypes.c_ulonglong(0))

    def do(self, name, *args):
        rc = getattr(self.cu, name)(*args)
        assert rc == 0, (name, rc)

    def chain(self):
        """Node types in order, and the types of the edges between them (one
        stream: every node has at most one successor)."""
        n = ctypes.c_size_t()
        self.do("cuGraphGetNodes", self.graph, None, ctypes.byref(n))
        nodes = (vp * n.value)()
        self.do("cuGraphGetNodes", self.graph, nodes, ctypes.byref(n))
        kinds = {}
        for node in nodes:
            t = ctypes.c_int()
            self.do("cuGraphNodeGetType", vp(node), ctypes.byref(t))
            kinds[node] = t.value
        m = ctypes.c_size_t()
        self.do("cuGraphGetEdges_v2", self.graph, None, None, None, ctypes.byref(m))
        src, dst, data = (vp * m.value)(), (vp * m.value)(), (EdgeData * m.value)()
        self.do("cuGraphGetEdges_v2", self.graph, src, dst, data, ctypes.byref(m))
        after = {s: (t, e.type) for s, t, e in zip(src, dst, data)}
        assert len(after) == m.value == len(kinds) - 1
        at = (set(kinds) - set(dst)).pop()
        order, edges = [kinds[at]], []
        while at in after:
            at, e = after[at]
            order.append(kinds[at])
            edges.append(e)
        return order, edges

    def replay(self):
        self.do("cuGraphLaunch", self.exec, vp(self.stream.cuda_stream))
        self.stream.synchronize()

    def close(self):
        self.do("cuGraphExecDestroy", self.exec)
        self.do("cuGraphDestroy", self.graph)


def test_scores_elsewhere_are_copied():
    """A layer's scores go into the caller's device array from the kernel, and
    into other memory (page-locked here) by a copy behind it."""
    wl = workloads.CONFIGS["tiny"].with_(layers=1)
    x = workloads.generate(wl, seed=5, device="cuda")
    ctx = bacon.Context(1, wl.kv_heads, wl.q_heads, wl.head_dim, wl.window, wl.pool, 64,
                        max_seq_len=wl.seq_len, max_requests=1)
    state = bacon.State(ctx)
    device = torch.empty(wl.kv_heads, wl.seq_len, device="cuda")
    host = torch.empty(wl.kv_heads, wl.seq_len, pin_memory=True)
    for out, copies in ((device, []), (host, [MEMCPY])):
        def body():
            state.reset()
            return state.score_layer(0, x.qwin[0, 0], x.k[0, 0], scores_out=out)

        g = Captured(body)
        assert g.chain()[0] == [KERNEL] * 3 + copies
        out.fill_(7)
        torch.cuda.synchronize()
        g.replay()
        g.close()
    assert torch.equal(host, device.cpu())
    state.close()
    ctx.close()


GQA = dict(layers=3, q_heads=8, kv_heads=2, head_dim=128, seq_len=1200, visual=(16, 1100))
ONE_PASS = dict(layers=3, q_heads=4, kv_heads=4, head_dim=64, seq_len=640)
SWEEP = [dict(m=4), dict(m=2, r=3), dict(rho=1)]


def _calls(wl, x, ctx, state, budget):
    """{name: (the call, its kernels per call of the library)}."""
    R, L, d = wl.requests, wl.layers, wl.head_dim
    two = (wl.q_heads // wl.kv_heads) * wl.window > 32 or wl.seq_len > 1024
    window = 3 if two else 1  # statistics, normalisers, scores; or one kernel
    lse = torch.logsumexp(torch.randn(R, L, wl.q_heads, wl.window, 8, device="cuda"), -1) + 3.0

    def layers():
        state.reset()
        out = []
        for l in range(L):
            S = state.score_layer(l, x.qwin[0, l], x.k[0, l], scores_out=True)
            idx = state.select(budget, wl.seq_len)
            out += [S, idx, *ctx.compact(x.k[0, l], x.v[0, l], idx)]
        return out

    def noalloc():
        out = [torch.empty(wl.kv_heads, wl.seq_len, device="cuda") for _ in range(3)]
        rc = bacon.load().bacon_window_scores_noalloc(
            wl.kv_heads, wl.q_heads, d, wl.window, x.qwin[0, 1].data_ptr(), x.k[0, 1].data_ptr(),
            wl.seq_len, *(t.data_ptr() for t in out), torch.cuda.current_stream().cuda_stream)
        assert rc == bacon.BACON_OK
        return out

    def pyramid():
        k, v, idx = ctx.compress_layer_budgets(x.qwin, x.k, x.v, [budget - 8 * l for l in range(L)])
        return [t for rows in (k, v, idx) for row in rows for t in row]

    return {
        "step": (lambda: list(ctx.compress_all_layers(x.qwin, x.k, x.v, budget)), [window + 2]),
        "lse": (lambda: list(ctx.compress_with_lse(x.qwin, x.k, x.v, lse, budget)), [4]),
        "pyramid": (pyramid, [window + 2]),
        "adaptive": (lambda: list(ctx.compress_adaptive(x.qwin, x.k, x.v, budget)), [window + 3]),
        "sweep": (lambda: list(ctx.sweep(x.qwin, x.k, budget, SWEEP)), [window + 2]),
        "layers": (layers, [3, 1, 1] * L),
        "noalloc": (noalloc, [3]),
    }


@pytest.mark.parametrize("over", [GQA, ONE_PASS], ids=["two_passes", "one_pass"])
@pytest.mark.parametrize("name", ["step", "lse", "pyramid", "adaptive", "sweep", "layers",
                                  "noalloc"])
def test_calls_meet_the_stream_with_full_edges(name, over):
    wl = workloads.CONFIGS["tiny"].with_(**over)
    x = workloads.generate(wl, seed=2, device="cuda")
    budget = wl.window + 60
    ctx = bacon.Context(wl.layers, wl.kv_heads, wl.q_heads, wl.head_dim, wl.window, wl.pool,
                        budget, max_seq_len=wl.seq_len, max_requests=1)
    state = bacon.State(ctx)
    call, kernels = _calls(wl, x, ctx, state, budget)[name]
    mark = torch.zeros(64, device="cuda")

    def body():
        mark.add_(1.0)  # the caller's kernels around the call
        out = call()
        mark.add_(1.0)
        return out

    g = Captured(body)
    order, edges = g.chain()
    assert order == [KERNEL] * (sum(kernels) + 2)
    want = [e for n in kernels for e in [FULL] + [PROGRAMMATIC] * (n - 1)] + [FULL]
    assert edges == want

    other = workloads.generate(wl, seed=3, device="cuda")
    for mine, new in ((x.qwin, other.qwin), (x.k, other.k), (x.v, other.v)):
        mine.copy_(new)
    for t in g.result:
        t.fill_(7)
    torch.cuda.synchronize()
    g.replay()
    for got, want in zip(g.result, call()):
        assert torch.equal(got, want)
    ctx.sync()
    g.close()
    state.close()
    ctx.close()
