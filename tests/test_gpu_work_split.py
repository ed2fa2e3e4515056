"""The window passes cut their work by the size of the call: pass 1 by chunk
of a unit or, when that leaves SMs idle, by row block of a chunk, pass 2 by
tile.  A call of many units and a call of one layer therefore take different
routes over the same tensors; their final scores must be the same bits."""

import pytest
import torch

from paper_2606_14782_gb300 import bacon, build, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    bacon.load()


# window rows G W: one to four row blocks, whole and half last ones, and rows
# that do not fill their 64-row box
@pytest.mark.parametrize("group,window,head_dim,seq_len", [
    (1, 64, 128, 1153),    # 64 rows: one block
    (4, 34, 64, 1025),     # 136: a half last block of 8 rows
    (3, 64, 128, 2047),    # 192
    (4, 64, 64, 1300),     # 256
    (5, 64, 128, 1100),    # 320
    (6, 64, 128, 1281),    # 384
    (7, 64, 64, 1537),     # 448
    (7, 63, 128, 1111),    # 441: a window that is not a multiple of 16
    (8, 64, 128, 1024),    # 512
])
def test_few_units_and_many_give_the_same_bits(group, window, head_dim, seq_len):
    layers, requests, hkv = 20, 4, 2  # at least 320 chunks: by chunk
    wl = workloads.CONFIGS["tiny"].with_(
        layers=layers, requests=requests, q_heads=group * hkv, kv_heads=hkv, head_dim=head_dim,
        seq_len=seq_len, window=window, visual=(16, seq_len - 200))
    x = workloads.generate(wl, seed=9, device="cuda")
    budget = window + 40
    ctx = bacon.Context(layers, hkv, group * hkv, head_dim, window, 7, budget,
                        max_seq_len=seq_len, max_requests=requests, keep_scores=1)
    _, _, idx = ctx.compress_all_layers(x.qwin, x.k, x.v, budget)
    whole = {n: ctx.scores(n).view(requests, layers, hkv, seq_len) for n in ("S", "B", "Q")}
    ctx.sync()
    st = bacon.State(ctx)
    for r in (0, requests - 1):
        st.reset()
        for l in range(3):
            S = st.score_layer(l, x.qwin[r, l], x.k[r, l], scores_out=True)
            assert torch.equal(S, whole["S"][r, l]), (r, l)
            assert torch.equal(st.select(budget, seq_len), idx[r, l]), (r, l)
    # the same two passes without a context
    B, Q, E = (torch.empty(hkv, seq_len, device="cuda") for _ in range(3))
    rc = bacon.load().bacon_window_scores_noalloc(
        hkv, group * hkv, head_dim, window, x.qwin[1, 2].data_ptr(), x.k[1, 2].data_ptr(), seq_len,
        B.data_ptr(), Q.data_ptr(), E.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == bacon.BACON_OK
    ctx.sync()
    assert torch.equal(B, whole["B"][1, 2]) and torch.equal(Q, whole["Q"][1, 2])
    st.close()
    ctx.close()


def _window_scores(q, k, window):
    """B, Q, E of one layer, q [Hq, W, d] and k [Hkv, N, d], without a context."""
    hkv, n, d = k.shape
    out = [torch.empty(hkv, n, device="cuda") for _ in range(3)]  # each 16-byte aligned
    rc = bacon.load().bacon_window_scores_noalloc(
        hkv, q.shape[0], d, window, q.data_ptr(), k.data_ptr(), n, *(t.data_ptr() for t in out),
        torch.cuda.current_stream().cuda_stream)
    assert rc == bacon.BACON_OK
    return torch.stack(out)


# Window rows that leave pass 2 two slots of them (and of their bias) in shared
# memory, and more tiles than SMs, so that a CTA's share ends one unit after
# one to a few tiles and goes on with the next.  A kv-head by itself has fewer
# tiles than there are SMs: every CTA then works on one tile of one unit.
@pytest.mark.parametrize("hkv,group,window,head_dim,seq_len", [
    (32, 1, 32, 128, 3000),
    (128, 1, 32, 128, 129),
    (128, 1, 32, 64, 257),
    (128, 1, 32, 128, 500),
    (32, 4, 32, 128, 700),
    (16, 2, 64, 128, 1537),
    (12, 4, 32, 64, 2049),
    (16, 4, 64, 64, 1500),
    (20, 5, 13, 128, 1100),  # any window
])
def test_shares_that_cross_short_units(hkv, group, window, head_dim, seq_len):
    g = torch.Generator(device="cuda").manual_seed(hkv * seq_len)
    q, k = (torch.randn(*shape, generator=g, device="cuda").to(torch.bfloat16)
            for shape in ((hkv * group, window, head_dim), (hkv, seq_len, head_dim)))
    got = _window_scores(q, k, window)
    for h in range(hkv):
        alone = _window_scores(q[h * group:(h + 1) * group], k[h:h + 1], window)
        assert torch.equal(got[:, h], alone[:, 0]), h


def test_whole_step_shares_that_cross_units():
    """The same with the normalisers from a launch of their own."""
    layers, requests, hkv, group, window, d, n = 6, 2, 8, 4, 32, 128, 700
    wl = workloads.CONFIGS["tiny"].with_(
        layers=layers, requests=requests, q_heads=group * hkv, kv_heads=hkv, head_dim=d,
        seq_len=n, window=window, visual=(16, n - 100))
    x = workloads.generate(wl, seed=13, device="cuda")
    ctx = bacon.Context(layers, hkv, group * hkv, d, window, 7, 100, max_seq_len=n,
                        max_requests=requests)
    ctx.compress_all_layers(x.qwin, x.k, x.v, 100)
    got = torch.stack([ctx.scores(s) for s in "BQE"]).view(3, requests, layers, hkv, n)
    ctx.sync()
    for r in range(requests):
        for l in range(layers):
            for h in range(hkv):
                alone = _window_scores(x.qwin[r, l, h * group:(h + 1) * group],
                                       x.k[r, l, h:h + 1], window)
                assert torch.equal(got[:, r, l, h], alone[:, 0]), (r, l, h)
    ctx.close()


@pytest.mark.parametrize("offset", [0, 1, 2, 4])
def test_scores_out_at_any_float_alignment(offset):
    """Aligned score rows are stored by the kernel, others copied: same bits."""
    hkv, n, w = 2, 1156, 32
    wl = workloads.CONFIGS["tiny"].with_(layers=1, q_heads=8, kv_heads=hkv, head_dim=64, seq_len=n,
                                         visual=(16, 1000))
    x = workloads.generate(wl, seed=3, device="cuda")
    ctx = bacon.Context(1, hkv, 8, 64, w, 7, 100, max_seq_len=n, max_requests=1)
    st = bacon.State(ctx)
    want = st.score_layer(0, x.qwin[0, 0], x.k[0, 0], scores_out=True)
    buf = torch.full((hkv * n + 8,), 7.0, device="cuda")
    st.reset()
    st.score_layer(0, x.qwin[0, 0], x.k[0, 0],
                   scores_out=buf[offset:offset + hkv * n].view(hkv, n))
    ctx.sync()
    assert torch.equal(buf[offset:offset + hkv * n].view(hkv, n), want)
    assert (buf[:offset] == 7.0).all() and (buf[offset + hkv * n:] == 7.0).all()
    st.close()
    ctx.close()


@pytest.mark.parametrize("layers,requests,seq_len", [(7, 2, 8192), (9, 1, 4099), (1, 1, 16384)])
def test_host_path_in_parts(layers, requests, seq_len):
    """Keys beyond one pipelined part: the last request goes in halves, and
    persistence reads the residuals of the parts before."""
    hkv, d, w, budget = 3, 128, 16, 200
    wl = workloads.CONFIGS["tiny"].with_(
        layers=layers, requests=requests, q_heads=2 * hkv, kv_heads=hkv, head_dim=d,
        seq_len=seq_len, window=w, visual=(16, seq_len - 200))
    x = workloads.generate(wl, seed=21, device="cuda")
    ctx = bacon.Context(layers, hkv, 2 * hkv, d, w, 7, budget, max_seq_len=seq_len,
                        max_requests=requests, keep_scores=1)
    want = ctx.compress_all_layers(x.qwin, x.k, x.v, budget)
    scores = {n: ctx.scores(n).clone() for n in ("B", "E", "V", "S", "lambda")}
    qh, kh, vh = (t.cpu().pin_memory() for t in (x.qwin, x.k, x.v))
    for _ in range(2):
        got = ctx.compress_host(qh, kh, vh, budget)
        for a, b in zip(got, want):
            assert torch.equal(a, b.cpu())
        for n, s in scores.items():
            assert torch.equal(ctx.scores(n), s), n
    ctx.close()
