"""The per-(request, layer) tensors of a whole-step call may sit anywhere:
one after the other, at one distance with gaps, at uneven distances or in
any order.  Evenly spaced ones share one TMA descriptor, the others take a
table of descriptors; every placement gives the same bits."""

import ctypes

import numpy as np
import pytest
import torch

from paper_2606_14782_gb300 import bacon, build, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    bacon.load()


def _place(t, how):
    """Per-pair views of t [R, L, ...] holding its values, placed as `how`."""
    pairs = t.flatten(0, 1)
    n, size = pairs.shape[0], pairs[0].numel()
    row = t.shape[-1]
    if how == "separate":  # one allocation each
        return [p.clone() for p in pairs]
    step = {"contiguous": size, "gaps": size + 3 * row, "reversed": size, "uneven": size}[how]
    # NaN in the gaps: nothing outside a pair's own tensor may be read into a score
    buf = torch.full((n * step + 7 * row,), float("nan"), dtype=t.dtype, device=t.device)
    out = []
    for i in range(n):
        at = (n - 1 - i if how == "reversed" else i) * step
        if how == "uneven" and i == n - 1:
            at += 7 * row
        out.append(buf[at:at + size].view(pairs[i].shape))
        out[-1].copy_(pairs[i])
    return out


@pytest.mark.parametrize("over", [
    dict(layers=3, q_heads=8, kv_heads=2, head_dim=128, seq_len=1200, visual=(16, 1100)),
    dict(layers=2, requests=2, q_heads=6, kv_heads=3, head_dim=64, seq_len=777, window=24,
         visual=(16, 700)),
    dict(layers=3, q_heads=4, kv_heads=4, head_dim=64, seq_len=640),  # one pass over K
    dict(layers=1, q_heads=4, kv_heads=4, head_dim=64, seq_len=640),  # a single pair
])
def test_placements_give_the_same_bits(over):
    wl = workloads.CONFIGS["tiny"].with_(**over)
    x = workloads.generate(wl, seed=4, device="cuda")
    budget = wl.window + 50
    ctx = bacon.Context(wl.layers, wl.kv_heads, wl.q_heads, wl.head_dim, wl.window, wl.pool,
                        budget, max_seq_len=wl.seq_len, max_requests=wl.requests, keep_scores=1)
    pairs = wl.requests * wl.layers
    want = None
    for how in ("contiguous", "gaps", "uneven", "reversed", "separate", "contiguous"):
        q, k, v = (_place(t, how) for t in (x.qwin, x.k, x.v))
        ko = torch.empty(pairs, wl.kv_heads, budget, wl.head_dim, dtype=torch.bfloat16,
                         device="cuda")
        vo = torch.empty_like(ko)
        idx = torch.empty(pairs, wl.kv_heads, budget, dtype=torch.int32, device="cuda")

        def table(ts):
            return (ctypes.c_void_p * pairs)(*[t.data_ptr() for t in ts])

        rc = bacon.load().bacon_compress_all_layers(
            ctx.handle, wl.requests, table(q), table(k), table(v), wl.seq_len, budget, table(ko),
            table(vo), idx.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == bacon.BACON_OK, how
        ctx._last_units, ctx._last_N = pairs * wl.kv_heads, wl.seq_len
        S = ctx.scores("S")
        ctx.sync()
        got = [t.cpu() for t in (idx, S, ko.view(torch.int16), vo.view(torch.int16))]
        assert np.isfinite(got[1].numpy()).all(), how
        if want is None:
            want = got
        for a, b in zip(got, want):
            assert torch.equal(a, b), how
    ctx.close()
