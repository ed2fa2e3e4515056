"""Pointer tables of the binding, with the library replaced by a recorder: each
(request, layer) entry is the address of t[r, l], also in tensors that hold
more layers or requests than the call uses, and a tensor that holds fewer is
refused."""

import types

import pytest
import torch

from paper_2606_14782_gb300 import bacon

R, L, HKV, HQ, W, D, N = 2, 3, 2, 4, 8, 64, 40
STREAM = types.SimpleNamespace(cuda_stream=0)


class Recorder:
    def bacon_compress_layer_budgets(self, handle, requests, q, k, v, *rest):
        self.tables = [[p for p in t[:R * L]] for t in (q, k, v)]
        return bacon.BACON_OK


@pytest.fixture
def ctx(monkeypatch):
    lib = Recorder()
    monkeypatch.setattr(bacon, "load", lambda: lib)
    c = bacon.Context.__new__(bacon.Context)
    c.handle, c.kv_heads, c.lib = None, HKV, lib
    return c


def _tensors(requests=R, layers=L):
    return [torch.zeros(requests, layers, *s, dtype=torch.bfloat16)
            for s in ((HKV, N, D), (HKV, N, D))]


@pytest.mark.parametrize("requests,layers", [(R, L), (R, L + 2), (R + 1, L), (R + 1, L + 1)])
def test_entries_are_the_pairs_addresses(ctx, requests, layers):
    q = torch.zeros(R, L, HQ, W, D, dtype=torch.bfloat16)
    k, v = _tensors(requests, layers)
    ctx.compress_layer_budgets(q, k, v, [16] * L, stream=STREAM)
    for table, t in zip(ctx.lib.tables, (q, k, v)):
        assert table == [t[r, l].data_ptr() for r in range(R) for l in range(L)]


@pytest.mark.parametrize("requests,layers", [(R, L - 1), (R - 1, L)])
def test_too_few_pairs_are_refused(ctx, requests, layers):
    q = torch.zeros(R, L, HQ, W, D, dtype=torch.bfloat16)
    k, v = _tensors(requests, layers)
    with pytest.raises(IndexError):
        ctx.compress_layer_budgets(q, k, v, [16] * L, stream=STREAM)


def test_views_of_a_larger_tensor(ctx):
    q = torch.zeros(R, L, HQ, W, D, dtype=torch.bfloat16)
    k, v = (t[:, 1:L + 1] for t in _tensors(R, L + 2))
    ctx.compress_layer_budgets(q, k, v, [16] * L, stream=STREAM)
    for table, t in zip(ctx.lib.tables, (q, k, v)):
        assert table == [t[r, l].data_ptr() for r in range(R) for l in range(L)]
