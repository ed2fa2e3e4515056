"""The calibration kernel's two selections at the edges of its size classes
and on scores with ties, against a stable sort of the kernel's own scores:
the kept positions exactly, and lambda from the members of the M best by the
pooled backbone in 64 bits."""

import pytest
import torch

from paper_2606_14782_gb300 import bacon, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    bacon.load()


def _best(x, k):
    return torch.sort(x, dim=-1, descending=True, stable=True).indices[..., :k].sort(-1).values


# distinct keys: 1 (every score ties), 5 (a boundary bin of hundreds of equal
# scores), 300 (runs of ties), 0 = all different
@pytest.mark.parametrize("distinct", [1, 5, 300, 0])
@pytest.mark.parametrize("n", [40, 1024, 1025, 2048, 2049, 4096, 4097, 8191, 8193, 16384, 16390])
def test_selections_match_a_stable_sort(n, distinct):
    g = torch.Generator(device="cuda").manual_seed(1000 * distinct + n)
    layers, h, d, w = 2, 2, 64, 8
    q = torch.randn(1, layers, h, w, d, generator=g, device="cuda").bfloat16()
    k = torch.randn(1, layers, h, n, d, generator=g, device="cuda")
    if distinct:
        pick = torch.randint(0, distinct, (n,), generator=g, device="cuda")
        k = k[..., :1, :].expand_as(k) if distinct == 1 else k[..., pick % n, :]
    k = k.bfloat16().contiguous()
    ncand = n - w
    for keep in sorted({1, 17, min(ncand - 1, max(1, n // 10)), ncand - 1}):
        ctx = bacon.Context(layers, h, h, d, w, 7, w + keep, max_seq_len=n, max_requests=1,
                            keep_scores=1)
        _, _, idx = ctx.compress_all_layers(q, k, k, w + keep)
        S, V, Bp = (ctx.scores(x).view(layers, h, n)[..., :ncand] for x in ("S", "V", "Bpool"))
        lam = ctx.scores("lambda").view(layers, h)
        ctx.sync()
        want = _best(S, keep)
        assert torch.equal(idx[0, ..., :keep].long(), want), keep
        assert torch.equal(idx[0, ..., keep:].long(),
                           torch.arange(ncand, n, device="cuda").expand(layers, h, w))
        top = _best(Bp, min(2 * keep, ncand))
        sb = Bp.double().gather(-1, top).std(-1, correction=0)
        sv = V.double().gather(-1, top).std(-1, correction=0)
        ref = sb / (sv + 1e-8)
        # fp32 moments about a member: a few ulp of the largest member, which
        # matters where the members hardly differ (std below 1e-6 of them)
        floor = 1e-6 * Bp.double().gather(-1, top).amax(-1) / (sv + 1e-8)
        assert ((lam.double() - ref).abs() <= 2e-4 * ref + floor).all(), (keep, lam, ref)
        ctx.close()


def _adaptive_reference(S, keep, sure):
    """Membership [H, ncand] of one layer: each head's own best, then the best
    of the rest jointly (ties to the lower head, then the lower position)."""
    h, ncand = S.shape
    taken = torch.zeros_like(S, dtype=torch.bool)
    if keep >= ncand:
        return ~taken
    if sure:
        taken.scatter_(1, _best(S, sure), True)
    rest = h * (keep - sure)
    if rest:
        free = (~taken).view(-1).nonzero()[:, 0]
        taken.view(-1)[free[_best(S.reshape(-1)[free], rest)]] = True
    return taken


@pytest.mark.parametrize("distinct", [1, 5, 0])
@pytest.mark.parametrize("n,h,win", [
    (12, 3, 8), (300, 1, 8), (1024, 32, 8), (1027, 5, 8), (2500, 4, 8), (8193, 3, 8),
    (16384, 4, 8), (16390, 2, 8), (1027, 5, 0),
])
def test_adaptive_matches_a_stable_sort(n, h, win, distinct):
    g = torch.Generator(device="cuda").manual_seed(77 * distinct + n)
    layers, d, w = 2, 64, 8
    q = torch.randn(1, layers, h, w, d, generator=g, device="cuda").bfloat16()
    k = torch.randn(1, layers, h, n, d, generator=g, device="cuda")
    if distinct:
        pick = torch.randint(0, distinct, (n,), generator=g, device="cuda")
        k = k[..., :1, :].expand_as(k) if distinct == 1 else k[..., pick % n, :]
    k = k.bfloat16().contiguous()
    ncand = n - win
    for budget in sorted({w, w + 4, min(n, (w + n // 12) // 4 * 4), n // 4 * 4, n - 1, n}):
        if budget < w or h * budget % 4:  # the binding's index blocks are 16-byte aligned
            continue
        ctx = bacon.Context(layers, h, h, d, w, 7, budget, max_seq_len=n, max_requests=1,
                            keep_window=int(win > 0))
        for alpha in (0.0, 0.2, 1.0):
            ko, vo, idx, counts = ctx.compress_adaptive(q, k, k, budget, alpha)
            S = ctx.scores("S").view(layers, h, n)[..., :ncand]
            ctx.sync()
            keep = budget - win
            sure = int(alpha * keep) if alpha in (0.0, 1.0) else int(
                torch.tensor(alpha, dtype=torch.float32).double().item() * keep)
            for l in range(layers):
                m = _adaptive_reference(S[l], keep, sure)
                tail = torch.arange(ncand, n, device="cuda")
                want = torch.cat([torch.cat([x.nonzero()[:, 0], tail]) for x in m])
                assert torch.equal(idx[0, l].long(), want), (budget, alpha, l)
                assert torch.equal(counts[0, l].long(), m.sum(1) + win), (budget, alpha, l)
                heads = torch.repeat_interleave(torch.arange(h, device="cuda"), counts[0, l].long())
                assert torch.equal(ko[0, l], k[0, l][heads, want])
        ctx.close()
