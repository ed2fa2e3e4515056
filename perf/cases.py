"""Measured cases: the compression calls that a serving program makes at the
end of a prefill, each through the Python binding.

A case names the call and the shape.  Calls (`call`):

  step      every layer of a batch of requests, one budget (the usual call)
  lse       the same when the prefill attention kept its rows' log-sum-exp
  pyramid   the same with one budget per layer
  adaptive  the same with head budgets shared inside each layer
  sweep     the ablation grid: many hyper-parameter sets over one prefill
  layers    layer by layer, as a prefill that compresses each layer when it
            is done with it (score, select, compact)
  noalloc   the window scores of one layer without a context
  host      the whole step on page-locked host buffers
"""

import math

import torch

from paper_2606_14782_gb300 import bacon, workloads

ALPHA = 0.2  # share of an adaptive layer budget that every head is sure of
BETA = 20    # steepness of the pyramid schedule

# The ablation grid over one prefill: the component variants, then the
# persistence depths and the coherence radii.
SWEEP = ([dict(use_E=e, use_L=l, use_T=t, m=4, r=5)
          for e, l, t in ((1, 1, 1), (0, 0, 0), (1, 0, 1), (1, 1, 0), (0, 1, 1))]
         + [dict(m=m, r=5) for m in (2, 6, 8)]
         + [dict(m=4, r=r) for r in (3, 7, 9)])


def _case(name, call, requests, layers, q_heads, kv_heads, head_dim, seq_len, window, budget,
          kind, pool=7, r=5, m=4, scores=False):
    c = dict(call=call, requests=requests, layers=layers, q_heads=q_heads, kv_heads=kv_heads,
             head_dim=head_dim, seq_len=seq_len, window=window, budget=budget, kind=kind,
             pool=pool, r=r, m=m, scores=scores)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a toy prompt: launches and host work are all there is
        _case("tiny_step", "step", 1, 2, 4, 4, 64, 640, 32, 64, "gaussian"),
        # one image in a multi-head model: many short heads
        _case("mha_image_step", "step", 1, 32, 32, 32, 128, 1024, 32, 256, "lowrank"),
        # one high-resolution image in a grouped-query model
        _case("gqa_image_step", "step", 1, 28, 28, 4, 128, 4096, 32, 512, "grid"),
        # two chat turns of ragged length, four query heads per kv-head
        _case("ragged_step", "step", 2, 16, 32, 8, 128, 3001, 32, 333, "lowrank"),
        # 32 frames of video
        _case("video_step", "step", 1, 28, 28, 4, 128, 6528, 64, 652, "video"),
        # four long screenshot prompts: the largest call, and the benchmark's
        _case("gui_step", "step", 4, 28, 28, 4, 128, 16384, 64, 1024, "heavytail"),
        # the same prompts when the prefill kept its normalisers
        _case("gui_lse", "lse", 4, 28, 28, 4, 128, 16384, 64, 1024, "heavytail"),
        # head budgets shared inside a layer
        _case("gqa_image_adaptive", "adaptive", 1, 28, 28, 4, 128, 4096, 32, 512, "grid"),
        # the ablation grid over one video
        _case("video_sweep", "sweep", 1, 28, 28, 4, 128, 6528, 64, 652, "video"),
        # a prefill that compresses every layer as it leaves it
        _case("video_layers", "layers", 1, 28, 28, 4, 128, 6528, 64, 652, "video", scores=True),
        # one long layer for an engine that owns all device memory
        _case("gui_layer_noalloc", "noalloc", 1, 1, 28, 4, 128, 16384, 64, 64, "heavytail"),
        # a cache that was offloaded to the host
        _case("gqa_image_host", "host", 1, 28, 28, 4, 128, 4096, 32, 512, "grid"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def _cost(c):
    """Elements of one pass of window logits, times the head dimension."""
    return (c["requests"] * c["layers"] * c["q_heads"] * c["window"] * c["seq_len"]
            * c["head_dim"])


MAX_COST = 4 * 28 * 28 * 64 * 16384 * 128  # the largest listed case


def draw(rng):
    while True:
        call = rng.choice(("step",) * 6 + ("lse", "pyramid", "adaptive", "sweep", "layers",
                                           "noalloc", "host"))
        q_heads, kv_heads = rng.choice(((4, 4), (8, 8), (32, 32), (28, 4), (32, 8), (16, 4),
                                        (8, 2), (6, 2), (12, 2)))
        window = rng.choice((8, 16, 32, 32, 32, 64, 64, rng.randint(1, 64)))
        seq_len = _log_int(rng, 320, 16384)
        if rng.random() < 0.3:  # prompts padded to a page of the cache
            seq_len = max(320, seq_len // 64 * 64)
        layers = rng.randint(2, 32)
        requests = rng.choice((1, 1, 1, 2, 3, 4))
        if call == "noalloc":
            layers = requests = 1
        elif call in ("layers", "host"):
            requests = 1
        if call == "pyramid":  # one list of outputs per layer: at most 64 of them
            layers, requests = min(layers, 20), 1
        budget = window + _log_int(rng, 16, max(17, (seq_len - window) // 2))
        c = _case(None, call, requests, layers, q_heads, kv_heads, rng.choice((64, 128, 128)),
                  seq_len, window, budget, rng.choice(("gaussian", "lowrank", "heavytail")),
                  pool=rng.choice((7, 7, 7, 5, 1)), r=rng.choice((5, 5, 5, 3, 7, 9)),
                  m=rng.choice((4, 4, 2, 6, 8)), scores=rng.random() < 0.5)
        rows = q_heads // kv_heads * window
        if rows > 512 or (call == "noalloc" and q_heads * window > 4096):
            continue
        if call == "adaptive" and kv_heads * (seq_len - window) > 190000:
            continue
        tokens = requests * layers * kv_heads * seq_len * c["head_dim"]
        if _cost(c) > MAX_COST or tokens > 4 * 28 * 4 * 16384 * 128:
            continue
        if call in ("sweep", "host") and tokens > 28 * 4 * 16384 * 128:
            continue
        return c


def _workload(c):
    n = c["seq_len"]
    planted = 16 if n >= 1024 else 4
    wl = workloads.Workload("case", c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"], n,
                            c["window"], c["pool"], (c["budget"],), c["requests"],
                            (16, n - max(c["window"], 32) - 32), c["kind"], planted)
    if c["kind"] == "grid":
        side = 60
        wl = wl.with_(grid=side, visual=(16, 16 + side * side))
    elif c["kind"] == "video":
        wl = wl.with_(frame_tokens=196, visual=(16, 16 + 32 * 196), planted=8)
    return wl


def _window_logits(c, qwin, k, dtype):
    """Masked, scaled logits of one (request, layer): [Hkv, G W, N]."""
    hkv, n, d = k.shape
    w = c["window"]
    x = torch.matmul(qwin.to(dtype).reshape(hkv, -1, d), k.to(dtype).transpose(1, 2))
    x *= 1.0 / math.sqrt(d)
    # window query j sits at position n - w + j and sees the keys up to it
    hidden = torch.ones(w, w, dtype=torch.bool, device=k.device).triu(1)
    x.view(hkv, -1, w, n)[..., n - w:].masked_fill_(hidden, float("-inf"))
    return x


def prepare(case, seed):
    c = case
    x = workloads.generate(_workload(c), seed=seed, device="cuda")
    s = dict(case=c, qwin=x.qwin, k=x.k, v=x.v)
    if c["call"] == "noalloc":
        s["lib"] = bacon.load()
        return s
    s["ctx"] = bacon.Context(c["layers"], c["kv_heads"], c["q_heads"], c["head_dim"],
                             c["window"], c["pool"], c["budget"], max_seq_len=c["seq_len"],
                             max_requests=c["requests"], r=c["r"], m=c["m"])
    if c["call"] == "lse":
        s["lse"] = torch.stack([torch.stack([
            torch.logsumexp(_window_logits(c, x.qwin[i, l], x.k[i, l], torch.float32), dim=-1)
            .reshape(c["q_heads"], c["window"])
            for l in range(c["layers"])]) for i in range(c["requests"])])
    elif c["call"] == "pyramid":
        s["budgets"] = bacon.pyramid_budgets(c["layers"], c["window"], c["budget"], BETA)
    elif c["call"] == "layers":
        s["state"] = bacon.State(s["ctx"])
        L, h, d, n = c["layers"], c["kv_heads"], c["head_dim"], c["seq_len"]
        kept = min(c["budget"], n)
        dev = x.k.device
        out = [torch.empty(L, h, kept, d, dtype=x.k.dtype, device=dev) for _ in range(2)]
        out.append(torch.empty(L, h, kept, dtype=torch.int32, device=dev))
        if c["scores"]:
            out.append(torch.empty(L, h, n, dtype=torch.float32, device=dev))
        s["out"] = out
        # a model holds one tensor per layer
        s["per_layer"] = [(x.qwin[0, l], x.k[0, l], x.v[0, l], out[0][l], out[1][l], out[2][l],
                           out[3][l] if c["scores"] else None) for l in range(L)]
    elif c["call"] == "host":
        for name in ("qwin", "k", "v"):
            s[name] = s[name].cpu().pin_memory()
        R, L, h, d = c["requests"], c["layers"], c["kv_heads"], c["head_dim"]
        kept = min(c["budget"], c["seq_len"])
        s["out"] = [torch.empty(R, L, h, kept, d, dtype=s["k"].dtype, pin_memory=True)
                    for _ in range(2)]
        s["out"].append(torch.empty(R, L, h, kept, dtype=torch.int32, pin_memory=True))
    return s


def _bits(t):
    """Copied cache rows as the bit patterns that they are."""
    return t.view(torch.int16)


def run(state):
    s, c = state, state["case"]
    call, budget = c["call"], c["budget"]
    if call == "noalloc":
        h, n = c["kv_heads"], c["seq_len"]
        B, Q, E = (torch.empty(h, n, dtype=torch.float32, device=s["k"].device)
                   for _ in range(3))
        status = s["lib"].bacon_window_scores_noalloc(
            h, c["q_heads"], c["head_dim"], c["window"], s["qwin"].data_ptr(),
            s["k"].data_ptr(), n, B.data_ptr(), Q.data_ptr(), E.data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        if status != bacon.BACON_OK:
            raise bacon.BaconError(status, "window scores")
        return {"B": B, "E": E, "Q": Q}
    ctx = s["ctx"]
    if call == "sweep":
        idx, lam = ctx.sweep(s["qwin"], s["k"], budget, SWEEP)
        return {"idx": idx, "lambda": lam}
    if call == "adaptive":
        k, v, idx, counts = ctx.compress_adaptive(s["qwin"], s["k"], s["v"], budget, ALPHA)
        return {"counts": counts, "idx": idx, "k": _bits(k), "v": _bits(v)}
    if call == "pyramid":
        k, v, idx = ctx.compress_layer_budgets(s["qwin"], s["k"], s["v"], s["budgets"])
        return {"idx": idx, "k": [[_bits(t) for t in row] for row in k],
                "v": [[_bits(t) for t in row] for row in v]}
    if call == "layers":
        st = s["state"]
        st.reset()
        n = c["seq_len"]
        for l, (q, k, v, ko, vo, idx, S) in enumerate(s["per_layer"]):
            st.score_layer(l, q, k, scores_out=S)
            st.select(budget, n, idx_out=idx)
            ctx.compact(k, v, idx, k_out=ko, v_out=vo)
        k, v, idx = s["out"][:3]
        out = {"idx": idx, "k": _bits(k), "v": _bits(v)}
        if c["scores"]:
            out["S"] = s["out"][3]
        return out
    if call == "host":
        k, v, idx = ctx.compress_host(s["qwin"], s["k"], s["v"], budget, *s["out"])
    elif call == "lse":
        k, v, idx = ctx.compress_with_lse(s["qwin"], s["k"], s["v"], s["lse"], budget)
    else:
        k, v, idx = ctx.compress_all_layers(s["qwin"], s["k"], s["v"], budget)
    return {"idx": idx, "k": _bits(k), "v": _bits(v)}


def _layer_budgets(c):
    if c["call"] != "pyramid":
        return [c["budget"]] * c["layers"]
    lo = (c["budget"] - c["window"]) // BETA
    hi = 2 * (c["budget"] - c["window"]) - lo
    if c["layers"] == 1 or c["budget"] <= c["window"]:
        return [c["budget"]] * c["layers"]
    return [c["window"] + lo + (c["layers"] - 1 - l) * (hi - lo) // (c["layers"] - 1)
            for l in range(c["layers"])]


def work(case):
    """Keys and window queries read once, the kept rows copied, the outputs
    written; one pass of window logits."""
    c = case
    n, d, pairs = c["seq_len"], c["head_dim"], c["requests"] * c["layers"]
    per_head = c["kv_heads"] * pairs
    bytes_ = 2 * d * (per_head * n + pairs * c["q_heads"] * c["window"])
    kept = c["requests"] * c["kv_heads"] * sum(min(b, n) for b in _layer_budgets(c))
    if c["call"] == "noalloc":
        bytes_ += 3 * 4 * per_head * n
    elif c["call"] == "sweep":
        bytes_ += len(SWEEP) * (4 * kept + 4 * per_head)
    else:
        bytes_ += kept * (4 * 2 * d + 4)
    if c["call"] == "lse":
        bytes_ += 4 * pairs * c["q_heads"] * c["window"]
    if c["call"] == "layers" and c["scores"]:
        bytes_ += 4 * per_head * n
    return {"bytes": bytes_, "flops": 2 * _cost(c)}


def tolerance(case):
    # Kept positions and copied rows are whole values.  Two scores that round
    # to either side of each other may swap at the selection's boundary, and
    # the positions between them then move by one: at most the values of one
    # head among a hundred.  The scores themselves carry the rounding of fp32
    # sums over the window rows and of the exponential unit: 7e-6 of the window
    # scores and 4e-6 of the final ones against 64 bits, stated four times.
    if case["call"] == "noalloc":
        return {"rel": 3e-5, "max": 1e-3}
    if case["call"] in ("sweep", "layers"):
        return {"rel": 1.5e-5, "max": 1e-3, "differ": 0.01}
    return {"rel": 0.0, "differ": 0.01}


def _exact_window(c, qwin, k):
    """B and Q of one (request, layer) in 64 bits: [Hkv, N] each."""
    hkv, n, w = c["kv_heads"], c["seq_len"], c["window"]
    a = torch.softmax(_window_logits(c, qwin, k, torch.float64), dim=-1).view(hkv, -1, w, n)
    return a.mean(dim=(1, 2)), a[:, :, -1].mean(dim=1)


def _exact_scores(c, B, E, before, keep, p):
    """lambda [Hkv] and S [Hkv, N - W] of one (request, layer); `before`: the
    residuals of the layers before it."""
    ncand = c["seq_len"] - c["window"]
    pooled = torch.nn.functional.max_pool1d(B[:, :ncand], c["pool"], 1, c["pool"] // 2)
    V = torch.zeros_like(E)
    if p["use_E"]:
        V = V + E
    if p["use_L"]:
        V = V + torch.nn.functional.avg_pool1d(E[None], 2 * p["r"] + 1, 1, p["r"],
                                               count_include_pad=False)[0]
    if p["use_T"] and before and p["m"]:
        V = V + torch.stack(before[-p["m"]:]).mean(dim=0)
    V = V[:, :ncand]
    M = min(2 * keep, ncand)
    top = torch.sort(pooled, dim=-1, descending=True, stable=True).indices[:, :M]
    lam = (pooled.gather(1, top).std(dim=1, correction=0)
           / (V.gather(1, top).std(dim=1, correction=0) + 1e-8))
    return lam, pooled + lam[:, None] * V


def _top(S, k):
    """Ascending positions of the k best, lower positions first among equals."""
    return torch.sort(S, dim=-1, descending=True, stable=True).indices[..., :k].sort(-1).values


def exact(case, seed):
    c = case
    if _cost(c) > MAX_COST // 2:
        return None  # only whole values come back, and 64-bit logits take long
    s = prepare(dict(c, call="noalloc"), seed)
    R, L, h, n, w = c["requests"], c["layers"], c["kv_heads"], c["seq_len"], c["window"]
    dev = s["k"].device
    if c["call"] == "noalloc":
        B, Q = _exact_window(c, s["qwin"][0, 0], s["k"][0, 0])
        return {"B": B, "E": (Q - B).clamp(min=0), "Q": Q}
    params = dict(r=c["r"], m=c["m"], use_E=1, use_L=1, use_T=1)
    sets = [dict(params, **v) for v in SWEEP] if c["call"] == "sweep" else [params]
    budgets = [min(b, n) for b in _layer_budgets(c)]
    tail = torch.arange(n - w, n, device=dev).expand(h, w)
    idx = [[[] for _ in range(R)] for _ in sets]
    lams = [[[] for _ in range(R)] for _ in sets]
    scores, counts = [], []
    for i in range(R):
        before = []
        for l in range(L):
            B, Q = _exact_window(c, s["qwin"][i, l], s["k"][i, l])
            E = (Q - B).clamp(min=0)
            keep = budgets[l] - w
            for j, p in enumerate(sets):
                lam, S = _exact_scores(c, B, E, before, keep, p)
                lams[j][i].append(lam)
                if c["call"] != "adaptive":
                    idx[j][i].append(torch.cat([_top(S, keep), tail], dim=1))
                    continue
                sure = math.floor(ALPHA * keep)
                taken = torch.zeros_like(S, dtype=torch.bool)
                taken.scatter_(1, _top(S, sure), True)
                rest = S.masked_fill(taken, float("-inf")).reshape(-1)
                taken.view(-1)[_top(rest, h * (keep - sure))] = True
                idx[j][i].append(torch.cat([torch.cat([t.nonzero()[:, 0], tail[0]])
                                            for t in taken]))
                counts.append(taken.sum(dim=1) + w)
            if c["call"] == "layers" and c["scores"]:
                scores.append(torch.nn.functional.pad(S, (0, w)))
            before.append(E)
    if c["call"] == "pyramid":
        none = [[None] * L for _ in range(R)]
        return {"idx": [[t.int() for t in row] for row in idx[0]], "k": none, "v": none}
    idx = torch.stack([torch.stack([torch.stack(row) for row in v]) for v in idx]).int()
    if c["call"] == "sweep":
        return {"idx": idx, "lambda": torch.stack([torch.stack([torch.stack(row) for row in v])
                                                   for v in lams])}
    if c["call"] == "layers":
        out = {"idx": idx[0, 0], "k": None, "v": None}
        if c["scores"]:
            out["S"] = torch.stack(scores)
        return out
    out = {"idx": idx[0], "k": None, "v": None}
    if c["call"] == "adaptive":
        out["counts"] = torch.stack(counts).view(R, L, h).int()
    return out
