"""Model of the selection kernels' membership rule, run on the CPU.

The calibration and adaptive-selection kernels choose "the k best" (larger
value first, equal values -> lower position first, as the oracle's stable
sort does) without sorting: a radix select finds the k-th best key tau and how
many of the keys equal to tau are taken (test_rank_select_model.py models it),
and every thread then decides its own run of consecutive positions.  This file
replays the kernels' integer key mapping, the runs and the scans over the
threads in Python, and checks the members against a plain stable sort on inputs
with many ties, narrow and wide key ranges, and k from 1 to n.  A mistake in
the tie rule fails it.
"""

import random
import struct

import numpy as np
import pytest

from test_rank_select_model import select


def float_key(f):
    """Order-preserving 32-bit key of an fp32 value (the kernels' mapping)."""
    u = struct.unpack("<I", struct.pack("<f", float(np.float32(f))))[0]
    return u ^ 0xFFFFFFFF if u & 0x80000000 else u | 0x80000000


def reference(values, k):
    order = sorted(range(len(values)), key=lambda i: (-float(np.float32(values[i])), i))
    return sorted(order[:k])


def cases():
    rng = random.Random(7)
    out = []
    for trial in range(60):
        n = rng.choice([1, 2, 31, 32, 33, 100, 640, 992, 2047, 4000])
        kind = trial % 6
        if kind == 0:    # heavy ties: few distinct values
            vals = [rng.choice([0.25, 0.5, 0.125, 1e-6]) for _ in range(n)]
        elif kind == 1:  # plateaus like a max-pooled score
            base = [rng.random() * 1e-3 for _ in range(n)]
            vals = [max(base[max(0, i - 3):i + 4]) for i in range(n)]
        elif kind == 2:  # wide dynamic range
            vals = [10 ** rng.uniform(-12, -1) for _ in range(n)]
        elif kind == 3:  # all equal
            vals = [3.0] * n
        elif kind == 4:  # signed values
            vals = [rng.gauss(0, 1) for _ in range(n)]
        else:            # near-equal keys (a few ulps apart)
            vals = [float(np.nextafter(np.float32(1.0), np.float32(2.0)) * (1 + rng.randint(0, 3) * 1e-7))
                    for _ in range(n)]
        for k in sorted({1, n, max(1, n // 3), max(1, n - 1), rng.randint(1, n)}):
            out.append((vals, k))
    return out


def test_float_key_orders_like_floats():
    xs = [-np.inf, -3.5, -1e-30, -0.0, 0.0, 1e-30, 2.0, np.inf]
    ks = [float_key(x) for x in xs]
    assert ks == sorted(ks)
    assert float_key(-0.0) < float_key(0.0)


def members_by_runs(keys, sel, T, PER):
    """Membership as the kernels decide it: every thread walks
    its own run in position order; its tie rank starts from the keys equal
    to tau in the runs of lower threads (an exclusive scan in thread order),
    and the members are written at the scan of the per-thread member counts."""
    tau, need, count_eq = sel
    n = len(keys)
    eq_counts = [sum(1 for i in range(t * PER, min(n, t * PER + PER)) if keys[i] == tau)
                 for t in range(T)]
    eq_before = [0] * T
    for t in range(1, T):
        eq_before[t] = eq_before[t - 1] + eq_counts[t - 1]
    masks = []
    for t in range(T):
        rank = eq_before[t] if need != count_eq else 0
        m = []
        for i in range(t * PER, min(n, t * PER + PER)):
            eq = keys[i] == tau
            if keys[i] > tau or (eq and (need == count_eq or rank < need)):
                m.append(i)
            rank += eq
        masks.append(m)
    out = [None] * sum(len(m) for m in masks)
    pos = 0
    for m in masks:              # exclusive scan of the member counts
        for j, i in enumerate(m):
            out[pos + j] = i
        pos += len(m)
    return out


@pytest.mark.parametrize("T,PER", [(128, 8), (256, 8), (512, 8), (1024, 8), (1024, 16), (1024, 24)])
def test_run_membership_matches_stable_sort(T, PER):
    for vals, k in cases():
        if len(vals) > T * PER:
            continue
        keys = [float_key(v) for v in vals]
        assert members_by_runs(keys, select(keys, k, T), T, PER) == reference(vals, k), (len(vals), k)


def test_run_membership_without_the_tie_scan_is_caught():
    """Ranking ties inside each run only (no scan over lower threads) keeps
    too many equal keys: the comparison above would fail."""
    vals = [1.0] * 64
    keys = [float_key(v) for v in vals]
    sel = select(keys, 10, 8)
    tau, need, count_eq = sel
    per_run_only = [i for t in range(8) for j, i in enumerate(range(t * 8, t * 8 + 8))
                    if keys[i] > tau or j < need]
    assert per_run_only != reference(vals, 10)
    assert members_by_runs(keys, sel, 8, 8) == reference(vals, 10)
