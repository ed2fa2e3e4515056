"""Model of the block-wide selection of the calibration and adaptive kernels,
run on the CPU: a histogram of four bins per thread over the keys' own range,
the boundary bin from a scan over the threads' pieces (highest first), narrowed
until the bin holds one key value or at most 256 keys, which then rank
themselves by counting.  Checked against a plain sort on inputs with ties,
plateaus and wide ranges."""

import random

import pytest

FEW = 256


def boundary(bins, remaining):
    """(bin, keys of it that are taken, its keys), as the pieces find it."""
    above = 0
    for piece in range(len(bins) // 4 - 1, -1, -1):
        c = bins[4 * piece:4 * piece + 4]
        left = remaining - above
        if 0 < left <= sum(c):
            b, n = 4 * piece + 3, c[3]
            if left > n:
                left, n, b = left - n, c[2], b - 1
            if b == 4 * piece + 2 and left > n:
                left, n, b = left - n, c[1], b - 1
            if b == 4 * piece + 1 and left > n:
                left, n, b = left - n, c[0], b - 1
            return b, left, n
        above += sum(c)
    raise AssertionError("no boundary bin")


def select(keys, k, threads):
    """(tau, keys equal to tau that are taken, keys equal to tau)."""
    nbins = 4 * threads
    log2 = nbins.bit_length() - 1
    lo, last = min(keys), max(keys) - min(keys)
    shift = max(0, (last | 1).bit_length() - log2)
    while True:
        bins = [0] * nbins
        for key in keys:
            if 0 <= key - lo <= last:
                bins[(key - lo) >> shift] += 1
        b, k, n = boundary(bins, k)
        lo += b << shift
        last = (1 << shift) - 1
        if shift == 0:
            return lo, k, n
        if n <= FEW:
            break
        shift = max(0, shift - log2)
    few = [key for key in keys if 0 <= key - lo <= last]
    assert len(few) == n
    found = {(key, k - gt, eq) for key in few
             for gt, eq in [(sum(o > key for o in few), few.count(key))]
             if gt < k <= gt + eq}
    assert len(found) == 1  # only equal keys publish, and they publish the same
    return found.pop()


def _cases():
    rng = random.Random(5)
    out = []
    for threads in (128, 256, 512, 1024):
        for kind in ("wide", "narrow", "plateaus", "equal", "extremes"):
            n = rng.randint(1, 16 * threads)
            if kind == "wide":
                keys = [rng.getrandbits(32) for _ in range(n)]
            elif kind == "narrow":
                keys = [0x80000000 + rng.randint(0, 700) for _ in range(n)]
            elif kind == "plateaus":
                values = [rng.getrandbits(32) for _ in range(5)]
                keys = [rng.choice(values) for _ in range(n)]
            elif kind == "equal":
                keys = [rng.getrandbits(32)] * n
            else:
                keys = [rng.choice((0, 0xffffffff, 1, 0xfffffffe, 0x80000000)) for _ in range(n)]
            out.append((threads, kind, keys))
    return out


@pytest.mark.parametrize("threads,kind,keys", _cases())
def test_rank_select_matches_a_sort(threads, kind, keys):
    order = sorted(keys, reverse=True)
    for k in sorted({1, len(keys) // 3 or 1, len(keys)}):
        tau, need, eq = select(keys, k, threads)
        assert tau == order[k - 1]
        assert eq == keys.count(tau)
        assert need == k - sum(x > tau for x in keys)
