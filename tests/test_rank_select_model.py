"""Model of the block-wide selection of the calibration and adaptive kernels,
run on the CPU: a histogram of four bins per thread over the keys' own range,
the boundary bin from a scan over the threads' pieces (highest first), narrowed
until the bin holds one key value or at most 256 keys, which then rank
themselves by counting.  Keys are 32-bit words and sums and differences wrap as
the kernels' do: a range may reach past the largest word, and no included key
may wrap into it.  Checked against a plain sort on inputs with ties, plateaus,
wide ranges and ranges that end at the top, and with words of six bits on every
pair of least and largest key.  A key below the given least one does wrap in,
and the model reports it."""

import random

import pytest

FEW = 256
TOP = 0xffffffff


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


def select(keys, k, threads, bits=32, few_max=FEW, least=None):
    """(tau, keys equal to tau that are taken, keys equal to tau); `least`: the
    lower end of the key range that the kernel is given."""
    word = (1 << bits) - 1
    nbins = 4 * threads
    log2 = nbins.bit_length() - 1
    lo = min(keys) if least is None else least
    last = max(keys) - lo
    shift = max(0, (last | 1).bit_length() - log2)
    while True:
        bins = [0] * nbins
        for key in keys:
            d = (key - lo) & word
            if d <= last:
                assert d >> shift < nbins  # the kernels' histogram has no more
                bins[d >> shift] += 1
        b, k, n = boundary(bins, k)
        lo = (lo + (b << shift)) & word
        last = (1 << shift) - 1
        if shift == 0:
            return lo, k, n
        if n <= few_max:
            break
        shift = max(0, shift - log2)
    few = [key for key in keys if ((key - lo) & word) <= last]
    assert len(few) == n  # the kernels' array has room for few_max
    found = {(key, k - gt, eq) for key in few
             for gt, eq in [(sum(o > key for o in few), few.count(key))]
             if gt < k <= gt + eq}
    assert len(found) == 1  # only equal keys publish, and they publish the same
    return found.pop()


def _top(rng, n):
    """Keys at both ends of the range of words: the last bin reaches past the
    largest word, to just below the least key."""
    return ([3, TOP] + [TOP - rng.randint(0, 1 << 19) for _ in range(n // 4)]
            + [3 + rng.randint(0, 1 << 19) for _ in range(n // 2)])


def _cases():
    rng = random.Random(5)
    out = []
    for threads in (128, 256, 512, 1024):
        for kind in ("wide", "narrow", "plateaus", "equal", "extremes", "top"):
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
            elif kind == "top":
                keys = _top(rng, n)
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


def _expected(keys, k):
    tau = sorted(keys, reverse=True)[k - 1]
    return tau, k - sum(x > tau for x in keys), keys.count(tau)


def test_every_range_of_six_bit_words():
    rng = random.Random(17)
    for lo in range(64):
        for hi in range(lo, 64):
            keys = [lo, hi] + [rng.choice((lo, hi, rng.randint(lo, hi))) for _ in range(10)]
            for k in range(1, len(keys) + 1):
                assert select(keys, k, 1, bits=6, few_max=2) == _expected(keys, k), (keys, k)


def test_a_key_below_the_given_range_is_caught():
    keys = [1, 61, 62]  # the top bin of [5, 62] is 53 ... 63 and, wrapped, 0 ... 4
    assert select(keys, 1, 1, bits=6, few_max=2) == _expected(keys, 1)
    with pytest.raises(AssertionError):
        select(keys, 1, 1, bits=6, few_max=2, least=5)


def test_boundary_matches_a_scan_from_the_top():
    rng = random.Random(11)
    for trial in range(400):
        n = 4 * rng.choice((128, 256, 512, 1024))
        bins = [0] * n
        if trial % 3 == 0:    # few occupied bins, long runs of zeros
            for _ in range(rng.randint(1, 40)):
                bins[rng.randrange(n)] += rng.randint(1, 50)
        elif trial % 3 == 1:  # dense
            bins = [rng.randint(0, 9) for _ in range(n)]
        else:                 # one heavy bin
            bins[rng.randrange(n)] = rng.randint(1, 16000)
        total = sum(bins)
        for remaining in sorted({1, total, max(1, total // 2)} - {0}):
            above = 0
            for b in range(n - 1, -1, -1):
                if above + bins[b] >= remaining:
                    break
                above += bins[b]
            assert boundary(bins, remaining) == (b, remaining - above, bins[b])
