// Block-wide selection building blocks shared by the calibration kernel and
// the adaptive (per-layer) selection kernel.
//
// "The k best" always means: larger value first, equal values -> lower index
// first.  Values are compared through order-preserving 32-bit keys
// (float_key).  A range-adaptive radix select finds the k-th best key tau
// and how many elements equal to tau are taken; membership is then key > tau,
// or key == tau among the first `need` equal keys in index order.
#pragma once

#include "common.cuh"

namespace bacon {
namespace sel {

struct SelectResult {
    uint32_t tau;  // key of the k-th best element
    int need;      // how many elements with key == tau are taken
    int count_eq;  // how many included elements have key == tau
    // every element equal to tau is taken: membership is key >= tau and
    // needs no index-ordered counting
    __device__ __forceinline__ bool all_ties_in() const { return need == count_eq; }
};

// Exclusive prefix sum of one int per thread, in thread order; total receives
// the sum.  One block barrier: every warp scans the warps' sums itself.
// warp_sums holds 32 ints and is not used again before the next barrier.
template <int T>
__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_sums, int& total)
{
    constexpr int kWarps = T / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    const int w = lane < kWarps ? warp_sums[lane] : 0;
    int wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += y;
    }
    total = __shfl_sync(0xffffffffu, wi, 31);
    return __shfl_sync(0xffffffffu, wi - w, warp) + incl - v;
}

// x[k] = src[i0 + k] for the thread's PER positions (0 at and past n), with
// 16-byte loads when the run is whole and aligned (n % 4 == 0).
template <int PER>
__device__ __forceinline__ void load_run(const float* __restrict__ src, int i0, int n, float* x)
{
    if ((n & 3) == 0 && i0 + PER <= n) {
        const float4* s4 = reinterpret_cast<const float4*>(src + i0);
#pragma unroll
        for (int q = 0; q < PER / 4; ++q) {
            const float4 v = __ldg(s4 + q);
            x[4 * q] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < PER; ++k) x[k] = i0 + k < n ? src[i0 + k] : 0.f;
    }
}

// The k-th best key: one histogram of kBins bins over the keys' own range,
// then the boundary bin is gathered, and its keys (at most kFew, else the
// range narrows by another histogram) find their own rank: a thread counts
// the gathered keys above and equal to its own, and the one whose ranks span
// k publishes the result.  Five block barriers in the usual case.
template <int T>
struct SelectScratch {
    // fewer keys need fewer bins, and one warp walks them all
    static constexpr int kBins = T >= 512 ? 2048 : (T >= 256 ? 1024 : 512);
    static constexpr int kFew = 256;  // keys that are ranked by counting
    __align__(16) int bins[kBins];
    __align__(16) uint32_t few[kFew];
    uint32_t lo[32], hi[32];  // per-warp key ranges
    int out[3];               // boundary bin, count above it left over, keys in it
    uint32_t tau;
    int need, eq;
    int nfew;
};

// By one warp: the highest bin from which the count from the top reaches
// `remaining`; out = {bin, how many of its keys are taken, its keys}.
template <int BINS>
__device__ __forceinline__ void boundary_bin(const int* bins, int remaining, int* out)
{
    constexpr int BL = BINS / 32;  // bins per lane
    static_assert(BL == 64 || BL == 32 || BL == 16, "two, one or half a bin per lane below");
    const int lane = threadIdx.x & 31;
    const int4* b4 = reinterpret_cast<const int4*>(bins) + (BL / 4) * lane;
    int mine = 0;
#pragma unroll
    for (int q = 0; q < BL / 4; ++q) {
        const int4 v = b4[(q + lane) & (BL / 4 - 1)];
        mine += v.x + v.y + v.z + v.w;
    }
    int incl = mine;  // keys in this lane's bins and above
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_down_sync(0xffffffffu, incl, o);
        if (lane + o < 32) incl += y;
    }
    const uint32_t hit = __ballot_sync(0xffffffffu, incl >= remaining);
    const int lb = hit ? 31 - __clz(hit) : 0;
    const int above = __shfl_sync(0xffffffffu, incl - mine, lb);
    // the boundary lane's bins: two, one or (below 32) at most one per lane
    constexpr int PL = BL == 64 ? 2 : 1;
    const int b0 = BL * lb + PL * lane;
    const bool held = PL * lane < BL;
    const int c0 = held ? bins[b0] : 0, c1 = (PL == 2) ? bins[b0 + 1] : 0;
    const int pair = c0 + c1;
    int inc2 = pair;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_down_sync(0xffffffffu, inc2, o);
        if (lane + o < 32) inc2 += y;
    }
    const uint32_t hit2 = __ballot_sync(0xffffffffu, held && above + inc2 >= remaining);
    const int l2 = hit2 ? 31 - __clz(hit2) : 0;
    if (lane == l2) {
        const int before = above + inc2 - pair;  // keys above this lane's bins
        const bool top = PL == 2 && before + c1 >= remaining;
        out[0] = top ? b0 + 1 : b0;
        out[1] = (PL == 1 || top) ? remaining - before : remaining - before - c1;
        out[2] = top ? c1 : c0;
    }
}

// each(f) calls f(included, key) for every element of the calling thread
// (a flag instead of a branch around the call: the loads of a thread's
// elements and their tests then overlap); 1 <= k <= the block's included keys; kmin / kmax: the thread's share of a key
// range that holds all of them.  Every thread returns the same result.  The
// scratch may be used again after the call's last barrier: a second call's
// first writes touch only what no thread reads after that barrier.
template <int T, typename EachFn>
__device__ __forceinline__ SelectResult select_each(EachFn each, int k, SelectScratch<T>& sc,
                                                    uint32_t kmin, uint32_t kmax)
{
    using S = SelectScratch<T>;
    constexpr int kWarps = T / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
        sc.lo[warp] = kmin;
        sc.hi[warp] = kmax;
    }
    if (threadIdx.x == 0) sc.nfew = 0;
    for (int b = threadIdx.x; b < S::kBins / 4; b += T)
        reinterpret_cast<int4*>(sc.bins)[b] = make_int4(0, 0, 0, 0);
    __syncthreads();
    uint32_t lo = __reduce_min_sync(0xffffffffu, lane < kWarps ? sc.lo[lane] : 0xffffffffu);
    uint32_t last = __reduce_max_sync(0xffffffffu, lane < kWarps ? sc.hi[lane] : 0u) - lo;
    // keys of the current range: [lo, lo + last]; bins of 2^shift keys
    int shift = max(0, 32 - __clz(last | 1u) - (31 - __clz(S::kBins)));
    int remaining = k;
    while (true) {
        each([&](bool in, uint32_t key) {
            const uint32_t d = key - lo;
            if (in && d <= last) atomicAdd(&sc.bins[d >> shift], 1);
        });
        __syncthreads();
        if (warp == 0) boundary_bin<S::kBins>(sc.bins, remaining, sc.out);
        __syncthreads();
        lo += (uint32_t)sc.out[0] << shift;
        remaining = sc.out[1];
        const int in_bin = sc.out[2];
        last = (1u << shift) - 1u;
        if (shift == 0) return {lo, remaining, in_bin};
        if (in_bin <= S::kFew) break;
        // many keys in one bin (plateaus of equal scores): narrow the range
        shift = max(0, shift - (31 - __clz(S::kBins)));
        for (int b = threadIdx.x; b < S::kBins / 4; b += T)
            reinterpret_cast<int4*>(sc.bins)[b] = make_int4(0, 0, 0, 0);
        __syncthreads();
    }
    const int n = sc.out[2];
    each([&](bool in, uint32_t key) {
        if (in && key - lo <= last) sc.few[atomicAdd(&sc.nfew, 1)] = key;
    });
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += T) {
        const uint32_t key = sc.few[i];
        int gt = 0, eq = 0;
        for (int j = 0; j < n; ++j) {
            const uint32_t o = sc.few[j];
            gt += o > key;
            eq += o == key;
        }
        if (gt < remaining && gt + eq >= remaining) {  // (equal keys write the same values)
            sc.tau = key;
            sc.need = remaining - gt;
            sc.eq = eq;
        }
    }
    __syncthreads();
    return {sc.tau, sc.need, sc.eq};
}

// The same over values in registers: x holds the thread's PER values, the
// first nv of them included.
template <int T, int PER>
__device__ __forceinline__ SelectResult select_runs(const float* x, int nv, int k,
                                                    SelectScratch<T>& sc, uint32_t kmin,
                                                    uint32_t kmax)
{
    return select_each<T>(
        [&](auto f) {
#pragma unroll
            for (int q = 0; q < PER; ++q)
                f(q < nv, float_key(x[q]));
        },
        k, sc, kmin, kmax);
}

}  // namespace sel
}  // namespace bacon
