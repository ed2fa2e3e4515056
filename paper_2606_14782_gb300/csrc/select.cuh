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

// Exclusive prefix sum of one int per thread, in thread order (x), and the
// sum of all (y).  One block barrier: every warp scans the warps' sums itself.
// warp_sums holds 32 ints and is not used again before the next barrier.  A
// call and not inlined: the kernels here run their code once per block, so
// that fetching it (about 200 cycles per 128 bytes that no earlier block has
// left in the instruction cache) costs more than executing it.
template <int T>
__device__ __noinline__ int2 block_exclusive_scan(int v, int* warp_sums)
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
    return make_int2(__shfl_sync(0xffffffffu, wi - w, warp) + incl - v,
                     __shfl_sync(0xffffffffu, wi, 31));
}

// x[k] = src[i0 + k] for the thread's PER positions (0 at and past n), with
// 16-byte loads when the run is whole and aligned (n % 4 == 0).
template <int PER>
__device__ __forceinline__ void load_run(const float* src, int i0, int n, float* x)
{
    if ((n & 3) == 0 && i0 + PER <= n) {
        const float4* s4 = reinterpret_cast<const float4*>(src + i0);
#pragma unroll
        for (int q = 0; q < PER / 4; ++q) {
            const float4 v = s4[q];
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
// k publishes the result.  Six block barriers in the usual case.
//
// Ranges are compared by 32-bit differences from their lower end.  The bins
// span at most 2^32 from the given range's lower end, so a top bin that
// reaches past the largest word wraps to words below that end, where no
// included key is.
template <int T>
struct SelectScratch {
    static constexpr int kBins = 4 * T;  // one 16-byte piece per thread
    static constexpr int kFew = 256;     // keys that are ranked by counting
    __align__(16) int bins[kBins];
    __align__(16) uint32_t few[kFew];
    uint32_t lo[32], hi[32];  // per-warp key ranges
    int sums[32];
    int out[3];               // boundary bin, how many of its keys are taken, its keys
    uint32_t tau;
    int need, eq;
    int nfew;
};

// The highest bin from which the count from the top reaches `remaining`, into
// sc.out: thread t holds four bins, the highest first, and the counts above
// them come from a block scan.  Two block barriers.
template <int T>
__device__ __forceinline__ void boundary_bin(SelectScratch<T>& sc, int remaining)
{
    const int piece = T - 1 - (int)threadIdx.x;
    const int4 c = reinterpret_cast<const int4*>(sc.bins)[piece];
    const int mine = c.x + c.y + c.z + c.w;
    int left = remaining - block_exclusive_scan<T>(mine, sc.sums).x;
    if (left > 0 && left <= mine) {
        int bin = 4 * piece + 3, n = c.w;
        if (left > n) { left -= n; n = c.z; --bin; }
        if (bin == 4 * piece + 2 && left > n) { left -= n; n = c.y; --bin; }
        if (bin == 4 * piece + 1 && left > n) { left -= n; n = c.x; --bin; }
        sc.out[0] = bin;
        sc.out[1] = left;
        sc.out[2] = n;
    }
    __syncthreads();
}

// each(f) calls f(included, key) for every element of the calling thread
// (a flag instead of a branch around the call: the loads of a thread's
// elements and their tests then overlap); 1 <= k <= the block's included keys;
// kmin / kmax: the thread's share of a key range that holds all of them.  Every
// thread returns the same result.  The scratch may be used again after the
// call's last barrier: a second call's first writes touch only what no thread
// reads after that barrier.
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
        boundary_bin<T>(sc, remaining);
        lo += (uint32_t)sc.out[0] << shift;
        remaining = sc.out[1];
        const int in_bin = sc.out[2];
        last = (1u << shift) - 1u;  // (the top bin may reach past 2^32, see above)
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
