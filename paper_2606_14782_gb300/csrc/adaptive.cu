// AdaKV-style adaptive head budgets (the base compressor of Sec. 5 / App. B
// that spreads a layer's budget over its kv-heads; BACON supplies the score,
// Eq. 16):
//   1. every head keeps its own top g = floor(alpha K) candidates (the
//      calibration kernel marks them while it still holds the head's scores);
//   2. the remaining Hkv K - Hkv g slots go to the best remaining candidates
//      of all heads together (larger S first; ties to the lower head, then
//      the lower position);
//   3. each head's kept positions are written in ascending order, followed
//      by the window, into one flat per-layer array (heads in order), and
//      the per-head counts are reported.
// The kept K/V rows are then gathered into the same flat layout.
//
// Steps 2 and 3 are one CTA per (request, layer), a latency-bound chain: a
// thread owns consecutive 8-position runs of the heads in order and reads
// them again (L1/L2) for each of three sweeps, so that ranks in (thread,
// run, slot) order are ranks in flattened order.  28 layers of 4 x 4064
// candidates: 14.6 us, and 4 us more in the calibration kernel; with one CTA
// making the heads' own selections too, one after the other, from global
// memory, it took 56 us.
#include "common.cuh"
#include "select.cuh"

namespace bacon {
namespace {

using namespace sel;

constexpr int kThreads = 1024;
constexpr int kRun = 8;  // positions per run: one byte of the bitmap

__global__ void __launch_bounds__(kThreads)
adaptive_select_kernel(Shape s, int keep_window, AdaptArgs a)
{
    extern __shared__ uint8_t kept_map[];  // [runs] members of each run
    __shared__ SelectScratch<kThreads> sel_sm;
    __shared__ int ties[32], offsets[32];

    after_previous();
    const int pair = blockIdx.x;
    const int H = s.hkv, N = s.N, W = s.W;
    const int win = keep_window ? W : 0;
    const int n_cand = N - win;
    const int kept_total = min(a.budget, N);
    const int keep = kept_total - win;
    const int rest = H * (keep - min(a.guaranteed, keep));
    const int runs = (n_cand + kRun - 1) / kRun;  // per head
    const int per = (H * runs + kThreads - 1) / kThreads;
    const int r0 = min(H * runs, (int)threadIdx.x * per), r1 = min(H * runs, r0 + per);
    const float* Sp = a.S + (size_t)pair * H * N;
    const uint8_t* Tp = a.taken + (size_t)pair * H * a.taken_stride;

    // f(run, head, first position, its candidates, those already taken)
    auto each_run = [&](auto f) {
        int h = runs > 0 ? r0 / runs : 0, i = r0 - h * runs;
        for (int r = r0; r < r1; ++r) {
            const int n = min(kRun, n_cand - kRun * i);
            f(r, h, kRun * i, n, (uint32_t)Tp[(size_t)h * a.taken_stride + i]);
            if (++i == runs) {
                i = 0;
                ++h;
            }
        }
    };
    // keys of the candidates that no head has taken for itself
    auto each_key = [&](auto f) {
        each_run([&](int, int h, int i0, int n, uint32_t taken) {
            float x[kRun];
            load_run<kRun>(Sp + (size_t)h * N, i0, N, x);
#pragma unroll
            for (int k = 0; k < kRun; ++k)
                f(k < n && !((taken >> k) & 1u), float_key(x[k]));
        });
    };

    // 2. the rest, jointly over the heads
    SelectResult sel = {0xffffffffu, 0, 0};  // takes nothing more
    int rank = 0;
    const bool all = keep >= n_cand;  // every candidate is marked
    if (!all && rest > 0) {
        uint32_t kmin = 0xffffffffu, kmax = 0u;
        for (int h = threadIdx.x; h < H; h += kThreads) {
            const uint2 kr = a.key_range[(size_t)pair * H + h];
            kmin = min(kmin, kr.x);
            kmax = max(kmax, kr.y);
        }
        sel = select_each<kThreads>(each_key, rest, sel_sm, kmin, kmax);
        if (!sel.all_ties_in()) {
            int eq = 0;
            each_key([&](bool in, uint32_t key) { eq += in && key == sel.tau; });
            rank = block_exclusive_scan<kThreads>(eq, ties).x;
        }
    }
    // 3. the members of every run, then their places
    int mine = 0;
    each_run([&](int r, int h, int i0, int n, uint32_t taken) {
        uint32_t m = taken;
        if (!all && rest > 0) {
            float x[kRun];
            load_run<kRun>(Sp + (size_t)h * N, i0, N, x);
#pragma unroll
            for (int k = 0; k < kRun; ++k) {
                if (k < n && !((taken >> k) & 1u)) {
                    const uint32_t key = float_key(x[k]);
                    const bool eq = key == sel.tau;
                    if (key > sel.tau || (eq && rank < sel.need)) m |= 1u << k;
                    rank += eq;
                }
            }
        }
        kept_map[r] = (uint8_t)m;
        mine += __popc(m);
    });
    const int2 at = block_exclusive_scan<kThreads>(mine, offsets);
    int pos = at.x;
    const int total = at.y;
    int32_t* out = a.idx[pair];
    int32_t* counts = a.counts + (size_t)pair * H;
    for (int r = r0; r < r1; ++r) {
        const int h = r / runs, i = r - h * runs;
        if (i == 0) counts[h] = pos;  // candidates kept by the heads before h
        for (uint32_t m = kept_map[r]; m; m &= m - 1u)
            out[h * win + pos++] = kRun * i + __ffs(m) - 1;
    }
    __syncthreads();
    auto start = [&](int h) { return runs == 0 ? 0 : (h < H ? counts[h] : total); };
    for (int e = threadIdx.x; e < H * win; e += kThreads) {
        const int h = e / win, w = e - h * win;
        out[h * win + start(h + 1) + w] = N - W + w;
    }
    // starts become counts, each read before it is replaced
    for (int h0 = 0; h0 < H; h0 += kThreads) {
        const int h = h0 + (int)threadIdx.x;
        const int n = h < H ? start(h + 1) - start(h) : 0;
        __syncthreads();
        if (h < H) counts[h] = n + win;
        __syncthreads();
    }
    if (threadIdx.x == 0 && total != H * keep && a.err) atomicCAS(a.err, 0, 2);
}

// Flat per-layer gather: output row j of a pair belongs to the head whose
// segment (per-head counts, heads in order) contains it.
__global__ void __launch_bounds__(256)
gather_flat_kernel(GatherTable tab, Shape s, const int32_t* counts, int* err)
{
    wait_previous();
    const int pair = blockIdx.y;
    const int total = tab.kept[pair];  // rows of the pair
    const int cpr = s.d / 8;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = e / cpr, q = e - j * cpr;
    if (j >= total) return;
    int h = 0, start = 0;
    while (h < s.hkv - 1 && j >= start + counts[(size_t)pair * s.hkv + h]) {
        start += counts[(size_t)pair * s.hkv + h];
        ++h;
    }
    const int src = tab.idx[pair][j];
    if (src < 0 || src >= s.N) {
        if (err) atomicCAS(err, 0, 1);
        return;
    }
    const size_t in_off = ((size_t)h * s.N + src) * s.d;
    const size_t out_off = (size_t)j * s.d;
    const uint4 kv = load_input(tab.k[pair] + in_off, q);
    const uint4 vv = load_input(tab.v[pair] + in_off, q);
    reinterpret_cast<uint4*>(tab.ko[pair] + out_off)[q] = kv;
    reinterpret_cast<uint4*>(tab.vo[pair] + out_off)[q] = vv;
}

}  // namespace

cudaError_t launch_adaptive_select(const Shape& s, int keep_window, const AdaptArgs& a,
                                   cudaStream_t st)
{
    const int n_cand = s.N - (keep_window ? s.W : 0);
    const size_t sm = (size_t)s.hkv * ((n_cand + kRun - 1) / kRun);
    cudaError_t e = cudaFuncSetAttribute(adaptive_select_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    return launch_after(adaptive_select_kernel, s.units / s.hkv, kThreads, sm, st, s, keep_window,
                        a);
}

cudaError_t launch_gather_flat(const GatherTable& tab, const Shape& s, const int32_t* counts,
                               int* err, cudaStream_t st)
{
    const int pairs = s.units / s.hkv;
    int rows = 0;
    for (int p = 0; p < pairs; ++p) rows = tab.kept[p] > rows ? tab.kept[p] : rows;
    if (rows <= 0) return cudaSuccess;
    dim3 grid((rows * (s.d / 8) + 255) / 256, pairs);
    return launch_after(gather_flat_kernel, grid, 256, 0, st, tab, s, counts, err);
}

}  // namespace bacon
