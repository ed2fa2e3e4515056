// Calibration and selection, one CTA per (request, layer, kv-head):
//   V = E + L + T                (Sec. 4.3, Eqs. 5-11)
//   B~ = max-pool of B over the candidates
//   M = min(rho K, |I|), the M best candidates by B~, lambda =
//       gamma Std(B~) / (Std(V) + eps) over them      (Sec. 4.4, Eqs. 12-15)
//   S = B~ + lambda V                                 (Eq. 16)
//   the K best candidates by S, ascending, then the window (Eq. 17)
// Both "best k" sets use one order: larger value first, equal values ->
// lower position first.  A range-adaptive radix select (select.cuh) finds
// the k-th best key and how many of the keys equal to it are taken; the
// members are then decided thread by thread in position order.
//
// Each thread owns PER consecutive positions, [t PER, t PER + PER), and
// keeps them in registers: the pooled backbone and then the final score (the
// keys of the two selections), and V.  The windows' neighbours come from the
// adjacent lanes' runs by warp shuffles (from global memory at a warp's two
// ends), and position order is (thread, slot) order, so one block-wide
// exclusive scan gives every thread its tie rank or its output offset.
//
// A unit is bound by latency: 15 dependent rounds of a block barrier each (6
// per selection, 2 sums, 1 scan; one more per selection whose last ties are
// split), one CTA per unit and at most one or two CTAs' worth of warps per SM.
// Keys in registers take the passes over all of them off shared memory, the
// boundary bin's keys are ranked by counting instead of a second histogram
// and a warp's sort, every warp finishes the block reductions itself (one
// barrier each instead of three), and runs of 8 positions load B and every
// residual they need at once.  With a shared-memory array of keys, two
// histogram passes and about 30 barriers: 110 -> 77 us (448 units x 16384
// tokens), 25 -> 17.5 (112 x 6528), 21 -> 14 (112 x 4096), 24 -> 14 (1024 x
// 1024).
//
// The standard deviations are fp32 sums over the members: B~'s moments
// about the M-th value (one walk), V's mean and then its squared
// deviations from it (two walks); neither loses precision to cancellation.
#include "common.cuh"
#include "select.cuh"

namespace bacon {
namespace {

using namespace sel;

// Threads per CTA and positions per thread depend on the prompt length only
// (so that every call on the same shape reduces in the same order and gives
// the same bits), sized so that threads x positions stays close to N: 8
// positions per thread on 128, 256, 512 or 1024 threads up to 1024, 2048,
// 4096 or 8192 tokens (several CTAs share an SM below 1024 threads), then
// 1024 threads of 16 positions up to 16384 tokens and of 24 up to kMaxPrompt.

// Block-wide fp32 sums of NV values in one round, by a shuffle tree (pairwise,
// so the rounding error grows with log2 of the count).  Every warp reduces
// the warps' sums itself, so a round costs one block barrier; `red` holds
// NV x 32 floats and is not used again before the next barrier.  FP64 is
// avoided: its rate on this part is a small fraction of fp32.
template <int T, int NV>
__device__ __forceinline__ void block_sums(float (&v)[NV], float* red)
{
    constexpr int kWarps = T / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) red[32 * i + warp] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = lane < kWarps ? red[32 * i + lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
}

// dst[i0 + k] = x[k] for the positions below n.
template <int PER>
__device__ __forceinline__ void store_run(float* dst, int i0, int n, const float* x)
{
    if ((n & 3) == 0 && i0 + PER <= n) {
        float4* d4 = reinterpret_cast<float4*>(dst + i0);
#pragma unroll
        for (int q = 0; q < PER / 4; ++q)
            d4[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (i0 + k < n) dst[i0 + k] = x[k];
    }
}

// Membership of the thread's candidates (its first nv slots) in the k best
// (bit k of the result): key > tau, or key == tau among the first `need` such
// keys in position order.  eq_before = keys equal to tau at lower positions
// (other threads).
template <int PER>
__device__ __forceinline__ uint32_t members(const float* x, int nv, const SelectResult& sel,
                                            int eq_before)
{
    uint32_t m = 0u;
    int rank = eq_before;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (k < nv) {
            const uint32_t key = float_key(x[k]);
            const bool eq = key == sel.tau;
            if (key > sel.tau || (eq && rank < sel.need)) m |= 1u << k;
            rank += eq;
        }
    }
    return m;
}

// Keys equal to tau at lower positions than this thread's run (0 without a
// scan when every tie is taken: membership then never needs the rank).
template <int T, int PER>
__device__ __forceinline__ int ties_before(const float* x, int nv, const SelectResult& sel,
                                           int* warp_sums)
{
    if (sel.all_ties_in()) return 0;
    int eq = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) eq += k < nv && float_key(x[k]) == sel.tau;
    return block_exclusive_scan<T>(eq, warp_sums).x;
}

// The residual E of the thread's run (x, 0 at and past N), added to v when
// use_E, and the coherence (Eqs. 5-7) with the radius R a constant:
// v[k] += the mean of E over [i - R, i + R] clipped to [0, N), for the run's
// positions i = i0 + k < N.  The R values on either side come from the
// neighbouring lanes' runs by shuffles (from global memory at a warp's two
// ends, loaded together with the run) and count as 0 outside [0, N).  The
// window sum slides along the run: drop i - R, add i + 1 + R.  Needs
// R <= PER and every lane of the warp.
template <int PER, int R>
__device__ __forceinline__ void coherence_run(const float* Ec, int i0, int N,
                                              bool use_E, const float* x, float* v)
{
    static_assert(R <= PER, "the halo must come from the adjacent run");
    const int lane = threadIdx.x & 31;
    float gl[R], gh[R];
#pragma unroll
    for (int m = 0; m < R; ++m) {
        const int jl = i0 - R + m, jh = i0 + PER + m;
        gl[m] = (lane == 0 && jl >= 0 && jl < N) ? Ec[jl] : 0.f;
        gh[m] = (lane == 31 && jh < N) ? Ec[jh] : 0.f;
    }
    if (use_E) {
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] += x[k];
    }
    float e[PER + 2 * R];
#pragma unroll
    for (int m = 0; m < R; ++m) {
        const int jl = i0 - R + m, jh = i0 + PER + m;
        const float lo = __shfl_up_sync(0xffffffffu, x[PER - R + m], 1);
        const float hi = __shfl_down_sync(0xffffffffu, x[m], 1);
        e[m] = lane == 0 ? gl[m] : (jl >= 0 ? lo : 0.f);
        e[R + PER + m] = lane == 31 ? gh[m] : (jh < N ? hi : 0.f);
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) e[R + k] = x[k];
    const float inv_full = 1.f / (float)(2 * R + 1);  // windows away from the ends
    float sum = 0.f;
#pragma unroll
    for (int j = 0; j <= 2 * R; ++j) sum += e[j];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = i0 + k;
        if (i < N) {
            const int cnt = min(N - 1, i + R) - max(0, i - R) + 1;
            float w = inv_full;
            if (cnt != 2 * R + 1) w = 1.f / (float)cnt;
            // the window sum of non-negative values: rounding in the slide
            // can leave ~1e-9 below zero after a large value leaves the
            // window, so it is clamped
            v[k] += fmaxf(sum, 0.f) * w;
        }
        if (k + 1 < PER) {
            sum -= e[k];
            sum += e[k + 2 * R + 1];
        }
    }
}

// The same for any radius, reading the window from global memory (L1).
template <int PER>
__device__ __forceinline__ void coherence_any(const float* Ec, int i0, int N, int r,
                                              float* v)
{
    const float inv_full = 1.f / (float)(2 * r + 1);
    int lo = max(0, i0 - r), hi = min(N - 1, i0 + r);
    float sum = 0.f;
    for (int j = lo; j <= hi; ++j) sum += Ec[j];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = i0 + k;
        if (i < N) {
            const int cnt = hi - lo + 1;
            v[k] += fmaxf(sum, 0.f) * (cnt == 2 * r + 1 ? inv_full : 1.f / (float)cnt);
            if (i - r >= 0) sum -= Ec[i - r];
            if (i + 1 + r <= N - 1) sum += Ec[i + 1 + r];
            lo = max(0, i + 1 - r);
            hi = min(N - 1, i + 1 + r);
        }
    }
}

// Whether the run with its halo (PER + 2 R floats) and V (PER floats) fit
// in the 64 registers a thread has, with room for the rest.
__host__ __device__ constexpr bool run_fits(int PER, int R) { return R <= PER && 2 * PER + 2 * R <= 56; }

// E (added to v when use_E) and its coherence, with the paper's radii (3, 5,
// 7, 9) compiled as constants where the registers allow.
template <int PER>
__device__ __forceinline__ void residual_and_coherence(const float* Ec, int i0, int N,
                                                       int r, bool use_E, const float* x, float* v)
{
    if constexpr (run_fits(PER, 3))
        if (r == 3) return coherence_run<PER, 3>(Ec, i0, N, use_E, x, v);
    if constexpr (run_fits(PER, 5))
        if (r == 5) return coherence_run<PER, 5>(Ec, i0, N, use_E, x, v);
    if constexpr (run_fits(PER, 7))
        if (r == 7) return coherence_run<PER, 7>(Ec, i0, N, use_E, x, v);
    if constexpr (run_fits(PER, 9))
        if (r == 9) return coherence_run<PER, 9>(Ec, i0, N, use_E, x, v);
    if (use_E) {
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] += x[k];
    }
    coherence_any<PER>(Ec, i0, N, r, v);
}

// The residuals that a unit reads: layer l's row is at base + (l % ring) *
// layer_stride.
struct Residuals {
    const float* base;
    long long layer_stride;
    int ring;
    __device__ __forceinline__ const float* row(int l) const
    {
        return base + (long long)(l % ring) * layer_stride;
    }
};

__device__ __forceinline__ Residuals residuals_of(const CalibArgs& a, const Shape& s, int rq, int h)
{
    return {a.Ering + (long long)rq * a.ring_req_stride + (long long)h * s.N,
            (long long)s.hkv * s.N, a.ring};
}

// v += the runs of layers [l0, l0 + n), in layer order; AHEAD layers' loads
// are in flight together.
template <int PER, int AHEAD>
__device__ __forceinline__ void add_layers(const Residuals& E, int l0, int n, int i0, int N,
                                           float* v)
{
    int slot = l0 % E.ring;
    if ((N & 3) == 0 && i0 + PER <= N) {
#pragma unroll AHEAD
        for (int j = 0; j < n; ++j) {
            const float4* p = reinterpret_cast<const float4*>(E.base + slot * E.layer_stride + i0);
#pragma unroll
            for (int q = 0; q < PER / 4; ++q) {
                const float4 e = p[q];
                v[4 * q] += e.x;
                v[4 * q + 1] += e.y;
                v[4 * q + 2] += e.z;
                v[4 * q + 3] += e.w;
            }
            if (++slot == E.ring) slot = 0;
        }
    } else {
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            const float* p = E.base + slot * E.layer_stride;
#pragma unroll
            for (int k = 0; k < PER; ++k)
                if (i0 + k < N) v[k] += p[i0 + k];
            if (++slot == E.ring) slot = 0;
        }
    }
}

// The evidence V = E + L + T of the thread's run (Eqs. 5-11) into v, 0 at and
// past N; x: the run of the layer's own residuals, at Ec (runs of 8: loaded
// by the caller, ahead of the layers before).
template <int PER>
__device__ __forceinline__ void evidence_run(const Calib& c, const Residuals& E, int layer, int i0,
                                             int N, const float* Ec, float* x,
                                             float* v)
{
#pragma unroll
    for (int k = 0; k < PER; ++k) v[k] = 0.f;
    // persistence: mean of E over the preceding min(m, l) layers (Eqs. 8-9)
    if (c.use_T) {
        const int nprev = min(c.m, layer);
        const float inv_prev = nprev > 0 ? 1.f / (float)nprev : 0.f;
        add_layers<PER, (PER <= 8 ? 4 : (PER <= 16 ? 2 : 1))>(E, layer - nprev, nprev, i0, N, v);
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] *= inv_prev;
    }
    // E, and the coherence: truncated radius-r box mean of E (Eqs. 5-7)
    if (PER > 8) load_run<PER>(Ec, i0, N, x);
    if (c.use_L) {
        residual_and_coherence<PER>(Ec, i0, N, c.r, c.use_E, x, v);
    } else if (c.use_E) {
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] += x[k];
    }
#pragma unroll
    for (int k = 0; k < PER; ++k)
        if (i0 + k >= N) v[k] = 0.f;
}

// The pooled backbone of the thread's run (max over [i - half, i + half] of
// the candidates, 0 past them) from Bu's run in b, in place; the key range of
// the candidates goes to kmin, kmax.
template <int PER>
__device__ __forceinline__ void pool_run(const float* Bu, int i0, int n_cand, int half,
                                         float* b, uint32_t& kmin, uint32_t& kmax)
{
    float p[PER];
    if (half == 3) {
        // width 7 (the default): the run and three positions either side in
        // registers (-inf outside the candidates; the neighbours' values by
        // shuffles, from global memory at a warp's two ends), each output a
        // maximum of seven by three max3
        const int lane = threadIdx.x & 31;
        float hl[3], hr[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int jl = i0 - 3 + m, jr = i0 + PER + m;
            hl[m] = (lane == 0 && jl >= 0 && jl < n_cand) ? Bu[jl] : -INFINITY;
            hr[m] = (lane == 31 && jr < n_cand) ? Bu[jr] : -INFINITY;
        }
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (i0 + k >= n_cand) b[k] = -INFINITY;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const float lo = __shfl_up_sync(0xffffffffu, b[PER - 3 + m], 1);
            const float hi = __shfl_down_sync(0xffffffffu, b[m], 1);
            if (lane != 0) hl[m] = lo;
            if (lane != 31) hr[m] = hi;
        }
        auto at = [&](int j) -> float { return j < 0 ? hl[j + 3] : (j >= PER ? hr[j - PER] : b[j]); };
#pragma unroll
        for (int k = 0; k < PER; ++k)
            p[k] = max3f(max3f(at(k - 3), at(k - 2), at(k - 1)), max3f(at(k), at(k + 1), at(k + 2)),
                         at(k + 3));
    } else {
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int i = i0 + k;
            p[k] = -INFINITY;
            if (i < n_cand) {
                const int lo = max(0, i - half), hi = min(n_cand - 1, i + half);
                for (int v = lo; v <= hi; ++v) p[k] = fmaxf(p[k], Bu[v]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        b[k] = 0.f;
        if (i0 + k < n_cand) {
            b[k] = p[k];
            kmin = min(kmin, float_key(p[k]));
            kmax = max(kmax, float_key(p[k]));
        }
    }
}

// lambda over the M members (Eqs. 13-15): sx and syy are B~'s moment sums
// about the M-th value (every member is at or above it, so the fp32
// differences stay small), sv the members' sum of V, whose mean square
// deviation from its mean takes one more reduction.
template <int T, int PER>
__device__ __forceinline__ float lambda_of(const Calib& c, int M, uint32_t mem, float sx, float syy,
                                           float sv, const float* v, float* red)
{
    const float inv_m = 1.f / (float)M;
    const float mb = sx * inv_m, mv = sv * inv_m;
    float dev[1] = {0.f};
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if ((mem >> k) & 1u) {
            const float dv = v[k] - mv;
            dev[0] = fmaf(dv, dv, dev[0]);
        }
    }
    block_sums<T, 1>(dev, red);
    const float varv = dev[0] * inv_m;
    const float stdb = sqrtf(fmaxf(syy * inv_m - mb * mb, 0.f));
    const float stdv = sqrtf(varv);
    return c.gamma * stdb / (stdv + c.eps);
}

// Eq. 17's output: the members (`mem`, `keep` of them in all), ascending,
// then the window.
template <int T, int PER>
__device__ __forceinline__ void emit(uint32_t mem, int i0, int n_cand, int keep, int win, int N,
                                     int* offsets, int32_t* out, int* err)
{
    if (keep >= n_cand) {
        for (int i = threadIdx.x; i < n_cand; i += T) out[i] = i;
    } else if (keep > 0) {
        const int2 at = block_exclusive_scan<T>(__popc(mem), offsets);
        int pos = at.x;
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if ((mem >> k) & 1u) out[pos++] = i0 + k;
        if (threadIdx.x == 0 && at.y != keep && err) atomicCAS(err, 0, 2);
    }
    for (int w = threadIdx.x; w < win; w += T) out[keep + w] = N - win + w;
}

// M of Eq. 12 for a pair's budget.
__device__ __forceinline__ int match_count(int rho, int budget, int N, int win, int n_cand)
{
    const int calib_keep = min(budget, N) - win;
    const long long M = (long long)rho * (long long)(calib_keep > 0 ? calib_keep : 0);
    return (int)(M < n_cand ? M : n_cand);
}

// One unit (request, layer, kv-head) u under hyper-parameters c.  lam_out
// (may be null) receives lambda; idx_pair is the pair's [Hkv][kept] output.
// N <= T PER.  The thread's run of the pooled backbone (then of the final
// score: the keys of the two selections) stays in registers, and so does V
// where a run is 8 positions; longer runs park V in the thread's own column
// of shared memory while the first selection needs the registers.  The two
// selections are two turns of one loop, so that the second finds its code in
// the instruction cache.
// ADAPT: the head's guaranteed share and its key range for the adaptive
// selection take the place of Eq. 17.
template <int T, int PER, bool ADAPT>
__device__ __forceinline__ void calibrate_unit(const Shape& s, const Calib& c, const CalibArgs& a,
                                               int u, float* lam_out, int32_t* idx_pair)
{
    constexpr bool kPark = PER > 8;
    extern __shared__ __align__(16) float sm[];  // kPark: [PER][T]
    __shared__ SelectScratch<T> sel_sm;
    __shared__ int ties[2][32], offsets[32];
    __shared__ float red_b[3 * 32], red_v[32];

    const int N = s.N, W = s.W;
    const int pair = u / s.hkv, h = u - pair * s.hkv;
    const int rq = pair / s.layers;
    const int layer = a.layer0 + (pair - rq * s.layers);
    const int win = c.keep_window ? W : 0;
    const int n_cand = N - win;
    const int kept_total = min(a.budget[pair], N);
    const int keep = kept_total - win;
    const int i0 = (int)threadIdx.x * PER;
    const int nv = max(0, min(PER, n_cand - i0));  // this thread's candidates

    float b[PER];  // pooled backbone B~, then the final score S
    float v[PER];  // evidence V
    uint32_t kmin = 0xffffffffu, kmax = 0u;  // range of b's keys over the candidates
    int M = 0;
    if (a.compute_scores) {
        // (runs of 8: B, the residuals and then the layers before are in
        // flight together)
        const float* Bu = a.B + (size_t)u * N;
        if (!kPark) load_run<PER>(Bu, i0, N, b);
        {
            float x[PER];
            const Residuals E = residuals_of(a, s, rq, h);
            const float* Ec = E.row(layer);
            if (!kPark) load_run<PER>(Ec, i0, N, x);
            evidence_run<PER>(c, E, layer, i0, N, Ec, x, v);
        }
        if (a.V) store_run<PER>(a.V + (size_t)u * N, i0, N, v);
        if (kPark) {
#pragma unroll
            for (int k = 0; k < PER; ++k) sm[k * T + threadIdx.x] = v[k];
        }
        if (kPark) load_run<PER>(Bu, i0, N, b);
        pool_run<PER>(Bu, i0, n_cand, c.pool / 2, b, kmin, kmax);
        if (a.Bp) store_run<PER>(a.Bp + (size_t)u * N, i0, N, b);
        M = match_count(c.rho, a.calib_budget[pair], N, win, n_cand);
    } else {
        load_run<PER>(a.S + (size_t)u * N, i0, N, b);
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            if (k < nv) {
                kmin = min(kmin, float_key(b[k]));
                kmax = max(kmax, float_key(b[k]));
            }
        }
    }

    // turn 0: the M best candidates by B~ (Eq. 12), lambda, S; turn 1: the
    // best by S
#pragma unroll 1
    for (int turn = a.compute_scores ? 0 : 1; turn < 2; ++turn) {
        int k_best = M;
        if (turn == 1) {
            if (!ADAPT && !a.do_select) return;
            k_best = ADAPT ? min(a.guaranteed, keep) : keep;
            if (keep >= n_cand) k_best = 0;  // every candidate is kept
        }
        uint32_t mem = 0u;
        float pb = 0.f;
        if (k_best > 0) {
            const SelectResult sel = select_runs<T, PER>(b, nv, k_best, sel_sm, kmin, kmax);
            mem = members<PER>(b, nv, sel, ties_before<T, PER>(b, nv, sel, ties[turn]));
            pb = key_float(sel.tau);
        }
        if (turn == 0) {
            if (kPark) {
#pragma unroll
                for (int k = 0; k < PER; ++k) v[k] = sm[k * T + threadIdx.x];
            }
            // lambda over the M members (Eqs. 13-15)
            float lam = 0.f;
            if (M > 0) {
                float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < PER; ++k) {
                    if ((mem >> k) & 1u) {
                        const float db = b[k] - pb;
                        acc[0] += db;
                        acc[1] = fmaf(db, db, acc[1]);
                        acc[2] += v[k];
                    }
                }
                block_sums<T, 3>(acc, red_b);
                lam = lambda_of<T, PER>(c, M, mem, acc[0], acc[1], acc[2], v, red_v);
            }
            if (threadIdx.x == 0 && lam_out) *lam_out = lam;
            // Eq. 16 over the candidates (0 elsewhere)
            kmin = 0xffffffffu;
            kmax = 0u;
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                if (k < nv) {
                    b[k] = fmaf(lam, v[k], b[k]);
                    kmin = min(kmin, float_key(b[k]));
                    kmax = max(kmax, float_key(b[k]));
                }
            }
            if (a.write_S) store_run<PER>(a.S + (size_t)u * N, i0, N, b);
            if (a.S_copy) store_run<PER>(a.S_copy + (size_t)u * N, i0, N, b);
        } else if constexpr (ADAPT) {
            // the head's own best candidates as a bitmap of positions, and the
            // key range of its scores
            if (keep >= n_cand) mem = (1u << nv) - 1u;
            uint8_t* map = a.taken + (size_t)u * a.taken_stride;
#pragma unroll
            for (int q = 0; q < PER / 8; ++q)
                if (i0 + 8 * q < n_cand) map[i0 / 8 + q] = (uint8_t)(mem >> (8 * q));
            __shared__ uint32_t ranges[2][32];
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            kmin = __reduce_min_sync(0xffffffffu, kmin);
            kmax = __reduce_max_sync(0xffffffffu, kmax);
            if (lane == 0) {
                ranges[0][warp] = kmin;
                ranges[1][warp] = kmax;
            }
            __syncthreads();
            if (warp == 0) {
                kmin = __reduce_min_sync(0xffffffffu, lane < T / 32 ? ranges[0][lane] : 0xffffffffu);
                kmax = __reduce_max_sync(0xffffffffu, lane < T / 32 ? ranges[1][lane] : 0u);
                if (lane == 0) a.key_range[u] = make_uint2(kmin, kmax);
            }
        } else {
            emit<T, PER>(mem, i0, n_cand, keep, win, N, offsets, idx_pair + (size_t)h * kept_total,
                         a.err);
        }
    }
}

template <int T, int PER, bool ADAPT>
__global__ void __launch_bounds__(T, 1024 / T)
calibrate_select_kernel(Shape s, Calib c, CalibArgs a)
{
    wait_previous();
    if (ADAPT || (a.compute_scores && a.do_select)) release_next();  // not the call's last
    const int u = blockIdx.x;
    calibrate_unit<T, PER, ADAPT>(s, c, a, u, a.lambda + u, a.idx[u / s.hkv]);
}

// Several hyper-parameter sets over the same B and residuals, in two kernels.
// What the variants of a unit share is formed once: the pooled backbone, and
// per distinct rho the M best by it (a bitmap of positions, position order =
// bit order) with B~'s moment sums over them.  CTA (u, v) then runs unit u
// under variant v from there; variant v's indices start v *
// idx_variant_stride elements after the single-variant layout and its
// lambdas v * units after a.lambda.  Both are bound by latency like the
// kernel above: 11 variants of 112 units x 6528 tokens take 87 us, where
// every (unit, variant) repeating the shared part took 125.
template <int T, int PER>
__global__ void __launch_bounds__(T, 1024 / T)
sweep_shared_kernel(Shape s, Calib c, SweepArgs sw, CalibArgs a)
{
    __shared__ SelectScratch<T> sel_sm;
    __shared__ int ties[32];
    __shared__ float red[2 * 32];
    after_previous();
    const int u = blockIdx.x, ri = blockIdx.y;
    const int N = s.N, win = c.keep_window ? s.W : 0, n_cand = N - win;
    const int i0 = (int)threadIdx.x * PER;
    const int nv = max(0, min(PER, n_cand - i0));
    const float* Bu = a.B + (size_t)u * N;
    float b[PER];
    load_run<PER>(Bu, i0, N, b);
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    pool_run<PER>(Bu, i0, n_cand, c.pool / 2, b, kmin, kmax);
    if (ri == 0) store_run<PER>(sw.pooled + (size_t)u * N, i0, N, b);
    const int M = match_count(sw.rho[ri], a.calib_budget[u / s.hkv], N, win, n_cand);
    if (M <= 0) return;
    const SelectResult sel = select_runs<T, PER>(b, nv, M, sel_sm, kmin, kmax);
    const uint32_t mem = members<PER>(b, nv, sel, ties_before<T, PER>(b, nv, sel, ties));
    const float pb = key_float(sel.tau);
    float acc[2] = {0.f, 0.f};
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if ((mem >> k) & 1u) {
            const float db = b[k] - pb;
            acc[0] += db;
            acc[1] = fmaf(db, db, acc[1]);
        }
    }
    uint8_t* map = sw.maps + ((size_t)ri * s.units + u) * sw.map_stride;
#pragma unroll
    for (int q = 0; q < PER / 8; ++q)
        if (i0 + 8 * q < n_cand) map[i0 / 8 + q] = (uint8_t)(mem >> (8 * q));
    block_sums<T, 2>(acc, red);
    if (threadIdx.x == 0) sw.moments[(size_t)ri * s.units + u] = make_float2(acc[0], acc[1]);
}

template <int T, int PER>
__global__ void __launch_bounds__(T, 1024 / T)
calibrate_sweep_kernel(Shape s, CalibTable t, SweepArgs sw, CalibArgs a)
{
    __shared__ SelectScratch<T> sel_sm;
    __shared__ int ties[32], offsets[32];
    __shared__ float red_s[32], red_v[32];
    wait_previous();
    const int u = blockIdx.x, j = blockIdx.y;
    const Calib& c = t.c[j];
    const int N = s.N, win = c.keep_window ? s.W : 0, n_cand = N - win;
    const int pair = u / s.hkv, h = u - pair * s.hkv;
    const int rq = pair / s.layers;
    const int layer = a.layer0 + (pair - rq * s.layers);
    const int kept_total = min(a.budget[pair], N);
    const int i0 = (int)threadIdx.x * PER;
    const int nv = max(0, min(PER, n_cand - i0));
    const int ri = sw.rho_of[j];
    const int M = match_count(c.rho, a.calib_budget[pair], N, win, n_cand);
    uint32_t mem = 0u;
    if (M > 0) {
        const uint8_t* map = sw.maps + ((size_t)ri * s.units + u) * sw.map_stride;
#pragma unroll
        for (int q = 0; q < PER / 8; ++q)
            if (i0 + 8 * q < n_cand) mem |= (uint32_t)map[i0 / 8 + q] << (8 * q);
    }
    float x[PER], v[PER], b[PER];
    const Residuals E = residuals_of(a, s, rq, h);
    const float* Ec = E.row(layer);
    if (PER <= 8) {
        load_run<PER>(sw.pooled + (size_t)u * N, i0, N, b);
        load_run<PER>(Ec, i0, N, x);
    }
    evidence_run<PER>(c, E, layer, i0, N, Ec, x, v);
    if (PER > 8) load_run<PER>(sw.pooled + (size_t)u * N, i0, N, b);
    float lam = 0.f;
    if (M > 0) {
        float sv[1] = {0.f};
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if ((mem >> k) & 1u) sv[0] += v[k];
        const float2 mo = sw.moments[(size_t)ri * s.units + u];
        block_sums<T, 1>(sv, red_s);
        lam = lambda_of<T, PER>(c, M, mem, mo.x, mo.y, sv[0], v, red_v);
    }
    if (threadIdx.x == 0 && a.lambda) a.lambda[(size_t)j * s.units + u] = lam;
    uint32_t skmin = 0xffffffffu, skmax = 0u;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (k < nv) {
            b[k] = fmaf(lam, v[k], b[k]);
            skmin = min(skmin, float_key(b[k]));
            skmax = max(skmax, float_key(b[k]));
        }
    }
    const int keep = kept_total - win;
    mem = 0u;
    if (keep > 0 && keep < n_cand) {
        const SelectResult sel = select_runs<T, PER>(b, nv, keep, sel_sm, skmin, skmax);
        mem = members<PER>(b, nv, sel, ties_before<T, PER>(b, nv, sel, ties));
    }
    emit<T, PER>(mem, i0, n_cand, keep, win, N, offsets,
                 a.idx[pair] + (size_t)j * a.idx_variant_stride + (size_t)h * kept_total, a.err);
}

template <int T, int PER>
constexpr size_t smem_bytes()
{
    return PER > 8 ? (size_t)T * PER * sizeof(float) : 0;
}

template <int T, int PER, bool ADAPT>
cudaError_t launch_select_t(const Shape& s, const Calib& c, const CalibArgs& a, cudaStream_t st)
{
    constexpr size_t sm = smem_bytes<T, PER>();
    cudaError_t e = cudaFuncSetAttribute(calibrate_select_kernel<T, PER, ADAPT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    return launch(!a.compute_scores, calibrate_select_kernel<T, PER, ADAPT>, s.units, T, sm, st, s,
                  c, a);
}

template <int T, int PER>
cudaError_t launch_sweep_t(const Shape& s, const CalibTable& t, int variants, const SweepArgs& sw,
                           const CalibArgs& a, cudaStream_t st)
{
    cudaError_t e = launch_after(sweep_shared_kernel<T, PER>, dim3(s.units, sw.rhos), T, 0, st, s,
                                 t.c[0], sw, a);
    if (e != cudaSuccess) return e;
    return launch_after(calibrate_sweep_kernel<T, PER>, dim3(s.units, variants), T, 0, st, s, t, sw,
                        a);
}

// The launch for a prompt of N tokens: F(T, PER) with the size class above.
template <typename F>
cudaError_t by_size(int N, F f)
{
    if (N <= 1024) return f.template run<128, 8>();
    if (N <= 2048) return f.template run<256, 8>();
    if (N <= 4096) return f.template run<512, 8>();
    if (N <= 8192) return f.template run<1024, 8>();
    if (N <= 16384) return f.template run<1024, 16>();
    if (N <= 1024 * 24) return f.template run<1024, 24>();
    static_assert(kMaxPrompt == 1024 * 24, "the largest size class");
    return cudaErrorInvalidValue;
}

struct SelectLaunch {
    const Shape& s;
    const Calib& c;
    const CalibArgs& a;
    cudaStream_t st;
    template <int T, int PER>
    cudaError_t run() const
    {
        return a.taken ? launch_select_t<T, PER, true>(s, c, a, st)
                       : launch_select_t<T, PER, false>(s, c, a, st);
    }
};

struct SweepLaunch {
    const Shape& s;
    const CalibTable& t;
    int variants;
    const SweepArgs& sw;
    const CalibArgs& a;
    cudaStream_t st;
    template <int T, int PER>
    cudaError_t run() const { return launch_sweep_t<T, PER>(s, t, variants, sw, a, st); }
};

}  // namespace

cudaError_t launch_calibrate_select(const Shape& s, const Calib& c, const CalibArgs& a,
                                    cudaStream_t st)
{
    return by_size(s.N, SelectLaunch{s, c, a, st});
}

cudaError_t launch_calibrate_sweep(const Shape& s, const CalibTable& t, int variants,
                                   SweepArgs sw, const CalibArgs& a, cudaStream_t st)
{
    sw.rhos = 0;
    for (int j = 0; j < variants; ++j) {
        int r = 0;
        while (r < sw.rhos && sw.rho[r] != t.c[j].rho) ++r;
        if (r == sw.rhos) sw.rho[sw.rhos++] = t.c[j].rho;
        sw.rho_of[j] = r;
    }
    return by_size(s.N, SweepLaunch{s, t, variants, sw, a, st});
}

}  // namespace bacon
