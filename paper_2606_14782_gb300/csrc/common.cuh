// Device helpers and launch interfaces shared by the BACON kernels (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bacon {

// Upper bound on requests * layers of one call: the per-(request, layer)
// tensor pointers travel as kernel parameters.
constexpr int kMaxPairs = 256;

// Longest prompt: the calibration kernel's largest size class (1024 threads of
// 24 positions).
constexpr int kMaxPrompt = 1024 * 24;

struct GatherTable {
    const uint16_t* k[kMaxPairs];
    const uint16_t* v[kMaxPairs];
    uint16_t* ko[kMaxPairs];
    uint16_t* vo[kMaxPairs];
    const int32_t* idx[kMaxPairs];  // [Hkv][kept] kept positions of the pair
    int kept[kMaxPairs];             // rows kept per kv-head
};

// Geometry of one call.  A "unit" is one (request, layer, kv-head); units
// are numbered ((request * layers) + layer) * kv_heads + head and the
// per-(request, layer) pointer index is unit / kv_heads.
struct Shape {
    int layers, hkv, group, d, W, N;
    int units;  // requests * layers * hkv
    int rows;   // group * W window rows per kv-head
};

// Calibration hyper-parameters (Sections 4.3-4.4).
struct Calib {
    int r, m, rho;
    float gamma, eps;
    int use_E, use_L, use_T;
    int keep_window;
    int pool;
};

// ---------------------------------------------------------------- PTX

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 2^x on the special-function unit (ex2.approx, flush-to-zero); 2^-inf = 0.
__device__ __forceinline__ float fast_exp2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}

// max(a, b, c) in one instruction.
__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Order-preserving map of a float to an unsigned key (larger float ->
// larger key), used by the radix selections, and its inverse.
__device__ __forceinline__ uint32_t float_key(float f)
{
    uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// ----------------------------------------------------------- launchers

// The kernels of one call overlap (programmatic stream serialisation): all but
// the first are launched by launch_after, their blocks may be placed while the
// kernel before them finishes, and wait before they touch global memory.
// griddepcontrol.wait returns once that one kernel has completed and its
// writes are visible; that all earlier work has completed too follows only
// because every block of every kernel of the call waits, and because the first
// kernel starts in plain stream order (launch_first).  Over a call's edges it
// would not: a caller's kernel that was itself launched programmatically may
// complete before the one in front of it, which wrote K.  For the same reason
// the last kernel of a call releases nobody early (wait_previous alone), so
// that a caller's kernel never runs beside one of the library's.
// us a pass without any overlap, with it inside the calls, and over their edges
// too: 28 layers of 6528 tokens one by one, three calls each, 1433, 1318 and
// 1130; 28 layers x 4096 tokens in one call 101, 96.6 and 93.3; one layer of
// 16384 tokens without a context 35.2, 29.1 and 27.5.
__device__ __forceinline__ void wait_previous()
{
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
// The next kernel's blocks may be placed once every block has got here.
__device__ __forceinline__ void release_next()
{
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
__device__ __forceinline__ void after_previous()
{
    wait_previous();
    release_next();
}

// Piece q of a row of the caller's K or V through the read-only path: the one
// place that uses it.  That path is defined for memory which nobody writes
// while the kernel is resident, and a kernel launched by launch_after is
// resident while the kernel before it writes, so all that the library's own
// kernels hand to one another (B, E, S, partial statistics, bitmaps, counts,
// positions) is read by ordinary loads, through pointers without __restrict__,
// which after_previous() orders.
__device__ __forceinline__ uint4 load_input(const uint16_t* row, int q)
{
    return __ldg(reinterpret_cast<const uint4*>(row) + q);
}

template <typename... P, typename... A>
cudaError_t launch(bool first, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                   cudaStream_t st, const A&... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = first ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
// A call's first kernel, and one that follows another of the same call.
template <typename... P, typename... A>
cudaError_t launch_first(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                         const A&... args)
{
    return launch(true, kernel, grid, block, smem, st, args...);
}
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                         const A&... args)
{
    return launch(false, kernel, grid, block, smem, st, args...);
}

// Calibration + selection per unit (Eqs. 5-17).  The residual of layer j of
// request rq, kv-head h is read from
//     Ering + rq * ring_req_stride + (j % ring) * hkv * N + h * N,
// which covers both the whole-step path (ring = layers: every layer kept)
// and the layer-by-layer path (ring = m + 1 slots per request).  The
// absolute layer of unit u is layer0 + (u / hkv) % layers.
struct CalibArgs {
    const float* B;      // [units][N] window score
    const float* Ering;  // residual store (see above)
    int ring;
    long long ring_req_stride;
    int layer0;
    float* S;            // [units][N] final score (written when write_S)
    float* S_copy = nullptr;  // optional [units][N], 16-byte aligned: S once more
    float* V;            // optional [units][N]
    float* Bp;           // optional [units][N]
    float* lambda;       // [units]
    int32_t* idx[kMaxPairs];     // per (request, layer): [Hkv][kept] (written when do_select)
    int budget[kMaxPairs];       // kept tokens per head (window included)
    int calib_budget[kMaxPairs]; // budget that sets K in Eq. 12
    long long idx_variant_stride = 0;  // sweep only: elements between variants' indices
    // adaptive head budgets (taken null otherwise; do_select is 0 then): each
    // unit's `guaranteed` best candidates as a bitmap of positions,
    // taken_stride bytes per unit, and the range of its candidates' keys
    uint8_t* taken = nullptr;
    int taken_stride = 0;
    int guaranteed = 0;
    uint2* key_range = nullptr;
    int compute_scores;  // 1: V, B~, lambda, S from B and the residuals; 0: the call's only kernel
    int do_select;       // 1: top-B selection into idx
    int write_S;
    int* err;
};
cudaError_t launch_calibrate_select(const Shape& s, const Calib& c, const CalibArgs& a,
                                    cudaStream_t st);

// Ablation / sensitivity sweep: every unit under each of `variants`
// hyper-parameter sets (compute_scores and do_select must be 1, write_S 0,
// V and Bp null).
constexpr int kMaxVariants = 32;
struct CalibTable {
    Calib c[kMaxVariants];
};
// What the variants share (the launch fills the rho lists).
struct SweepArgs {
    float* pooled;    // [units][N] pooled backbone
    uint8_t* maps;    // [rhos][units] bitmaps of the M members, map_stride bytes each
    int map_stride;
    float2* moments;  // [rhos][units] B~'s moment sums over them
    int rhos;
    int rho[kMaxVariants];     // the distinct values
    int rho_of[kMaxVariants];  // each variant's place among them
};
cudaError_t launch_calibrate_sweep(const Shape& s, const CalibTable& t, int variants,
                                   SweepArgs sw, const CalibArgs& a, cudaStream_t st);

// AdaKV-style selection over the heads of each (request, layer), after the
// calibration has marked each head's guaranteed candidates.
struct AdaptArgs {
    const float* S;              // [units][N] final scores (0 off-candidates)
    const uint8_t* taken;        // CalibArgs' bitmap, taken_stride bytes per unit
    int taken_stride;
    const uint2* key_range;      // [units]
    int budget;                  // average per-head budget (window included)
    int guaranteed;              // g = floor(alpha K) candidates per head first
    int32_t* idx[kMaxPairs];     // per pair: flat [Hkv * kept] positions, heads in order
    int32_t* counts;             // [pairs][Hkv] kept per head (window included)
    int* err;
};
cudaError_t launch_adaptive_select(const Shape& s, int keep_window, const AdaptArgs& a,
                                   cudaStream_t st);
// Most candidates of one (request, layer), over its kv-heads, that the
// adaptive selection takes.
constexpr int kMaxAdaptive = 200 * 1024;
// Gather into the flat per-layer layout of the adaptive selection.
cudaError_t launch_gather_flat(const GatherTable& tab, const Shape& s, const int32_t* counts,
                               int* err, cudaStream_t st);

// Gather of the kept K/V rows (kept counts may differ between pairs); `first`:
// nothing of the same call comes before it.
cudaError_t launch_gather(const GatherTable& tab, const Shape& s, int* err, cudaStream_t st,
                          bool first = false);

}  // namespace bacon
