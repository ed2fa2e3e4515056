// Interface of the tcgen05 window-score kernels (window_tc.cu).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "common.cuh"

namespace bacon {

// The TMA descriptors travel as kernel parameters: when the (request, layer)
// pairs' tensors follow each other at one distance (a contiguous batch, or a
// single pair) one 3-D map, whose outermost coordinate is the pair, covers
// them all, and nothing has to be copied to the device before the launch.
// Per pair it reads exactly what a map of that pair alone reads (rows beyond
// the pair's own are zero).  A table of one map per pair has to be encoded and
// copied first, and the next call waits for that copy: without it, 28 layers of
// a 6528-token prompt scored one by one took 2.35 instead of 2.64 ms (before
// the other changes to that path).  Pairs at uneven distances take the table of
// one map each.  (The maps are a parameter of their own: inside TcArgs, whose
// address would then escape, the window kernels spilled and a 4 x 16384-token
// step took 1 % longer.)
struct TcMaps {
    CUtensorMap k;  // [pairs][Hkv * N][d]
    CUtensorMap q;  // [pairs][Hq * W][d]
};

// One launch covers every (request, layer, kv-head) unit of a call.
struct TcArgs {
    const CUtensorMap* kmaps;  // device table [pairs], each one pair's K, or null (TcMaps)
    const CUtensorMap* qmaps;  // device table [pairs] of the window queries, or null (TcMaps)
    Shape s;
    int chunks;                // 1024-token chunks per unit
    int total_chunks;          // units * chunks
    int items;                 // work items of the launch (set by it)
    float2* partial;           // pass 1 output [units][chunks][rows]
    const float* lse2;         // pass 2 input  [units][rows]; null: from `partial`
    float* B;                  // pass 2 outputs [units][N]
    float* Q;
    float* E;
    int* err;                  // device error word (timeouts)
    int fault = 0;             // test-only fault injection: 1 = CTA 0 of pass 1 never
                               // issues its first K-tile load (a missing arrival)
};

constexpr int kTcChunkTokens = 1024;

// Largest G * W the tcgen05 kernels take.
int window_tc_max_rows();

// Pass 1 / pass 2 on the tensor cores, and the merge between them.
cudaError_t launch_window_stats_tc(const TcArgs& a, const TcMaps& m, cudaStream_t st);
cudaError_t launch_window_scores_tc(const TcArgs& a, const TcMaps& m, cudaStream_t st);
cudaError_t launch_window_combine(const Shape& s, int chunks, const float2* partial, float* lse2,
                                  cudaStream_t st);

// One pass over K for units whose logits fit in tensor memory (at most 32
// window rows and 1024 tokens): B, Q and E as the two passes give them,
// without the partial statistics or the merge.
bool window_onepass_fits(const Shape& s);
cudaError_t launch_window_onepass(const TcArgs& a, const TcMaps& m, cudaStream_t st);

// Per (request, layer) natural-log softmax normalisers of the window rows,
// [Hq][W] fp32, as a prefill attention kernel produces them.
struct LseTable {
    const float* lse[kMaxPairs];
};
cudaError_t launch_lse_from_prefill(const Shape& s, const LseTable& t, float* lse2,
                                    cudaStream_t st);

// Tensor map over `pairs` blocks of `rows` rows of d bf16 values, the first at
// `base`, `pair_bytes` apart (a multiple of the row's bytes, at least a
// block's, below 2^40): boxes of 64 columns x box_rows rows of one block,
// 128-byte swizzle, zero fill out of bounds.
bool encode_rows_map(CUtensorMap* out, const void* base, int d, long long rows, int pairs,
                     long long pair_bytes, int box_rows);

// Box heights of the K maps (one 128-token tile) and window-query maps.
constexpr int kTcKBoxRows = 128;
constexpr int kTcQBoxRows = 64;

}  // namespace bacon
