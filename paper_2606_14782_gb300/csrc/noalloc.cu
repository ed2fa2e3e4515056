// Window scores of one layer without any device allocation.
//
// Some callers cannot call cudaMalloc: a serving engine that reserves all of
// HBM for its KV cache up front and forbids side allocations, or code that
// must not pay the implicit device-wide synchronisation of cudaMalloc /
// cudaFree in the middle of prefill.  For them, bacon_window_scores_noalloc
// runs the same window kernels as the context-based calls, but keeps
// their scratch (pass-1 partial statistics) in one file-scope __device__
// array instead of context-owned buffers.
//
// The call returns before its kernels run, so a device-side failure (a
// bounded pipeline wait that ran out) cannot come back as its status.  The
// same array holds an error word for that: the window kernels latch a timeout
// in it, and a last small kernel, when it is set, fills B, Q and E with NaN
// and clears it, so that a caller never reads partial scores as
// valid ones.
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "bacon.h"
#include "common.cuh"
#include "window_tc.h"

using namespace bacon;

namespace {

constexpr int kMaxTotalRows = 4096;   // kv_heads * (q_heads / kv_heads) * window
constexpr int kMaxSeq = 16384;        // tokens per call
constexpr int kChunk = 1024;          // pass-1 token chunk, as in the context path
constexpr int kMaxChunks = kMaxSeq / kChunk;
constexpr int kMaxDevices = 64;

constexpr int kErrSlots = 2;          // 16 bytes holding the error word

// [units][chunks][rows] partial (max, sum) pairs, then the device error word.
// About 512 KiB, held by every GPU that loads the library until the process
// exits.
static __device__ __align__(256) float2 g_scratch[kMaxTotalRows * kMaxChunks + kErrSlots];

std::mutex g_setup_mutex;
void* g_scratch_addr[kMaxDevices] = {};

// Test-only fault injection: when BACON_FAULT=missing_arrival is set at the
// first call of the process, that call's pass 1 withholds one K-tile load,
// so its bounded waits run out (nothing faults).  -1 = not read yet.
std::atomic<int> g_fault_pending{-1};

int take_fault()
{
    int s = g_fault_pending.load();
    if (s < 0) {
        const char* f = std::getenv("BACON_FAULT");
        g_fault_pending.compare_exchange_strong(s, (f && std::strcmp(f, "missing_arrival") == 0) ? 1 : 0);
    }
    int one = 1;
    return g_fault_pending.compare_exchange_strong(one, 0) ? 1 : 0;
}

// B, Q and E become NaN when a window kernel of this call latched an error,
// and the error word is cleared for the next call (one block: it has nothing
// to do unless a wait ran out, and the clearing needs no launch of its own).
__global__ void __launch_bounds__(1024)
poison_on_error_kernel(int* err, float* B, float* Q, float* E, size_t n)
{
    wait_previous();
    if (*reinterpret_cast<const volatile int*>(err) == 0) return;
    const float nan = __int_as_float(0x7fc00000);
    for (size_t i = threadIdx.x; i < n; i += blockDim.x) {
        B[i] = nan;
        Q[i] = nan;
        E[i] = nan;
    }
    __syncthreads();
    if (threadIdx.x == 0) *err = 0;
}

}  // namespace

extern "C" {

bacon_status bacon_window_scores_noalloc(int kv_heads, int q_heads, int head_dim, int window,
                                         const void* q_win, const void* k, int seq_len,
                                         float* B_out, float* Q_out, float* E_out,
                                         bacon_stream stream)
{
    // malformed arguments
    if (kv_heads < 1 || q_heads < 1 || q_heads % kv_heads) return BACON_EINVAL;
    if (head_dim != 64 && head_dim != 128) return BACON_EINVAL;
    if (window < 1 || seq_len < window) return BACON_EINVAL;
    const void* ps[] = {q_win, k, B_out, Q_out, E_out};
    for (const void* p : ps)
        if (!p || (reinterpret_cast<uintptr_t>(p) & 15u)) return BACON_EINVAL;
    // sizes beyond what the static scratch (or the kernels) can hold
    const long long rows = (long long)(q_heads / kv_heads) * window;
    if (seq_len > kMaxSeq || rows * kv_heads > kMaxTotalRows || rows > window_tc_max_rows())
        return BACON_EUNSUPPORTED;

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return BACON_ECUDA;
    float2* scratch = nullptr;
    {
        // one-time set-up per device, with that device current: the host-side
        // name of the array is not a device address, so look the address up
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_scratch_addr[dev]) {
            void* addr = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&addr, g_scratch);
            if (e != cudaSuccess || !addr) return BACON_ECUDA;
            g_scratch_addr[dev] = addr;
        }
        scratch = static_cast<float2*>(g_scratch_addr[dev]);
    }

    Shape s;
    s.layers = 1;
    s.hkv = kv_heads;
    s.group = q_heads / kv_heads;
    s.d = head_dim;
    s.W = window;
    s.N = seq_len;
    s.units = kv_heads;
    s.rows = (int)rows;
    const int chunks = (seq_len + kChunk - 1) / kChunk;
    float2* partial = scratch;
    int* err = reinterpret_cast<int*>(scratch + (size_t)kMaxTotalRows * kMaxChunks);
    const long long krows = (long long)kv_heads * seq_len, qrows = (long long)q_heads * window;
    TcArgs a;
    TcMaps m;  // the TMA descriptors are kernel parameters
    if (!encode_rows_map(&m.k, k, head_dim, krows, 1, krows * head_dim * 2, kTcKBoxRows) ||
        !encode_rows_map(&m.q, q_win, head_dim, qrows, 1, qrows * head_dim * 2, kTcQBoxRows))
        return BACON_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    a.kmaps = a.qmaps = nullptr;
    a.s = s;
    a.chunks = chunks;
    a.total_chunks = s.units * chunks;
    a.partial = partial;
    a.lse2 = nullptr;  // pass 2 forms the row normalisers from the partials
    a.B = B_out;
    a.Q = Q_out;
    a.E = E_out;
    a.err = err;
    TcArgs a1 = a;
    a1.fault = take_fault();
    cudaError_t e = launch_window_stats_tc(a1, m, st);
    if (e == cudaSuccess) e = launch_window_scores_tc(a, m, st);
    if (e == cudaSuccess)
        e = launch_after(poison_on_error_kernel, 1, 1024, 0, st, err, B_out, Q_out, E_out,
                         (size_t)kv_heads * seq_len);
    // without that kernel, what this call latched must not reach the next one
    if (e != cudaSuccess) cudaMemsetAsync(err, 0, sizeof(int), st);
    return e == cudaSuccess ? BACON_OK : BACON_ECUDA;
}

}  // extern "C"
