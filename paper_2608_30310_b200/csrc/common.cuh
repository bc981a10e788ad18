// Shared declarations of the GDN tail-replay CUDA library (host + device).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "gdn_tail_replay.h"

namespace gdn {

// Device-side view of one forward call; all pointers are device pointers.
struct Problem {
    const void* q;            // [T, Hq, dk] io dtype
    const void* k;            // [T, Hq, dk]
    const void* v;            // [T, Hv, dv]
    const float* g;           // [T, Hv]  log-decay
    const float* beta;        // [T, Hv]
    const int32_t* cu;        // [N + 1]
    const float* init_state;  // [N, Hv, dk, dv] or nullptr
    void* out_o;              // [T, Hv, dv] io dtype or nullptr
    float* out_state;         // [N, Hv, dk, dv] or nullptr
    int32_t* status_word;     // optional device int32
    int32_t num_seqs, Hq, Hv, dk, dv;
    int32_t input_raw;        // 1: q, k un-normalised, g = gate pre-activation, beta = pre-activation (fused input stage)
    int64_t total_tokens;
};

constexpr float kNormEps = 1.0e-6f;   // added to the squared norm of q and k rows in the fused input stage

// Operand ring of the tensor-core path for few chains (see gdn_tc.cu): slots per cluster, and the largest number of
// clusters (four CTAs each), hence of chains, that it is used for.
constexpr uint32_t kRingSlots = 9, kRingSlotBytes = 32768 + 512;
constexpr int64_t kRingClusters = 37;

// Scheduler scratch at the head of the workspace.
struct SchedHeader {
    uint32_t reserved[64];
};
static_assert(sizeof(SchedHeader) == 256, "header is one 256-byte line");

// Work list: requests ordered longest-first (paper is silent on scheduling; ragged tails from
// concurrent cache hits differ up to 8x in length, so long chains must start first).
struct Sched {
    int32_t* order;           // [N] request indices, longest first, from the scheduler kernel; null: every CTA orders the
                              // requests itself (up to kSelfSort of them)
    uint8_t* ring;            // kRingSlots * kRingSlotBytes per chain, for calls of up to kRingClusters chains on the
                              // tensor-core path; null: none (the call then runs without clusters)
};

// Kernel launch that may begin while the kernel before it in the stream is still running (programmatic dependent launch): the
// launch itself and a kernel's start-up pass under the tail of its predecessor.  Every kernel so launched calls
// wait_for_predecessor() before its first access to global memory, and allow_successor() as early as it likes.
template <typename... P, typename... A>
inline cudaError_t launch_kernel(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream, unsigned cluster, A&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cfg.attrs = at; cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Up to this many requests the kernels order the requests themselves, each CTA for itself: two lengths per lane, a rank is two
// ballots, so the whole order costs one load of cu and a few hundred cycles, less than the scheduler kernel's turn in the stream
// (a microsecond a call, although its launch is hidden).  Beyond two lengths per lane the calls are long and the scheduler kernel
// does it once.
constexpr int kSelfSort = 64;
// table[rank] = (first row, end row, request), longest first, ties by index.  All warps of the CTA call it, then synchronise.
static __device__ __noinline__ void sort_requests(const int32_t* cu, int num_seqs, int4* table, int warp, int nwarps, int lane)
{
    int len[2], row[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int n = lane + 32 * i;
        row[i] = n < num_seqs ? cu[n] : 0;
        len[i] = n < num_seqs ? cu[n + 1] - row[i] : (int)0x80000000;      // (longer than no request)
    }
    for (int n = warp; n < num_seqs; n += nwarps) {
        const int ln = __shfl_sync(0xffffffffu, n < 32 ? len[0] : len[1], n & 31);
        const int rn = __shfl_sync(0xffffffffu, n < 32 ? row[0] : row[1], n & 31);
        const int rank = __popc(__ballot_sync(0xffffffffu, len[0] > ln || (len[0] == ln && lane < n))) +
                         __popc(__ballot_sync(0xffffffffu, len[1] > ln || (len[1] == ln && lane + 32 < n)));
        if (lane == 0) table[rank] = make_int4(rn, rn + ln, n, 0);
    }
}
// Whether the CTAs have to call sort_requests; a single request needs no order.
__device__ __forceinline__ bool self_sorted(const Problem& p, const Sched& s) { return !s.order && p.num_seqs > 1; }
// (first row, end row, request) of place `i` in the order
__device__ __forceinline__ int4 request_at(const Problem& p, const Sched& s, const int4* table, uint32_t i)
{
    if (self_sorted(p, s)) return table[i];
    const int n = s.order ? s.order[i] : 0;
    return make_int4(p.cu[n], p.cu[n + 1], n, 0);
}

cudaError_t launch_scheduler(const int32_t* cu, int32_t num_seqs, const Sched& s, cudaStream_t stream);
cudaError_t launch_simt(const Problem& p, const Sched& s, int io_dtype, cudaStream_t stream, int* launches);
// Whether the tensor-core path can run this problem; launch_tcgen05 returns cudaErrorNotSupported when it cannot.
bool tcgen05_supported(const Problem& p);
cudaError_t launch_tcgen05(const Problem& p, const Sched& s, cudaStream_t stream, int* launches);
// One token per request from a given state (state_in and state_out may alias).
cudaError_t launch_decode(const void* q, const void* k, const void* v, const float* g, const float* beta,
                          const float* state_in, float* state_out, void* out_o, int32_t num_seqs, int32_t Hq,
                          int32_t Hv, int32_t dk, int32_t dv, int io_dtype, cudaStream_t stream);

}  // namespace gdn
