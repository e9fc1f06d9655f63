// Shared by all sources of the SNIP library: status handling, argument checks, chains of dependent launches.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "snip.h"

namespace snip {

// Thread-local text of the last CUDA error observed inside the library.
char *last_error_buffer();
void set_last_error(const char *where, cudaError_t e);

#define SNIP_CUDA_TRY(expr)                                   \
    do {                                                      \
        cudaError_t _e = (expr);                              \
        if (_e != cudaSuccess) {                              \
            ::snip::set_last_error(#expr, _e);                \
            return SNIP_ERR_CUDA;                             \
        }                                                     \
    } while (0)

static inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
static inline bool valid_fmt(int f) { return f >= SNIP_FMT_BF16 && f <= SNIP_FMT_FP4_E2M1; }
static inline bool valid_block(int b) { return b >= SNIP_BLOCK_ROW_1x128 && b <= SNIP_BLOCK_BLK_128x128; }
static inline bool valid_dim(int64_t d) { return d > 0 && (d % 64) == 0; }

// One output of the two-output quantizer (quantize.cu: quantize_dual_impl).
struct DualOut {
    int fmt;
    void *codes;
    float *scales;
    void *sf;             // optional UE8M0 atoms (power-of-two rule only)
    snip_stats_t *stats;  // optional; both outputs or neither
    int sr = 0;           // 1: stochastic rounding (FP4 only)
    uint64_t seed = 0;
};

// A linear-layer call enqueues a chain of kernels by programmatic dependent launch: quantizers, then GEMMs.
//   CHAIN_NONE  : a call of its own (starts after the kernel ahead of it on the stream; a quantizer launches its own statistics
//                 reduction)
//   CHAIN_FIRST : starts after the kernel ahead of it has completed, then lets the next one start beside it
//   CHAIN_BESIDE: reads nothing that the member directly ahead of it writes: starts beside it and waits for it only before it ends,
//                 so that "the last member has completed" keeps meaning "all of them have"
//   CHAIN_AFTER : its prologue runs beside the members ahead of it, its work after they have completed
// What a CHAIN_BESIDE member does read was written further ahead: the second and third quantizer read tensors made before the call, the
// second and third GEMM read what the quantizers left.  That is complete when the member starts, because a grid is scheduled only when
// every CTA of the one ahead has let it be, and a FIRST or AFTER member does so after its own wait (chain_start).  Hence the order of a
// chain: FIRST, then BESIDE for further quantizers, AFTER for the first GEMM, BESIDE for the others.  The waits made those writes visible
// to the grids that waited, not to the one that starts beside them: its SM's L1 may still hold an earlier call's values.  The quantizers
// read past L1 (cp.async.cg, __ldcg); the GEMMs, which read scale factors and bounds through it, begin with an acquire (chain_acquire).
enum ChainRole { CHAIN_NONE = 0, CHAIN_FIRST = 1, CHAIN_BESIDE = 2, CHAIN_AFTER = 3 };

// First thing in a GEMM, ahead of the CTA's first barrier, which passes it on to all threads: an acquiring load of the status word (the
// chain's first quantizer has cleared it), behind which nothing stale is read from L1, and a proxy fence that orders the TMA unit's reads of
// the operands behind it too.  By a thread of a warp that has nothing to set up, beside the allocation of tensor memory.  A layer of 1152
// tokens, 1216 -> 576: 26.43 us without it, 26.60 so, 26.96 with fence.acq_rel.gpu in its place (which waits for a full round of its own).
__device__ __forceinline__ void chain_acquire(int role, const uint32_t *status)
{
    if (role == CHAIN_BESIDE && threadIdx.x == 96) {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n\tfence.proxy.async.global;" : "=r"(v) : "l"(status) : "memory");
    }
}
// Start of every kernel that may be a member of a chain, by all threads, before they touch memory that a kernel ahead writes.
__device__ __forceinline__ void chain_start(int role)
{
    if (role != CHAIN_BESIDE) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// End of it.
__device__ __forceinline__ void chain_finish(int role)
{
    if (role == CHAIN_BESIDE) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Statistics partials left by the quantizers of a chain; the GEMM behind them reduces them in warps it has to spare (otherwise a
// launch per quantizer, in the way of everything behind it).
struct StatJob {
    const void *partials;   // CtaPartial[n] (quant_device.cuh)
    snip_stats_t *out;
    int32_t n;
};
struct StatJobs {
    StatJob job[6];
    int32_t count = 0;
};

// Workspace of one GEMM: status word, and (optional) arrival counters and partial sums of sliced tiles.  cleared: the status word and
// the counters are already zero, or will be by the time the kernel starts.
struct GemmWs {
    uint32_t *status = nullptr;
    uint32_t *counters = nullptr;
    float *partials = nullptr;
    bool cleared = false;   // false: the kernel clears the status word itself (status_begin)
};

// Non-zero mark of a launch that clears its status word itself; 0 where the word has been cleared.
uint32_t status_mark(bool cleared);

// What a chain passes along: the first quantizer clears `zero_words` words at `zero` (GEMM status word and slice counters).
struct ChainLink {
    int role = CHAIN_NONE;
    uint32_t *zero = nullptr;
    int32_t zero_words = 0;
    StatJobs *jobs = nullptr;   // quantizers append, the next GEMM takes them
    int32_t *ctas = nullptr;    // [3], zero at first: what the chain's GEMMs under the paper's rule launched, in order
};

// One tensor of the two-output quantizer (quantize.cu: quantize_dual_impl, quantize_xwd_impl).
constexpr int kDualTwoLevel = 16;   // kind beyond snip_dual_kind_t: 1x16 / 16x1 tiles of the two-level option
struct DualTask {
    const void *x;
    int64_t rows, cols, ld;
    int kind;                  // snip_dual_kind_t or kDualTwoLevel
    int pow2;
    const float *tensor_amax;  // two-level option only
    DualOut a, b;
    void *ws;                  // statistics scratch
    size_t ws_bytes;
};
inline DualTask two_level_task(const void *x, int64_t rows, int64_t cols, int64_t ld, const float *amax, void *codes_a, void *sf_a, snip_stats_t *stats_a,
                               void *codes_b, void *sf_b, snip_stats_t *stats_b, int rounding, uint64_t seed, void *ws, size_t ws_bytes)
{
    const int sr = rounding == SNIP_ROUND_STOCHASTIC ? 1 : 0;
    return {x, rows, cols, ld, kDualTwoLevel, 0, amax, DualOut{SNIP_FMT_FP4_E2M1, codes_a, nullptr, sf_a, stats_a, sr, seed},
            DualOut{SNIP_FMT_FP4_E2M1, codes_b, nullptr, sf_b, stats_b, sr, seed}, ws, ws_bytes};
}

// Fails with SNIP_ERR_UNSUPPORTED unless the current device is compute capability 10.x.
int require_sm100();

// Launch of a GEMM with the attribute that lets it start beside the kernel ahead of it (griddepcontrol in the kernel decides what
// waits: on its own, everything but the prologue).
template <typename... KArgs, typename... Args>
int launch_chained(void (*kern)(KArgs...), int grid, int threads, size_t smem_bytes, cudaStream_t st, int cluster, const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    if (cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs++].val.clusterDim.z = 1;
    }
    SNIP_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, args...));
    return SNIP_OK;
}

}  // namespace snip
