// Block-scaled GEMMs on the tcgen05 tensor cores:  out[Mo,No] = A[Mo,Kc] . B[No,Kc]^T with both
// operands contraction-major, FP32 accumulation in tensor memory, and the paper's FP32 tile
// scales applied per 128-long chunk of the contraction (Sec. 2.3: "the output is scaled back by
// dividing by the same scaling factor"; Fig. 5 for the three GEMMs of a linear layer).
//
// Structure of one CTA (persistent, one per SM, 384 threads):
//   warp 0      : TMA producer - streams 128-byte-wide operand tiles into a shared-memory ring
//   warp 1      : MMA issuer   - one thread issues tcgen05.mma; owns the tensor-memory allocation
//   warps 2..3  : weight-gradient product: loaders of the per-row / per-column scale factors (one ring of ready
//                 reciprocals for the CTA); warp 2 also adds up the statistics of quantizers ahead.  They give their
//                 registers to the epilogue warps
//   warps 4..11 : promotion / epilogue - pull each chunk's partial sums out of tensor memory,
//                 multiply by 1/(S_a*S_b) of that chunk and add into FP32 register accumulators
//                 (so the scaling overlaps the next chunk's MMAs, which write the other
//                 tensor-memory buffer), then round and store the tile.
// Three forms, chosen by shape in gemm_impl: 128-row tiles of 256 (192) or of 128 columns on one CTA, 256-row tiles on a
// pair of CTAs (tcgen05.mma.cta_group::2; the leader's MMA warp and barriers serve both).  128-wide tiles of the weight gradient have a
// fourth, in which the slices of a tile are the CTAs of a cluster.
// All hand-offs use mbarriers with bounded waits; on a timeout the CTA raises a status word and
// leaves cleanly (tensor memory is always released).
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>

#include "common.cuh"
#include "quant_device.cuh"
#include "sm100.cuh"
#include "work_items.cuh"

namespace snip {

using namespace sm100;

namespace {

constexpr int CM = 128;   // output rows of a CTA
constexpr int kGemmThreads = 384;  // warps 0-3: producer, MMA issuer, 2 scale loaders (wgrad) or idle; warps 4-11: epilogue
constexpr int kNumEpiWarps = 8;
static_assert(kNumEpiWarps == kSliceWarps, "slice counters");
// Contraction slices of the weight-gradient product's last wave: no shorter than kMinSliceStages, and only where they shorten the CTAs' sequence
// of stages by what the exchange of the partial sums takes (8-13 us; 2048 tokens x 256 x 2048: 15.6 us whole, 20.6 us in two slices).
constexpr int kMinSliceStages = 8, kMinSavedStages = 20;
// Slices in a cluster exchange their sums through shared memory: about 3 us, ten stages of a 128-wide tile (2048 tokens x 256 x 2048, where
// two slices save eight: 12.0 us whole, 12.6 us sliced).  256-wide tiles keep the exchange through L2: there are half as many of them as
// narrow ones, and two slices of 64 such tiles come out level with 128 whole narrow ones (8192 x 1024 x 2048: 32.9 / 32.5 us).
constexpr int kMinSavedStagesCluster = 12;
// What the exchange through the workspace takes for 128-wide tiles, in the same measure: about 5 us more (see prefer_clusters).
constexpr int kWorkspaceExchangeChunks = 24;
constexpr int kSfCols = 32;  // tensor-memory columns holding constant scale factors (kind::mxf4)

enum ScaleMode { SCALE_BLOCK_B = 1, SCALE_VEC_B = 2 };

struct GemmArgs {
    int32_t Mo, No, Kc;        // output rows / cols, contraction length in elements
    const float *sa;           // A scales [chunks][Mo]
    int64_t sa_chunk_stride;
    const float *sb;           // B scales: SCALE_BLOCK_B [blk*sb_blk_stride + chunk*sb_chunk_stride]
    int64_t sb_chunk_stride;   //           SCALE_VEC_B   [chunk*sb_chunk_stride + n]
    int64_t sb_blk_stride;
    void *out;
    int64_t ldo;
    int32_t accumulate;
    uint32_t stage_tx_bytes;   // bytes the two TMA loads of one stage report to the barrier
    uint32_t tx_skew;          // testing hook, part of stage_tx_bytes: in a cluster of slices the first slice's only
    uint64_t wait_limit_ns;    // bound of every device-side wait
    uint32_t *status;
    uint32_t status_mark;      // see status_begin
    WorkSplit work;
    float *partials;           // [tail tile r][slice j][epilogue warp][column quad][row lane][4]: FP32 sums of a slice
    uint32_t *counters;        // [tail tile r][epilogue warp]: slices that have delivered their sums (zero at launch)
    int32_t chain;             // ChainRole
    StatJobs stats;            // reductions left by the quantizers ahead
};

template <MmaKind KIND, int BN, int SCALE, bool PAIR>
struct Cfg {
    static constexpr int kCtas = PAIR ? 2 : 1;
    static constexpr int BM = CM * kCtas;                                    // rows of a tile
    static constexpr int kBLines = BN / kCtas;                               // B lines fetched by a CTA
    static constexpr int kStageElemsX = 128;                                 // TMA x step per stage
    static constexpr int kChunkElems = 128;                                  // scale granularity
    static constexpr int kStageK = KIND == MmaKind::F8F6F4 ? 128 : 256;
    static constexpr int kABytes = CM * 128;
    static constexpr int kBBytes = kBLines * 128;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kStages = PAIR ? 6 : BN <= 128 ? (SCALE == 1 ? 5 : 6) : (BN >= 256 || SCALE == 1) ? 4 : 5;
    // block mode (fwd / dgrad) fetches four chunks of scale factors per instruction into two alternating group slots:
    // [4 chunks][32 rows] S_a, then [2 blocks][4 chunks] S_b
    static constexpr int kGroupFloats = 144;
    static constexpr int kRingFloatsPerWarp = 2 * kGroupFloats;
    // vector mode (wgrad): ONE ring for the CTA, filled by the two loader warps: per chunk 128 row factors 1/S_a and BN column
    // factors 1/S_b, kVecDepth chunks deep, handed over kVecBlock chunks at a time.  A slot is laid out for the fragments of the
    // promotion warps: rows [32-row quarter][row % 8][row / 8 % 4]; columns [column half][column % 4][column / 4], the four
    // residues kVecQuad floats apart (16 bytes more than their data: their 16-byte reads hit distinct banks)
    static constexpr int kVecDepth = 16, kVecBlock = 4, kVecAhead = 8;
    static constexpr int kVecQuad = BN / 8 + 4;
    static constexpr int kVecSlotFloats = 128 + 8 * kVecQuad;
    static constexpr int kSbInvBytes = (SCALE == 2) ? (kVecDepth * kVecSlotFloats * 4 + 1023) / 1024 * 1024 : kNumEpiWarps * kRingFloatsPerWarp * 4;
    // block mode (fwd / dgrad) writes its output through kOutSlots 2 KB staging tiles per warp and TMA stores; where shared
    // memory has room for a warp's whole bf16 tile no store is waited for before the next tile's sums
    static constexpr bool kTmaOut = (SCALE == 1);
    static constexpr int kOutSlots = (BN == 192) ? 3 : (BN == 128) ? 2 : 1;
    static constexpr int kOutStageBytes = kTmaOut ? kNumEpiWarps * kOutSlots * 2048 : 0;
    static constexpr int kSmemBytes = kStages * kStageBytes + kSbInvBytes + kOutStageBytes + 256 + 1024;  // + barriers + alignment slack
    static_assert(kSmemBytes <= 232448, "shared memory budget");
    static_assert(kStageBytes % 1024 == 0 && kSbInvBytes % 1024 == 0, "staging tiles must stay 1024-byte aligned");
    static constexpr bool kClusterSlices = SCALE == 2 && BN == 128 && !PAIR;   // see plan_clusters
    static constexpr int kAccCols = 2 * BN;
    static constexpr int kSfCol0 = kAccCols;
    static constexpr int kTmemCols = 512;
    static_assert(kAccCols + (KIND == MmaKind::MXF4 ? kSfCols : 0) <= 512, "tensor memory budget");
};

// Reciprocal from the special-function unit (one instruction, ~1 ulp; a subnormal result is flushed to zero,
// which only affects products of scales beyond FP32's range).
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// Store 32 consecutive output values of one row.
template <bool OUT_F32>
__device__ __forceinline__ void store32(const GemmArgs &g, int64_t row, int col, const float *v)
{
    if (OUT_F32) {
        float *dst = static_cast<float *>(g.out) + row * g.ldo + col;
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
            if (col + i < g.No) {
                float4 o = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                if (g.accumulate) {
                    const float4 p = *reinterpret_cast<const float4 *>(dst + i);
                    o.x += p.x; o.y += p.y; o.z += p.z; o.w += p.w;
                }
                *reinterpret_cast<float4 *>(dst + i) = o;
            }
        }
    } else {
        __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(g.out) + row * g.ldo + col;
#pragma unroll
        for (int i = 0; i < 32; i += 8) {
            if (col + i < g.No) {
                uint4 o = make_uint4(pack_bf16x2(v[i], v[i + 1]), pack_bf16x2(v[i + 2], v[i + 3]),
                                     pack_bf16x2(v[i + 4], v[i + 5]), pack_bf16x2(v[i + 6], v[i + 7]));
                *reinterpret_cast<uint4 *>(dst + i) = o;
            }
        }
    }
}

// 4 x 4 transpose of words over the four lanes of a quad: afterwards w[k] is lane k's former w[lane % 4].
__device__ __forceinline__ void quad_transpose(uint32_t (&w)[4], int lane)
{
#pragma unroll
    for (int m = 1; m <= 2; m <<= 1) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k & m) continue;
            const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, up ? w[k] : w[k + m], m);
            if (up) w[k] = got; else w[k + m] = got;
        }
    }
}

// Stores a fragment of 16 rows x 32 columns in the register order of tmem_ld_frag: rows `row` and `row + 8`, columns
// col + 4 i + lane % 4.  The lanes of a quad swap so that each stores four consecutive columns of every sixteen.
template <bool OUT_F32>
__device__ __forceinline__ void store_frag(const GemmArgs &g, int64_t row, int col, const float *v, int lane)
{
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int64_t r = row + 8 * b;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int c = col + 16 * k + 4 * (lane & 3);
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = __float_as_uint(v[2 * (4 * k + i) + b]);
            quad_transpose(w, lane);
            if (r < g.Mo && c < g.No) {
                float4 o = make_float4(__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]), __uint_as_float(w[3]));
                if (OUT_F32) {
                    float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(g.out) + r * g.ldo + c);
                    if (g.accumulate) { const float4 p = *dst; o.x += p.x; o.y += p.y; o.z += p.z; o.w += p.w; }
                    *dst = o;
                } else {
                    *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(g.out) + r * g.ldo + c) = make_uint2(pack_bf16x2(o.x, o.y), pack_bf16x2(o.z, o.w));
                }
            }
        }
    }
}

// CLUSTER: the CTAs of a cluster hold the slices of one tile, an item each (plan_clusters).  An instantiation of its own: with the cluster
// barriers in the code of the others, unused, a 512 x 512 x 512 layer takes 17.0 instead of 16.0 us.
template <MmaKind KIND, int BN, int SCALE, bool PAIR, bool OUT_F32, bool CLUSTER>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmO,
            const GemmArgs g, const uint32_t idesc)
{
    using C = Cfg<KIND, BN, SCALE, PAIR>;
    constexpr int S = C::kStages, BM = C::BM;
    constexpr int HALF = BN / 2;     // columns handled by one epilogue warp
    // registers per tensor-memory load: 16 in vector mode (wgrad: 16 rows x 32 columns as a fragment), 32 otherwise (32 rows x
    // 32 columns; fwd / dgrad: 2.5 % faster than 16)
    constexpr int GC = (SCALE == SCALE_VEC_B) ? 16 : 32;
    constexpr int G = HALF / GC;     // groups handled by one epilogue warp per chunk
    // A chunk's sums are waited for with one vote (wait_warp), except on 128-wide tiles of kind::mxf4 in fwd / dgrad, where that is the
    // slower way: 1024 x 4096 x 4096 18.3 us without, 19.2 us with it (192-wide pairs, 5376 x 1536 x 4096: 36.3 without, 35.6 with it).
    constexpr bool kOneVote = !(KIND == MmaKind::MXF4 && BN == 128 && SCALE == SCALE_BLOCK_B);
    constexpr int D = (SCALE == SCALE_VEC_B) ? (G < 6 ? G : 4) : (BN <= 192) ? G : 2;   // groups of staging registers next to the accumulators
    static_assert(!CLUSTER || C::kClusterSlices, "slices in clusters: 128-wide tiles of the weight gradient");
    // (tiles of up to 192 columns: at most 96 accumulators leave room for the whole chunk, so the buffer goes back before any multiplication)

    extern __shared__ uint8_t smem_raw[];
    chain_acquire(g.chain, g.status);
    // operand tiles need 1024-byte alignment for the 128-byte swizzle
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t smem_a0 = smem_base;
    const uint32_t smem_b0 = smem_base + S * C::kABytes;
    float *scale_ring = reinterpret_cast<float *>(smem_gen + S * C::kStageBytes);
    const uint32_t out_stage0 = smem_base + S * C::kStageBytes + C::kSbInvBytes;   // 1024-byte aligned
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_gen + S * C::kStageBytes + C::kSbInvBytes + C::kOutStageBytes);
    const uint32_t bar0 = smem_base + S * C::kStageBytes + C::kSbInvBytes + C::kOutStageBytes;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * S + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * S + 2 + a); };
    constexpr int kVBlocks = C::kVecDepth / C::kVecBlock;
    auto vfull_bar = [&](int k) { return bar0 + 8u * (2 * S + 4 + k); };              // vector mode: ring block k holds its chunks' factors
    auto vempty_bar = [&](int k) { return bar0 + 8u * (2 * S + 4 + kVBlocks + k); };  // vector mode: the eight epilogue warps are done with block k
    static_assert((2 * S + 4 + 2 * kVBlocks) * 8 + 8 <= 256, "barrier area");
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * S + 4 + 2 * kVBlocks);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;   // 0 = leader: its barriers and its MMA warp serve the pair
    const int unit = (int)blockIdx.x / C::kCtas, units = (int)gridDim.x / C::kCtas;
    const int num_m = (g.Mo + BM - 1) / BM, num_n = (g.No + BN - 1) / BN;
    const int num_chunks = (g.Kc + C::kChunkElems - 1) / C::kChunkElems;
    const int num_kstages = (g.Kc + C::kStageK - 1) / C::kStageK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), kNumEpiWarps * C::kCtas); }
        for (int k = 0; k < kVBlocks; ++k) { mbar_init(vfull_bar(k), 2); mbar_init(vempty_bar(k), kNumEpiWarps); }
        *abort_flag = 0u;
        fence_barrier_init();
        prefetch_tensormap(&tmA);
        prefetch_tensormap(&tmB);
    }
    if (warp == 1) {
        tmem_alloc<PAIR>(smem_u32(tmem_slot), C::kTmemCols);
        tmem_relinquish<PAIR>();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // everything up to here touches nothing that a kernel ahead on the stream writes
    chain_start(g.chain);

    if (KIND == MmaKind::MXF4) {
        // constant scale factors 2^0 (UE8M0 byte 127) for every row of A and B
        if (warp >= 4 && warp < 8) {
            const uint32_t q = warp & 3;
            for (int c = 0; c < kSfCols; ++c) tmem_st1(tmem_base + ((q * 32u) << 16) + C::kSfCol0 + c, 0x7F7F7F7Fu);
            tmem_st_wait();
        }
        tc_fence_before_sync();
        __syncthreads();
        tc_fence_after_sync();
    }

    if (PAIR) {   // both CTAs' barriers and tensor memory (constant scale factors included) are ready before anyone signals across the pair
        tc_fence_before_sync();
        cluster_sync();
        tc_fence_after_sync();
    }
    // Bounded wait; a failed one raises the abort flag of both CTAs.
    auto wait1 = [&](uint32_t bar, uint32_t parity) {
        const bool got = mbar_wait(bar, parity, abort_flag, g.wait_limit_ns);
        if (PAIR && !got) st_cluster_u32(mapa(smem_u32(const_cast<uint32_t *>(abort_flag)), rank ^ 1u), 1u);
        return got;
    };
    // The same for a converged warp, one vote deciding for all lanes.  try_wait itself holds the thread until the phase completes (or a
    // time limit passes), so the bounded loop behind it is hardly ever entered; going through it costs 35 cycles more per wait, also where
    // the phase completed long ago (145 -> 110 cycles).
    auto wait_warp = [&](uint32_t bar, uint32_t parity) {
        if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) return true;
        const bool got = wait1(bar, parity);
        return (bool)__all_sync(0xFFFFFFFFu, got);
    };

    if (warp < 4) {
      reg_dealloc<40>();  // frees (168-40)*128 = 16384 registers
      if (warp == 0) {
        // ================= TMA producer =================
        status_begin(g.status, g.status_mark);
        const uint32_t lead_full0 = PAIR ? mapa(full_bar(0), 0) : 0u;
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int w = unit; w < g.work.num_items && ok; w += units) {
                const WorkItem wi = work_item<SCALE == SCALE_VEC_B>(g.work, w, num_kstages);
                int m_idx, n_idx;
                tile_coords(wi.t, num_m, num_n, m_idx, n_idx);
                const uint32_t tx_bytes = C::kCtas * g.stage_tx_bytes - (CLUSTER && wi.slice > 0 ? g.tx_skew : 0u);
                for (int ks = wi.ks0; ks < wi.ks1; ++ks, ++it) {
                    const int s = it % S;
                    const uint32_t ph = (it / S) & 1u;
                    if (!wait1(empty_bar(s), ph ^ 1u)) { ok = false; break; }
                    if (rank == 0) mbar_arrive_expect_tx(full_bar(s), tx_bytes);
                    const int row = m_idx * BM + (int)rank * CM, col = n_idx * BN + (int)rank * C::kBLines;
                    if (PAIR) {   // each CTA fetches its own share (no multicast); the leader's barrier counts the bytes of both
                        tma_load_2d_pair(smem_a0 + s * C::kABytes, &tmA, lead_full0 + 8u * s, ks * C::kStageElemsX, row);
                        tma_load_2d_pair(smem_b0 + s * C::kBBytes, &tmB, lead_full0 + 8u * s, ks * C::kStageElemsX, col);
                    } else {
                        tma_load_2d(smem_a0 + s * C::kABytes, &tmA, full_bar(s), ks * C::kStageElemsX, row);
                        tma_load_2d(smem_b0 + s * C::kBBytes, &tmB, full_bar(s), ks * C::kStageElemsX, col);
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        // Block mode: an elected lane, under which the operands of the tcgen05 instructions stay in uniform registers (issue of a chunk
        // 204 -> 55 cycles, 2-4 % of the FP4 kernels); in vector mode it costs the promotion warps registers and gains nothing.
        if (rank == 0 && (SCALE == SCALE_BLOCK_B ? elect_one() : lane == 0)) {
            uint32_t it = 0, cc = 0;
            bool ok = true;
            const uint32_t sfa = tmem_base + C::kSfCol0, sfb = tmem_base + C::kSfCol0 + 16;
            for (int w = unit; w < g.work.num_items && ok; w += units) {
                const WorkItem wi = work_item<SCALE == SCALE_VEC_B>(g.work, w, num_kstages);
                for (int ks = wi.ks0; ks < wi.ks1 && ok; ++ks, ++it) {
                    const int s = it % S;
                    const uint32_t ph = (it / S) & 1u;
                    if (!wait1(full_bar(s), ph)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint64_t adesc = make_smem_desc_k128(smem_a0 + s * C::kABytes);
                    const uint64_t bdesc = make_smem_desc_k128(smem_b0 + s * C::kBBytes);
                    if (KIND == MmaKind::F8F6F4) {
                        const uint32_t a = cc & 1u;
                        if (!wait1(tempty_bar(a), ((cc >> 1) & 1u) ^ 1u)) { ok = false; break; }
                        tc_fence_after_sync();
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            mma_ss<KIND, PAIR>(tmem_base + a * BN, adesc + 2 * k, bdesc + 2 * k, idesc, k > 0 ? 1u : 0u, 0, 0);
                        // one commit serves both hand-offs (a stage is one chunk here): the producer takes it as
                        // "stage s is free", the epilogue warps as "the chunk's partial sums are complete"
                        tc_commit<PAIR>(empty_bar(s));
                        ++cc;
                    } else {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (2 * ks + h < num_chunks) {
                                const uint32_t a = cc & 1u;
                                if (!wait1(tempty_bar(a), ((cc >> 1) & 1u) ^ 1u)) { ok = false; break; }
                                tc_fence_after_sync();
#pragma unroll
                                for (int k = 0; k < 2; ++k)
                                    mma_ss<KIND, PAIR>(tmem_base + a * BN, adesc + 2 * (2 * h + k), bdesc + 2 * (2 * h + k), idesc,
                                                 k > 0 ? 1u : 0u, sfa, sfb);
                                tc_commit<PAIR>(tfull_bar(a));
                                ++cc;
                            }
                        }
                        tc_commit<PAIR>(empty_bar(s));
                    }
                }
            }
        }
      } else if (SCALE != SCALE_VEC_B) {
        // ================= warp 2: statistics of the quantizers ahead =================
        if (warp == 2)
            for (int i = blockIdx.x; i < g.stats.count; i += gridDim.x) reduce_stats_warp(g.stats.job[i], lane);
      } else {
        // ================= warps 2, 3: scale loaders of the weight-gradient product =================
        // Both factors of a chunk are vectors here (1/S_a per output row, 1/S_b per output column).  Warp 2 brings the 128
        // row scales, warp 3 the BN column scales of every chunk into one ring for the CTA (cp.async, kVecAhead chunks
        // ahead), turns them into reciprocals in place and publishes them kVecBlock chunks at a time, so that the epilogue
        // warps only read ready factors: no copies, reciprocals or warp barriers of their own on the per-chunk path.
        const bool rows_side = (warp == 2);
        constexpr int kChunksPerStage = C::kStageK / C::kChunkElems;
        uint32_t total = 0;            // chunks of all of this CTA's work items
        for (int w = unit; w < g.work.num_items; w += units) {
            const WorkItem wi = work_item<SCALE == SCALE_VEC_B>(g.work, w, num_kstages);
            total += (uint32_t)(min(kChunksPerStage * wi.ks1, num_chunks) - kChunksPerStage * wi.ks0);
        }
        const uint32_t ring_u32 = smem_u32(scale_ring);
        int pw = unit, pj = 0, pn = 0;   // work item and chunk of the next request, chunks of that item
        uint32_t pc = 0;               // its position in the sequence of this CTA's chunks
        bool ok = true;
        const float *src0 = nullptr, *src1 = nullptr;
        int64_t stride = 0;
        auto item_sources = [&]() {
            const WorkItem wi = work_item<SCALE == SCALE_VEC_B>(g.work, pw < g.work.num_items ? pw : unit, num_kstages);
            int m_idx, n_idx;
            tile_coords(wi.t, num_m, num_n, m_idx, n_idx);
            const int c0 = kChunksPerStage * wi.ks0;
            pn = min(kChunksPerStage * wi.ks1, num_chunks) - c0;
            // rows / columns outside the matrix repeat the last four factors (their sums are never stored)
            if (rows_side) {
                stride = g.sa_chunk_stride;
                src0 = g.sa + c0 * stride + min(m_idx * BM + (int)rank * CM + 4 * lane, g.Mo - 4);
            } else {
                stride = g.sb_chunk_stride;
                src0 = g.sb + c0 * stride + min(n_idx * BN + 4 * lane, g.No - 4);
                src1 = g.sb + c0 * stride + min(n_idx * BN + 128 + 4 * lane, g.No - 4);
            }
        };
        item_sources();
        auto request = [&]() {
            if (pc < total && ok) {
                const uint32_t d = pc % C::kVecDepth;
                if ((pc % C::kVecBlock) == 0 && !__all_sync(0xFFFFFFFFu, wait1(vempty_bar(d / C::kVecBlock), ((pc / C::kVecDepth) & 1u) ^ 1u))) ok = false;
                else {
                    const uint32_t slot = ring_u32 + d * (C::kVecSlotFloats * 4);
                    if (rows_side) {
                        cp_async_16(slot + 16u * lane, src0);
                    } else {
                        cp_async_16(slot + 512u + 16u * lane, src0);
                        if (128 + 4 * lane < BN) cp_async_16(slot + 1024u + 16u * lane, src1);
                    }
                    src0 += stride;
                    src1 += stride;
                    if (++pj == pn) { pj = 0; pw += units; item_sources(); }
                }
            }
            ++pc;
            cp_async_commit();   // one group per position, empty past the end, so that the wait below stays uniform
        };
        for (int i = 0; i < C::kVecAhead; ++i) request();
        for (uint32_t cc = 0; cc < total && ok; ++cc) {
            request();                       // position cc + kVecAhead
            cp_async_wait<C::kVecAhead>();   // this lane's copies of position cc have landed
            const uint32_t d = cc % C::kVecDepth;
            // raw factors of four consecutive lines per lane -> reciprocals in the fragment order of the slot
            float *slot = scale_ring + d * C::kVecSlotFloats;
            const float4 *raw = reinterpret_cast<const float4 *>(slot + (rows_side ? 0 : 128) + 4 * lane);
            const float4 v = raw[0];
            float4 w = v;
            if (!rows_side && 128 + 4 * lane < BN) w = raw[32];
            __syncwarp();                    // every lane has read its raw values
            if (rows_side) {
                // rows 4*lane .. +3: quarter lane / 8, row / 8 = lane / 2 % 4, row % 8 = 4 * (lane % 2) + t
                float *dst = slot + (lane >> 3) * 32 + (lane & 1) * 16 + ((lane >> 1) & 3);
                dst[0] = rcp_approx(v.x); dst[4] = rcp_approx(v.y); dst[8] = rcp_approx(v.z); dst[12] = rcp_approx(v.w);
            } else {
                auto put = [&](int col, const float4 &x) {   // col: a multiple of four
                    const int hh = col / HALF;
                    float *dst = slot + 128 + 4 * hh * C::kVecQuad + (col - hh * HALF) / 4;
                    dst[0] = rcp_approx(x.x); dst[C::kVecQuad] = rcp_approx(x.y); dst[2 * C::kVecQuad] = rcp_approx(x.z); dst[3 * C::kVecQuad] = rcp_approx(x.w);
                };
                put(4 * lane, v);
                if (128 + 4 * lane < BN) put(128 + 4 * lane, w);
            }
            __syncwarp();
            // a block is published when its last slot (or the last chunk of all) is ready
            if (lane == 0 && ((cc % C::kVecBlock) == C::kVecBlock - 1 || cc + 1 == total)) mbar_arrive(vfull_bar(d / C::kVecBlock));
        }
        cp_async_wait<0>();
        if (warp == 2)
            for (int i = blockIdx.x; i < g.stats.count; i += gridDim.x) reduce_stats_warp(g.stats.job[i], lane);
      }
      if (CLUSTER) {   // the two barriers of the slices' exchange (below)
          __syncwarp();
          cluster_sync();
          cluster_sync();
      }
    } else {
        reg_alloc<232>();    // needs (232-168)*256 = 16384 <= 16384 (an unsatisfiable request would block forever)
        // ================= promotion / epilogue warps =================
        const uint32_t lead_tempty0 = PAIR ? mapa(tempty_bar(0), 0) : 0u;
        const int e = warp - 4;          // 0..7
        const int q = warp & 3;          // tensor-memory lane quarter this warp may access
        const int h = e >> 2;            // column half
        // Block mode: per-warp scale-factor buffers, filled ahead with cp.async so that no global-memory latency
        // sits between two chunks.  S_a of this warp's 32 rows comes four chunks at a time into two alternating
        // group slots [4 chunks][32 rows], with the S_b of its one or two 128-column blocks next to them
        // ([2 blocks][4 chunks] at float 128 of the group).  Vector mode reads the CTA's ring of ready factors.
        float *ring = scale_ring + e * C::kRingFloatsPerWarp;
        const uint32_t ring_u32 = smem_u32(ring);
        const uint32_t stage_u32 = out_stage0 + e * (C::kOutSlots * 2048);   // this warp's staging tiles: 32 rows x 64 bytes each
        uint32_t cc = 0;
        bool ok = true;
        for (int w = unit; w < g.work.num_items && ok; w += units) {
            const WorkItem wi = work_item<SCALE == SCALE_VEC_B>(g.work, w, num_kstages);
            int m_idx, n_idx;
            tile_coords(wi.t, num_m, num_n, m_idx, n_idx);
            const int row0 = m_idx * BM + (int)rank * CM + q * 32;
            const int row = row0 + lane;
            const int col0 = n_idx * BN + h * HALF;
            const bool row_ok = row < g.Mo;
            constexpr int kChunksPerStage = C::kStageK / C::kChunkElems;
            const int nacc = min(kChunksPerStage * wi.ks1, num_chunks) - kChunksPerStage * wi.ks0;
            const int blk0 = col0 >> 7;
            const int blk_last = (g.No - 1) >> 7;

            // Block mode: the scale factors of four consecutive chunks with two instructions per warp.  Lane L
            // fetches 16 bytes = S_a of rows 4*(L%8) .. +3 of chunk 4*gn + L/8 (the warp's 32 rows lie inside or
            // outside the matrix together: row counts are multiples of 64); lanes 0..3 (0..7 with two blocks)
            // fetch S_b of one chunk each.  Group gn lands in slot gn % 2; groups are requested in order, so the source pointers
            // only step (64-bit index products and bounds per request: 3-6 % of the FP4 kernels).
            constexpr int kBlocksPerWarp = ((HALF % 128) == 0 || (128 % HALF) == 0) ? 1 : 2;
            const float *pa = g.sa + (int64_t)(lane >> 3) * g.sa_chunk_stride + row0 + (lane & 7) * 4;
            const float *pb = g.sb + (int64_t)min(blk0 + (lane >> 2), blk_last) * g.sb_blk_stride + (int64_t)(lane & 3) * g.sb_chunk_stride;
            const int64_t pa_step = 4 * g.sa_chunk_stride, pb_step = 4 * g.sb_chunk_stride;
            int left_a = (row0 < g.Mo) ? nacc - (lane >> 3) : 0, left_b = (lane < 4 * kBlocksPerWarp) ? nacc - (lane & 3) : 0;
            auto prefetch_group = [&](int gn) {
                const uint32_t slot = ring_u32 + (gn & 1) * C::kGroupFloats * 4;
                if (left_a > 0) cp_async_16(slot + lane * 16, pa);
                if (left_b > 0) cp_async_4(slot + (128 + lane) * 4, pb);
                pa += pa_step; pb += pb_step; left_a -= 4; left_b -= 4;
                cp_async_commit();
            };

            float2 acc[HALF / 2];
#pragma unroll
            for (int i = 0; i < HALF / 2; ++i) acc[i] = make_float2(0.0f, 0.0f);
            if (SCALE == SCALE_BLOCK_B) {
                // out-of-range rows / columns read 1.0 (their products are zero anyway)
                for (int i = lane; i < C::kRingFloatsPerWarp; i += 32) ring[i] = 1.0f;
                __syncwarp();
                prefetch_group(0);
                prefetch_group(1);
            }
            // Block mode: the reciprocal factors 1/(S_a*S_b) of the four chunks of group gn, from its slot (which must
            // have landed and been made visible to the warp), into a register queue that the chunk loop shifts.
            float fq[kBlocksPerWarp][4];
            auto load_factors = [&](int gn) {
                const float *sl = ring + (gn & 1) * C::kGroupFloats;
                const float4 b0 = *reinterpret_cast<const float4 *>(sl + 128);
                const float sb0[4] = {b0.x, b0.y, b0.z, b0.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float sa = sl[j * 32 + lane];
                    fq[0][j] = rcp_approx(sa * sb0[j]);
                    if (kBlocksPerWarp == 2) fq[1][j] = rcp_approx(sa * sl[132 + j]);
                }
            };
            if (SCALE == SCALE_BLOCK_B) {
                cp_async_wait<1>();   // group 0
                __syncwarp();
                load_factors(0);
            }
            for (int c = 0; c < nacc; ++c, ++cc) {
                const uint32_t a = cc & 1u;
                float f[G];
                // Vector mode: this chunk's slot of the CTA's factor ring (filled by warps 2 and 3), taken over a block at a time.
                // A thread's fragment is 4 rows (lane / 4 + 8 b) x HALF / 4 columns (4 j + lane % 4), so it needs 4 + HALF / 4 factors:
                // 9 shared-memory reads of 16 bytes per chunk and warp.  With a row per lane (the 32x32b loads of fwd / dgrad) it was
                // one broadcast read per four columns, 33 in all: about 600 cycles of the shared-memory pipe per 128 x 256 chunk, next to
                // the 770 that the operands' way in and out takes.
                const uint32_t vd = cc % C::kVecDepth;
                const float *vslot = scale_ring + vd * C::kVecSlotFloats;
                if (SCALE == SCALE_VEC_B && (cc % C::kVecBlock) == 0) {
                    if (!wait_warp(vfull_bar(vd / C::kVecBlock), (cc / C::kVecDepth) & 1u)) { ok = false; break; }
                }
                float4 rf = make_float4(0.0f, 0.0f, 0.0f, 0.0f), cf[2][2];   // row factors; column factors of two 32-column blocks
                const float4 *cfs = reinterpret_cast<const float4 *>(vslot + 128 + (4 * h + (lane & 3)) * C::kVecQuad);
                if (SCALE == SCALE_VEC_B) {
                    rf = *reinterpret_cast<const float4 *>(vslot + q * 32 + (lane >> 2) * 4);
                    cf[0][0] = cfs[0]; cf[0][1] = cfs[1];
                    cf[1][0] = cfs[2]; cf[1][1] = cfs[3];
                }
#pragma unroll
                for (int gi = 0; gi < G; ++gi) {
                    if (SCALE == SCALE_BLOCK_B) f[gi] = (kBlocksPerWarp == 1 || ((col0 + 32 * gi) >> 7) == blk0) ? fq[0][0] : fq[kBlocksPerWarp - 1][0];
                }
                if (SCALE == SCALE_BLOCK_B) {
#pragma unroll
                    for (int b = 0; b < kBlocksPerWarp; ++b) { fq[b][0] = fq[b][1]; fq[b][1] = fq[b][2]; fq[b][2] = fq[b][3]; }
                }
                // barrier that announces this chunk's partial sums (see the MMA issuer)
                const uint32_t done_bar = (KIND == MmaKind::F8F6F4) ? empty_bar(cc % S) : tfull_bar(a);
                const uint32_t done_par = (KIND == MmaKind::F8F6F4) ? ((cc / S) & 1u) : ((cc >> 1) & 1u);
                if (!(kOneVote ? wait_warp(done_bar, done_par) : (bool)__all_sync(0xFFFFFFFFu, wait1(done_bar, done_par)))) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + a * BN + h * HALF;
                uint32_t v[D][GC];
                auto load_group = [&](int gi, uint32_t (&dst)[GC]) {
                    // vector mode: rows 16 * (gi % 2) .., columns 32 * (gi / 2) ..
                    if constexpr (SCALE == SCALE_VEC_B) tmem_ld_frag(taddr + ((uint32_t)(16 * (gi & 1)) << 16) + 32 * (gi >> 1), dst);
                    else tmem_ld32(taddr + GC * gi, dst);
                };
#pragma unroll
                for (int gi = 0; gi < D; ++gi) load_group(gi, v[gi]);
                // In the shadow of the first load.  Block mode: with the last chunk of a group of four the register
                // queue is empty; the next group's slot (requested four chunks ago) is turned into the next four
                // factors and the slot of the group just finished is refilled two groups ahead.  One warp barrier
                // per four chunks: between the copies of all lanes and the reads of all lanes.
                if (SCALE == SCALE_BLOCK_B) {
                    if ((c & 3) == 3 && c + 1 < nacc) {
                        cp_async_wait<0>();
                        __syncwarp();
                        load_factors((c >> 2) + 1);
                        prefetch_group((c >> 2) + 2);
                    }
                }
                // all of this warp's reads of buffer `a` are done: hand it back to the MMA warp
                auto release_buffer = [&]() {
                    tc_fence_before_sync();
                    __syncwarp();
                    // (one CTA on 256 columns hands back between two groups, where the branch is the cheaper one: 1024 x 4096 x 4096 FP8
                    // 17.6 us elected, 17.4 us so)
                    if (PAIR) mbar_arrive_cluster_relaxed_elected(lead_tempty0 + 8u * a);
                    else if (SCALE == SCALE_VEC_B || G <= D) mbar_arrive_elected(tempty_bar(a));
                    else if (lane == 0) mbar_arrive(tempty_bar(a));
                };
                auto consume_group = [&](int gi, const uint32_t (&cur)[GC]) {
                    if (SCALE == SCALE_BLOCK_B) {
                        const float2 ff = make_float2(f[gi], f[gi]);
#pragma unroll
                        for (int i = 0; i < GC / 2; ++i)
                            acc[(GC / 2) * gi + i] = __ffma2_rn(make_float2(__uint_as_float(cur[2 * i]), __uint_as_float(cur[2 * i + 1])), ff, acc[(GC / 2) * gi + i]);
                    } else {
                        // group gi: rows 16 * (gi % 2) + {lane / 4, + 8}, columns 32 * (gi / 2) + 4 i + lane % 4
                        const float2 r2 = (gi & 1) ? make_float2(rf.z, rf.w) : make_float2(rf.x, rf.y);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float4 c4 = cf[(gi >> 1) & 1][i >> 2];
                            const float c = (i & 3) == 0 ? c4.x : (i & 3) == 1 ? c4.y : (i & 3) == 2 ? c4.z : c4.w;
                            // (two scalar FMAs instead of the packed one: 1092 instead of 1066 cycles per 128 x 256 chunk)
                            const float2 p = __fmul2_rn(make_float2(__uint_as_float(cur[2 * i]), __uint_as_float(cur[2 * i + 1])), r2);
                            acc[8 * gi + i] = __ffma2_rn(p, make_float2(c, c), acc[8 * gi + i]);
                        }
                    }
                };
                tmem_ld_wait();
                if (G <= D) release_buffer();
#pragma unroll
                for (int gi = 0; gi < G; ++gi) {
                    consume_group(gi, v[gi % D]);
                    if constexpr (D == G) {
                        // the whole chunk was loaded at once
                    } else if constexpr (SCALE == SCALE_VEC_B) {
                        // D loads from the start, the others as registers become free, and one wait for all of them: the buffer goes
                        // back after G - D groups' worth of multiplications (waiting for the last load later, with the buffer handed back
                        // later too: 2-4 % slower)
                        if ((gi & 1) && (gi >> 1) + 2 < G / 2) { cf[(gi >> 1) & 1][0] = cfs[gi + 3]; cf[(gi >> 1) & 1][1] = cfs[gi + 4]; }
                        if (gi + D < G) load_group(gi + D, v[gi % D]);
                        if (gi + D == G - 1) { tmem_ld_wait(); release_buffer(); }
                    } else {
                        // Two loads are in flight from the start; each group's FMAs free its registers for the load two groups
                        // on.  A load is waited for one group after it was issued, before the next one is issued (the wait covers
                        // every outstanding load of the thread), so that its latency lies under that group's FMAs and no group is
                        // consumed before its load has been waited for.  The buffer goes back to the MMA warp when the last load
                        // has landed; the last group follows the release.
                        if (gi >= 1 && gi + 1 < G) tmem_ld_wait();                   // group gi+1 has landed
                        if (gi + 2 < G) load_group(gi + 2, v[gi & 1]);
                        if (G > 2 && gi + 2 == G) release_buffer();                  // ... and it was the chunk's last load
                    }
                }
                if (SCALE == SCALE_VEC_B && (cc % C::kVecBlock) == C::kVecBlock - 1) {
                    __syncwarp();                        // every lane has read the block's slots
                    if (lane == 0) mbar_arrive(vempty_bar(vd / C::kVecBlock));
                }
            }
            if constexpr (CLUSTER) {
                // A slice of a tile whose other slices are in this cluster (the CTA's only item).  The sums of fragment group gi belong to
                // slice gi * nsl / G: every CTA writes the groups of the others into their stage memory, which no copy or MMA uses any
                // more once all CTAs are here, and then adds its own groups in slice order and stores them.  Nothing is sent through L2
                // and no CTA adds the whole tile: 8192 tokens x 256 x 2048 20.6 -> 16.5 us, 16384 x 512 x 1024 28.7 -> 22.9 us.  A CTA that gave
                // up a wait takes part in both barriers all the same; before the second one it raises the abort flag of every CTA here, because
                // none of them has the tile's sums then.
                const int me = wi.slice, nsl = wi.nsl, per = (G + nsl - 1) / nsl;
                float *av = reinterpret_cast<float *>(acc);
                auto owner = [&](int gi) { return gi * nsl / G; };
                auto slot = [&](int from, int gi) {   // of group gi, sent by slice `from`, in its owner's stage memory: [sender][warp][group][quad][lane]
                    const int k = gi - (owner(gi) * G + nsl - 1) / nsl;
                    return (uint32_t)((((from * kNumEpiWarps + e) * per + k) * 4) * 512 + lane * 16);
                };
                cluster_sync();
                if (e == 0 && lane < nsl && *abort_flag) st_cluster_u32(mapa(smem_u32(const_cast<uint32_t *>(abort_flag)), (uint32_t)lane), 1u);
                if (ok) {
#pragma unroll
                    for (int gi = 0; gi < G; ++gi) {
                        if (owner(gi) != me) {
                            const uint32_t dst = mapa(smem_base + slot(me, gi), (uint32_t)owner(gi));
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                st_cluster_v4(dst + 512u * j, make_float4(av[16 * gi + 4 * j], av[16 * gi + 4 * j + 1], av[16 * gi + 4 * j + 2], av[16 * gi + 4 * j + 3]));
                        }
                    }
                }
                cluster_sync();
                ok = !*abort_flag;
                if (ok) {
#pragma unroll
                    for (int gi = 0; gi < G; ++gi) {
                        if (owner(gi) == me) {
                            float t[16];
                            for (int sl = 0; sl < nsl; ++sl) {
                                float u[16];
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    const float4 x = sl == me ? make_float4(av[16 * gi + 4 * j], av[16 * gi + 4 * j + 1], av[16 * gi + 4 * j + 2], av[16 * gi + 4 * j + 3])
                                                              : *reinterpret_cast<const float4 *>(smem_gen + slot(sl, gi) + 512 * j);
                                    u[4 * j] = x.x; u[4 * j + 1] = x.y; u[4 * j + 2] = x.z; u[4 * j + 3] = x.w;
                                }
#pragma unroll
                                for (int j = 0; j < 16; ++j) t[j] = sl == 0 ? u[j] : t[j] + u[j];
                            }
                            store_frag<OUT_F32>(g, row0 + 16 * (gi & 1) + (lane >> 2), col0 + 32 * (gi >> 1), t, lane);
                        }
                    }
                }
            } else {
                cp_async_wait<0>();
                if (ok) {
                    if (C::kTmaOut && !g.accumulate) {
                        // round, stage 32 rows x 64 bytes in shared memory (16-byte chunks XOR-swizzled the way
                        // the output tensor map's 64-byte swizzle expects) and let the TMA unit write each box;
                        // rows and columns outside the matrix are clipped by the hardware
                        constexpr int kPerBox = OUT_F32 ? 16 : 32;   // output columns per 64-byte box row
#pragma unroll
                        for (int b = 0; b < HALF / kPerBox; ++b) {
                            if (lane == 0) bulk_wait_read<C::kOutSlots - 1>();     // the box that was in this staging tile has left it
                            __syncwarp();
                            const float *src = reinterpret_cast<const float *>(acc) + b * kPerBox;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                uint4 o;
                                if (OUT_F32) o = make_uint4(__float_as_uint(src[4 * j]), __float_as_uint(src[4 * j + 1]), __float_as_uint(src[4 * j + 2]), __float_as_uint(src[4 * j + 3]));
                                else o = make_uint4(pack_bf16x2(src[8 * j], src[8 * j + 1]), pack_bf16x2(src[8 * j + 2], src[8 * j + 3]),
                                                    pack_bf16x2(src[8 * j + 4], src[8 * j + 5]), pack_bf16x2(src[8 * j + 6], src[8 * j + 7]));
                                st_shared_v4(stage_u32 + (b % C::kOutSlots) * 2048 + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4), o);
                            }
                            fence_proxy_async();
                            __syncwarp();
                            const int col = col0 + b * kPerBox;
                            if (lane == 0) {
                                if (col < g.No && row0 < g.Mo) tma_store_2d(&tmO, stage_u32 + (b % C::kOutSlots) * 2048, col, row0);
                                bulk_commit();   // one group per box, empty outside the matrix: the wait above counts groups
                            }
                        }
                    } else {
                        bool write_out = true;
                        if (SCALE == SCALE_VEC_B && wi.nsl > 1) {
                            // A slice of a sliced tile: this warp's 32 x HALF sums go to the slice's slot (512 contiguous bytes
                            // per store instruction); the warp that delivers a sub-tile's last slice adds all slices in slice
                            // order, whoever came last, so the result does not depend on the order of arrival.
                            float *av = reinterpret_cast<float *>(acc);
                            constexpr size_t kWarpFloats = 32 * HALF;
                            constexpr int kWarps = kNumEpiWarps * C::kCtas;   // promotion warps of a tile
                            const int ew = (int)rank * kNumEpiWarps + e;
                            float *first = g.partials + (size_t)(wi.tail * wi.nsl) * kWarps * kWarpFloats + ew * kWarpFloats + lane * 4;
                            float *mine = first + (size_t)wi.slice * kWarps * kWarpFloats;
#pragma unroll
                            for (int j4 = 0; j4 < HALF / 4; ++j4)
                                __stcg(reinterpret_cast<float4 *>(mine + j4 * 128), make_float4(av[4 * j4], av[4 * j4 + 1], av[4 * j4 + 2], av[4 * j4 + 3]));
                            __threadfence();
                            __syncwarp();
                            uint32_t old = 0;
                            if (lane == 0) old = atomicAdd(g.counters + wi.tail * kWarps + ew, 1u);
                            old = __shfl_sync(0xFFFFFFFFu, old, 0);
                            write_out = (old == (uint32_t)wi.nsl - 1u);
                            if (write_out) {
                                __threadfence();
                                // The loads of half a warp's share of a slice are in flight together: 2 L2 round trips per slice (one per 16
                                // bytes: 25 us at the end of every sliced launch).  Narrow tiles have registers for half a share of all slices
                                // (22.5 -> 20.6 us for 8192 tokens x 256 x 2048; with 128 sums per thread it would spill).
                                if constexpr (HALF <= 64) {
                                    constexpr int kBatch = HALF / 8;
#pragma unroll
                                    for (int b0 = 0; b0 < HALF / 4; b0 += kBatch) {
                                        float4 u[kMaxSlices][kBatch];
#pragma unroll
                                        for (int sl = 0; sl < kMaxSlices; ++sl) {
                                            const float *src = first + (size_t)sl * kWarps * kWarpFloats + b0 * 128;
                                            if (sl < wi.nsl) {
#pragma unroll
                                                for (int j = 0; j < kBatch; ++j) u[sl][j] = __ldcg(reinterpret_cast<const float4 *>(src + j * 128));
                                            }
                                        }
#pragma unroll
                                        for (int j = 0; j < kBatch; ++j) {
                                            float4 t = u[0][j];
#pragma unroll
                                            for (int sl = 1; sl < kMaxSlices; ++sl)
                                                if (sl < wi.nsl) { t.x += u[sl][j].x; t.y += u[sl][j].y; t.z += u[sl][j].z; t.w += u[sl][j].w; }
                                            float *d = av + 4 * (b0 + j);
                                            d[0] = t.x; d[1] = t.y; d[2] = t.z; d[3] = t.w;
                                        }
                                    }
                                } else {
#pragma unroll
                                    for (int b0 = 0; b0 < HALF / 4; b0 += HALF / 8) {
                                        for (int sl = 0; sl < wi.nsl; ++sl) {
                                            const float *src = first + (size_t)sl * kWarps * kWarpFloats + b0 * 128;
                                            float4 u[HALF / 8];
#pragma unroll
                                            for (int j = 0; j < HALF / 8; ++j) u[j] = __ldcg(reinterpret_cast<const float4 *>(src + j * 128));
#pragma unroll
                                            for (int j = 0; j < HALF / 8; ++j) {
                                                float *d = av + 4 * (b0 + j);
                                                if (sl == 0) { d[0] = u[j].x; d[1] = u[j].y; d[2] = u[j].z; d[3] = u[j].w; }
                                                else { d[0] += u[j].x; d[1] += u[j].y; d[2] += u[j].z; d[3] += u[j].w; }
                                            }
                                        }
                                    }
                                }
                            }
                        }
                        if constexpr (SCALE == SCALE_VEC_B) {
                            if (write_out) {
#pragma unroll
                                for (int gi = 0; gi < G; ++gi)
                                    store_frag<OUT_F32>(g, row0 + 16 * (gi & 1) + (lane >> 2), col0 + 32 * (gi >> 1), reinterpret_cast<const float *>(acc) + 16 * gi, lane);
                            }
                        } else if (write_out && row_ok) {
#pragma unroll
                            for (int gi = 0; gi < HALF / 32; ++gi) store32<OUT_F32>(g, row, col0 + 32 * gi, reinterpret_cast<const float *>(acc) + 32 * gi);
                        }
                    }
                }
                __syncwarp();
            }
        }
        if (lane == 0) bulk_wait_all0();   // outstanding output stores have read their staging tiles
    }

    // ---- teardown: every role ends here, tensor memory is always released ------------------
    __syncwarp();
    chain_finish(g.chain);
    tc_fence_before_sync();
    __syncthreads();
    if (PAIR) cluster_sync();   // no more arrivals from the other CTA, and the pair's MMAs read no more of this CTA's memory
    if (*abort_flag) {
        // give copies and MMAs still in flight time to land before the CTA's resources go away
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
        if (threadIdx.x == 0) status_report(g.status, g.status_mark, (uint32_t)SNIP_ERR_TIMEOUT, g.wait_limit_ns);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc<PAIR>(tmem_base, C::kTmemCols);
    }
}

// ---- host side ---------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Tensor map over a row-major [rows][kc] operand whose rows are `row_bytes` apart, fetched in
// boxes of (128 bytes of K) x box_rows with the 128-byte swizzle.
int make_operand_map(CUtensorMap *map, const void *ptr, CUtensorMapDataType dt, int64_t rows, int64_t kc_elems,
                     int64_t row_bytes, int box_x_elems, int box_rows, CUtensorMapSwizzle swz = CU_TENSOR_MAP_SWIZZLE_128B)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) { snprintf(last_error_buffer(), 256, "cuTensorMapEncodeTiled entry point not found"); return SNIP_ERR_CUDA; }
    cuuint64_t dims[2] = {(cuuint64_t)kc_elems, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
    cuuint32_t box[2] = {(cuuint32_t)box_x_elems, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, dt, 2, const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(last_error_buffer(), 256, "cuTensorMapEncodeTiled failed: CUresult %d (rows %lld, k %lld, row bytes %lld, dtype %d)",
                 (int)r, (long long)rows, (long long)kc_elems, (long long)row_bytes, (int)dt);
        return SNIP_ERR_CUDA;
    }
    return SNIP_OK;
}

int sm_count()
{
    static thread_local int dev_cached = -1, n = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != dev_cached) { cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev); dev_cached = dev; }
    return n;
}

// Clusters of `size` CTAs of the 128-wide weight-gradient kernel that find a place on the current device together (a cluster's CTAs share
// a GPC, so this is less than SMs / size); 0 if it cannot be told.  The occupancy query answers for an idle device.  Clusters of two and
// four fit up to that number also where they take over SMs one by one from the kernel ahead (74 and 33 of them, 60 runs each behind CTAs
// that ended at random), but three CTAs are one and a half pairs of SMs: of 45 clusters up to four were left waiting for others to end,
// 42 had one left in 1 run of 10, 41 none.  So odd sizes keep a tenth back.  4096 tokens, 45 tiles of 128 x 128, calls in a row: three
// slices 27.2 us, two 16.0 us.
int max_clusters(int size)
{
    static thread_local int dev_cached = -1, n[kMaxSlices + 1];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != dev_cached) {
        for (int c = 2; c <= kMaxSlices; ++c) {
            using C = Cfg<MmaKind::F8F6F4, 128, SCALE_VEC_B, false>;
            auto kern = gemm_kernel<MmaKind::F8F6F4, 128, SCALE_VEC_B, false, false, true>;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)c; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(c * (sm_count() / c)));
            cfg.blockDim = dim3(kGemmThreads);
            cfg.dynamicSmemBytes = C::kSmemBytes;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            n[c] = 0;
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&n[c], kern, &cfg) != cudaSuccess) {
                n[c] = 0;
                cudaGetLastError();
            }
            if (c & 1) n[c] -= n[c] / 10;
        }
        dev_cached = dev;
    }
    return size >= 2 && size <= kMaxSlices ? n[size] : 0;
}

// All tiles in slices, the slices of a tile in a cluster, where all clusters run at the same time and slicing saves what the exchange costs;
// nsplit == 1: not so.  128-wide tiles on one CTA each.  In a chain the product starts beside others, on free_sms SMs: where its whole tiles
// fit there and its slices do not, those that would wait for an SM cost more than a few stages saved (one layer, FP8, us whole / in two slices:
// 3072 tokens 256 -> 4608 48.0 / 56.8, 1024 -> 1024 35.3 / 37.7; where neither fits, 3584 tokens 1152 -> 1024 44.2 / 41.1).
WorkSplit plan_clusters(int num_tiles, int num_stages, bool slice, int free_sms)
{
    for (int ns = kMaxSlices; slice && ns > 1; --ns) {
        const int saved = num_stages - num_stages / ns;
        if (num_stages / ns < kMinSliceStages || saved < kMinSavedStagesCluster || num_tiles > max_clusters(ns)) continue;
        if (saved < kMinSavedStages && num_tiles <= free_sms && num_tiles * ns > free_sms) continue;
        return {0, ns, num_tiles * ns};
    }
    return {num_tiles, 1, num_tiles};
}

// SMs that a chain's third GEMM, the weight gradient, finds free when it starts (which is when all CTAs of the second one have started): all
// but those on which a CTA of the second one had to wait for one of the first to end.  ctas: what the first two launched.
int free_beside(const int32_t *ctas, int sms)
{
    const int late = ctas[1] - (sms - ctas[0]);
    return late > 0 ? sms - late : sms;
}

// Host side of a launch.
struct LaunchEnv {
    bool cleared;       // status word and slice counters are zero when the kernel starts
    int32_t free_sms;   // SMs that are free when it starts
    int32_t *ctas;      // a chain's count of this GEMM's CTAs, or null
    cudaStream_t st;
};

thread_local int last_gemm[4];   // see snip_debug_last_gemm

// 128-wide tiles: slices in clusters, or fewer chunks each and the dearer exchange through the workspace?  Clusters fill the chip less well
// (45 tiles: two slices each, 90 of 148 SMs, against three), so long contractions go through the workspace.  us, clusters / workspace: 45
// tiles of 64 chunks 22.0 / 22.9, 76 24.6 / 24.6, 118 33.2 / 30.9, 256 61.5 / 50.4; 36 tiles (three against four) of 118 26.3 / 26.7, 160
// 32.0 / 31.6, 256 44.7 / 41.6.
bool prefer_clusters(const WorkSplit &clusters, const WorkSplit &workspace, int num_chunks)
{
    if (clusters.nsplit == 1 || workspace.nsplit == 1) return clusters.nsplit > 1;   // (whole tiles: plan_clusters has weighed them)
    return (float)num_chunks / clusters.nsplit + kMinSavedStagesCluster <= (float)num_chunks / workspace.nsplit + kWorkspaceExchangeChunks;
}

template <MmaKind KIND, int BN, int SCALE, bool PAIR, bool OUT_F32>
int launch_gemm(const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmO, const GemmArgs &g, uint32_t idesc, const LaunchEnv &env)
{
    using C = Cfg<KIND, BN, SCALE, PAIR>;
    const int num_tiles = (int)(ceil_div(g.Mo, C::BM) * ceil_div(g.No, BN)), num_stages = (int)ceil_div(g.Kc, C::kStageK);
    const int units = sm_count() / C::kCtas;
    const bool slice = SCALE == SCALE_VEC_B && g.partials;
    GemmArgs ga = g;
    auto launch = [&](auto kern, int cluster) -> int {
        // a per-function, per-device attribute; setting it on every launch is cheap and correct on any device
        SNIP_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes));
        const int grid = (ga.work.num_items < units ? ga.work.num_items : units) * C::kCtas;
        last_gemm[0] = BN; last_gemm[1] = C::kCtas; last_gemm[2] = ga.work.nsplit; last_gemm[3] = cluster;
        if (env.ctas) *env.ctas = grid;
        return launch_chained(kern, grid, kGemmThreads, C::kSmemBytes, env.st, cluster, tmA, tmB, tmO, ga, idesc);
    };
    ga.work = plan_work(num_tiles, num_stages, units, kMinSliceStages, kMinSavedStages, slice, kMaxSlicedItems / C::kCtas);
    if constexpr (C::kClusterSlices) {
        const WorkSplit cl = plan_clusters(num_tiles, num_stages, slice, env.free_sms);
        if (prefer_clusters(cl, ga.work, (int)ceil_div(g.Kc, C::kChunkElems))) {
            ga.work = cl;
            return launch(gemm_kernel<KIND, BN, SCALE, PAIR, OUT_F32, true>, cl.nsplit);
        }
    }
    if (ga.work.nsplit > 1 && !env.cleared)
        SNIP_CUDA_TRY(cudaMemsetAsync(g.counters, 0, (size_t)(num_tiles - ga.work.split_first) * kNumEpiWarps * C::kCtas * sizeof(uint32_t), env.st));
    return launch(gemm_kernel<KIND, BN, SCALE, PAIR, OUT_F32, false>, C::kCtas);
}

template <MmaKind KIND, int BN, int SCALE>
int launch_gemm_form(bool pair, bool out_f32, const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmO, const GemmArgs &g, uint32_t idesc,
                     const LaunchEnv &env)
{
    if (pair)
        return out_f32 ? launch_gemm<KIND, BN, SCALE, true, true>(tmA, tmB, tmO, g, idesc, env)
                       : launch_gemm<KIND, BN, SCALE, true, false>(tmA, tmB, tmO, g, idesc, env);
    return out_f32 ? launch_gemm<KIND, BN, SCALE, false, true>(tmA, tmB, tmO, g, idesc, env)
                   : launch_gemm<KIND, BN, SCALE, false, false>(tmA, tmB, tmO, g, idesc, env);
}
template <MmaKind KIND, int BN>
int launch_gemm_scale(int scale, bool pair, bool out_f32, const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmO, const GemmArgs &g,
                      uint32_t idesc, const LaunchEnv &env)
{
    return scale == SCALE_BLOCK_B ? launch_gemm_form<KIND, BN, SCALE_BLOCK_B>(pair, out_f32, tmA, tmB, tmO, g, idesc, env)
                                  : launch_gemm_form<KIND, BN, SCALE_VEC_B>(pair, out_f32, tmA, tmB, tmO, g, idesc, env);
}

// 128-wide tiles, one CTA each.
template <MmaKind KIND>
int launch_gemm_narrow(int scale, bool out_f32, const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmO, const GemmArgs &g, uint32_t idesc,
                     const LaunchEnv &env)
{
    if (scale == SCALE_BLOCK_B)
        return out_f32 ? launch_gemm<KIND, 128, SCALE_BLOCK_B, false, true>(tmA, tmB, tmO, g, idesc, env)
                       : launch_gemm<KIND, 128, SCALE_BLOCK_B, false, false>(tmA, tmB, tmO, g, idesc, env);
    return out_f32 ? launch_gemm<KIND, 128, SCALE_VEC_B, false, true>(tmA, tmB, tmO, g, idesc, env)
                   : launch_gemm<KIND, 128, SCALE_VEC_B, false, false>(tmA, tmB, tmO, g, idesc, env);
}

}  // namespace

size_t gemm_ws_bytes() { return 256; }
// Workspace with which the weight-gradient product may slice the tiles of its last wave along the contraction:
// status word, arrival counters, one FP32 tile per slice.
size_t gemm_ws_bytes_sliced() { return kSliceCountersOffset + kSliceCountersBytes + (size_t)kMaxSlicedItems * CM * 256 * sizeof(float); }

// (gemm_bf16.cu slices the same way.)
// The parts of a workspace of gemm_ws_bytes() or gemm_ws_bytes_sliced(), for one GEMM.
GemmWs gemm_ws(void *ws, size_t ws_bytes)
{
    GemmWs w;
    w.status = static_cast<uint32_t *>(ws);
    if (ws_bytes >= gemm_ws_bytes_sliced()) {
        w.counters = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(ws) + kSliceCountersOffset);
        w.partials = reinterpret_cast<float *>(static_cast<uint8_t *>(ws) + kSliceCountersOffset + kSliceCountersBytes);
    }
    return w;
}
// What a chain's first kernel clears of it: status word and counters.
int32_t gemm_ws_zero_words() { return (int32_t)((kSliceCountersOffset + kSliceCountersBytes) / sizeof(uint32_t)); }

// Testing hooks (snip_debug_set): process-wide, off by default.
namespace {
std::atomic<long long> g_wait_limit_ns{2000000000ll};   // bound of every device-side wait of the GEMM kernels
std::atomic<int> g_tx_skew{0};                           // bytes added to what a stage's barrier expects (a wait that cannot complete)
std::atomic<int> g_slicing{1};                           // 0: the weight-gradient product never slices its last wave
std::atomic<int> g_kernel_choice{0};                     // 0 = by shape, 1 = single-CTA form, 2 = CTA-pair form, 3 = 128-wide tiles (paper-rule kernels)
}  // namespace

// The hooks' current values, for the other GEMM families (gemm_mx.cu).
void gemm_debug_hooks(uint64_t *wait_limit_ns, int *tx_skew)
{
    *wait_limit_ns = (uint64_t)g_wait_limit_ns.load();
    *tx_skew = g_tx_skew.load();
}

bool gemm_slicing_enabled() { return g_slicing.load() != 0; }

int gemm_bf16_impl(const void *a, bool a_mn, const void *b, bool b_mn, int64_t Mo, int64_t No, int64_t Kc, void *out, int out_dtype, int accumulate,
                   const GemmWs &w, cudaStream_t st, const ChainLink &link);   // gemm_bf16.cu

uint32_t status_mark(bool cleared)
{
    static std::atomic<uint32_t> next{1};
    if (cleared) return 0;
    const uint32_t m = next.fetch_add(1);
    return m ? m : next.fetch_add(1);
}

// Shared with the power-of-two-scale GEMMs: 2-D tiled tensor map over a row-major matrix.
int make_tiled_map_2d(CUtensorMap *map, const void *ptr, int dtype, int64_t rows, int64_t inner_elems, int64_t row_bytes, int box_x_elems,
                      int box_rows, int swizzle)
{
    return make_operand_map(map, ptr, static_cast<CUtensorMapDataType>(dtype), rows, inner_elems, row_bytes, box_x_elems, box_rows,
                            static_cast<CUtensorMapSwizzle>(swizzle));
}
int gemm_sm_count() { return sm_count(); }

// Core GEMM over stored operands.  a_codes: [Mo][Kc] and b_codes: [No][Kc], contraction-major.
// scale_mode: SCALE_BLOCK_B (fwd / dgrad) or SCALE_VEC_B (wgrad); unused for BF16.  mn: BF16 operands stored [Kc][lines] instead (bit 0: A,
// bit 1: B).
int gemm_impl(int fmt_a, int fmt_b, const void *a_codes, const void *b_codes, int64_t Mo, int64_t No, int64_t Kc, const float *sa,
              int64_t sa_chunk_stride, const float *sb, int64_t sb_chunk_stride, int64_t sb_blk_stride, int scale_mode, void *out,
              int out_dtype, int accumulate, const GemmWs &w, cudaStream_t st, const ChainLink &link, int mn)
{
    if (!a_codes || !b_codes || !out) return SNIP_ERR_ARG;
    if (!valid_dim(Mo) || !valid_dim(No) || !valid_dim(Kc) || Mo > INT32_MAX || No > INT32_MAX || Kc > INT32_MAX) return SNIP_ERR_SHAPE;
    if (out_dtype != SNIP_OUT_BF16 && out_dtype != SNIP_OUT_FP32) return SNIP_ERR_ARG;
    if (accumulate && out_dtype != SNIP_OUT_FP32) return SNIP_ERR_UNSUPPORTED;
    if (!w.status) return SNIP_ERR_WORKSPACE;
    if (!aligned16(a_codes) || !aligned16(b_codes) || !aligned16(out) || !aligned16(w.status)) return SNIP_ERR_ALIGN;
    const bool a16 = fmt_a == SNIP_FMT_BF16, b16 = fmt_b == SNIP_FMT_BF16;
    if (a16 != b16) return SNIP_ERR_UNSUPPORTED;
    if (!a16 && (!sa || !sb)) return SNIP_ERR_ARG;
    if (!a16 && (!aligned16(sa) || !aligned16(sb))) return SNIP_ERR_ALIGN;   // scale factors are fetched 16 bytes at a time
    int rc = require_sm100();
    if (rc != SNIP_OK) return rc;
    if (a16) return gemm_bf16_impl(a_codes, mn & 1, b_codes, mn & 2, Mo, No, Kc, out, out_dtype, accumulate, w, st, link);

    GemmArgs g;
    g.Mo = (int32_t)Mo; g.No = (int32_t)No; g.Kc = (int32_t)Kc;
    g.sa = sa; g.sa_chunk_stride = sa_chunk_stride;
    g.sb = sb; g.sb_chunk_stride = sb_chunk_stride; g.sb_blk_stride = sb_blk_stride;
    g.out = out; g.ldo = No; g.accumulate = accumulate;
    g.status = w.status;
    g.status_mark = status_mark(w.cleared);
    g.chain = link.role;
    if (link.jobs) g.stats = *link.jobs;
    g.partials = nullptr; g.counters = nullptr;
    if (scale_mode == SCALE_VEC_B && w.partials && g_slicing.load()) {
        g.counters = w.counters;
        g.partials = w.partials;
    }
    g.stage_tx_bytes = 0;
    g.tx_skew = (uint32_t)g_tx_skew.load();
    g.wait_limit_ns = (uint64_t)g_wait_limit_ns.load();
    const bool f32 = out_dtype == SNIP_OUT_FP32;
    LaunchEnv env = {w.cleared, sm_count(), nullptr, st};
    if (link.ctas) {
        int i = 0;
        while (i < 2 && link.ctas[i]) ++i;
        env.ctas = link.ctas + i;
        if (i == 2) env.free_sms = free_beside(link.ctas, sm_count());
    }

    // Pairs of CTAs on 256-row tiles halve a CTA's share of B and keep six stages instead of four: forward and input gradient 2-4 % faster
    // (FP8 16384x12288x4096 837 -> 808 us, 8192x8640x3200 248 -> 239 us, FP4 655 -> 635 us).  The weight gradient, whose promotion sets the pace,
    // gains nothing (FP8 1062 / 1059 us, FP4 950 / 956 us) and neither do shapes with fewer such tiles than pairs of SMs.
    const int choice = g_kernel_choice.load();
    auto use_pair = [&](int tile_n) {
        if (choice != 0) return choice == 2;
        return scale_mode == SCALE_BLOCK_B && ceil_div(Mo, 256) * ceil_div(No, tile_n) >= sm_count() / 2;
    };

    // Tiles 128 columns wide, one CTA each, where they shorten the launch: as a rule where the wider tiles leave more than half of the SMs idle,
    // so that twice the tiles still are one wave (forward FP8 1024x2048x4096 18.0 -> 12.5 us, 8192x256x2048 11.2 -> 8.3 us, 512x512x512 6.6 -> 5.2
    // us; FP4 1024x4096x4096, two waves either way, 24.8 -> 18.6 us; weight gradient 8192x256x2048 28.6 -> 20.6 us).  A launch lasts as long as
    // the pipeline stages that its SMs run one after the other (kMinSavedStages more where its last wave is sliced) times what a stage of a narrow
    // tile takes next to a wide one's: measured 0.64-0.68 forward and input gradient (one-CTA forms; against pairs FP8 is at 0.57-0.63 by now, three waves to two of
    // 4096 features 29.8 us narrow, 32.4 us wide, and still goes by 0.68), 0.69-0.79 weight gradient.  FP4 against pairs 192 wide
    // 0.70-0.72 (1536 columns of 22-132 row tiles over 4096 features, us narrow / wide: 2 waves to 2 18.3 / 24.9, 5 to 4 41 / 46, 4 to 3 33.4 / 35.6, 11 to 8 87 / 89,
    // 7 to 5 55.9 / 56.8, 3 to 2 25.8 / 25.0).  In a layer the next product takes over the SMs that a last wave leaves idle, so that whole waves
    // count for less there and the line lies at 0.76 (one layer, us with it at 0.72 / 0.76: 8192 x 8640 -> 3200, 11 to 8, 714 / 706, 2816 x 2496 ->
    // 3200, 4 to 3, 109.4 / 104.1, 4864 x 1920 -> 1792, 4 to 3, 92.5 / 94.1), and in the weight gradient, whose narrow stages take more (3264
    // tokens, 2112 -> 3904 131.6 / 124.0 us).
    auto use_narrow = [&](int tile_n, int stage_k, float ratio) {
        if (choice != 0) return choice == 3;
        auto stages = [&](int bn) {
            const int sms = sm_count(), tiles = (int)(ceil_div(Mo, CM) * ceil_div(No, bn)), per_tile = (int)ceil_div(Kc, stage_k);
            const bool slice = scale_mode == SCALE_VEC_B && g.partials;
            const WorkSplit sp = plan_work(tiles, per_tile, sms, kMinSliceStages, kMinSavedStages, slice);
            const WorkSplit cl = plan_clusters(tiles, per_tile, slice && bn == 128, env.free_sms);
            if (prefer_clusters(cl, sp, (int)ceil_div(Kc, 128))) return (float)per_tile / cl.nsplit + kMinSavedStagesCluster;
            if (sp.nsplit > 1) return (float)(sp.split_first / sms) * per_tile + (float)per_tile / sp.nsplit + kMinSavedStages;
            return (float)ceil_div(tiles, sms) * per_tile;
        };
        return stages(128) * ratio < stages(tile_n);
    };

    CUtensorMap tmA, tmB, tmO;
    // output boxes of 32 rows x 64 bytes for the TMA stores of the block-mode epilogue
    rc = f32 ? make_operand_map(&tmO, out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, Mo, No, No * 4, 16, 32, CU_TENSOR_MAP_SWIZZLE_64B)
             : make_operand_map(&tmO, out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Mo, No, No * 2, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
    if (rc) return rc;
    if (fmt_a == SNIP_FMT_FP4_E2M1 && fmt_b == SNIP_FMT_FP4_E2M1 && (scale_mode == SCALE_BLOCK_B || (Kc % 128) != 0)) {
        // Packed FP4 on both sides, forward / input gradient, or a contraction length ending in a 64-wide tile: kind::mxf4 on the
        // packed bytes (fetched as plain u8, exact extents).  Its 128x192 tile (what tensor memory allows next to the scale
        // factors) does a quarter less per hand-off than the 128x256 tile of kind::f8f6f4, but a chunk's sums fit in the promotion
        // warps' registers at once, and with half the operand bytes and a quarter of the tensor time it stays below the power
        // cap: 16384x12288x4096 755 -> 673 us, 8192x3200x8640 215 -> 193 us, 8192x2048x256 16.4 -> 14.5 us.  The weight gradient over
        // whole chunks takes the path below: with two operations per element the wider tile is as fast or faster.
        const bool narrow = use_narrow(192, 256, scale_mode == SCALE_BLOCK_B && !link.ctas ? 0.72f : 0.76f);
        const int BN = narrow ? 128 : 192;
        const bool pair = !narrow && use_pair(BN);
        const int ctas = pair ? 2 : 1;
        rc = make_operand_map(&tmA, a_codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, Mo, Kc / 2, Kc / 2, 128, CM);
        if (rc) return rc;
        rc = make_operand_map(&tmB, b_codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, No, Kc / 2, Kc / 2, 128, BN / ctas);
        if (rc) return rc;
        const uint32_t idesc = make_idesc_block_scaled(1, 1, CM * ctas, BN);
        g.stage_tx_bytes = (CM + BN / ctas) * 128 + g.tx_skew;
        if (narrow) return launch_gemm_narrow<MmaKind::MXF4>(scale_mode, f32, tmA, tmB, tmO, g, idesc, env);
        return launch_gemm_scale<MmaKind::MXF4, 192>(scale_mode, pair, f32, tmA, tmB, tmO, g, idesc, env);
    }
    // FP8 x FP8, the mixed pairs and the FP4 x FP4 weight gradient over whole chunks: kind::f8f6f4; FP4 operands are expanded by
    // the TMA unit to one 16-byte-aligned group per 16 elements, which is the layout this MMA kind reads
    const bool narrow = use_narrow(256, 128, scale_mode == SCALE_BLOCK_B ? 0.68f : 0.75f);
    const int BN = narrow ? 128 : 256;
    const bool pair = !narrow && use_pair(BN);
    const int ctas = pair ? 2 : 1;
    const bool a4 = fmt_a == SNIP_FMT_FP4_E2M1, b4 = fmt_b == SNIP_FMT_FP4_E2M1;
    // The expanding 4-bit tensor-map type only accepts an inner extent that is a multiple of 128
    // elements.  A contraction length ending in a 64-wide tile is therefore declared rounded up: the
    // extra 64 codes of each row are the first codes of the next row (for the last row, 32 bytes of
    // the slack that snip_quantize_sizes reserves); they meet zero-filled FP8 codes of the other
    // operand, whose map has the exact extent, so they contribute nothing.  (Two FP4 operands with such a
    // length never get here: both maps would be padded.)
    const int64_t kpad = ceil_div(Kc, 128) * 128;
    rc = make_operand_map(&tmA, a_codes, a4 ? CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B : CU_TENSOR_MAP_DATA_TYPE_UINT8, Mo, a4 ? kpad : Kc,
                          a4 ? Kc / 2 : Kc, 128, CM);
    if (rc) return rc;
    rc = make_operand_map(&tmB, b_codes, b4 ? CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B : CU_TENSOR_MAP_DATA_TYPE_UINT8, No, b4 ? kpad : Kc,
                          b4 ? Kc / 2 : Kc, 128, BN / ctas);
    if (rc) return rc;
    const uint32_t idesc = make_idesc(a4 ? 5 : 0, b4 ? 5 : 0, CM * ctas, BN);
    // an FP4 operand expanded by the TMA unit occupies 128 B per row in shared memory but reports
    // only its 64 packed source bytes to the barrier
    g.stage_tx_bytes = CM * (a4 ? 64 : 128) + BN / ctas * (b4 ? 64 : 128) + g.tx_skew;
    if (narrow) return launch_gemm_narrow<MmaKind::F8F6F4>(scale_mode, f32, tmA, tmB, tmO, g, idesc, env);
    return launch_gemm_scale<MmaKind::F8F6F4, 256>(scale_mode, pair, f32, tmA, tmB, tmO, g, idesc, env);
}

}  // namespace snip

extern "C" int snip_gemm_quantized(int op, const snip_qtensor_t *a, const snip_qtensor_t *b, void *out, int out_dtype,
                                   int accumulate, void *ws, size_t ws_bytes, void *stream)
{
    using namespace snip;
    if (!a || !b || op < SNIP_OP_FWD || op > SNIP_OP_WGRAD) return SNIP_ERR_ARG;
    if (!valid_fmt(a->fmt) || !valid_fmt(b->fmt)) return SNIP_ERR_ARG;
    const bool q = a->fmt != SNIP_FMT_BF16;
    int64_t Mo, No, Kc;
    const float *sa = a->scales, *sb = b->scales;
    int64_t sa_cs, sb_cs, sb_bs;
    int mode;
    if (op == SNIP_OP_FWD) {
        // A = X[M,K] ROW tiles, B = W[N,K] blocks
        if (a->cols != b->cols || a->transposed || b->transposed) return SNIP_ERR_SHAPE;
        if (q && (a->block != SNIP_BLOCK_ROW_1x128 || b->block != SNIP_BLOCK_BLK_128x128)) return SNIP_ERR_UNSUPPORTED;
        Mo = a->rows; No = b->rows; Kc = a->cols;
        sa_cs = Mo; sb_bs = ceil_div(Kc, 128); sb_cs = 1; mode = SCALE_BLOCK_B;
    } else if (op == SNIP_OP_DGRAD) {
        // A = dY[M,N] ROW tiles, B = W[N,K] blocks stored transposed ([K,N])
        if (a->cols != b->rows || a->transposed || !b->transposed) return SNIP_ERR_SHAPE;
        if (q && (a->block != SNIP_BLOCK_ROW_1x128 || b->block != SNIP_BLOCK_BLK_128x128)) return SNIP_ERR_UNSUPPORTED;
        Mo = a->rows; No = b->cols; Kc = a->cols;
        sa_cs = Mo; sb_bs = 1; sb_cs = ceil_div(No, 128); mode = SCALE_BLOCK_B;
    } else {
        // A = dY[M,N] COL tiles stored transposed ([N,M]), B = X[M,K] COL tiles stored transposed ([K,M])
        if (a->rows != b->rows || !a->transposed || !b->transposed) return SNIP_ERR_SHAPE;
        if (q && (a->block != SNIP_BLOCK_COL_128x1 || b->block != SNIP_BLOCK_COL_128x1)) return SNIP_ERR_UNSUPPORTED;
        Mo = a->cols; No = b->cols; Kc = a->rows;
        sa_cs = Mo; sb_cs = No; sb_bs = 0; mode = SCALE_VEC_B;
    }
    if (!ws || ws_bytes < gemm_ws_bytes()) return SNIP_ERR_WORKSPACE;
    return gemm_impl(a->fmt, b->fmt, a->codes, b->codes, Mo, No, Kc, sa, sa_cs, sb, sb_cs, sb_bs, mode, out, out_dtype, accumulate,
                     gemm_ws(ws, ws_bytes), static_cast<cudaStream_t>(stream), ChainLink(), 0);
}

extern "C" int snip_debug_set(int key, long long value)
{
    using namespace snip;
    switch (key) {
        case SNIP_DEBUG_WAIT_LIMIT_NS: if (value <= 0) return SNIP_ERR_ARG; g_wait_limit_ns.store(value); return SNIP_OK;
        case SNIP_DEBUG_TX_SKEW_BYTES: if (value < 0 || value > 4096 || (value % 16) != 0) return SNIP_ERR_ARG; g_tx_skew.store((int)value); return SNIP_OK;
        case SNIP_DEBUG_GEMM_KERNEL: if (value < 0 || value > 3) return SNIP_ERR_ARG; g_kernel_choice.store((int)value); return SNIP_OK;
        case SNIP_DEBUG_GEMM_SLICING: if (value < 0 || value > 1) return SNIP_ERR_ARG; g_slicing.store((int)value); return SNIP_OK;
        default: return SNIP_ERR_ARG;
    }
}

extern "C" int snip_debug_last_gemm(int plan_host[4])
{
    if (!plan_host) return SNIP_ERR_ARG;
    for (int i = 0; i < 4; ++i) plan_host[i] = snip::last_gemm[i];
    return SNIP_OK;
}

extern "C" int snip_poll_status(const void *ws, int *status_host)
{
    using namespace snip;
    if (!ws || !status_host) return SNIP_ERR_ARG;
    uint32_t v = 0;
    SNIP_CUDA_TRY(cudaMemcpy(&v, ws, sizeof(v), cudaMemcpyDeviceToHost));
    *status_host = (int)v;
    return SNIP_OK;
}
