// BF16 GEMM of the linear layers' BF16-tagged products:  out[Mo,No] = A . B^T with FP32 accumulation on tcgen05.mma kind::f16.
//
// Each operand is read as it lies in memory: [lines][contraction] ("K-major") or [contraction][lines] ("MN-major", the tensor
// core's other operand order for 16-bit types), so the input gradient (W[N,K] contracted over N) and the weight gradient (dY[M,N]
// and X[M,K] contracted over M) need no transposed copies.
//
// One CTA per SM, persistent, 384 threads; tiles of 256 x 256 shared by a pair of CTAs (tcgen05.mma.cta_group::2: each CTA holds 128
// rows of A and of the accumulator and half of B's lines), or 128 x 256 on one CTA where there are few tiles.  Warp 0 streams 64-long
// stages of both operands (TMA, 128-byte swizzle), warp 1 (of the pair's leader) issues the MMAs (one elected lane) into one of two
// 256-column accumulators, warp 2 reduces statistics left by the quantizers ahead, warps 4-11 drain the other accumulator, round and
// store through the TMA unit.  The tiles of the last wave are cut into contraction slices (work_items.cuh) where the workspace has
// room.  Every wait is bounded, as in gemm.cu.
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "quant_device.cuh"
#include "sm100.cuh"
#include "work_items.cuh"

namespace snip {

using namespace sm100;

namespace {

constexpr int CM = 128, BN = 256, HALF = BN / 2;   // rows of a CTA, columns of a tile
constexpr int kThreads = 384, kNumEpiWarps = kSliceWarps;
constexpr int kStageK = 64;                      // elements of the contraction per stage: 128-byte rows
constexpr int kBoxBytes = kStageK * 128;         // MN-major: a box is 64 contraction rows of 64 lines
constexpr int kOutSlots = 2;                     // 2 KB staging tiles per epilogue warp
constexpr int kOutStageBytes = kNumEpiWarps * kOutSlots * 2048;
template <bool PAIR>
struct Cfg {
    static constexpr int kCtas = PAIR ? 2 : 1;
    static constexpr int BM = CM * kCtas;            // rows of a tile
    static constexpr int kBLines = BN / kCtas;       // B lines fetched by a CTA
    static constexpr int kABytes = CM * 128, kBBytes = kBLines * 128, kStageBytes = kABytes + kBBytes;
    static constexpr int kStages = PAIR ? 6 : 4;
    static constexpr int kSmemBytes = kStages * kStageBytes + kOutStageBytes + 256 + 1024;
    static_assert(kSmemBytes <= 232448, "shared memory budget");
};
// Contraction slices: see gemm.cu (0.30 us a stage; 4096 x 1024 x 2048 weight gradient 23.9 us whole, 26.6 us in two slices that save 32 stages)
constexpr int kMinSliceStages = 16, kMinSavedStages = 40;

struct Bf16Args {
    int32_t Mo, No, Kc;
    float *out_acc;            // FP32 output to add to (accumulate), else null: the output map is written
    uint32_t stage_tx_bytes;
    uint64_t wait_limit_ns;
    uint32_t *status;
    uint32_t status_mark;      // see status_begin
    WorkSplit work;
    float *partials;           // see gemm.cu
    uint32_t *counters;
    int32_t chain;
    StatJobs stats;
};

__device__ __forceinline__ uint32_t bf16x2(uint32_t lo, uint32_t hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(lo), __uint_as_float(hi));
    return *reinterpret_cast<uint32_t *>(&v);
}

template <bool PAIR, bool A_MN, bool B_MN, bool OUT_F32>
__global__ void __launch_bounds__(kThreads, 1)
gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmO,
                 const Bf16Args g, const uint32_t idesc)
{
    using C = Cfg<PAIR>;
    constexpr int S = C::kStages, kStageBytes = C::kStageBytes, kABytes = C::kABytes, BM = C::BM;
    extern __shared__ uint8_t smem_raw[];
    chain_acquire(g.chain, g.status);
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    auto a_tile = [&](int s) { return smem_base + s * kStageBytes; };
    auto b_tile = [&](int s) { return smem_base + s * kStageBytes + kABytes; };
    const uint32_t out_stage0 = smem_base + S * kStageBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_gen + S * kStageBytes + kOutStageBytes);
    const uint32_t bar0 = smem_base + S * kStageBytes + kOutStageBytes;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * S + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * S + 2 + a); };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * S + 4);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_m = (g.Mo + BM - 1) / BM, num_n = (g.No + BN - 1) / BN;
    const int num_kstages = g.Kc / kStageK;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;   // 0 = leader: its barriers and its MMA warp serve the pair
    const int unit = (int)blockIdx.x / C::kCtas, units = (int)gridDim.x / C::kCtas;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), kNumEpiWarps * C::kCtas); }
        *abort_flag = 0u;
        fence_barrier_init();
        prefetch_tensormap(&tmA);
        prefetch_tensormap(&tmB);
        prefetch_tensormap(&tmO);
    }
    if (warp == 1) {
        tmem_alloc<PAIR>(smem_u32(tmem_slot), 512);
        tmem_relinquish<PAIR>();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (PAIR) cluster_sync();   // both CTAs' barriers and tensor memory exist before anyone signals across the pair
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // everything up to here touches nothing that a kernel ahead on the stream writes
    chain_start(g.chain);
    status_begin(g.status, g.status_mark);

    // a whole converged warp waits, with one answer for all its lanes; a failed wait raises the abort flag of both CTAs
    auto wait_all = [&](uint32_t bar, uint32_t parity) {
        const bool got = mbar_wait(bar, parity, abort_flag, g.wait_limit_ns);
        if (PAIR && !got) st_cluster_u32(mapa(smem_u32(const_cast<uint32_t *>(abort_flag)), rank ^ 1u), 1u);
        return __all_sync(0xFFFFFFFFu, got) != 0;
    };

    if (warp == 0) {
        // ================= TMA producer (every CTA, into its own shared memory; bytes counted by the leader's barrier) =================
        const uint32_t lead_full0 = PAIR ? mapa(full_bar(0), 0) : 0u;
        uint32_t it = 0;
        bool ok = true;
        for (int w = unit; w < g.work.num_items && ok; w += units) {
            const WorkItem wi = work_item<true>(g.work, w, num_kstages);
            int m_idx, n_idx;
            tile_coords(wi.t, num_m, num_n, m_idx, n_idx);
            for (int ks = wi.ks0; ks < wi.ks1; ++ks, ++it) {
                const int s = it % S;
                if (!wait_all(empty_bar(s), ((it / S) & 1u) ^ 1u)) { ok = false; break; }
                if (elect_one()) {
                    if (rank == 0) mbar_arrive_expect_tx(full_bar(s), C::kCtas * g.stage_tx_bytes);
                    const int row = m_idx * BM + (int)rank * CM, col = n_idx * BN + (int)rank * C::kBLines;
                    auto load = [&](uint32_t dst, const CUtensorMap *m, int c0, int c1) {
                        if (PAIR) tma_load_2d_pair(dst, m, lead_full0 + 8u * s, c0, c1);   // no multicast: each CTA fetches its own share
                        else tma_load_2d(dst, m, full_bar(s), c0, c1);
                    };
                    if (A_MN) {
#pragma unroll
                        for (int i = 0; i < CM / 64; ++i) load(a_tile(s) + i * kBoxBytes, &tmA, row + 64 * i, ks * kStageK);
                    } else {
                        load(a_tile(s), &tmA, ks * kStageK, row);
                    }
                    if (B_MN) {
#pragma unroll
                        for (int i = 0; i < C::kBLines / 64; ++i) load(b_tile(s) + i * kBoxBytes, &tmB, col + 64 * i, ks * kStageK);
                    } else {
                        load(b_tile(s), &tmB, ks * kStageK, col);
                    }
                }
                __syncwarp();
            }
        }
    } else if (warp == 1) {
      // ================= MMA issuer (leader; whole warp in the loop, one elected lane issues) =================
      if (rank == 0) {
        uint32_t it = 0, done = 0;
        bool ok = true;
        for (int w = unit; w < g.work.num_items && ok; w += units, ++done) {
            const WorkItem wi = work_item<true>(g.work, w, num_kstages);
            const uint32_t a = done & 1u;
            if (!wait_all(tempty_bar(a), ((done >> 1) & 1u) ^ 1u)) { ok = false; break; }
            tc_fence_after_sync();
            for (int ks = wi.ks0; ks < wi.ks1; ++ks, ++it) {
                const int s = it % S;
                if (!wait_all(full_bar(s), (it / S) & 1u)) { ok = false; break; }
                tc_fence_after_sync();
                const uint64_t adesc = A_MN ? make_smem_desc_mn128(a_tile(s), kBoxBytes) : make_smem_desc_k128(a_tile(s));
                const uint64_t bdesc = B_MN ? make_smem_desc_mn128(b_tile(s), kBoxBytes) : make_smem_desc_k128(b_tile(s));
                // 16 elements of the contraction per MMA: 32 bytes of a K-major row, or 16 rows of 128 bytes
                constexpr uint64_t kAStep = (A_MN ? 2048 : 32) >> 4, kBStep = (B_MN ? 2048 : 32) >> 4;
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        mma_ss<MmaKind::F16, PAIR>(tmem_base + a * BN, adesc + kAStep * k, bdesc + kBStep * k, idesc, (ks > wi.ks0 || k > 0) ? 1u : 0u, 0, 0);
                    tc_commit<PAIR>(empty_bar(s));
                    if (ks == wi.ks1 - 1) {
                        tc_commit<PAIR>(tfull_bar(a));
                    }
                }
                __syncwarp();
            }
        }
      }
    } else if (warp == 2) {
        // ================= statistics of the quantizers ahead =================
        for (int i = blockIdx.x; i < g.stats.count; i += gridDim.x) reduce_stats_warp(g.stats.job[i], lane);
    } else if (warp >= 4) {
        // ================= epilogue: drain, add slices, round, store =================
        const int e = warp - 4, q = warp & 3, h = e >> 2;
        const uint32_t stage_u32 = out_stage0 + e * (kOutSlots * 2048);
        const uint32_t lead_tempty0 = PAIR ? mapa(tempty_bar(0), 0) : 0u;
        uint32_t done = 0;
        bool ok = true;
        for (int w = unit; w < g.work.num_items && ok; w += units, ++done) {
            const WorkItem wi = work_item<true>(g.work, w, num_kstages);
            int m_idx, n_idx;
            tile_coords(wi.t, num_m, num_n, m_idx, n_idx);
            const int row0 = m_idx * BM + (int)rank * CM + q * 32, col0 = n_idx * BN + h * HALF;
            const uint32_t a = done & 1u;
            if (!wait_all(tfull_bar(a), (done >> 1) & 1u)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + a * BN + h * HALF;
            uint32_t v[4][32];
#pragma unroll
            for (int gi = 0; gi < 4; ++gi) tmem_ld32(taddr + 32 * gi, v[gi]);
            tmem_ld_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) {
                if (PAIR) mbar_arrive_cluster_relaxed(lead_tempty0 + 8u * a);
                else mbar_arrive(tempty_bar(a));
            }
            bool write_out = true;
            if (wi.nsl > 1) {
                constexpr size_t kWarpFloats = 32 * HALF;
                constexpr int kWarps = kNumEpiWarps * C::kCtas;   // epilogue warps of a tile
                const int ew = (int)rank * kNumEpiWarps + e;
                float *first = g.partials + (size_t)(wi.tail * wi.nsl) * kWarps * kWarpFloats + ew * kWarpFloats + lane * 4;
                float *mine = first + (size_t)wi.slice * kWarps * kWarpFloats;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    __stcg(reinterpret_cast<uint4 *>(mine + j * 128), make_uint4(v[j >> 3][4 * (j & 7)], v[j >> 3][4 * (j & 7) + 1], v[j >> 3][4 * (j & 7) + 2], v[j >> 3][4 * (j & 7) + 3]));
                __threadfence();
                __syncwarp();
                uint32_t old = 0;
                if (lane == 0) old = atomicAdd(g.counters + wi.tail * kWarps + ew, 1u);
                old = __shfl_sync(0xFFFFFFFFu, old, 0);
                write_out = (old == (uint32_t)wi.nsl - 1u);
                if (write_out) {
                    __threadfence();
#pragma unroll
                    for (int gi = 0; gi < 4; ++gi) {
                        for (int sl = 0; sl < wi.nsl; ++sl) {
                            const float *src = first + (size_t)sl * kWarps * kWarpFloats + gi * 8 * 128;
                            float4 u[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) u[j] = __ldcg(reinterpret_cast<const float4 *>(src + j * 128));
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float x[4] = {u[j].x, u[j].y, u[j].z, u[j].w};
#pragma unroll
                                for (int i = 0; i < 4; ++i) v[gi][4 * j + i] = __float_as_uint(sl == 0 ? x[i] : __uint_as_float(v[gi][4 * j + i]) + x[i]);
                            }
                        }
                    }
                }
            }
            if (!write_out) continue;
            if (OUT_F32 && g.out_acc) {
                if (row0 < g.Mo) {
                    float *dst = g.out_acc + (int64_t)(row0 + lane) * g.No + col0;
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        if (col0 + 4 * j < g.No) {
                            float4 p = *reinterpret_cast<const float4 *>(dst + 4 * j);
                            p.x += __uint_as_float(v[j >> 3][4 * (j & 7)]);     p.y += __uint_as_float(v[j >> 3][4 * (j & 7) + 1]);
                            p.z += __uint_as_float(v[j >> 3][4 * (j & 7) + 2]); p.w += __uint_as_float(v[j >> 3][4 * (j & 7) + 3]);
                            *reinterpret_cast<float4 *>(dst + 4 * j) = p;
                        }
                    }
                }
                continue;
            }
            // 32 rows x 64 bytes at a time through shared memory (16-byte pieces swizzled the way the output map expects); rows and
            // columns outside the matrix are clipped by the hardware
            constexpr int kPerBox = OUT_F32 ? 16 : 32;
#pragma unroll
            for (int b = 0; b < HALF / kPerBox; ++b) {
                if (lane == 0) bulk_wait_read<kOutSlots - 1>();   // the box that was in this staging tile has left it
                __syncwarp();
                const uint32_t slot = stage_u32 + (b % kOutSlots) * 2048;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint4 o;
                    if (OUT_F32) {
                        const uint32_t *src = &v[(b * 16) / 32][(b * 16) % 32 + 4 * j];
                        o = make_uint4(src[0], src[1], src[2], src[3]);
                    } else {
                        const uint32_t *src = &v[b & 3][8 * j];
                        o = make_uint4(bf16x2(src[0], src[1]), bf16x2(src[2], src[3]), bf16x2(src[4], src[5]), bf16x2(src[6], src[7]));
                    }
                    st_shared_v4(slot + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4), o);
                }
                fence_proxy_async();
                __syncwarp();
                const int col = col0 + b * kPerBox;
                if (lane == 0) {
                    if (col < g.No && row0 < g.Mo) tma_store_2d(&tmO, slot, col, row0);
                    bulk_commit();   // one group per box, empty outside the matrix: the wait above counts groups
                }
            }
        }
        if (lane == 0) bulk_wait_all0();
    }

    // ---- teardown: every role ends here, tensor memory is always released ----
    __syncwarp();
    chain_finish(g.chain);
    tc_fence_before_sync();
    __syncthreads();
    if (PAIR) cluster_sync();   // no more arrivals from the other CTA, and the pair's MMAs read no more of this CTA's memory
    if (*abort_flag) {
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
        if (threadIdx.x == 0) status_report(g.status, g.status_mark, (uint32_t)SNIP_ERR_TIMEOUT, g.wait_limit_ns);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc<PAIR>(tmem_base, 512);
    }
}

template <bool PAIR, bool A_MN, bool B_MN, bool OUT_F32>
int launch_bf16(const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmO, const Bf16Args &g, uint32_t idesc, int grid, cudaStream_t st)
{
    auto kern = gemm_bf16_kernel<PAIR, A_MN, B_MN, OUT_F32>;
    SNIP_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<PAIR>::kSmemBytes));
    return launch_chained(kern, grid, kThreads, Cfg<PAIR>::kSmemBytes, st, PAIR ? 2 : 1, tmA, tmB, tmO, g, idesc);
}
template <bool PAIR>
int launch_bf16_order(bool a_mn, bool b_mn, bool f32, const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmO, const Bf16Args &g,
                      uint32_t idesc, int grid, cudaStream_t st)
{
    if (!a_mn && !b_mn) return f32 ? launch_bf16<PAIR, false, false, true>(tmA, tmB, tmO, g, idesc, grid, st) : launch_bf16<PAIR, false, false, false>(tmA, tmB, tmO, g, idesc, grid, st);
    if (!a_mn) return f32 ? launch_bf16<PAIR, false, true, true>(tmA, tmB, tmO, g, idesc, grid, st) : launch_bf16<PAIR, false, true, false>(tmA, tmB, tmO, g, idesc, grid, st);
    if (b_mn) return f32 ? launch_bf16<PAIR, true, true, true>(tmA, tmB, tmO, g, idesc, grid, st) : launch_bf16<PAIR, true, true, false>(tmA, tmB, tmO, g, idesc, grid, st);
    return SNIP_ERR_UNSUPPORTED;
}

}  // namespace

int make_tiled_map_2d(CUtensorMap *map, const void *ptr, int dtype, int64_t rows, int64_t inner_elems, int64_t row_bytes, int box_x_elems,
                      int box_rows, int swizzle);
int gemm_sm_count();
void gemm_debug_hooks(uint64_t *wait_limit_ns, int *tx_skew);
bool gemm_slicing_enabled();

// a: [Mo][Kc], or [Kc][Mo] if a_mn; b: [No][Kc], or [Kc][No] if b_mn.  Arguments have been checked by the caller (gemm_impl).
int gemm_bf16_impl(const void *a, bool a_mn, const void *b, bool b_mn, int64_t Mo, int64_t No, int64_t Kc, void *out, int out_dtype, int accumulate,
                   const GemmWs &w, cudaStream_t st, const ChainLink &link)
{
    const bool f32 = out_dtype == SNIP_OUT_FP32;
    Bf16Args g;
    g.Mo = (int32_t)Mo; g.No = (int32_t)No; g.Kc = (int32_t)Kc;
    g.out_acc = accumulate ? static_cast<float *>(out) : nullptr;
    g.status = w.status;
    g.status_mark = status_mark(w.cleared);
    g.counters = w.counters; g.partials = w.partials;
    g.chain = link.role;
    if (link.jobs) g.stats = *link.jobs;
    int tx_skew = 0;
    gemm_debug_hooks(&g.wait_limit_ns, &tx_skew);
    CUtensorMap tmA, tmB, tmO;
    int rc = f32 ? make_tiled_map_2d(&tmO, out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, Mo, No, No * 4, 16, 32, CU_TENSOR_MAP_SWIZZLE_64B)
                 : make_tiled_map_2d(&tmO, out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Mo, No, No * 2, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
    if (rc) return rc;
    auto map = [&](CUtensorMap *m, const void *p, bool mn, int64_t lines, int box_lines) {
        return mn ? make_tiled_map_2d(m, p, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Kc, lines, lines * 2, 64, kStageK, CU_TENSOR_MAP_SWIZZLE_128B)
                  : make_tiled_map_2d(m, p, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, lines, Kc, Kc * 2, kStageK, box_lines, CU_TENSOR_MAP_SWIZZLE_128B);
    };
    const int sms = gemm_sm_count();
    // The pair form halves a CTA's share of B (shared-memory writes, L2 reads, power): 16384x12288x4096 1322 -> 1210 us, 8192x5632x2048
    // 160 -> 147 us.  With fewer 256-row tiles than pairs of SMs the single form spreads the work better (2048x1024x1024 14.3 -> 12.3 us).
    const bool pair = ceil_div(Mo, 256) * ceil_div(No, BN) >= sms / 2;
    const int ctas = pair ? 2 : 1, tile_m = CM * ctas;
    rc = map(&tmA, a, a_mn, Mo, CM);
    if (rc) return rc;
    rc = map(&tmB, b, b_mn, No, BN / ctas);
    if (rc) return rc;
    g.stage_tx_bytes = (pair ? Cfg<true>::kStageBytes : Cfg<false>::kStageBytes) + tx_skew;
    const uint32_t idesc = make_idesc(1, 1, tile_m, BN) | (a_mn ? 1u << 15 : 0u) | (b_mn ? 1u << 16 : 0u);
    const int num_tiles = (int)(ceil_div(Mo, tile_m) * ceil_div(No, BN));
    g.work = plan_work(num_tiles, (int)(Kc / kStageK), sms / ctas, kMinSliceStages, kMinSavedStages, w.partials != nullptr && gemm_slicing_enabled(), kMaxSlicedItems / ctas);
    if (g.work.nsplit > 1 && !w.cleared)
        SNIP_CUDA_TRY(cudaMemsetAsync(w.counters, 0, (size_t)(num_tiles - g.work.split_first) * kNumEpiWarps * ctas * sizeof(uint32_t), st));
    const int units = sms / ctas, grid = (g.work.num_items < units ? g.work.num_items : units) * ctas;
    return pair ? launch_bf16_order<true>(a_mn, b_mn, f32, tmA, tmB, tmO, g, idesc, grid, st)
                : launch_bf16_order<false>(a_mn, b_mn, f32, tmA, tmB, tmO, g, idesc, grid, st);
}

}  // namespace snip
