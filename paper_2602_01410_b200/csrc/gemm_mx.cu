// GEMMs for the power-of-two scale option: out[Mo,No] = A[Mo,Kc] . B[No,Kc]^T where every 128-long
// chunk of the contraction carries a power-of-two scale per operand line.  The tensor core applies
// the scales itself (tcgen05.mma ... block_scale with UE8M0 scale factors in tensor memory), so the
// whole contraction accumulates in tensor memory and the epilogue runs once per output tile.
// (Power-of-two block scales are the MX-format convention the paper cites in Sec. 2.3; the paper's own
// rule FPX_MAX/amax needs the per-chunk FP32 promotion of gemm.cu.)
//
// One CTA per SM, persistent, 384 threads; tiles of 256x256 shared by a pair of CTAs (tcgen05.mma.cta_group::2: each holds 128
// rows and fetches half of B's lines), or 128x256 on one CTA where there are few.  Warp 0 streams operand tiles and 512-byte
// scale-factor atoms into a shared-memory ring (both through tensor maps, so that a CTA can report them to its leader's
// barrier); warp 1 copies each stage's atoms into tensor memory (tcgen05.cp) and issues the MMAs; warps 4-11 drain the FP32 accumulator
// (one buffer: 256 columns, next to 12 or 24 scale-factor columns), round, and store through the TMA unit.
// Warps 0 and 1 walk their loops as whole warps and one elected lane issues.  Every wait is bounded, as in gemm.cu.
//
// The bytes may differ within a chunk (32-long tiles: byte k belongs to the k-th 32 elements; the MMA of that step
// selects it through the descriptor's scale-factor id).  A third instantiation serves the two-level option in the
// style of NVFP4: E2M1 codes, an E4M3 scale byte per 16 elements (a word per line and 64-long MMA step, two atoms per
// chunk), tcgen05.mma kind::mxf4nvf4 with scale_vec::4X, and one division by the two per-tensor factors at the end.
#include <cuda.h>
#include <cuda_bf16.h>
#include <float.h>

#include "common.cuh"
#include "quant_device.cuh"
#include "sm100.cuh"
#include "work_items.cuh"

namespace snip {

using namespace sm100;

namespace {

constexpr int CM = 128;   // rows of a CTA
constexpr int BN = 256;
constexpr int kThreads = 384;
constexpr int kNumEpiWarps = 8;
constexpr int kSfaCol = 256;   // tensor-memory columns: accumulator 0..255, SFA 256..259, SFB 260..267
constexpr int kSfbCol = 260;
constexpr int kNvSfbCol = 264; // two-level option: a word per line and MMA: SFA 256..263 (two MMAs), SFB 264..279
constexpr int kTmemCols = 512;

struct MxMaps {
    CUtensorMap a, b, o, sfa, sfb;
};
struct MxArgs {
    int32_t Mo, No, Kc;
    int32_t n_atoms_a, n_atoms_b;   // ceil(Mo/128), ceil(No/128): line tiles of the scale-factor atoms [line tile][chunk]
    uint32_t stage_tx_bytes;   // bytes reported to a stage's barrier (operands + scale-factor atoms)
    uint32_t *status;
    uint32_t status_mark;      // see status_begin
    const float *amax_a, *amax_b;   // two-level option: the tensors' magnitude bounds (device); else null
    uint64_t wait_limit_ns;    // bound of every device-side wait
    int32_t chain;             // ChainRole
    StatJobs stats;            // reductions left by the quantizers ahead
};

template <MmaKind KIND, bool PAIR>
struct MxCfg {
    static constexpr int kCtas = PAIR ? 2 : 1;
    static constexpr int BM = CM * kCtas;          // rows of a tile
    static constexpr int kBLines = BN / kCtas;     // B lines fetched by a CTA
    static constexpr bool kNv = KIND == MmaKind::NVF4;
    static constexpr int kChunksPerStage = (KIND == MmaKind::MXF4 || kNv) ? 2 : 1;   // packed FP4: 256 elements per 128-byte row
    static constexpr int kABytes = CM * 128;
    static constexpr int kBBytes = kBLines * 128;
    // per chunk: SFA 512 + SFB 2 x 512 (+ pad); two-level option: an atom per 64 elements, SFA 2 x 512 + SFB 4 x 512
    static constexpr int kSfChunkBytes = kNv ? 3072 : 2048;
    static constexpr int kSfBytes = kSfChunkBytes * kChunksPerStage;
    static constexpr int kStageBytes = kABytes + kBBytes + kSfBytes;
    static constexpr int kStages = PAIR ? (KIND == MmaKind::MXF8 ? 6 : 5) : kNv ? 3 : 4;
    static constexpr int kOutStageBytes = kNumEpiWarps * 2048;
    static constexpr int kSmemBytes = kStages * kStageBytes + kOutStageBytes + 256 + 1024;
    static_assert(kSmemBytes <= 232448, "shared memory budget");
    static_assert(kStageBytes % 1024 == 0, "operand tiles must stay 1024-byte aligned");
};

__device__ __forceinline__ uint32_t mx_pack_bf16x2(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

template <MmaKind KIND, bool PAIR, bool OUT_F32>
__global__ void __launch_bounds__(kThreads, 1)
gemm_mx_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmO,
               const __grid_constant__ CUtensorMap tmSfa, const __grid_constant__ CUtensorMap tmSfb, const MxArgs g, const uint32_t idesc)
{
    using C = MxCfg<KIND, PAIR>;
    constexpr int S = C::kStages, BM = C::BM;
    constexpr int CPS = C::kChunksPerStage;
    constexpr int HALF = BN / 2;

    extern __shared__ uint8_t smem_raw[];
    chain_acquire(g.chain, g.status);
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    auto a_tile = [&](int s) { return smem_base + s * C::kStageBytes; };
    auto b_tile = [&](int s) { return smem_base + s * C::kStageBytes + C::kABytes; };
    auto sf_tile = [&](int s) { return smem_base + s * C::kStageBytes + C::kABytes + C::kBBytes; };
    const uint32_t out_stage0 = smem_base + S * C::kStageBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_gen + S * C::kStageBytes + C::kOutStageBytes);
    const uint32_t bar0 = smem_base + S * C::kStageBytes + C::kOutStageBytes;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    const uint32_t tfull_bar = bar0 + 8u * (2 * S), tempty_bar = bar0 + 8u * (2 * S + 1);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * S + 2);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_m = (g.Mo + BM - 1) / BM, num_n = (g.No + BN - 1) / BN;
    const int num_tiles = num_m * num_n;
    const int num_chunks = (g.Kc + 127) / 128;
    const int num_kstages = (num_chunks + CPS - 1) / CPS;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;   // 0 = leader: its barriers and its MMA warp serve the pair
    const int unit = (int)blockIdx.x / C::kCtas, units = (int)gridDim.x / C::kCtas;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        mbar_init(tfull_bar, 1);
        mbar_init(tempty_bar, kNumEpiWarps * C::kCtas);
        *abort_flag = 0u;
        fence_barrier_init();
        prefetch_tensormap(&tmA);
        prefetch_tensormap(&tmB);
        prefetch_tensormap(&tmO);
        prefetch_tensormap(&tmSfa);
        prefetch_tensormap(&tmSfb);
    }
    if (warp == 1) {
        tmem_alloc<PAIR>(smem_u32(tmem_slot), kTmemCols);
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
        // ================= producer: operand tiles and scale-factor atoms =================
        // (every CTA, into its own shared memory; bytes counted by the leader's barrier; whole warp in the loop, one elected lane issues)
        {
            const uint32_t lead_full0 = PAIR ? mapa(full_bar(0), 0) : 0u;
            uint32_t it = 0;
            bool ok = true;
            for (int t = unit; t < num_tiles && ok; t += units) {
                int m_idx, n_idx;
                tile_coords(t, num_m, num_n, m_idx, n_idx);
                const int row = m_idx * BM + (int)rank * CM, col = n_idx * BN + (int)rank * C::kBLines;
                // line tiles of the scale factors: this CTA's rows, and both column blocks (every CTA of a pair holds those of the whole
                // tile); beyond the matrix the last one again
                const int na = min(row / CM, g.n_atoms_a - 1), nb0 = 2 * n_idx, nb1 = min(2 * n_idx + 1, g.n_atoms_b - 1);
                for (int ks = 0; ks < num_kstages; ++ks, ++it) {
                    const int s = it % S;
                    if (!wait_all(empty_bar(s), ((it / S) & 1u) ^ 1u)) { ok = false; break; }
                    if (elect_one()) {
                        if (rank == 0) mbar_arrive_expect_tx(full_bar(s), C::kCtas * g.stage_tx_bytes);
                        auto load = [&](uint32_t dst, const CUtensorMap *m, int c0, int c1) {
                            if (PAIR) tma_load_2d_pair(dst, m, lead_full0 + 8u * s, c0, c1);   // no multicast: each CTA fetches its own share
                            else tma_load_2d(dst, m, full_bar(s), c0, c1);
                        };
                        load(a_tile(s), &tmA, ks * 128, row);
                        load(b_tile(s), &tmB, ks * 128, col);
#pragma unroll
                        for (int h = 0; h < CPS; ++h) {
                            const int c = min(ks * CPS + h, num_chunks - 1);   // a stage's unused second chunk reloads a valid atom
                            constexpr uint32_t kAtom = C::kNv ? 1024 : 512;    // two-level option: two halves per chunk
                            const uint32_t dst = sf_tile(s) + h * C::kSfChunkBytes;
                            load(dst, &tmSfa, 0, na * num_chunks + c);
                            load(dst + kAtom, &tmSfb, 0, nb0 * num_chunks + c);
                            load(dst + 2 * kAtom, &tmSfb, 0, nb1 * num_chunks + c);
                        }
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp == 1) {
        // ================= scale-factor copies and MMA issue =================
        // The whole warp walks the loop and one elected lane issues: under `elect.sync` the operands of the tcgen05
        // instructions stay in uniform registers, which makes each of them several times cheaper for the issuing thread than
        // under a `lane == 0` branch; with up to seventeen of them per stage that thread is what the tensor core waits for.
        if (rank == 0) {
            uint32_t it = 0, tiles_done = 0;
            bool ok = true;
            const uint32_t sfa = tmem_base + kSfaCol, sfb = tmem_base + (C::kNv ? kNvSfbCol : kSfbCol);
            for (int t = unit; t < num_tiles && ok; t += units, ++tiles_done) {
                // the single accumulator must have been drained by the epilogue of the previous tile
                if (!wait_all(tempty_bar, (tiles_done & 1u) ^ 1u)) { ok = false; break; }
                tc_fence_after_sync();
                for (int ks = 0; ks < num_kstages && ok; ++ks, ++it) {
                    const int s = it % S;
                    if (!wait_all(full_bar(s), (it / S) & 1u)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint64_t adesc = make_smem_desc_k128(a_tile(s));
                    const uint64_t bdesc = make_smem_desc_k128(b_tile(s));
                    if (elect_one()) {
#pragma unroll
                        for (int h = 0; h < CPS; ++h) {
                            if (ks * CPS + h < num_chunks) {
                                const uint32_t sf = sf_tile(s) + h * C::kSfChunkBytes;
                                if (C::kNv) {
                                    // MMA k of the chunk reads a whole word per line: SFA columns 4k.., SFB columns 8k.. (two 128-line groups)
                                    tmem_cp_sf_atom<PAIR>(sfa, sf);             tmem_cp_sf_atom<PAIR>(sfa + 4, sf + 512);
                                    tmem_cp_sf_atom<PAIR>(sfb, sf + 1024);      tmem_cp_sf_atom<PAIR>(sfb + 8, sf + 1536);
                                    tmem_cp_sf_atom<PAIR>(sfb + 4, sf + 2048);  tmem_cp_sf_atom<PAIR>(sfb + 12, sf + 2560);
                                } else {
                                    tmem_cp_sf_atom<PAIR>(sfa, sf);
                                    tmem_cp_sf_atom<PAIR>(sfb, sf + 512);
                                    tmem_cp_sf_atom<PAIR>(sfb + 4, sf + 1024);
                                }
                                constexpr int kMmas = 4 / CPS;   // 32 bytes of K per MMA: four per 128-byte row
#pragma unroll
                                for (int k = 0; k < kMmas; ++k) {
                                    const int kk = h * kMmas + k;
                                    // which of the line's four scale bytes this MMA applies: byte k for the 32-long blocks of
                                    // kind::mxf8f6f4, bytes 2k and 2k+1 for the two halves of kind::mxf4's 64-long step
                                    // (descriptor fields b_sf_id at bit 4, a_sf_id at bit 29); the two-level option reads whole words
                                    const uint32_t sf_id = C::kNv ? 0u : (KIND == MmaKind::MXF4) ? 2u * k : (uint32_t)k;
                                    mma_ss<KIND, PAIR>(tmem_base, adesc + 2 * kk, bdesc + 2 * kk, idesc | (sf_id << 4) | (sf_id << 29),
                                                        (ks > 0 || kk > 0) ? 1u : 0u, sfa + (C::kNv ? 4 * k : 0), sfb + (C::kNv ? 8 * k : 0));
                                }
                            }
                        }
                        tc_commit<PAIR>(empty_bar(s));
                        if (ks == num_kstages - 1) {
                            tc_commit<PAIR>(tfull_bar);
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
        // ================= epilogue: drain, round, store =================
        const int e = warp - 4, q = warp & 3, h = e >> 2;
        const uint32_t stage_u32 = out_stage0 + e * 2048;
        const uint32_t lead_tempty = PAIR ? mapa(tempty_bar, 0) : 0u;
        uint32_t tiles_done = 0;
        bool ok = true;
        // two-level option: the sums carry both tensors' factors 2688 / bound; they are divided out here, once per output
        float out_scale = 1.0f;
        if (C::kNv) {
            const float ba = *g.amax_a, bb = *g.amax_b;
            const float ea = ba == 0.0f ? 1.0f : fminf(__fdiv_rn(2688.0f, ba), FLT_MAX), eb = bb == 0.0f ? 1.0f : fminf(__fdiv_rn(2688.0f, bb), FLT_MAX);
            out_scale = __fdiv_rn(1.0f, ea * eb);
        }
        for (int t = unit; t < num_tiles && ok; t += units, ++tiles_done) {
            int m_idx, n_idx;
            tile_coords(t, num_m, num_n, m_idx, n_idx);
            const int row0 = m_idx * BM + (int)rank * CM + q * 32;
            const int col0 = n_idx * BN + h * HALF;
            if (!wait_all(tfull_bar, tiles_done & 1u)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + h * HALF;
            uint32_t v[4][32];
#pragma unroll
            for (int gi = 0; gi < 4; ++gi) tmem_ld32(taddr + 32 * gi, v[gi]);
            tmem_ld_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) {   // the next tile's MMAs may start
                if (PAIR) mbar_arrive_cluster_relaxed(lead_tempty);
                else mbar_arrive(tempty_bar);
            }
            if (C::kNv) {
#pragma unroll
                for (int gi = 0; gi < 4; ++gi)
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[gi][i] = __float_as_uint(__uint_as_float(v[gi][i]) * out_scale);
            }
            constexpr int kPerBox = OUT_F32 ? 16 : 32;   // output columns per 64-byte box row
#pragma unroll
            for (int b = 0; b < HALF / kPerBox; ++b) {
                if (lane == 0) bulk_wait_read0();
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint4 o;
                    if (OUT_F32) {
                        const uint32_t *src = &v[(b * 16) / 32][(b * 16) % 32 + 4 * j];
                        o = make_uint4(src[0], src[1], src[2], src[3]);
                    } else {
                        const uint32_t *src = &v[b][8 * j];
                        o = make_uint4(mx_pack_bf16x2(__uint_as_float(src[0]), __uint_as_float(src[1])), mx_pack_bf16x2(__uint_as_float(src[2]), __uint_as_float(src[3])),
                                       mx_pack_bf16x2(__uint_as_float(src[4]), __uint_as_float(src[5])), mx_pack_bf16x2(__uint_as_float(src[6]), __uint_as_float(src[7])));
                    }
                    st_shared_v4(stage_u32 + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4), o);
                }
                fence_proxy_async();
                __syncwarp();
                const int col = col0 + b * kPerBox;
                if (lane == 0 && col < g.No && row0 < g.Mo) { tma_store_2d(&tmO, stage_u32, col, row0); bulk_commit(); }
            }
        }
        if (lane == 0) bulk_wait_all0();
    }

    // ---- teardown ----
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
        tmem_dealloc<PAIR>(tmem_base, kTmemCols);
    }
}


template <MmaKind KIND, bool PAIR, bool OUT_F32>
int launch_mx(const MxMaps &m, const MxArgs &g, uint32_t idesc, int sms, cudaStream_t st)
{
    using C = MxCfg<KIND, PAIR>;
    auto kern = gemm_mx_kernel<KIND, PAIR, OUT_F32>;
    // a per-function, per-device attribute; setting it on every launch is cheap and correct on any device
    SNIP_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes));
    const int num_tiles = (int)(ceil_div(g.Mo, C::BM) * ceil_div(g.No, BN));
    const int units = sms / C::kCtas, grid = (num_tiles < units ? num_tiles : units) * C::kCtas;
    return launch_chained(kern, grid, kThreads, C::kSmemBytes, st, C::kCtas, m.a, m.b, m.o, m.sfa, m.sfb, g, idesc);
}

}  // namespace

int make_tiled_map_2d(CUtensorMap *map, const void *ptr, int dtype, int64_t rows, int64_t inner_elems, int64_t row_bytes, int box_x_elems,
                      int box_rows, int swizzle);
GemmWs gemm_ws(void *ws, size_t ws_bytes);
int gemm_sm_count();
void gemm_debug_hooks(uint64_t *wait_limit_ns, int *tx_skew);   // testing hooks of snip_debug_set (gemm.cu)

namespace {

// What the three forms share: checks, output and scale-factor maps, the choice between one CTA and a pair per tile, the launch.
// sf_words: 32-bit words of a scale-factor atom (128, two-level option 256); operand maps of `box_a` / `box_b` elements are set by `operand`.
template <MmaKind KIND, class Operand>
int run_mx(const void *a_codes, const void *b_codes, const void *sfa, const void *sfb, const float *amax_a, const float *amax_b, int64_t Mo, int64_t No,
           int64_t Kc, void *out, int out_dtype, const GemmWs &w, cudaStream_t st, const ChainLink &link, int sf_words, uint32_t row_bytes_a, uint32_t row_bytes_b,
           uint32_t idesc_base, Operand operand)
{
    const bool f32 = out_dtype == SNIP_OUT_FP32;
    MxArgs g;
    g.Mo = (int32_t)Mo; g.No = (int32_t)No; g.Kc = (int32_t)Kc;
    g.n_atoms_a = (int32_t)ceil_div(Mo, 128);
    g.n_atoms_b = (int32_t)ceil_div(No, 128);
    g.status = w.status;
    g.status_mark = status_mark(w.cleared);
    g.chain = link.role;
    if (link.jobs) g.stats = *link.jobs;
    int tx_skew = 0;
    gemm_debug_hooks(&g.wait_limit_ns, &tx_skew);
    g.amax_a = amax_a; g.amax_b = amax_b;
    const int sms = gemm_sm_count();
    // Pairs halve a CTA's share of B, as in gemm_bf16.cu; with fewer 256-row tiles than pairs the single form spreads the work better.
    const bool pair = ceil_div(Mo, 256) * ceil_div(No, BN) >= sms / 2;
    const int ctas = pair ? 2 : 1, lines_b = BN / ctas;
    const int64_t chunks = ceil_div(Kc, 128);
    MxMaps m;
    int rc = f32 ? make_tiled_map_2d(&m.o, out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, Mo, No, No * 4, 16, 32, CU_TENSOR_MAP_SWIZZLE_64B)
                 : make_tiled_map_2d(&m.o, out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Mo, No, No * 2, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
    if (rc) return rc;
    rc = operand(&m.a, a_codes, Mo, CM, true);
    if (rc) return rc;
    rc = operand(&m.b, b_codes, No, lines_b, false);
    if (rc) return rc;
    rc = make_tiled_map_2d(&m.sfa, sfa, CU_TENSOR_MAP_DATA_TYPE_UINT32, g.n_atoms_a * chunks, sf_words, sf_words * 4, sf_words, 1, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (rc) return rc;
    rc = make_tiled_map_2d(&m.sfb, sfb, CU_TENSOR_MAP_DATA_TYPE_UINT32, g.n_atoms_b * chunks, sf_words, sf_words * 4, sf_words, 1, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (rc) return rc;
    g.stage_tx_bytes = CM * row_bytes_a + lines_b * row_bytes_b + MxCfg<KIND, false>::kChunksPerStage * 3 * sf_words * 4 + tx_skew;
    const uint32_t idesc = idesc_base | ((uint32_t)((CM * ctas) >> 4) << 24);
    if (pair) return f32 ? launch_mx<KIND, true, true>(m, g, idesc, sms, st) : launch_mx<KIND, true, false>(m, g, idesc, sms, st);
    return f32 ? launch_mx<KIND, false, true>(m, g, idesc, sms, st) : launch_mx<KIND, false, false>(m, g, idesc, sms, st);
}

int check_mx(const void *a_codes, const void *b_codes, const void *sfa, const void *sfb, int64_t Mo, int64_t No, int64_t Kc, const void *out, int out_dtype,
             const GemmWs &w)
{
    if (!a_codes || !b_codes || !sfa || !sfb || !out) return SNIP_ERR_ARG;
    if (!valid_dim(Mo) || !valid_dim(No) || !valid_dim(Kc) || Mo > INT32_MAX || No > INT32_MAX || Kc > INT32_MAX) return SNIP_ERR_SHAPE;
    if (ceil_div(Mo > No ? Mo : No, 128) * ceil_div(Kc, 128) > INT32_MAX) return SNIP_ERR_SHAPE;   // atoms are addressed by a 32-bit index
    if (out_dtype != SNIP_OUT_BF16 && out_dtype != SNIP_OUT_FP32) return SNIP_ERR_ARG;
    if (!w.status) return SNIP_ERR_WORKSPACE;
    if (!aligned16(a_codes) || !aligned16(b_codes) || !aligned16(sfa) || !aligned16(sfb) || !aligned16(out) || !aligned16(w.status)) return SNIP_ERR_ALIGN;
    return SNIP_OK;
}

}  // namespace

// a_codes [Mo][Kc], b_codes [No][Kc] contraction-major; sfa / sfb: UE8M0 atoms [line tile][chunk][512].
int gemm_mx_impl(int fmt_a, int fmt_b, const void *a_codes, const void *b_codes, const void *sfa, const void *sfb, int64_t Mo, int64_t No,
                 int64_t Kc, void *out, int out_dtype, const GemmWs &w, cudaStream_t st, const ChainLink &link)
{
    int rc = check_mx(a_codes, b_codes, sfa, sfb, Mo, No, Kc, out, out_dtype, w);
    if (rc) return rc;
    if (fmt_a == SNIP_FMT_BF16 || fmt_b == SNIP_FMT_BF16) return SNIP_ERR_UNSUPPORTED;
    rc = require_sm100();
    if (rc != SNIP_OK) return rc;
    const bool a4 = fmt_a == SNIP_FMT_FP4_E2M1, b4 = fmt_b == SNIP_FMT_FP4_E2M1;
    if (a4 && b4) {
        // packed FP4: kind::mxf4, 256 elements per 128-byte row, two scale chunks per stage
        auto operand = [&](CUtensorMap *m, const void *p, int64_t lines, int box, bool) {
            return make_tiled_map_2d(m, p, CU_TENSOR_MAP_DATA_TYPE_UINT8, lines, Kc / 2, Kc / 2, 128, box, CU_TENSOR_MAP_SWIZZLE_128B);
        };
        return run_mx<MmaKind::MXF4>(a_codes, b_codes, sfa, sfb, nullptr, nullptr, Mo, No, Kc, out, out_dtype, w, st, link, 128, 128, 128,
                                     make_idesc_block_scaled(1, 1, 0, BN), operand);
    }
    const int64_t kpad = ceil_div(Kc, 128) * 128;   // see gemm.cu: the expanding 4-bit map wants a multiple of 128
    auto operand = [&](CUtensorMap *m, const void *p, int64_t lines, int box, bool is_a) {
        const bool f4 = is_a ? a4 : b4;
        return make_tiled_map_2d(m, p, f4 ? CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B : CU_TENSOR_MAP_DATA_TYPE_UINT8, lines, f4 ? kpad : Kc, f4 ? Kc / 2 : Kc, 128, box,
                                 CU_TENSOR_MAP_SWIZZLE_128B);
    };
    return run_mx<MmaKind::MXF8>(a_codes, b_codes, sfa, sfb, nullptr, nullptr, Mo, No, Kc, out, out_dtype, w, st, link, 128, a4 ? 64 : 128, b4 ? 64 : 128,
                                 make_idesc_block_scaled(a4 ? 5 : 0, b4 ? 5 : 0, 0, BN), operand);
}

// Two-level option: packed E2M1 codes, E4M3 scale bytes per 16-long tile as atoms [line tile][chunk][half][512], and the
// two tensors' magnitude bounds (device pointers).  out = (sum of block-scaled products) / (enc_a * enc_b), enc = 2688 / bound.
int gemm_nvfp4_impl(const void *a_codes, const void *b_codes, const void *sfa, const void *sfb, const float *amax_a, const float *amax_b,
                    int64_t Mo, int64_t No, int64_t Kc, void *out, int out_dtype, const GemmWs &w, cudaStream_t st, const ChainLink &link)
{
    if (!amax_a || !amax_b) return SNIP_ERR_ARG;
    int rc = check_mx(a_codes, b_codes, sfa, sfb, Mo, No, Kc, out, out_dtype, w);
    if (rc) return rc;
    if ((reinterpret_cast<uintptr_t>(amax_a) & 3u) || (reinterpret_cast<uintptr_t>(amax_b) & 3u)) return SNIP_ERR_ALIGN;
    rc = require_sm100();
    if (rc != SNIP_OK) return rc;
    auto operand = [&](CUtensorMap *m, const void *p, int64_t lines, int box, bool) {
        return make_tiled_map_2d(m, p, CU_TENSOR_MAP_DATA_TYPE_UINT8, lines, Kc / 2, Kc / 2, 128, box, CU_TENSOR_MAP_SWIZZLE_128B);
    };
    return run_mx<MmaKind::NVF4>(a_codes, b_codes, sfa, sfb, amax_a, amax_b, Mo, No, Kc, out, out_dtype, w, st, link, 256, 128, 128,
                                 make_idesc_block_scaled_e4m3(1, 1, 0, BN), operand);
}

}  // namespace snip

// A quantized operand of the power-of-two option: codes as in snip_qtensor_t plus its UE8M0 atoms.
extern "C" int snip_gemm_mx(int op, const snip_qtensor_t *a, const void *sf_a, const snip_qtensor_t *b, const void *sf_b, void *out,
                            int out_dtype, void *ws, size_t ws_bytes, void *stream)
{
    using namespace snip;
    if (!a || !b || op < SNIP_OP_FWD || op > SNIP_OP_WGRAD) return SNIP_ERR_ARG;
    if (!valid_fmt(a->fmt) || !valid_fmt(b->fmt)) return SNIP_ERR_ARG;
    int64_t Mo, No, Kc;
    if (op == SNIP_OP_FWD) {
        if (a->cols != b->cols || a->transposed || b->transposed) return SNIP_ERR_SHAPE;
        // the paper's tiles, or 32-long tiles along the contraction on both sides
        if (!((a->block == SNIP_BLOCK_ROW_1x128 && b->block == SNIP_BLOCK_BLK_128x128) || (a->block == SNIP_BLOCK_ROW_1x32 && b->block == SNIP_BLOCK_ROW_1x32)))
            return SNIP_ERR_UNSUPPORTED;
        Mo = a->rows; No = b->rows; Kc = a->cols;
    } else if (op == SNIP_OP_DGRAD) {
        if (a->cols != b->rows || a->transposed || !b->transposed) return SNIP_ERR_SHAPE;
        if (!((a->block == SNIP_BLOCK_ROW_1x128 && b->block == SNIP_BLOCK_BLK_128x128) || (a->block == SNIP_BLOCK_ROW_1x32 && b->block == SNIP_BLOCK_COL_32x1)))
            return SNIP_ERR_UNSUPPORTED;
        Mo = a->rows; No = b->cols; Kc = a->cols;
    } else {
        if (a->rows != b->rows || !a->transposed || !b->transposed) return SNIP_ERR_SHAPE;
        if (!((a->block == SNIP_BLOCK_COL_128x1 && b->block == SNIP_BLOCK_COL_128x1) || (a->block == SNIP_BLOCK_COL_32x1 && b->block == SNIP_BLOCK_COL_32x1)))
            return SNIP_ERR_UNSUPPORTED;
        Mo = a->cols; No = b->cols; Kc = a->rows;
    }
    if (!ws || ws_bytes < 256) return SNIP_ERR_WORKSPACE;
    return gemm_mx_impl(a->fmt, b->fmt, a->codes, b->codes, sf_a, sf_b, Mo, No, Kc, out, out_dtype, gemm_ws(ws, 256), static_cast<cudaStream_t>(stream), ChainLink());
}

extern "C" int snip_gemm_nvfp4(int op, const snip_qtensor_t *a, const void *sf_a, const float *amax_a, const snip_qtensor_t *b, const void *sf_b,
                               const float *amax_b, void *out, int out_dtype, void *ws, size_t ws_bytes, void *stream)
{
    using namespace snip;
    if (!a || !b || op < SNIP_OP_FWD || op > SNIP_OP_WGRAD) return SNIP_ERR_ARG;
    if (a->fmt != SNIP_FMT_FP4_E2M1 || b->fmt != SNIP_FMT_FP4_E2M1) return SNIP_ERR_UNSUPPORTED;
    int64_t Mo, No, Kc;
    if (op == SNIP_OP_FWD) {
        if (a->cols != b->cols || a->transposed || b->transposed) return SNIP_ERR_SHAPE;
        if (a->block != SNIP_BLOCK_ROW_1x16 || b->block != SNIP_BLOCK_ROW_1x16) return SNIP_ERR_UNSUPPORTED;
        Mo = a->rows; No = b->rows; Kc = a->cols;
    } else if (op == SNIP_OP_DGRAD) {
        if (a->cols != b->rows || a->transposed || !b->transposed) return SNIP_ERR_SHAPE;
        if (a->block != SNIP_BLOCK_ROW_1x16 || b->block != SNIP_BLOCK_COL_16x1) return SNIP_ERR_UNSUPPORTED;
        Mo = a->rows; No = b->cols; Kc = a->cols;
    } else {
        if (a->rows != b->rows || !a->transposed || !b->transposed) return SNIP_ERR_SHAPE;
        if (a->block != SNIP_BLOCK_COL_16x1 || b->block != SNIP_BLOCK_COL_16x1) return SNIP_ERR_UNSUPPORTED;
        Mo = a->cols; No = b->cols; Kc = a->rows;
    }
    if (!ws || ws_bytes < 256) return SNIP_ERR_WORKSPACE;
    return gemm_nvfp4_impl(a->codes, b->codes, sf_a, sf_b, amax_a, amax_b, Mo, No, Kc, out, out_dtype, gemm_ws(ws, 256), static_cast<cudaStream_t>(stream), ChainLink());
}
