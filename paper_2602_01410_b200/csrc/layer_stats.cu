// Layer statistics in one read per tensor (paper Sec. 3.1, Step 1): sum x^2 of a bf16 tensor and,
// for the tensors that get quantized (X, W, dY), the error sums  sum (x - code/S)^2  under every
// candidate format (FP8 E4M3, FP4 E2M1) and every tile kind the tensor is consumed with
// (X, dY: 1x128 along the columns and 128x1 along the rows; W: 128x128), all from the same
// registers.  The scheme-generation step needs the error of every option (Sec. 4.4), not only of
// the format currently in use.
//
// One persistent launch for all six tensors, three CTAs of 256 threads per SM.  X, W and dY are bound by instruction issue (66 % of the
// slots, with two CTA barriers a tile; no pipe is full), Y, dX and dW, of which only the norm is wanted, by HBM; so every SM
// works on both kinds at once, some CTAs on tiles of the first, some streaming the second.  Tiles are 128x128, each thread an 8x8
// sub-block that it fetches itself (cp.async into a private slot, one tile ahead).  Scales and codes are the quantizer's: S =
// FPX_MAX/amax (binary32 quotient, one division per tile and format, shared through shared memory), code = RNE_fmt(fl32(x*S)); the error
// term is x - value(code)/S for FP8 (per element pair a product, two packed FMAs, a conversion to the format and three back) and
// value(code) - fl32(x*S) for FP4 (two additions for one of the FMAs and two of the conversions, weighed by S^-2 per tile line).  A
// reduction of the CTAs' sums follows.
// Six tensors of an 8192 x 3200 x 9600 linear: 250 -> 135 us, X with four options 16384 x 4096: 92 -> 68 us (before: thirteen launches of one
// tile per CTA, every thread dividing for all of its rows and columns).
#include <stddef.h>

#include "common.cuh"
#include "quant_device.cuh"

namespace snip {

int gemm_sm_count();  // gemm.cu

namespace {

constexpr int kTile = 128;
constexpr int kThreads = 256;
constexpr int kCtas = 3;             // per SM
constexpr int kSlotBytes = kTile * kTile * 2;

enum { MODE_PLAIN = 0, MODE_BLK = 1, MODE_ROWCOL = 2 };
constexpr int kChunk = kThreads * 64;   // elements a CTA takes at a time of a tensor without error sums

// per CTA: [0] sum x^2; [1] FP8 kind A; [2] FP8 kind B; [3] FP4 kind A; [4] FP4 kind B
// (ROWCOL: A = ROW, B = COL; BLK: A = BLK, B unused)
struct StatsPartial {
    double v[8];
};

struct StatsTensor {
    const uint16_t *x;
    int32_t rows, cols, tiles_c;
    int32_t nitems;                  // tiles, or chunks (MODE_PLAIN)
    int32_t mode;
    StatsPartial *partials;          // one per CTA that has items of it
};
// Tensors with error sums (heavy) and without (light); each list is one sequence of items dealt in turn to the CTAs that work on it.
struct LayerStatsArgs {
    StatsTensor t[6];
    int32_t nheavy, nlight;          // t[0 .. nheavy), t[nheavy .. nheavy + nlight)
    int32_t light_ctas;              // the first CTAs stream the light tensors, the others take tiles
};

struct Scales {                      // of one tile line: scale and negated reciprocal for both formats
    float s8, n8, s4, n4;
};
struct Shared {
    uint32_t col_amax[8][kTile / 2];  // packed bf16 pairs, one row per warp
    __align__(16) Scales row[kTile];
    __align__(16) float col[4][kTile];   // the four values apart: a thread reads eight consecutive columns (interleaved, 8-way bank conflicts)
    uint32_t blk_amax[2][8];
    double red[8][5];
    __align__(16) uint8_t slot[2][kSlotBytes];   // the tile at hand and the next one; not there in a launch without heavy tensors
};

// (The reciprocal is the correctly rounded one of S itself: FP4's weighs whole sums, in which a bias like that of amax * fl(1/FPX_MAX)
// would stay.)
template <bool F8, bool F4>
__device__ __forceinline__ Scales scales_of(float am)
{
    Scales s = {0.0f, 0.0f, 0.0f, 0.0f};
    if (F8) { s.s8 = tile_scale<SNIP_FMT_FP8_E4M3>(am, 0); s.n8 = -__frcp_rn(s.s8); }
    if (F4) { s.s4 = tile_scale<SNIP_FMT_FP4_E2M1>(am, 0); s.n4 = -__frcp_rn(s.s4); }
    return s;
}

// Adds the squared error of an element pair under FP8; n = -1/S.
__device__ __forceinline__ void err_pair_f8(const float2 x, const float2 s, const float2 n, float2 &se2)
{
    const float2 t = __fmul2_rn(x, s);
    const float2 e = __ffma2_rn(dec_e4m3x2(cvt_e4m3x2(t.x, t.y)), n, x);
    se2 = __ffma2_rn(e, e, se2);
}
// Under FP4, in units of 1/S^2 ...
__device__ __forceinline__ void err_pair_f4(const float2 x, const float2 s, float2 &se2)
{
    const float2 e = fp4_scaled_rounding_err(__fmul2_rn(x, s));
    se2 = __ffma2_rn(e, e, se2);
}
// ... and back to the units of x (two multiplications: 1/S^2 alone may leave binary32 where the product does not).
__device__ __forceinline__ float unscale(const float2 se2, float n, float sum) { return fmaf((se2.x + se2.y) * n, n, sum); }

__device__ __forceinline__ void fetch(const StatsTensor &t, int tile, uint8_t *slot)
{
    if (tile < t.nitems) {
        const int tid = threadIdx.x, tr = tile / t.tiles_c, tc = tile - tr * t.tiles_c;
        const int r = tr * kTile + 8 * (tid >> 4), c = tc * kTile + 8 * (tid & 15);
        const bool ok = r < t.rows && c < t.cols;    // dims are multiples of 64: all 64 elements or none
        const uint16_t *src = t.x + (ok ? (int64_t)r * t.cols + c : 0);
        const uint32_t step = ok ? (uint32_t)t.cols : 0u, dst = (uint32_t)__cvta_generic_to_shared(slot) + tid * 16;
        const int nbytes = ok ? 16 : 0;              // 0: the slot is zero-filled, nothing is read
#pragma unroll
        for (int p = 0; p < 8; ++p)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + p * (kThreads * 16)), "l"(src + p * step), "r"(nbytes) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The CTA's sums of one tensor -> its partial (block reduction in a fixed order); the sums start again at zero.
__device__ __forceinline__ void flush(const StatsTensor &t, int slot, Shared &sh, double (&acc)[5])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc[k] += __shfl_xor_sync(0xFFFFFFFFu, acc[k], off);
    }
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 5; ++k) sh.red[warp][k] = acc[k];
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        double d = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) d += sh.red[w][threadIdx.x];
        t.partials[slot].v[threadIdx.x] = d;
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) acc[k] = 0.0;
}

// Sum of squares of 64 elements per thread (eight 16-byte pieces).
__device__ __forceinline__ float sumsq64(const uint4 (&v)[8])
{
    float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        const uint32_t w[4] = {v[p].x, v[p].y, v[p].z, v[p].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 x = make_float2(bf16lo(w[i]), bf16hi(w[i]));
            s = __ffma2_rn(x, x, s);
        }
    }
    return s.x + s.y;
}

// The light tensors: contiguous arrays, streamed.
__device__ __forceinline__ void run_light(const LayerStatsArgs &a, int cta, int ctas, Shared &sh)
{
    int first = cta;
    for (int j = a.nheavy; j < a.nheavy + a.nlight; ++j) {
        const StatsTensor &t = a.t[j];
        const int64_t n = (int64_t)t.rows * t.cols;
        double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        int c = first;
        for (; c < t.nitems; c += ctas) {
            const int64_t base = (int64_t)c * kChunk + threadIdx.x * 8;
            uint4 v[8];
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const int64_t at = base + p * (kThreads * 8);
                v[p] = at < n ? __ldg(reinterpret_cast<const uint4 *>(t.x + at)) : make_uint4(0, 0, 0, 0);
            }
            acc[0] += (double)sumsq64(v);
        }
        if (first < t.nitems) flush(t, first, sh, acc);
        first = c - t.nitems;   // the deal goes on where this tensor ended
    }
}

template <bool F8, bool F4>
__global__ void __launch_bounds__(kThreads, kCtas) layer_stats_kernel(const __grid_constant__ LayerStatsArgs a)
{
    extern __shared__ __align__(128) uint8_t smem[];
    Shared &sh = *reinterpret_cast<Shared *>(smem);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;

    if ((int)blockIdx.x < a.light_ctas) { run_light(a, (int)blockIdx.x, a.light_ctas, sh); return; }
    const int ctas = (int)gridDim.x - a.light_ctas;
    int first = (int)blockIdx.x - a.light_ctas, parity = 0;
    for (int j = 0; j < a.nheavy; ++j) {
        const StatsTensor &t = a.t[j];
        if (first >= t.nitems) { first -= t.nitems; continue; }
        const bool rowcol = t.mode == MODE_ROWCOL;
        double hacc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        int tile = first;
        int buf = 0;
        fetch(t, tile, sh.slot[0]);
        for (; tile < t.nitems; tile += ctas) {
            fetch(t, tile + ctas, sh.slot[buf ^ 1]);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            const uint4 *slot = reinterpret_cast<const uint4 *>(sh.slot[buf]) + threadIdx.x;
            buf ^= 1;
            float2 sx2 = make_float2(0.0f, 0.0f);
            float2 e8a = make_float2(0.0f, 0.0f), e8b = e8a;
            float e4a = 0.0f, e4b = 0.0f;
            // maxima (signs are garbage until masked: max.xorsign.abs keeps magnitudes only)
            uint32_t rmax[8], cm[4] = {0, 0, 0, 0};
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const uint4 v = slot[p * kThreads];
                rmax[p] = absmax2x(absmax2x(v.x, v.y), absmax2x(v.z, v.w));
                cm[0] = absmax2x(cm[0], v.x);
                cm[1] = absmax2x(cm[1], v.y);
                cm[2] = absmax2x(cm[2], v.z);
                cm[3] = absmax2x(cm[3], v.w);
            }
            if (rowcol) {
                // rows: exchange-halving butterfly over the 16 lanes of a row group; lane tx ends up with rows 4 bit3 + 2 bit2 + {0, 1}
                // and derives the scales of the one its bit 0 names
                uint32_t pk[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    pk[q] = max2(__byte_perm(rmax[2 * q], rmax[2 * q + 1], 0x5410) & 0x7FFF7FFFu, __byte_perm(rmax[2 * q], rmax[2 * q + 1], 0x7632) & 0x7FFF7FFFu);
                const bool b3 = (tx & 8) != 0, b2 = (tx & 4) != 0;
                uint32_t k0 = b3 ? pk[2] : pk[0], k1 = b3 ? pk[3] : pk[1];
                const uint32_t g0 = b3 ? pk[0] : pk[2], g1 = b3 ? pk[1] : pk[3];
                k0 = max2(k0, __shfl_xor_sync(0xFFFFFFFFu, g0, 8));
                k1 = max2(k1, __shfl_xor_sync(0xFFFFFFFFu, g1, 8));
                uint32_t k = b2 ? k1 : k0;
                const uint32_t g = b2 ? k0 : k1;
                k = max2(k, __shfl_xor_sync(0xFFFFFFFFu, g, 4));
                k = max2(k, __shfl_xor_sync(0xFFFFFFFFu, k, 2));
                k = max2(k, __shfl_xor_sync(0xFFFFFFFFu, k, 1));
                const float am = (tx & 1) ? bf16hi(k) : bf16lo(k);
                const Scales rs = scales_of<F8, F4>(am);
                if (!(tx & 2)) sh.row[8 * ty + ((tx >> 3) & 1) * 4 + ((tx >> 2) & 1) * 2 + (tx & 1)] = rs;
                // columns: the two row groups of a warp, then the 8 warps through shared memory
#pragma unroll
                for (int q = 0; q < 4; ++q) cm[q] = absmax2x(cm[q], __shfl_xor_sync(0xFFFFFFFFu, cm[q], 16));
                if (lane < 16) *reinterpret_cast<uint4 *>(&sh.col_amax[warp][4 * tx]) = make_uint4(cm[0], cm[1], cm[2], cm[3]);
                __syncthreads();
                if (tid < kTile) {
                    const uint16_t *h = reinterpret_cast<const uint16_t *>(&sh.col_amax[0][0]);
                    uint32_t m = 0;
#pragma unroll
                    for (int w = 0; w < 8; ++w) m = max(m, (uint32_t)h[w * kTile + tid] & 0x7FFFu);   // non-negative bf16: integer order
                    const Scales cs = scales_of<F8, F4>(__uint_as_float(m << 16));
                    sh.col[0][tid] = cs.s8; sh.col[1][tid] = cs.n8; sh.col[2][tid] = cs.s4; sh.col[3][tid] = cs.n4;
                }
                __syncthreads();
                float2 cs8[4], cn8[4], cs4[4], c4[4];   // c4: FP4 errors squared of the column pairs, in units of their scales
                auto get = [&](int k, float2 (&d)[4]) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float4 c = *reinterpret_cast<const float4 *>(&sh.col[k][8 * tx + 4 * i]);
                        d[2 * i] = make_float2(c.x, c.y);
                        d[2 * i + 1] = make_float2(c.z, c.w);
                    }
                };
                if (F8) { get(0, cs8); get(1, cn8); }
                if (F4) get(2, cs4);
#pragma unroll
                for (int i = 0; i < 4; ++i) c4[i] = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    const uint4 v = slot[p * kThreads];
                    const float4 r = *reinterpret_cast<const float4 *>(&sh.row[8 * ty + p]);
                    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
                    float2 r4 = make_float2(0.0f, 0.0f);   // of this row
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 x = make_float2(bf16lo(w[i]), bf16hi(w[i]));
                        sx2 = __ffma2_rn(x, x, sx2);
                        if (F8) {
                            err_pair_f8(x, make_float2(r.x, r.x), make_float2(r.y, r.y), e8a);
                            err_pair_f8(x, cs8[i], cn8[i], e8b);
                        }
                        if (F4) {
                            err_pair_f4(x, make_float2(r.z, r.z), r4);
                            err_pair_f4(x, cs4[i], c4[i]);
                        }
                    }
                    if (F4) e4a = unscale(r4, r.w, e4a);
                }
                if (F4) {
                    // (the column scales of this tile stay in place until every warp has passed the next tile's first barrier)
                    float2 n[4];
                    get(3, n);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        e4b = fmaf(c4[i].x * n[i].x, n[i].x, e4b);
                        e4b = fmaf(c4[i].y * n[i].y, n[i].y, e4b);
                    }
                }
            } else {
                uint32_t m = absmax2x(absmax2x(cm[0], cm[1]), absmax2x(cm[2], cm[3])) & 0x7FFF7FFFu;
                m = __reduce_max_sync(0xFFFFFFFFu, max(m & 0xFFFFu, m >> 16));
                parity ^= 1;   // the other half may still be read by warps that are behind
                if (lane == 0) sh.blk_amax[parity][warp] = m;
                __syncthreads();
                uint32_t bm = sh.blk_amax[parity][0];
#pragma unroll
                for (int w = 1; w < 8; ++w) bm = max(bm, sh.blk_amax[parity][w]);
                const Scales s = scales_of<F8, F4>(__uint_as_float(bm << 16));
                const float2 s8 = make_float2(s.s8, s.s8), n8 = make_float2(s.n8, s.n8), s4 = make_float2(s.s4, s.s4);
                float2 b4 = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    const uint4 v = slot[p * kThreads];
                    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 x = make_float2(bf16lo(w[i]), bf16hi(w[i]));
                        sx2 = __ffma2_rn(x, x, sx2);
                        if (F8) err_pair_f8(x, s8, n8, e8a);
                        if (F4) err_pair_f4(x, s4, b4);
                    }
                }
                e4a = unscale(b4, s.n4, e4a);
            }
            hacc[0] += (double)(sx2.x + sx2.y);
            if (F8) { hacc[1] += (double)(e8a.x + e8a.y); hacc[2] += (double)(e8b.x + e8b.y); }
            if (F4) { hacc[3] += (double)e4a; hacc[4] += (double)e4b; }
        }
        flush(t, first, sh, hacc);
        first = tile - t.nitems;
    }
}

// Fixed-order sums of the CTAs' partials, one block per tensor of the result; every value of the result is written (0 for what was not
// asked for).
struct ReduceArgs {
    const StatsPartial *partials[6];   // null: tensor not given
    int32_t n[6];
    uint32_t fmt_mask;
    snip_layer_stats_t *out;
};
__global__ void __launch_bounds__(256) layer_stats_reduce_kernel(const ReduceArgs a)
{
    __shared__ double sh[8][5];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int i = blockIdx.x;
    double d[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (a.partials[i]) {
        for (int k = threadIdx.x; k < a.n[i]; k += 256) {
#pragma unroll
            for (int c = 0; c < 5; ++c) d[c] += a.partials[i][k].v[c];
        }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) d[c] += __shfl_xor_sync(0xFFFFFFFFu, d[c], off);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < 5; ++c) sh[warp][c] = d[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            t[c] = 0.0;
            for (int w = 0; w < 8; ++w) t[c] += sh[w][c];
        }
        a.out->sumsq[i] = t[0];
        const int q = i == 0 ? 0 : i == 1 ? 1 : i == 3 ? 2 : -1;   // X, W, dY have error sums
        if (q >= 0) {
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                const bool on = (a.fmt_mask & (2u << f)) != 0;
                a.out->sumsq_err[q][f][SNIP_BLOCK_ROW_1x128] = on && q != 1 ? t[1 + 2 * f] : 0.0;
                a.out->sumsq_err[q][f][SNIP_BLOCK_COL_128x1] = on && q != 1 ? t[2 + 2 * f] : 0.0;
                a.out->sumsq_err[q][f][SNIP_BLOCK_BLK_128x128] = on && q == 1 ? t[1 + 2 * f] : 0.0;
            }
        }
    }
}

size_t tensor_ws_bytes(int64_t rows, int64_t cols)
{
    return align_up((size_t)(ceil_div(rows, kTile) * ceil_div(cols, kTile)) * sizeof(StatsPartial), 256);
}

template <bool F8, bool F4>
int launch_stats(const LayerStatsArgs &a, int grid, cudaStream_t st)
{
    const size_t smem = a.nheavy ? sizeof(Shared) : offsetof(Shared, slot);
    auto kern = layer_stats_kernel<F8, F4>;
    SNIP_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared)));
    kern<<<grid, kThreads, smem, st>>>(a);
    SNIP_CUDA_TRY(cudaGetLastError());
    return SNIP_OK;
}

}  // namespace
}  // namespace snip

extern "C" int snip_layer_stats_workspace(int64_t M, int64_t N, int64_t K, size_t *ws_bytes)
{
    using namespace snip;
    if (!ws_bytes) return SNIP_ERR_ARG;
    if (!valid_dim(M) || !valid_dim(N) || !valid_dim(K)) return SNIP_ERR_SHAPE;
    *ws_bytes = 2 * (tensor_ws_bytes(M, K) + tensor_ws_bytes(N, K) + tensor_ws_bytes(M, N));
    return SNIP_OK;
}

extern "C" int snip_layer_stats(const snip_layer_tensors_t *t, uint32_t fmt_mask, snip_layer_stats_t *out, void *ws, size_t ws_bytes,
                                void *stream)
{
    using namespace snip;
    if (!t || !out || !ws) return SNIP_ERR_ARG;
    if (fmt_mask & ~6u) return SNIP_ERR_ARG;
    size_t need = 0;
    int rc = snip_layer_stats_workspace(t->M, t->N, t->K, &need);
    if (rc) return rc;
    if (ws_bytes < need) return SNIP_ERR_WORKSPACE;
    if (!aligned16(ws) || !aligned16(out)) return SNIP_ERR_ALIGN;
    rc = require_sm100();
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t M = t->M, N = t->N, K = t->K;
    struct T { const void *p; int64_t r, c; int mode; } tens[6] = {
        {t->X, M, K, MODE_ROWCOL}, {t->W, N, K, MODE_BLK}, {t->Y, M, N, MODE_PLAIN}, {t->dY, M, N, MODE_ROWCOL}, {t->dX, M, K, MODE_PLAIN}, {t->dW, N, K, MODE_PLAIN}};
    // every argument is checked before anything is enqueued
    LayerStatsArgs a = {};
    ReduceArgs red = {};
    red.fmt_mask = fmt_mask;
    red.out = out;
    int64_t total = 0;
    uint8_t *cursor = static_cast<uint8_t *>(ws);
    StatsPartial *parts[6];
    for (int i = 0; i < 6; ++i) {
        parts[i] = reinterpret_cast<StatsPartial *>(cursor);
        cursor += tensor_ws_bytes(tens[i].r, tens[i].c);
        if (!tens[i].p) continue;
        if (!aligned16(tens[i].p)) return SNIP_ERR_ALIGN;
        if (ceil_div(tens[i].r, kTile) > 65535) return SNIP_ERR_SHAPE;
        const int64_t n = ceil_div(tens[i].r, kTile) * ceil_div(tens[i].c, kTile);
        if (n > INT32_MAX || tens[i].c > INT32_MAX) return SNIP_ERR_SHAPE;
        total += n;
    }
    const int64_t cap = kCtas * (int64_t)gemm_sm_count();
    const int grid = (int)(total < cap ? total : cap);
    for (int heavy = 1; heavy >= 0; --heavy) {
        for (int i = 0; i < 6; ++i) {
            const int mode = fmt_mask ? tens[i].mode : MODE_PLAIN;
            if (!tens[i].p || (mode != MODE_PLAIN) != (heavy == 1)) continue;
            StatsTensor &s = a.t[a.nheavy + a.nlight];
            s.x = static_cast<const uint16_t *>(tens[i].p);
            s.rows = (int32_t)tens[i].r; s.cols = (int32_t)tens[i].c;
            s.tiles_c = (int32_t)ceil_div(tens[i].c, kTile);
            s.nitems = heavy ? (int32_t)(ceil_div(tens[i].r, kTile) * s.tiles_c) : (int32_t)ceil_div(tens[i].r * tens[i].c, (int64_t)kChunk);
            s.mode = mode;
            s.partials = parts[i];
            red.partials[i] = parts[i];
            if (heavy) ++a.nheavy; else ++a.nlight;
        }
    }
    // CTAs of each kind by their cost per 128x128 elements, measured: about 5 (1x128 and 128x1 tiles), 3 (128x128) and 1 (norm only).  FP4
    // alone costs a little less than that (16384 x 4096 x 4096 136.6 us at 5 : 3 : 1, 132.2 us so; 8192 x 3200 x 9600 119.3, 116.8 us).
    const bool f4_alone = fmt_mask == 4u;
    int64_t cost[2] = {0, 0};
    for (int i = 0; i < a.nheavy + a.nlight; ++i)
        cost[i < a.nheavy ? 0 : 1] += (int64_t)a.t[i].nitems * (a.t[i].mode == MODE_ROWCOL ? (f4_alone ? 47 : 50) : a.t[i].mode == MODE_BLK ? (f4_alone ? 29 : 30) : 10);
    a.light_ctas = a.nheavy == 0 ? grid : 0;
    if (a.nheavy && a.nlight) {
        a.light_ctas = (int32_t)(grid * cost[1] / (cost[0] + cost[1]));
        // (past about 108 of 444 the launch takes 15-30 % longer, with any option: 512 x 8192 x 28672 179 us at 107, 239 us at 110)
        if (f4_alone && a.light_ctas > grid * 6 / 25) a.light_ctas = grid * 6 / 25;
        if (a.light_ctas < 1) a.light_ctas = 1;
        if (a.light_ctas > grid - 1) a.light_ctas = grid - 1;
    }
    for (int i = 0, h = 0; i < 6; ++i) {
        if (!tens[i].p) continue;
        h = 0;
        while (a.t[h].partials != parts[i]) ++h;
        const int ctas = h < a.nheavy ? grid - a.light_ctas : a.light_ctas;
        red.n[i] = a.t[h].nitems < ctas ? a.t[h].nitems : ctas;
    }
    if (grid > 0) {
        const bool f8 = (fmt_mask & 2u) != 0, f4 = (fmt_mask & 4u) != 0;
        rc = f8 && f4 ? launch_stats<true, true>(a, grid, st) : f8 ? launch_stats<true, false>(a, grid, st) : launch_stats<false, true>(a, grid, st);
        if (rc) return rc;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(6);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SNIP_CUDA_TRY(cudaLaunchKernelEx(&cfg, layer_stats_reduce_kernel, red));
    return SNIP_OK;
}
