// Thin wrappers over the sm_100a PTX used by the GEMM kernels: mbarrier, TMA (bulk tensor
// copies), tcgen05 (tensor memory allocation, MMA issue, commit, load) and the descriptors
// the tensor core reads.  Every wait in here is bounded.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace snip {
namespace sm100 {

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Status word of a GEMM (word[0]) cleared by the launch itself, in place of a memset ahead of it (which cost the kernel a 4 us gap):
// CTA 0 clears it and leaves the launch's mark in word[1]; a CTA that gives up later reports only once that mark is there, so that the
// clearing cannot erase the report (bounded: a CTA 0 that never came to run would hold it up for `limit_ns` at most).
// A replayed graph repeats the mark: there CTA 0, scheduled first, has the whole limit of the wait that ran out to clear the word in.
__device__ __forceinline__ void status_begin(uint32_t *word, uint32_t mark)
{
    if (mark != 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        atomicExch(word, 0u);
        __threadfence();
        atomicExch(word + 1, mark);
    }
}
__device__ __forceinline__ void status_report(uint32_t *word, uint32_t mark, uint32_t value, uint64_t limit_ns)
{
    const uint64_t t0 = globaltimer_ns();
    while (mark != 0 && atomicAdd(word + 1, 0u) != mark && globaltimer_ns() - t0 < limit_ns) __nanosleep(1000);
    atomicExch(word, value);
}

// Move registers between warpgroups (all four warps of an aligned group must execute it).
template <int N> __device__ __forceinline__ void reg_alloc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void reg_dealloc() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

// One lane of a converged warp (the same one every time), chosen in a way the compiler knows to be
// warp-uniform: code under `if (elect_one())` keeps its operands in uniform registers, which is what
// the TMA and tcgen05 instructions read (a `lane == 0` branch forces a move per operand per instruction).
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xFFFFFFFF;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(pred));
    return pred != 0;
}

// ---- thread-block clusters (pairs of CTAs sharing one MMA; the two to four slices of a weight-gradient tile) ----
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Address of the same shared-memory offset in CTA `rank` of the cluster (shared::cluster window).
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// All threads of the cluster's CTAs arrive and wait (hardware barrier; every path that reaches it is bounded).
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrive on an mbarrier given by its shared::cluster address (own CTA or the other CTA of the pair), without release semantics: for
// hand-offs that publish no ordinary memory (a tensor-memory buffer whose loads have been waited for; shared-memory values that have
// already been consumed).  A release at cluster scope would first wait for every earlier memory operation of the thread.
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Arrivals by one lane of a converged warp, predicated by elect.sync: a `lane == 0` branch around the instruction, at the end of every
// chunk of a GEMM, costs 2-6 % of its cycles (but is the cheaper form between two groups of a chunk: see release_buffer in gemm.cu).
__device__ __forceinline__ void mbar_arrive_cluster_relaxed_elected(uint32_t cluster_addr)
{
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\t@p mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];\n\t}" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void mbar_arrive_elected(uint32_t bar)
{
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar) : "memory");
}
// Plain 32-bit store into the shared memory of a CTA of the cluster.
__device__ __forceinline__ void st_cluster_u32(uint32_t cluster_addr, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}

__device__ __forceinline__ void st_cluster_v4(uint32_t cluster_addr, const float4 &v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// ---- mbarrier ------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait.  Returns false if `*abort_flag` was raised by another thread or if the wait
// exceeded `limit_ns`; in the latter case it raises the flag itself.  Never spins forever.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag,
                                          uint64_t limit_ns = 2000000000ull)
{
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;   // after a failed wait anywhere in the CTA every later wait returns at once
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t i = 0;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 15u) == 15u) {
            if (*abort_flag) return false;
            if (globaltimer_ns() - t0 > limit_ns) {
                *abort_flag = 1u;
                return false;
            }
        }
    }
}

// ---- cp.async (per-thread asynchronous copies, used for the small scale-factor prefetch) ----
__device__ __forceinline__ void cp_async_4(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---- TMA --------------------------------------------------------------------------------
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *m)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// 2-D tile load global -> shared (this CTA), completion counted in bytes on `bar`.
// c0 is the innermost (contiguous) coordinate; c0 * element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *m, uint32_t bar, int32_t c0, int32_t c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}

// Same load issued by a CTA of a pair: the data lands in this CTA's shared memory, the byte count
// is reported to the barrier at `bar_cluster` (a shared::cluster address, normally the pair leader's).
// No multicast: each CTA fetches its own tiles.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *m, uint32_t bar_cluster, int32_t c0, int32_t c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar_cluster), "r"(c0), "r"(c1)
        : "memory");
}

// 2-D tile store shared -> global (bulk async group); out-of-range parts of the box are clipped.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *m, uint32_t src, int32_t c0, int32_t c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(src), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// ---- tensor memory ---------------------------------------------------------------------
// Allocate `ncols` (power of two >= 32) columns; the base address is written to shared memory.
// Must be executed by one full warp.
// PAIR = true: the allocation is made for a CTA pair (both CTAs execute it with the same warp).
template <bool PAIR>
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    if constexpr (PAIR) asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
    else asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tmem_relinquish()
{
    if constexpr (PAIR) asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    else asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    if constexpr (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Make `bar` receive one arrival when all MMAs issued so far by this thread have completed.  With PAIR the MMAs tracked are those of the
// CTA pair, and the barrier at the same offset in both CTAs of the cluster of two receives one: one instruction for both, because the
// second of two separate commits waits in the issuing thread behind the first (16384x12288x4096 FP4 forward 625 -> 619 us, 11008 x 4096 FP4
// input gradient 548 -> 538 us; FP8 8192x8192x4096 231 -> 226 us).
template <bool PAIR>
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    if constexpr (PAIR) asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((uint16_t)3) : "memory");
    else asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Load 32 consecutive columns of this warp's 32 lanes: thread i gets lane (base lane + i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// Load 16 lanes x 32 columns (lane base a multiple of 16 within the warp's 32) as a fragment: thread T gets r[2i] = lane T/4,
// column 4i + T%4 and r[2i+1] = lane T/4 + 8, the same column.  (Half the rate of the 32x32b shape; the 16x256b shape, whose
// fragments hold column pairs, has a quarter of it: 134 / 256 / 512 cycles measured for 128 x 256 words on one SM.)
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x128b.x8.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
// Wait for this thread's outstanding tcgen05.ld.  ptxas tracks the destination registers of the
// asynchronous load up to this instruction, so uses of them stay behind it.
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Store one 32-bit word per lane into `n` consecutive columns (used to fill constants).
__device__ __forceinline__ void tmem_st1(uint32_t taddr, uint32_t v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(v) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Copy a 512-byte scale-factor atom (32 rows x 16 bytes, rows contiguous) from shared memory into
// four tensor-memory columns, replicated into the four 32-lane quarters.  Runs in the tensor core's
// queue, in issue order with the MMAs of the same thread.
template <bool PAIR = false>
__device__ __forceinline__ void tmem_cp_sf_atom(uint32_t taddr, uint32_t smem_addr)
{
    // shared-memory matrix descriptor without swizzle: 8-row groups 128 bytes apart, one 16-byte column
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(16 >> 4) << 16;     // leading byte offset (a single 16-byte column: unused)
    d |= (uint64_t)(128 >> 4) << 32;    // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;             // descriptor version for sm_100
    // PAIR: one instruction copies in both CTAs of the pair, each from its own shared memory (same offset)
    if constexpr (PAIR) asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(d) : "memory");
    else asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(d) : "memory");
}

// ---- descriptors -----------------------------------------------------------------------
// Shared-memory matrix descriptor for a K-major operand tile whose rows are 128 bytes long and
// stored with the 128-byte swizzle (what a TMA box of 128 bytes x rows produces): rows 128 B
// apart, groups of 8 rows 1024 B apart.  The tile base must be 1024-byte aligned; stepping
// along K inside the 128-byte row is done by adding the byte offset to the start address.
__device__ __forceinline__ uint64_t make_smem_desc_k128(uint32_t smem_addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);  // start address, 16-byte units
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused with swizzle)
    d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset: 8 rows * 128 B
    d |= (uint64_t)1 << 46;                          // descriptor version for sm_100
    d |= (uint64_t)2 << 61;                          // 128-byte swizzle
    return d;
}

// Shared-memory matrix descriptor for an MN-major 16-bit operand tile: boxes of 64 lines (128 bytes, contiguous) x contraction rows,
// 128-byte swizzle, rows 128 B apart (so 8 rows of the contraction are 1024 B), boxes box_bytes apart along the lines.  Base
// 1024-byte aligned; 16 rows of the contraction are a step of 2048 bytes.
__device__ __forceinline__ uint64_t make_smem_desc_mn128(uint32_t smem_addr, uint32_t box_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(box_bytes >> 4) << 16;           // leading byte offset: to the next 64 lines
    d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset: to the next 8 rows of the contraction
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor for kind::f16 / kind::f8f6f4, FP32 accumulate, K-major A and B.
//   a_fmt / b_fmt: kind::f16: 0 = f16, 1 = bf16;  kind::f8f6f4: 0 = e4m3, 1 = e5m2, 5 = e2m1
__host__ __device__ constexpr uint32_t make_idesc(uint32_t a_fmt, uint32_t b_fmt, uint32_t M, uint32_t N)
{
    return (1u << 4) | (a_fmt << 7) | (b_fmt << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}
// Instruction descriptor for the block-scaled kinds (kind::mxf4 here: formats = 1 for e2m1),
// UE8M0 scale factors, scale-factor ids 0.
__host__ __device__ constexpr uint32_t make_idesc_block_scaled(uint32_t a_fmt, uint32_t b_fmt, uint32_t M, uint32_t N)
{
    return (a_fmt << 7) | (b_fmt << 10) | ((N >> 3) << 17) | (1u << 23) | ((M >> 4) << 24);
}
// The same with E4M3 scale factors (bit 23 clear), as kind::mxf4nvf4 with scale_vec::4X takes them.
__host__ __device__ constexpr uint32_t make_idesc_block_scaled_e4m3(uint32_t a_fmt, uint32_t b_fmt, uint32_t M, uint32_t N)
{
    return (a_fmt << 7) | (b_fmt << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

enum class MmaKind { F16, F8F6F4, MXF4, MXF8, NVF4 };   // MXF8 = kind::mxf8f6f4 with hardware block scales; NVF4 = kind::mxf4nvf4, E4M3 scale per 16

template <MmaKind KIND, bool PAIR>
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate,
                                       uint32_t sfa_tmem, uint32_t sfb_tmem)
{
#define SNIP_MMA(GROUP)                                                                                                        \
    if constexpr (KIND == MmaKind::F16) {                                                                                      \
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                                                       \
                     "tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),                      \
                     "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");                                        \
    } else if constexpr (KIND == MmaKind::F8F6F4) {                                                                            \
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                                                       \
                     "tcgen05.mma.cta_group::" GROUP ".kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),                   \
                     "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");                                        \
    } else if constexpr (KIND == MmaKind::MXF8) {                                                                              \
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                                                       \
                     "tcgen05.mma.cta_group::" GROUP ".kind::mxf8f6f4.block_scale [%0], %1, %2, %3, [%5], [%6], p;\n\t}"        \
                     ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)         \
                     : "memory");                                                                                              \
    } else if constexpr (KIND == MmaKind::NVF4) {                                                                              \
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                                                       \
                     "tcgen05.mma.cta_group::" GROUP ".kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%5], [%6], p;\n\t}" \
                     ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)         \
                     : "memory");                                                                                              \
    } else {                                                                                                                   \
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                                                       \
                     "tcgen05.mma.cta_group::" GROUP ".kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}" \
                     ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)         \
                     : "memory");                                                                                              \
    }
    if constexpr (PAIR) { SNIP_MMA("2") } else { SNIP_MMA("1") }
#undef SNIP_MMA
}

}  // namespace sm100
}  // namespace snip
