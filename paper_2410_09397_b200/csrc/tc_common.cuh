// sm_100a building blocks used by the tensor-core kernels: mbarriers with bounded
// waits, TMA tile loads, tensor-memory (TMEM) allocation and access, tcgen05.mma issue,
// and the shared-memory / instruction descriptors.  Inline PTX only.
//
// Waiting never blocks for ever: every wait polls for at most Abort::limit_ns (kWaitNs) nanoseconds, then
// raises the CTA's abort flag and the global status word and returns false.  After an
// abort all later waits of the CTA return at once, the kernel runs to its normal end
// (its results are then meaningless, and the caller sees ATTN_ERR_DEVICE_TIMEOUT), what is
// in flight is given time to land, TMEM is freed and the CTA exits.  Nothing is in order between the roles by then: a thread that
// loads stops at its first wait that fails, and a stage is released only by a thread that has
// seen its load land, since a barrier must not be armed twice in one phase.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "tc_units.cuh"

namespace attn {
namespace tc {

constexpr unsigned long long kWaitNs = 1000000000ull;   // 1 s per wait

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// ------------------------------------------------------------------ mbarrier
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Per-CTA abort state: `flag` lives in shared memory, `status` is the workspace word, `limit_ns` is how
// long one wait may poll (the kernels of the library leave it at kWaitNs).
struct Abort {
    volatile uint32_t *flag;
    uint32_t *status;
    unsigned long long limit_ns = kWaitNs;
};

// Returns true when the phase with the given parity has completed.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, const Abort &ab)
{
    if (mbar_try_wait(bar, parity)) return true;
    if (*ab.flag) return false;
    const unsigned long long t0 = globaltimer();
    uint32_t spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 63u) == 0) {
            if (*ab.flag) return false;
            if (globaltimer() - t0 > ab.limit_ns) {
                *ab.flag = 1u;
                atomicExch(ab.status, 10u);   // ATTN_ERR_DEVICE_TIMEOUT
                return false;
            }
        }
    }
    return true;
}

// For a loading thread: the stage has been released and the load before, for which `full` was armed, has landed, which a release that
// comes early because the CTA is giving up does not tell.  (Only where the role that releases the stage does not itself wait for the
// load.)  Both in one go: a wait of the loading thread takes long while the products stream their operands.
__device__ __forceinline__ bool mbar_reload(uint64_t *full, uint64_t *empty, uint32_t parity, const Abort &ab)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %3;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 q, [%2], %3;\n\t"
        "and.pred p, p, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(full)), "r"(smem_u32(empty)), "r"(parity)
        : "memory");
    return ok != 0 || (mbar_wait(full, parity, ab) && mbar_wait(empty, parity, ab));
}

// ------------------------------------------------------------------ fences
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tcgen05_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tcgen05_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ------------------------------------------------------------------ TMA (tiled; every load is issued by one CTA for itself)
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *m)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// x = innermost coordinate (elements; x * element size must be a multiple of 16 bytes)
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *m, uint64_t *bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *m, uint64_t *bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *m, const void *src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(src)), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *m, const void *src, int x, int y, int z)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// ------------------------------------------------------------------ TMEM
// One warp allocates `cols` (power of two, 32..512) columns; the base address lands in *dst_smem.
__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// The end of a kernel that holds tensor memory.  In the usual course every load and product has been waited for by now.  A CTA that
// gives up may have some in flight, which must not land in the shared or tensor memory of its successor: it holds both for kSettleNs
// more.  The longest queue of products and the slowest load take some ten microseconds.
constexpr unsigned long long kSettleNs = 1000000ull;
__device__ __forceinline__ void tmem_leave(uint32_t taddr, uint32_t cols, int warp, const Abort &ab)
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        if (__any_sync(0xffffffffu, *ab.flag != 0)) {
            const unsigned long long t0 = globaltimer();
            while (globaltimer() - t0 < kSettleNs) __nanosleep(1000);
            __syncwarp();
        }
        tmem_dealloc(taddr, cols);
    }
}

// 32 lanes x 32 consecutive 32-bit columns: thread t of the warp gets lane (base lane + t),
// v[k] = column (base column + k).  The lane field of taddr must be the warp's own
// quarter: 32 * (warp index % 4).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]),
        "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]),
        "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------------ descriptors
// Shared-memory matrix descriptor (64 bit): start address >> 4 in bits 0-13, leading
// byte offset >> 4 in 16-29, stride byte offset >> 4 in 32-45, descriptor version 1 in
// 46-47, swizzle mode in 61-63 (2 = 128-byte swizzle).  Operand tiles here are always
// what a 128-byte-swizzled TMA load of a [rows][64 bf16] box produces: row r at byte
// r * 128, 16-byte chunk c of a row stored at chunk (c xor (r mod 8)); tile bases are
// 1024-byte aligned.  Such a tile is
//   * a K-major operand when the contraction runs along the 64 contiguous elements
//     (8-row groups 1024 bytes apart = stride byte offset; a K step of 16 elements
//     advances the start address by 32 bytes), and
//   * an MN-major operand when the contraction runs along the rows (8-row groups again
//     1024 bytes apart; further 64-element slabs of the M/N dimension are `slab_bytes`
//     apart = leading byte offset; a K step of 16 rows advances the start by 2048 bytes).
__device__ __forceinline__ uint64_t smem_desc_kmajor(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ uint64_t smem_desc_mnmajor(uint32_t saddr, uint32_t slab_bytes)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(slab_bytes >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Instruction descriptor for kind::f16 with bf16 operands and fp32 accumulation.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn_major, int b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ------------------------------------------------------------------ MMA issue (one thread)
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The same issue with the descriptors given as their low 32-bit words.  Every operand
// tile in this library has a stride byte offset of 1024, descriptor version 1 and the
// 128-byte swizzle, so the high word is the constant kDescHi; the low word is
// (address >> 4) | (leading byte offset >> 4) << 16, and stepping through a tile is one
// 32-bit add of (byte offset >> 4).  This keeps the single issuing thread short.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo_kmajor(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ uint32_t desc_lo_mnmajor(uint32_t saddr, uint32_t slab_bytes)
{
    return ((saddr & 0x3FFFFu) >> 4) | ((slab_bytes >> 4) << 16);
}
__device__ __forceinline__ void mma_ss_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "mov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi)
        : "memory");
}
__device__ __forceinline__ void mma_ts_lo(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi)
        : "memory");
}
// Arrives on `bar` once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// Byte offset of element (row, col) inside a 128-byte-swizzled [rows][64 bf16] slab.
__device__ __forceinline__ uint32_t sw128_offset(uint32_t row, uint32_t col)
{
    return row * 128u + ((((col >> 3) ^ (row & 7u)) << 4) | ((col & 7u) << 1));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// v * s + n and p * (v * s + n) of two entries, an instruction each (the roundings of the scalar forms)
__device__ __forceinline__ uint64_t fma_pair(uint32_t v0, uint32_t v1, float s, float n0, float n1)
{
    uint64_t x, y, z;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(v0), "r"(v1));
    asm("mov.b64 %0, {%1, %1};" : "=l"(y) : "f"(s));
    asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(n0), "f"(n1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(x) : "l"(x), "l"(y), "l"(z));
    return x;
}
__device__ __forceinline__ void mul_pair(uint64_t x, uint32_t p0, uint32_t p1, float &d0, float &d1)
{
    uint64_t w;
    asm("mov.b64 %0, {%1, %2};" : "=l"(w) : "r"(p0), "r"(p1));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(x) : "l"(x), "l"(w));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d0), "=f"(d1) : "l"(x));
}

// What two fp32 values lose when they are packed as `hi` (pack_bf16), packed the same way: x = hi + lo up to 2^-17 |x|.
__device__ __forceinline__ uint32_t pack_bf16_rest(float x, float y, uint32_t hi)
{
    return pack_bf16(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
}

// ------------------------------------------------------------------ schedule
// The hardware's scheduler hands CTAs of the grid that have not started yet to CTAs that run (cluster launch control): the
// answer, 16 bytes, arrives in shared memory and reports to `bar`.  After an answer without work no further one may be asked for.
__device__ __forceinline__ void clc_request(void *answer, uint64_t *bar)
{
    mbar_expect_tx(bar, 16);
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 ::"r"(smem_u32(answer)), "r"(smem_u32(bar)) : "memory");
}
// The block index that was handed over; false: there is none left.
__device__ __forceinline__ bool clc_answer(const void *answer, int &bx, int &by)
{
    uint32_t ok, x, y;
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b128 r;\n\t.reg .b32 z, w;\n\t"
        "ld.shared.b128 r, [%3];\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t"
        "mov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, %2, z, w}, r;\n\t}"
        : "=r"(ok), "=r"(x), "=r"(y) : "r"(smem_u32(answer)) : "memory");
    bx = (int)x; by = (int)y;
    fence_proxy_async_smem();   // read before the next answer is written
    return ok != 0;
}

template <int kGroup = 0>   // threads that take units together (named barrier 1)
struct UnitIo {   // UnitQueue on the hardware
    Abort ab;
    __device__ __forceinline__ bool wait(uint64_t *bar, uint32_t parity) const { return mbar_wait(bar, parity, ab); }
    __device__ __forceinline__ bool late() const { return *ab.flag != 0; }
    __device__ __forceinline__ bool all(bool x) const { return __all_sync(0xffffffffu, x); }
    __device__ __forceinline__ bool all_warps(bool x) const
    {
        uint32_t y;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                     : "=r"(y) : "r"((uint32_t)x), "n"(kGroup) : "memory");
        return y != 0;
    }
    __device__ __forceinline__ void arrive(uint64_t *bar) const { mbar_arrive(bar); }
    __device__ __forceinline__ void request(void *answer, uint64_t *bar) const { clc_request(answer, bar); }
    __device__ __forceinline__ bool answer(const void *from, int &bx, int &by) const { return clc_answer(from, bx, by); }
};

// 32 bytes to global memory (a whole sector); `wide`: the address is a multiple of 32, else of 16
__device__ __forceinline__ void store32(void *to, const uint32_t (&v)[8], bool wide)
{
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(to), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                     "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
    } else {
        reinterpret_cast<uint4 *>(to)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<uint4 *>(to)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

}  // namespace tc

// ------------------------------------------------------------------ host: tensor maps
// rank-3 bf16 tensor [dim2][dim1][dim0] (dim0 contiguous), box [1][box1][64], 128-byte swizzle,
// out-of-range elements read as zero.  Returns false if the driver refuses.
bool make_tmap_bf16_3d(CUtensorMap *out, const void *base, uint64_t dim0, uint64_t dim1, uint64_t dim2, uint32_t box1);
// rank-3 fp32 tensor [dim2][dim1][dim0], box [1][box1][32] (128 bytes a row), 128-byte swizzle
bool make_tmap_f32_3d(CUtensorMap *out, const void *base, uint64_t dim0, uint64_t dim1, uint64_t dim2, uint32_t box1);
// the same as the first with the row pitch (elements), the box [1][box1][box0] and the swizzle span (64 or 128 bytes;
// box0 * 2 bytes must not exceed it) given: the maps of the tiles that TMA stores write
bool make_tmap_bf16_3d_box(CUtensorMap *out, const void *base, uint64_t dim0, uint64_t dim1, uint64_t dim2, uint64_t pitch_elems,
                           uint32_t box0, uint32_t box1, int swizzle_bytes);
// rank-2 bf16 matrix [rows][cols] with row pitch `pitch_bytes`, box [box_rows][64].
bool make_tmap_bf16_2d(CUtensorMap *out, const void *base, uint64_t cols, uint64_t rows, uint64_t pitch_bytes,
                       uint32_t box_rows);

}  // namespace attn
