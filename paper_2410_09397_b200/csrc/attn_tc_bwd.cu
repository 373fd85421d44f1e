// Fused backward for bf16 on the 5th-generation tensor cores (large-cache regime of
// Appendix D: no n x n matrix ever leaves the SM).
//
// The loops of the paper's phase-2 algorithm are swapped: a CTA owns one tile of 128
// KEYS j (K_j, V_j stay in shared memory, dK_j and dV_j stay in tensor memory) and walks
// the kept QUERY tiles i.  Per (i, j) pair, with everything transposed so that the
// tensor-memory lane is the key index:
//
//   S^T  = K_j Q_i^T                         (tcgen05.mma, both operands K-major smem)
//   dP^T = V_j dO_i^T                        (same)
//   P^T  = exp2(S^T * scale*log2e - LSE_i*log2e)        (256 threads, fp32)
//   dS^T = scale * P^T o (dP^T - D_i)                   (Definition B.9, p = f o q - diag(v) f;
//                                                        the scale of dQ and dK is folded in here)
//   dV_j += P^T  dO_i      A = P^T  in tensor memory (bf16), B = dO_i MN-major smem
//   dK_j += dS^T Q_i       A = dS^T K-major smem,            B = Q_i  MN-major smem
//   dQ_i += dS K_j         computed as dQ^T = K_j^T dS^T (lane = head-dimension index), so that
//                          the fp32 reductions into global memory are coalesced; at d = 64 the
//                          product is padded to M = 128 with an all-zero slab
//
// dQ partial tiles are added into an fp32 accumulator in the workspace with
// red.global.add (the one place where summation order is not fixed); a small kernel
// converts it to bf16 at the end.  Tensor memory (512 columns): 128 take S^T and dP^T in turn (fused kernel, d = 64: S^T
// alone, dP^T has 128 of its own), 128 take P^T and dQ^T (dK/dV kernel: P^T and dS^T), dV d, dK d.
//
// Two kernels: tc_bwd_fused_kernel (all five products, the default) and tc_bwd_dkdv_kernel
// (without the dQ product; `deterministic = 1`, and lengths that are no multiple of 8, pair it with the
// query-stationary dQ kernel of attn_tc_bwd_dq.cu).  Warp roles are described at each kernel.  All waits are bounded
// (tc_common.cuh).
#include "tc_bwd_common.cuh"

namespace attn {
namespace {

using namespace tc;
using namespace bwdk;

constexpr int TQ = 128;
template <int HD>
struct BwdSmem {
    static constexpr int NS = HD == 64 ? 3 : 2;           // stages of Q, dO and the row statistics
    static constexpr int NdS = HD == 64 ? 2 : 1;          // buffers of dS^T
    static constexpr uint32_t kSlabs = HD / 64;
    static constexpr uint32_t kTile = kSlabs * SLAB;      // one [128][HD] bf16 tile
    static constexpr uint32_t oK = 0;
    static constexpr uint32_t oV = oK + kTile;
    static constexpr uint32_t oQ = oV + kTile;            // NS stages
    static constexpr uint32_t odO = oQ + NS * kTile;
    static constexpr uint32_t odS = odO + NS * kTile;     // [128 keys][128 queries] bf16, 2 slabs
    static constexpr uint32_t oLSE = odS + NdS * 2 * SLAB;
    static constexpr uint32_t oD = oLSE + NS * 128 * 4;
    static constexpr uint32_t oBar = oD + NS * 128 * 4;    // mbarriers (8 bytes each)
    static constexpr uint32_t oWork = oBar + 32 * 8;      // two slots of KeyWork, the answer of the scheduler
    static constexpr uint32_t oTile = oWork + 2 * 32 + 16;// query tile of the last four loads
    static constexpr uint32_t oMisc = oTile + 16;         // tmem base, abort flag
    static constexpr uint32_t kBytes = oMisc + 16;
    static_assert(kBytes <= 227 * 1024, "shared memory budget");
};

// barrier indices of the fused kernel; P exists once per 64-query half of a tile
enum { V2_KF = 0, V2_KE = 1, V2_VF = 2, V2_VE = 3, V2_QFULL = 4, V2_QEMPTY = 7, V2_S = 10, V2_DP = 11, V2_DQ = 12, V2_CLC = 13, V2_WF = 14,
       V2_WE = 16, V2_SLD = 18, V2_DPLD = 19, V2_DS = 20, V2_P = 21, V2_DQDONE = 23, V2_DQREL = 24, V2_NOBODY = 25 };

// One unit of work: a key tile of one head and the query tiles that it visits
struct KeyWork {
    int tile, bh, count; // tile = -1: there is no more work
    int first;           // the first query tile, or its place in the list
    const int *rows;     // query blocks of a mask with lists
    int pad[2];
};
static_assert(sizeof(KeyWork) == 32, "two slots in shared memory");


// ---------------------------------------------------------------------------------------
// dK and dV only: the key-stationary half of the path without atomics (dQ comes from the
// query-stationary kernel).  Without the dQ product dS^T never has to be in shared memory.
// Tensor memory: region A (128 columns) receives S^T and dP^T in turn; an exp / dS thread copies its
// 32 columns into registers with one load and releases the region at once.  Region B (128 columns)
// holds P^T and dS^T as bf16 pairs (per 64-query half: P^T in columns 64 h .. 64 h + 31, dS^T in
// 64 h + 32 .. 64 h + 63), from where dV += P^T dO and dK += dS^T Q take them as their A operand.
// Two MMA-issuing threads: A issues dP^T(k) (once S^T(k) has been copied out and dK(k-1) has left
// dS^T(k-1)) and S^T(k+1) (once dP^T(k) has been copied out); B issues dV(k) and dK(k).  The 32 KB that
// dS^T does not take in shared memory hold a third Q stage; Q, dO and the row statistics are released
// separately (dO after dV, Q after dK, LSE / D after the dS phase).
//
// A CTA takes the key tiles of CTAs that have not started yet, as in the fused kernel.  32 heads, n = 4096, d = 128, causal: 293 ->
// 267 us; 32 heads, n = 1024, d = 64, causal: 35.2 -> 33.1; 24 heads, n = 3000, d = 64, no mask: 205 -> 202; two terms, 16 heads,
// n = 2047, d = 128, causal: 65.8 -> 63.9.
//
// SPLIT: P and dS enter their products as two bf16 terms each, x = hi + lo up to 2^-17, for calls whose P and dS must not be
// rounded to one (bf16 storage whose length is no multiple of 8): six product units instead of four.  P^T then fills region B,
// per half 32 columns of leading terms and 32 of rests.  dS^T has 128 columns of its own at d = 64; at d = 128 there are none
// left, and it goes over P^T once dV(k) has consumed that, and P^T(k+1) over it once dK(k) has.  16 heads, n = 2047, causal:
// 64 us at d = 128, 52 us at d = 64; the FMA kernel, which forms dQ too, takes 2170 and 1605 us.
template <int HD> struct DkdvSmem {
    static constexpr uint32_t kSlabs = HD / 64;
    static constexpr uint32_t kTile = kSlabs * SLAB;        // one [128][HD] bf16 tile
    static constexpr uint32_t oK = 0;
    static constexpr uint32_t oV = oK + kTile;
    static constexpr uint32_t oQ = oV + kTile;              // 3 stages
    static constexpr uint32_t odO = oQ + 3 * kTile;         // 2 stages
    static constexpr uint32_t oLSE = odO + 2 * kTile;       // 2 stages x 128 floats
    static constexpr uint32_t oD = oLSE + 2 * 128 * 4;
    static constexpr uint32_t oBar = oD + 2 * 128 * 4;
    static constexpr uint32_t oWork = oBar + 40 * 8;        // two slots of KeyWork, the answer of the scheduler
    static constexpr uint32_t oMisc = oWork + 2 * 32 + 16;
    static constexpr uint32_t kBytes = oMisc + 16;
    static_assert(kBytes <= 227 * 1024, "shared memory budget");
};
enum { KD_KV = 0, KD_QFULL = 1, KD_QEMPTY = 4, KD_OFULL = 7, KD_OEMPTY = 9, KD_LFULL = 11, KD_S = 13, KD_DP = 14, KD_DONE = 15,
       KD_KVE = 16, KD_CLC = 17, KD_WF = 18, KD_LEMPTY = 20, KD_SLD = 22, KD_DPLD = 23, KD_DS = 24, KD_P = 25, KD_WE = 27, KD_COUNT = 29 };
constexpr int kThreadsDkdv = 512 + 128;   // 16 exp/dS warps, issuer A, TMA producer, issuer B, one idle warp

// The query tiles of a key tile: places first .. first + count - 1 of `rows` (a mask with lists) or the tiles themselves.  By a
// whole warp.
__device__ __forceinline__ void query_range(const BwdArgs &a, int jt, int bh, int lane, const int *&rows, int &first, int &count)
{
    const bool causal = mask_is_causal(a.mask_kind);
    if (!mask_is_block(a.mask_kind)) {
        first = causal ? jt : 0;
        count = (a.n + TQ - 1) / TQ - first;
        return;
    }
    // the lists ascend: what lies beyond n is at their end, and (block mask AND causal) what ends before the key tile begins at
    // their start
    const int sub = a.block / TQ, J = jt / (a.block / TK);
    const long mh = a.mask_heads == 1 ? 0 : bh;
    const int *cp = a.col_ptr + mh * 2 * a.nb + 2 * J;
    const int start = cp[0], raw = (cp[1] - start) * sub;
    rows = a.row_idx + mh * (long)a.nb * a.nb + start;
    int before = 0, within = 0;
    for (int e = lane; e < raw; e += 32) {
        const int it = rows[e / sub] * sub + e % sub;
        before += causal && it < jt;
        within += it * TQ < a.n;
    }
    first = __reduce_add_sync(0xffffffffu, before);
    count = max((int)__reduce_add_sync(0xffffffffu, within) - first, 0);
}

template <int HD, bool SPLIT>
__global__ void __launch_bounds__(kThreadsDkdv, 1)
tc_bwd_dkdv_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK_,
                   const __grid_constant__ CUtensorMap mV, const __grid_constant__ CUtensorMap mdO, const BwdArgs a)
{
    constexpr int kExpWarps = 16, kHalfWarps = 8;
    using L = DkdvSmem<HD>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::oBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(smem + L::oMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + L::oMisc + 4);
    const Abort ab{abort_flag, a.status};

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int n = a.n;
    const bool lists = mask_is_block(a.mask_kind), causal = mask_is_causal(a.mask_kind);
    const int sub = lists ? a.block / TQ : 1;
    volatile KeyWork *slots = reinterpret_cast<volatile KeyWork *>(smem + L::oWork);

    if ((smem_u32(smem) & 1023u) != 0) {
        chain_wait();
        if (tid == 0) atomicExch(a.status, 9u);
        return;
    }
    if (tid == 0) {
        *abort_flag = 0;
        for (int b = 0; b < KD_COUNT; ++b)   // WE: both issuers and the exp / dS warps
            mbar_init(&bars[b], b >= KD_WE ? 2 + kExpWarps : b >= KD_P ? kHalfWarps : b >= KD_LEMPTY ? kExpWarps : 1);
        fence_barrier_init();
        prefetch_tensormap(&mQ); prefetch_tensormap(&mK_); prefetch_tensormap(&mV); prefetch_tensormap(&mdO);
    }
    chain_wait();
    if (warp == 0) tmem_alloc(tmem_base_s, 512);
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    chain_release();
    const uint32_t tm = *tmem_base_s;
    const uint32_t T_A = tm, T_B = tm + 128, T_dV = tm + 256, T_dK = tm + 256 + HD;
    constexpr bool kShareB = SPLIT && HD == 128;   // P^T and dS^T in turn in region B
    const uint32_t T_dS = !SPLIT ? T_B + 32 : kShareB ? T_B : tm + 384;
    constexpr uint32_t HALF_ROWS = 64 * 128;   // byte offset of rows 64.. inside a [128][64] slab

    // the units of work of this CTA as the loading warp publishes them
    const UnitQueue<KeyWork, UnitIo<>> units{slots, &bars[KD_WF], &bars[KD_WE], &bars[KD_CLC], smem + L::oWork + 2 * sizeof(KeyWork), {ab}};
    auto query_tile = [&](const int *rows, int e) { return !lists ? e : sub == 1 ? rows[e] : rows[e / sub] * sub + e % sub; };

    // In every role k counts the query tiles of all units of work so far (a wait for what belongs to a tile before the first
    // returns at once); units follow one another as in the fused kernel.

    if (warp == 17) {
        // ------------------------------------------------------------ TMA producer, and the schedule
        int bx = blockIdx.x, by = blockIdx.y;
        int k = 0, nkv = 0;
        bool more = true;
        for (int t = 0; more; ++t) {
            const int jt = bx / a.group, bh = by * a.group + bx % a.group, j0 = jt * TK;
            int count, first;
            const int *rows = nullptr;
            query_range(a, jt, bh, lane, rows, first, count);
            auto load_unit = [&]() -> bool {   // false: there is no further unit, or the kernel is giving up
                volatile KeyWork *to = units.claim(t);
                if (!to) return false;
                to->tile = jt; to->bh = bh; to->count = count; to->first = first; to->rows = rows;
                units.publish(t);
                if (count > 0) {
                    if (!mbar_reload(&bars[KD_KV], &bars[KD_KVE], (nkv - 1) & 1, ab)) return false;   // S^T and dP^T of the unit before
                    ++nkv;
                    mbar_expect_tx(&bars[KD_KV], 2 * L::kTile);
#pragma unroll
                    for (uint32_t sl = 0; sl < L::kSlabs; ++sl) {
                        tma_load_3d(smem + L::oK + sl * SLAB, &mK_, &bars[KD_KV], sl * 64, j0, bh);
                        tma_load_3d(smem + L::oV + sl * SLAB, &mV, &bars[KD_KV], sl * 64, j0, bh);
                    }
                } else {
                    units.ask();
                }
                for (int e = 0; e < count; ++e, ++k) {
                    const int i0 = query_tile(rows, first + e) * TQ, sq = k % 3, s2 = k & 1;
                    const uint32_t nrows = min(TQ, a.ns - i0);
                    if (e == max(count - 2, 0)) units.ask();
                    if (k >= 3 && !mbar_reload(&bars[KD_QFULL + sq], &bars[KD_QEMPTY + sq], ((k / 3) - 1) & 1, ab)) return false;
                    mbar_expect_tx(&bars[KD_QFULL + sq], L::kTile);
#pragma unroll
                    for (uint32_t sl = 0; sl < L::kSlabs; ++sl)
                        tma_load_3d(smem + L::oQ + sq * L::kTile + sl * SLAB, &mQ, &bars[KD_QFULL + sq], sl * 64, i0, bh);
                    if (k >= 2 && !mbar_reload(&bars[KD_LFULL + s2], &bars[KD_LEMPTY + s2], ((k >> 1) - 1) & 1, ab)) return false;
                    mbar_expect_tx(&bars[KD_LFULL + s2], 2 * nrows * 4);
                    bulk_load_1d(smem + L::oLSE + s2 * 512, a.nLSE2 + (size_t)bh * a.ns + i0, nrows * 4, &bars[KD_LFULL + s2]);
                    bulk_load_1d(smem + L::oD + s2 * 512, a.nDs + (size_t)bh * a.ns + i0, nrows * 4, &bars[KD_LFULL + s2]);
                    if (k >= 2 && !mbar_reload(&bars[KD_OFULL + s2], &bars[KD_OEMPTY + s2], ((k >> 1) - 1) & 1, ab)) return false;
                    mbar_expect_tx(&bars[KD_OFULL + s2], L::kTile);
#pragma unroll
                    for (uint32_t sl = 0; sl < L::kSlabs; ++sl)
                        tma_load_3d(smem + L::odO + s2 * L::kTile + sl * SLAB, &mdO, &bars[KD_OFULL + s2], sl * 64, i0, bh);
                }
                return units.next(t, bx, by);
            };
            if (lane == 0) more = load_unit();
            __syncwarp();
            more = __shfl_sync(0xffffffffu, (int)more, 0) != 0;
            bx = __shfl_sync(0xffffffffu, bx, 0);
            by = __shfl_sync(0xffffffffu, by, 0);
        }
    } else if (warp == 16) {
        // ------------------------------------------------------------ MMA issuer A: the products into region A
        if (lane == 0) {
            constexpr uint32_t idesc_s = idesc_bf16(128, 128, 0, 0);       // S^T, dP^T
            const uint32_t kK = desc_lo_kmajor(smem_u32(smem + L::oK)), kV = desc_lo_kmajor(smem_u32(smem + L::oV));
            constexpr uint32_t kSlab = SLAB >> 4;
            int k = 0, nkv = 0;
            for (int t = 0; units.take_alone(t); ++t) {
                const int end = k + slots[t & 1].count;
                mbar_arrive(&bars[KD_WE + (t & 1)]);
                if (k == end) continue;
                mbar_wait(&bars[KD_KV], nkv & 1, ab);
                ++nkv;
                for (; k < end; ++k) {
                    // S^T(k) as soon as dP^T(k-1) has been copied out
                    mbar_wait(&bars[KD_QFULL + k % 3], (k / 3) & 1, ab);
                    mbar_wait(&bars[KD_DPLD], (k - 1) & 1, ab);
                    tcgen05_fence_after();
                    const uint32_t kQ = desc_lo_kmajor(smem_u32(smem + L::oQ + (k % 3) * L::kTile));
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        const uint32_t off = (kk / 4) * kSlab + (kk % 4) * 2;
                        mma_ss_lo(T_A, kK + off, kQ + off, idesc_s, kk > 0);
                    }
                    mma_commit(&bars[KD_S]);
                    // dP^T(k) into region A: S^T(k) copied out, dO(k) landed, and -- because the exp / dS warps store
                    // dS^T(k) as soon as they have seen dP^T(k) -- the dK product of tile k-1 done with dS^T(k-1)
                    mbar_wait(&bars[KD_OFULL + (k & 1)], (k >> 1) & 1, ab);
                    if (k > 0) mbar_wait(&bars[KD_QEMPTY + (k - 1) % 3], ((k - 1) / 3) & 1, ab);
                    mbar_wait(&bars[KD_SLD], k & 1, ab);
                    tcgen05_fence_after();
                    const uint32_t kdO = desc_lo_kmajor(smem_u32(smem + L::odO + (k & 1) * L::kTile));
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        const uint32_t off = (kk / 4) * kSlab + (kk % 4) * 2;
                        mma_ss_lo(T_A, kV + off, kdO + off, idesc_s, kk > 0);
                    }
                    mma_commit(&bars[KD_DP]);
                }
                mma_commit(&bars[KD_KVE]);
            }
        }
    } else if (warp == 18) {
        // ------------------------------------------------------------ MMA issuer B: dV += P^T dO, dK += dS^T Q
        if (lane == 0) {
            constexpr uint32_t idesc_dv = idesc_bf16(128, HD, 0, 1);       // A in tensor memory, B MN-major
            constexpr uint32_t kHalf = HALF_ROWS >> 4;
            int k = 0;
            for (int t = 0; units.take_alone(t); ++t) {
              const int begin = k, end = k + slots[t & 1].count;
              mbar_arrive(&bars[KD_WE + (t & 1)]);
              if (k == end) continue;
              // the first dV of a unit overwrites the accumulator of the unit before: both halves' warps have read it
              mbar_wait(&bars[KD_P + 1], k & 1, ab);
              for (; k < end; ++k) {
                const uint32_t mdO_ = desc_lo_mnmajor(smem_u32(smem + L::odO + (k & 1) * L::kTile), SLAB);
                const uint32_t mQ_ = desc_lo_mnmajor(smem_u32(smem + L::oQ + (k % 3) * L::kTile), SLAB);
                // P^T of one term is handed over by warps that have seen dP^T(k), so dO(k) is there; dS^T(k) follows both loads
                if constexpr (SPLIT) mbar_wait(&bars[KD_OFULL + (k & 1)], (k >> 1) & 1, ab);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    mbar_wait(&bars[KD_P + h], k & 1, ab);
                    tcgen05_fence_after();
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        mma_ts_lo(T_dV, T_B + 64 * h + kk * 8, mdO_ + h * kHalf + kk * 128, idesc_dv, (k > begin) || (h > 0) || (kk > 0));
                    if constexpr (SPLIT) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_ts_lo(T_dV, T_B + 64 * h + 32 + kk * 8, mdO_ + h * kHalf + kk * 128, idesc_dv, 1);
                    }
                }
                mma_commit(&bars[KD_OEMPTY + (k & 1)]);
                mbar_wait(&bars[KD_DS], k & 1, ab);
                tcgen05_fence_after();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        mma_ts_lo(T_dK, T_dS + 64 * h + kk * 8, mQ_ + h * kHalf + kk * 128, idesc_dv, (k > begin) || (h > 0) || (kk > 0));
                    if constexpr (SPLIT) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_ts_lo(T_dK, T_dS + 64 * h + 32 + kk * 8, mQ_ + h * kHalf + kk * 128, idesc_dv, 1);
                    }
                }
                mma_commit(&bars[KD_QEMPTY + k % 3]);
              }
              mma_commit(&bars[KD_DONE]);
            }
        }
    } else if (warp < 16) {
        // ------------------------------------------------------------ warpgroup 2h + qq owns queries 64 h + 32 qq .. + 31
        const int h = warp / 8, qq = (warp / 4) & 1;
        const int row = (warp % 4) * 32 + lane;        // tensor-memory lane = key row inside the tile
        const uint32_t lane_addr = (uint32_t)((warp % 4) * 32) << 16;
        const float sl2 = a.sl2;
        const bool wide = (((uintptr_t)a.dK | (uintptr_t)a.dV) & 31) == 0;
        const uint32_t c0 = h * 64 + qq * 32;          // this thread's first column of S^T / dP^T in region A
        const uint32_t cP = h * 64 + qq * 16;          // of its bf16 pairs of P^T in region B; dS^T 32 columns further
        int k = 0, done = 0;
        for (int t = 0; units.take(t); ++t) {
          const int jt = slots[t & 1].tile, bh = slots[t & 1].bh, count = slots[t & 1].count, begin = k - slots[t & 1].first, end = k + count;
          const int *rows = slots[t & 1].rows;
          int it0 = slots[t & 1].first;
          warp_arrive(&bars[KD_WE + (t & 1)], lane);
          const int j0 = jt * TK, jg = j0 + row;
          for (; k < end; ++k) {
            const int it = !lists ? it0++ : query_tile(rows, k - begin);
            const int s2 = k & 1, i0 = it * TQ;
            const float4 *sNL = reinterpret_cast<const float4 *>(smem + L::oLSE + s2 * 512 + h * 256 + qq * 128);
            const float4 *sDs = reinterpret_cast<const float4 *>(smem + L::oD + s2 * 512 + h * 256 + qq * 128);
            const bool diag = causal && it == jt;
            const int ig0 = i0 + h * 64 + qq * 32;
            // a mask finer than the tile: the keep bits of this thread's key row and its 32 query columns
            uint32_t kw = 0xffffffffu;
            if (a.fine.mode) kw = (ig0 < n && jg < n) ? fine_word(a.fine, a.mask_heads, bh, false, jg, ig0) : 0u;
            const bool masked = diag || i0 + TQ > n || j0 + TK > n || a.fine.mode != 0;
            mbar_wait(&bars[KD_S], k & 1, ab);
            tcgen05_fence_after();
            if constexpr (SPLIT) {
                float p[32];   // P stays in fp32: dS is formed from it
                {
                    uint32_t sv[32];
                    tmem_ld32(T_A + lane_addr + c0, sv);
                    tmem_wait_ld();
                    tcgen05_fence_before();
                    warp_arrive(&bars[KD_SLD], lane);   // region A may take dP^T
                    mbar_wait(&bars[KD_LFULL + s2], (k >> 1) & 1, ab);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 nl = sNL[q];
                        p_pair(sv[q * 4 + 0], sv[q * 4 + 1], sl2, nl.x, nl.y, p[q * 4 + 0], p[q * 4 + 1]);
                        p_pair(sv[q * 4 + 2], sv[q * 4 + 3], sl2, nl.z, nl.w, p[q * 4 + 2], p[q * 4 + 3]);
                    }
                    if (masked) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            const int ig = ig0 + e;
                            p[e] = ig < n && jg < n && (!diag || jg <= ig) && ((kw >> e) & 1u) ? p[e] : 0.f;
                        }
                    }
                }
                // P^T(k) over P^T(k-1), which dV(k-1) has consumed, or (kShareB) over dS^T(k-1), which dK(k-1) has.  Either
                // completion is the newest its barrier can have: the next one of that stage needs P^T(k)
                if (k > 0) {
                    if (kShareB) mbar_wait(&bars[KD_QEMPTY + (k - 1) % 3], ((k - 1) / 3) & 1, ab);
                    else mbar_wait(&bars[KD_OEMPTY + ((k - 1) & 1)], ((k - 1) >> 1) & 1, ab);
                    tcgen05_fence_after();
                }
                {
                    uint32_t hi[16], lo[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        hi[e] = pack_bf16(p[2 * e], p[2 * e + 1]);
                        lo[e] = pack_bf16_rest(p[2 * e], p[2 * e + 1], hi[e]);
                    }
                    tmem_st16(T_B + lane_addr + cP, hi);
                    tmem_st16(T_B + lane_addr + cP + 32, lo);
                    tmem_wait_st();
                    tcgen05_fence_before();
                    warp_arrive(&bars[KD_P + h], lane);
                }
                mbar_wait(&bars[KD_DP], k & 1, ab);
                tcgen05_fence_after();
                uint32_t hi[16], lo[16];
#pragma unroll
                for (int part = 0; part < 2; ++part) {   // 16 query columns at a time
                    uint32_t dv[16];
                    tmem_ld16(T_A + lane_addr + c0 + part * 16, dv);
                    tmem_wait_ld();
                    if (part == 1) {
                        tcgen05_fence_before();
                        warp_arrive(&bars[KD_DPLD], lane);   // region A may take the next S^T
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 dsc = sDs[part * 4 + q];
                        const float *p4 = &p[part * 16 + q * 4];
                        float d0, d1, d2, d3;
                        mul_pair(fma_pair(dv[q * 4 + 0], dv[q * 4 + 1], a.scale, dsc.x, dsc.y), __float_as_uint(p4[0]), __float_as_uint(p4[1]), d0, d1);
                        mul_pair(fma_pair(dv[q * 4 + 2], dv[q * 4 + 3], a.scale, dsc.z, dsc.w), __float_as_uint(p4[2]), __float_as_uint(p4[3]), d2, d3);
                        if (masked) {   // stale tail entries of the row vectors may be anything: select, do not multiply
                            d0 = p4[0] != 0.f ? d0 : 0.f; d1 = p4[1] != 0.f ? d1 : 0.f;
                            d2 = p4[2] != 0.f ? d2 : 0.f; d3 = p4[3] != 0.f ? d3 : 0.f;
                        }
                        const int to = part * 8 + q * 2;
                        hi[to] = pack_bf16(d0, d1);
                        hi[to + 1] = pack_bf16(d2, d3);
                        lo[to] = pack_bf16_rest(d0, d1, hi[to]);
                        lo[to + 1] = pack_bf16_rest(d2, d3, hi[to + 1]);
                    }
                }
                // dS^T(k): over dS^T(k-1), whose dK product the issuer of dP^T(k) has seen complete, or (kShareB) over P^T(k)
                if (kShareB) {
                    mbar_wait(&bars[KD_OEMPTY + s2], (k >> 1) & 1, ab);   // dV(k); the stage's next completion needs P^T(k+2)
                    tcgen05_fence_after();
                }
                tmem_st16(T_dS + lane_addr + cP, hi);
                tmem_st16(T_dS + lane_addr + cP + 32, lo);
                tmem_wait_st();
            } else {
                uint32_t ppack[16];
                {
                    uint32_t sv[32];
                    tmem_ld32(T_A + lane_addr + c0, sv);
                    tmem_wait_ld();
                    tcgen05_fence_before();
                    warp_arrive(&bars[KD_SLD], lane);   // region A may take dP^T
                    mbar_wait(&bars[KD_LFULL + s2], (k >> 1) & 1, ab);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 nl = sNL[q];
                        float p[4];
                        p_pair(sv[q * 4 + 0], sv[q * 4 + 1], sl2, nl.x, nl.y, p[0], p[1]);
                        p_pair(sv[q * 4 + 2], sv[q * 4 + 3], sl2, nl.z, nl.w, p[2], p[3]);
                        if (masked) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int ig = ig0 + q * 4 + e;
                                const bool ok = ig < n && jg < n && (!diag || jg <= ig) && ((kw >> (q * 4 + e)) & 1u);
                                p[e] = ok ? p[e] : 0.f;
                            }
                        }
                        ppack[q * 2 + 0] = pack_bf16(p[0], p[1]);
                        ppack[q * 2 + 1] = pack_bf16(p[2], p[3]);
                    }
                }
                // P^T(k) over P^T(k-1): the dV product of the previous tile must have consumed it.  Stored ahead of the wait for dP^T
                if (k > 0) {
                    mbar_wait(&bars[KD_OEMPTY + ((k - 1) & 1)], ((k - 1) >> 1) & 1, ab);
                    tcgen05_fence_after();
                }
                tmem_st16(T_B + lane_addr + cP, ppack);
                mbar_wait(&bars[KD_DP], k & 1, ab);
                tcgen05_fence_after();
                uint32_t dv[32];
                tmem_ld32(T_A + lane_addr + c0, dv);
                tmem_wait_ld();
                tcgen05_fence_before();
                warp_arrive(&bars[KD_DPLD], lane);   // region A may take the next S^T
                tmem_wait_st();
                tcgen05_fence_before();
                warp_arrive(&bars[KD_P + h], lane);
                {
                    uint32_t dpack[16];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 dsc = sDs[q];
                        // a masked entry has p = 0 and a finite dP, so its dS is an exact zero
                        const uint32_t pa = ppack[q * 2], pb = ppack[q * 2 + 1];
                        float d0, d1, d2, d3;
                        ds_pair(pa, dv[q * 4 + 0], dv[q * 4 + 1], a.scale, dsc.x, dsc.y, d0, d1);
                        ds_pair(pb, dv[q * 4 + 2], dv[q * 4 + 3], a.scale, dsc.z, dsc.w, d2, d3);
                        if (masked) {   // stale tail entries of the row vectors may be anything: select, do not multiply
                            d0 = (pa & 0xffffu) != 0u ? d0 : 0.f; d1 = (pa >> 16) != 0u ? d1 : 0.f;
                            d2 = (pb & 0xffffu) != 0u ? d2 : 0.f; d3 = (pb >> 16) != 0u ? d3 : 0.f;
                        }
                        dpack[q * 2 + 0] = pack_bf16(d0, d1);
                        dpack[q * 2 + 1] = pack_bf16(d2, d3);
                    }
                    // dS^T(k) over dS^T(k-1): the issuer of dP^T(k) has seen the dK product of tile k-1 complete
                    tmem_st16(T_dS + lane_addr + cP, dpack);
                    tmem_wait_st();
                }
            }
            tcgen05_fence_before();
            warp_arrive(&bars[KD_DS], lane);
            warp_arrive(&bars[KD_LEMPTY + s2], lane);
          }
          // ---------------------------------------------------------- epilogue: dV_j, dK_j (32 columns per warpgroup)
          if (count > 0) {
              mbar_wait(&bars[KD_DONE], done & 1, ab);
              ++done;
              tcgen05_fence_after();
          }
          const int cq = (warp / 4) * 32;       // d = 64: the upper two warpgroups have no columns
          if (cq < HD) {
              const int jc = jg < n ? jg : 0;
#pragma unroll
              for (int which = 0; which < 2; ++which) {
                  __nv_bfloat16 *po = (which == 0 ? a.dV : a.dK) + ((size_t)bh * n + jc) * HD + cq;
#pragma unroll
                  for (int e0 = 0; e0 < 32; e0 += 16) {
                      uint32_t v[16], y[8];
                      tmem_ld16((which == 0 ? T_dV : T_dK) + lane_addr + cq + e0, v);
                      tmem_wait_ld();
#pragma unroll
                      for (int u = 0; u < 8; ++u)   // without a query tile nothing has been accumulated
                          y[u] = count > 0 ? pack_bf16(__uint_as_float(v[2 * u]), __uint_as_float(v[2 * u + 1])) : 0u;
                      if (jg < n) store32(po + e0, y, wide);
                  }
              }
              tcgen05_fence_before();
          }
        }
    }
    tmem_leave(tm, 512, warp, ab);
}

// ---------------------------------------------------------------------------------------
// The fused kernel.  The exp / dS warps handle a 128-query tile as two halves of 64 queries (P^T is handed
// over per half, everything else per tile).  Warps 0-15: exp / dS (warpgroups 2h and 2h+1 own the two 32-query quarters of half
// h, so each scheduler has four such warps to hide tensor-memory and MUFU latency); warps 16-23:
// reducers, which do nothing but move finished dQ^T tiles from tensor memory into the fp32
// accumulator, so that the red.global.add queue stalls them and not the warps on the tile loop;
// warp 24 lane 0 issues the products into region A (S^T, dP^T), warp 26 lane 0 the products that read
// P^T and dS^T (dV, dQ^T, dK), warp 25 lane 0 every TMA load; warp 27 only completes that warpgroup.
//
// Tensor memory: region A (128 columns) receives S^T and dP^T in turn, region B (128 columns) holds
// P^T (bf16 pairs, 32 columns per half) and then dQ^T.  An exp / dS thread copies its 32 columns of
// S^T (and later of dP^T) into registers at once and releases region A right away, so the next
// product into A runs while the exponentials (or the dS arithmetic) are still being computed:
//
//   issuer A:  dP^T(k) -> A  (once S^T(k) has been copied out)  |  S^T(k+1) -> A  (once dP^T(k) has been)
//   issuer B:  dV += P^T(k) dO  (P^T(k) written in B)  |  dK += dS^T(k) Q, dQ^T(k) -> B  (dS^T(k) in shared
//              memory, the reducers done with dQ^T(k-1)); dK goes first at d = 128, where it releases one of two
//              Q / dO stages, dQ^T at d = 64
//
// The exp / dS warps keep P only as the bf16 pairs they hand to the dV product, and form dS from
// those, two entries an instruction (fma.rn.f32x2: the roundings of the scalar forms; -scale D comes from the pre-pass).
// Registers are traded between the warpgroups after launch (setmaxnreg).
//
// A CTA stays on its SM and takes the block indices of CTAs that have not started yet (cluster launch control); the loading
// warp publishes each key tile in one of two slots, and K_j, V_j, the first Q and dO and S^T of the next key tile come while dK
// and dV of this one are written out.  With a CTA per key tile 8.7 us a CTA passed outside its tiles.  What an issuing thread
// does between its products counts twice: testing for the first tile of a unit inside the loop, instead of ahead of it, cost
// 3.5 % at d = 128 and 13 % at d = 64; barriers merged to save it two waits a tile made no difference at d = 128 and cost 7 %
// at d = 64 (dV then competes with S^T and dP^T for the pipe).
// Before and now, kernel alone: 32 heads, n = 8192, d = 128, causal 1347 -> 1291 us; the same, d = 64, no mask 1897 -> 1664; 64
// heads, n = 2048, d = 64 272 -> 238; window of 512 keys, 16 heads, n = 4096, d = 128 109 -> 83 (half of it from the keep words,
// applied to the packed pairs and only in warps that drop something); blocks of 64, 10 %, 16 heads, n = 8192, d = 64 559 -> 449.
template <int N> __device__ __forceinline__ void setmaxnreg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void setmaxnreg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
constexpr int kThreadsFused = 512 + 256 + 128;  // 16 exp/dS warps, 8 reducer warps, two issuer warps, TMA producer warp, 1 idle warp
// 72 registers everywhere at launch (896 x 72 = 64,512).  The reducers give up 24 each and work through their
// 64 columns in two steps, the issuer's warpgroup gives up 16, the exp / dS warps take 16:
// 512 x 88 + 256 x 48 + 128 x 56 = 64,512.
struct FusedRegs {
    static constexpr int kExp = 88, kReduce = 48, kIssue = 56;
};
template <int HD, bool FINE>
__global__ void __launch_bounds__(kThreadsFused, 1)
tc_bwd_fused_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK_,
                 const __grid_constant__ CUtensorMap mV, const __grid_constant__ CUtensorMap mdO, const BwdArgs a)
{
    // d = 64: the dQ^T product needs M = 128, so the K tile's second 64-wide slab of M is an all-zero slab
    using L = BwdSmem<HD>;
    constexpr uint32_t oZero = (L::kBytes + 1023u) & ~1023u;
    constexpr int kHalfWarps = 8;     // exp / dS warps per half
    constexpr int kReduceWarps = HD / 32;   // reducer warps per half that have rows of dQ^T (d = 64: lanes 64..127 of the padded product hold zeros)
    constexpr int NS = L::NS;
    auto stage_of = [](int kt) { return NS == 2 ? kt & 1 : kt % 3; };
    auto phase_of = [](int kt) { return NS == 2 ? (kt >> 1) & 1 : (kt / 3) & 1; };
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::oBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(smem + L::oMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + L::oMisc + 4);
    volatile KeyWork *slots = reinterpret_cast<volatile KeyWork *>(smem + L::oWork);
    const Abort ab{abort_flag, a.status};

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int n = a.n;
    const bool lists = mask_is_block(a.mask_kind), causal = mask_is_causal(a.mask_kind);
    const int sub = lists ? a.block / TQ : 1;

    if ((smem_u32(smem) & 1023u) != 0) {
        chain_wait();
        if (tid == 0) atomicExch(a.status, 9u);
        return;
    }
    if (tid == 0) {
        *abort_flag = 0;
        for (int b = 0; b < V2_SLD; ++b) mbar_init(&bars[b], b >= V2_WE ? 2 + 2 * kHalfWarps + 2 * kReduceWarps : 1);   // WE: every reader of a slot
        mbar_init(&bars[V2_SLD], 2 * kHalfWarps);
        mbar_init(&bars[V2_DPLD], 2 * kHalfWarps);
        mbar_init(&bars[V2_DS], 2 * kHalfWarps);
        mbar_init(&bars[V2_P], kHalfWarps);
        mbar_init(&bars[V2_P + 1], kHalfWarps);
        mbar_init(&bars[V2_DQDONE], 2 * kReduceWarps);
        mbar_init(&bars[V2_DQREL], 2 * kReduceWarps);
        mbar_init(&bars[V2_NOBODY], 1);   // takes the release of a stage whose load has not landed
        fence_barrier_init();
        *reinterpret_cast<int4 *>(smem + L::oTile) = make_int4(0, 0, 0, 0);   // whatever becomes of the loads, a tile that exists
        prefetch_tensormap(&mQ); prefetch_tensormap(&mK_); prefetch_tensormap(&mV); prefetch_tensormap(&mdO);
    }
    if (HD == 64) {
        for (uint32_t i = tid; i < SLAB / 16; i += kThreadsFused) reinterpret_cast<uint4 *>(smem + oZero)[i] = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
    }
    chain_wait();
    if (warp == 0) tmem_alloc(tmem_base_s, 512);
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    chain_release();
    const uint32_t tm = *tmem_base_s;
    const uint32_t T_A = tm, T_B = tm + 128, T_dV = tm + 256, T_dK = tm + 256 + HD;
    // d = 64 leaves 128 columns free: dP^T gets a region of its own there, so that S^T(k+1) does not wait for dP^T(k)
    // to be copied out of region A and dP^T(k+1) does not wait for S^T(k+1)
    constexpr bool kSplitA = HD == 64;
    const uint32_t T_A2 = kSplitA ? tm + 384 : T_A;
    constexpr uint32_t HALF_ROWS = 64 * 128;   // byte offset of rows 64.. inside a [128][64] slab

    // the units of work of this CTA as the loading warp publishes them; one stays in its slot until both issuers, the exp / dS warps
    // and the reducers have arrived on WE
    const UnitQueue<KeyWork, UnitIo<>> units{slots, &bars[V2_WF], &bars[V2_WE], &bars[V2_CLC], smem + L::oWork + 2 * sizeof(KeyWork), {ab}};
    auto query_tile = [&](const int *rows, int e) { return !lists ? e : sub == 1 ? rows[e] : rows[e / sub] * sub + e % sub; };
    // query tile of the kt-th load, for the exp / dS warps; the fourth load after it follows dK(kt + 1) at the latest, by when they
    // are past it
    volatile int *tiles = reinterpret_cast<volatile int *>(smem + L::oTile);

    // In every role kt counts the query tiles of all units of work so far (a wait for what belongs to tile -1 returns at once: a
    // new barrier counts as complete in the phase before its first): the barriers run on from one unit to the next, and
    // what the next one needs first is loaded and formed while dK and dV of this one are written out.
    if (warp >= 24) {
        setmaxnreg_dec<FusedRegs::kIssue>();
        if (warp == 25) {
            // ------------------------------------------------------------ TMA producer, and the schedule
            // launch order: heads in groups of `a.group`, inside a group key tile major -- with a causal
            // mask the CTAs of a group then start longest first, which evens out the tail of the grid
            int bx = blockIdx.x, by = blockIdx.y;
            int kt = 0, nkv = 0;   // query tiles and key tiles loaded so far
            bool more = true;
            for (int t = 0; more; ++t) {
                const int jt = bx / a.group, bh = by * a.group + bx % a.group, j0 = jt * TK;
                int count, first;
                const int *rows = nullptr;
                query_range(a, jt, bh, lane, rows, first, count);
                auto load_unit = [&]() -> bool {   // false: there is no further unit, or the kernel is giving up
                    volatile KeyWork *to = units.claim(t);
                    if (!to) return false;
                    int it = count > 0 ? query_tile(rows, first) : 0;
                    to->tile = jt; to->bh = bh; to->count = count; to->first = first; to->rows = rows;
                    units.publish(t);
                    // The loop is left by its condition, and what releases a stage is chosen by its barrier: how this thread and the
                    // issuing ones go on decides in which order the products queue, and other forms of the same checks (returns,
                    // two waits a stage, branches around commits) took 1,680 to 2,090 us for 1,660 at 32 heads, n = 8192, d = 64.
                    bool go = true;
                    for (int k = 0; k < count && go; ++k, ++kt) {
                        const int s = stage_of(kt), here = it, i0 = it * TQ;
                        if (k + 1 < count) it = query_tile(rows, first + k + 1);
                        if (k == max(count - 2, 0)) units.ask();
                        if (k == 0) {
                            if (!mbar_wait(&bars[V2_VE], (nkv - 1) & 1, ab)) return false;   // dP^T of the unit before
                            mbar_expect_tx(&bars[V2_VF], L::kTile);
#pragma unroll
                            for (uint32_t sl = 0; sl < L::kSlabs; ++sl)
                                tma_load_3d(smem + L::oV + sl * SLAB, &mV, &bars[V2_VF], sl * 64, j0, bh);
                        }
                        if (kt < NS || (go = mbar_wait(&bars[V2_QEMPTY + s], phase_of(kt - NS), ab))) {   // last read by dK of tile kt - NS
                            // negative: position drops some of its entries (causal, or beyond n)
                            tiles[kt & 3] = (causal && here == jt) || i0 + TQ > n || j0 + TK > n ? here - (1 << 30) : here;
                            const uint32_t nrows = min(TQ, a.ns - i0);
                            uint64_t *bar = &bars[V2_QFULL + s];
                            mbar_expect_tx(bar, 2 * L::kTile + 2 * nrows * 4);
#pragma unroll
                            for (uint32_t sl = 0; sl < L::kSlabs; ++sl) {
                                tma_load_3d(smem + L::oQ + s * L::kTile + sl * SLAB, &mQ, bar, sl * 64, i0, bh);
                                tma_load_3d(smem + L::odO + s * L::kTile + sl * SLAB, &mdO, bar, sl * 64, i0, bh);
                            }
                            bulk_load_1d(smem + L::oLSE + s * 512, a.nLSE2 + (size_t)bh * a.ns + i0, nrows * 4, bar);
                            bulk_load_1d(smem + L::oD + s * 512, a.nDs + (size_t)bh * a.ns + i0, nrows * 4, bar);
                        }
                        if (k == 0) {
                            if (!mbar_wait(&bars[V2_KE], (nkv - 1) & 1, ab)) return false;   // dQ^T of the unit before
                            mbar_expect_tx(&bars[V2_KF], L::kTile);
#pragma unroll
                            for (uint32_t sl = 0; sl < L::kSlabs; ++sl)
                                tma_load_3d(smem + L::oK + sl * SLAB, &mK_, &bars[V2_KF], sl * 64, j0, bh);
                        }
                    }
                    if (!go) return false;
                    if (count > 0) ++nkv;
                    else units.ask();
                    return units.next(t, bx, by);
                };
                if (lane == 0) more = load_unit();
                __syncwarp();
                more = __shfl_sync(0xffffffffu, (int)more, 0) != 0;
                bx = __shfl_sync(0xffffffffu, bx, 0);
                by = __shfl_sync(0xffffffffu, by, 0);
            }
        } else if (warp == 24 && lane == 0) {
            // ------------------------------------------------------------ MMA issuer A: the products into region A (S^T, dP^T)
            constexpr uint32_t idesc_s = idesc_bf16(128, 128, 0, 0);
            constexpr uint32_t kSlab = SLAB >> 4;   // low descriptor words (tc_common.cuh): per-step offsets are added as (bytes >> 4)
            int kt = 0, nkv = 0;
            for (int t = 0; units.take_alone(t); ++t) {
                const int count = slots[t & 1].count;
                mbar_arrive(&bars[V2_WE + (t & 1)]);
                const uint32_t kK = desc_lo_kmajor(smem_u32(smem + L::oK)), kV = desc_lo_kmajor(smem_u32(smem + L::oV));
                bool landed = count > 0;
                if (landed) {
                    landed = mbar_wait(&bars[V2_VF], nkv & 1, ab);
                    mbar_wait(&bars[V2_KF], nkv & 1, ab);
                }
                for (int k = 0; k < count; ++k, ++kt) {
                    const int s = stage_of(kt);
                    // S^T = K_j Q_i^T once region A is free: dP^T of the tile before (d = 64: its S^T) has been copied out
                    mbar_wait(&bars[kSplitA ? V2_SLD : V2_DPLD], (kt - 1) & 1, ab);
                    mbar_wait(&bars[V2_QFULL + s], phase_of(kt), ab);
                    tcgen05_fence_after();
                    const uint32_t kQ = desc_lo_kmajor(smem_u32(smem + L::oQ + s * L::kTile));
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        const uint32_t off = (kk / 4) * kSlab + (kk % 4) * 2;
                        mma_ss_lo(T_A, kK + off, kQ + off, idesc_s, kk > 0);
                    }
                    mma_commit(&bars[V2_S]);
                    // dP^T = V_j dO_i^T once every exp / dS warp holds its part of S^T in registers (d = 64: of the dP^T before)
                    if (!kSplitA) mbar_wait(&bars[V2_SLD], kt & 1, ab);
                    else mbar_wait(&bars[V2_DPLD], (kt - 1) & 1, ab);
                    tcgen05_fence_after();
                    const uint32_t kdO = desc_lo_kmajor(smem_u32(smem + L::odO + s * L::kTile));
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        const uint32_t off = (kk / 4) * kSlab + (kk % 4) * 2;
                        mma_ss_lo(T_A2, kV + off, kdO + off, idesc_s, kk > 0);
                    }
                    mma_commit(&bars[V2_DP]);
                }
                if (landed) {
                    mma_commit(&bars[V2_VE]);
                    ++nkv;
                }
            }
        } else if (warp == 26 && lane == 0) {
            // ------------------------------------------------------------ MMA issuer B: the products that read P^T and dS^T
            // (dV, dQ^T into region B, dK).  Two issuing threads, because a thread that waits on a barrier or commits
            // cannot keep the short queue of the tensor pipe filled; everything that orders A's products against B's
            // goes through the exp / dS warps' barriers.
            constexpr uint32_t idesc_dv = idesc_bf16(128, HD, 0, 1);       // dV (A tmem), dK (A K-major smem)
            constexpr uint32_t idesc_dq = idesc_bf16(128, 128, 1, 1);      // dQ^T
            const uint32_t kdS = desc_lo_kmajor(smem_u32(smem + L::odS)), mdS = desc_lo_mnmajor(smem_u32(smem + L::odS), SLAB);
            constexpr uint32_t kHalf = HALF_ROWS >> 4, kSlab = SLAB >> 4;
            int kt = 0, nkv = 0;
            for (int t = 0; units.take_alone(t); ++t) {
                const int count = slots[t & 1].count;
                mbar_arrive(&bars[V2_WE + (t & 1)]);
                const uint32_t mK = desc_lo_mnmajor(smem_u32(smem + L::oK), HD == 64 ? oZero - L::oK : SLAB);
                if (count > 0) {
                    if (!mbar_wait(&bars[V2_KF], nkv & 1, ab)) break;
                    // the first dV of a unit overwrites the accumulator of the unit before: both halves' warps have read it
                    mbar_wait(&bars[V2_P + 1], kt & 1, ab);
                }
                for (int k = 0; k < count; ++k, ++kt) {
                    const int s = stage_of(kt);
                    const uint32_t mdO_ = desc_lo_mnmajor(smem_u32(smem + L::odO + s * L::kTile), SLAB);
                    const uint32_t mQ_ = desc_lo_mnmajor(smem_u32(smem + L::oQ + s * L::kTile), SLAB);
                    const bool landed = mbar_wait(&bars[V2_QFULL + s], phase_of(kt), ab);
                    // dV += P_h^T dO_h, P_h^T in columns 64 h .. 64 h + 31 of region B
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        mbar_wait(&bars[V2_P + h], kt & 1, ab);
                        tcgen05_fence_after();
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_ts_lo(T_dV, T_B + 64 * h + kk * 8, mdO_ + h * kHalf + kk * 128, idesc_dv, (k > 0) || (h > 0) || (kk > 0));
                    }
                    // dQ^T = K_j^T dS^T into region B (this thread's products execute in issue order, so dV has consumed P^T by
                    // then) and dK += dS^T Q_i.  d = 128: dK first, its completion releases the Q / dO stage, and with two stages
                    // the load of the tile after next is what the next S^T ends up waiting for.  d = 64: three stages and a
                    // second buffer of dS^T, so dQ^T, which P^T of the next tile waits for, goes first
                    // (n = 8192, 32 heads, no mask: 1762 -> 1691 us).
                    // That the reducers have read all of the previous dQ^T is waited for ahead of dS, which the tile is waiting for
                    mbar_wait(&bars[V2_DQDONE], (kt - 1) & 1, ab);
                    mbar_wait(&bars[V2_DS], kt & 1, ab);
                    tcgen05_fence_after();
                    const uint32_t ds = L::NdS == 2 ? (kt & 1) * (2 * SLAB >> 4) : 0;
                    auto issue_dK = [&] {
#pragma unroll
                        for (int kk = 0; kk < TQ / 16; ++kk)
                            mma_ss_lo(T_dK, kdS + ds + (kk / 4) * kSlab + (kk % 4) * 2, mQ_ + kk * 128, idesc_dv, (k > 0) || (kk > 0));
                        mma_commit(&bars[landed ? V2_QEMPTY + s : V2_NOBODY]);
                    };
                    if (L::NdS == 1) issue_dK();
#pragma unroll
                    for (int kk = 0; kk < TK / 16; ++kk)
                        mma_ss_lo(T_B, mK + kk * 128, mdS + ds + kk * 128, idesc_dq, kk > 0);
                    mma_commit(&bars[V2_DQ]);
                    if (L::NdS == 2) issue_dK();
                }
                if (count > 0) {
                    mma_commit(&bars[V2_KE]);
                    ++nkv;
                }
            }
            // every product has completed before the CTA leaves: the last dQ^T is awaited by the reducers, this thread's last
            // commit comes after it
            if (nkv > 0) mbar_wait(&bars[V2_KE], (nkv - 1) & 1, ab);
        }
    } else if (warp >= 16) {
        setmaxnreg_dec<FusedRegs::kReduce>();
        // ------------------------------------------------------------ reducers: dQ_h^T tile -> fp32 accumulator
        // lanes = head-dimension index c, columns = queries: one warp instruction adds 128 contiguous bytes.
        // 32 columns at a time (the reducers run on 48 registers); the half is released after the second load
        const int h = (warp - 16) / 4;
        const uint32_t lane_addr = (uint32_t)((warp % 4) * 32) << 16;
        int kt = 0;
        for (int t = 0; warp % 4 < kReduceWarps && units.take(t); ++t) {
            const int count = slots[t & 1].count;
            for (int k = 0; k < count; ++k, ++kt) {
                // the slot is read anew for every tile, ahead of the wait, to save registers
                const int left = n - query_tile(slots[t & 1].rows, slots[t & 1].first + k) * TQ - h * 64;   // rows of this half that exist
                float *base = a.dQ_acc + ((size_t)slots[t & 1].bh * n + (n - left)) * HD + (warp % 4) * 32 + lane;
                mbar_wait(&bars[V2_DQ], kt & 1, ab);
                tcgen05_fence_after();
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    uint32_t v0[32];
                    tmem_ld32(T_B + lane_addr + h * 64 + part * 32, v0);
                    tmem_wait_ld();
                    tcgen05_fence_before();
                    // part 0: the 32 columns that take P^T of the next tile are free; part 1: the whole half is
                    warp_arrive(&bars[part == 0 ? V2_DQREL : V2_DQDONE], lane);
                    if (left >= 64) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) red_add_f32(base + (part * 32 + e) * HD, __uint_as_float(v0[e]));
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (part * 32 + e < left) red_add_f32(base + (part * 32 + e) * HD, __uint_as_float(v0[e]));
                    }
                }
            }
            warp_arrive(&bars[V2_WE + (t & 1)], lane);
        }
    } else {
        // ------------------------------------------------------------ warps 0-15: exp / dS; warpgroup 2h + qq owns queries 64 h + 32 qq .. + 31
        setmaxnreg_inc<FusedRegs::kExp>();
        // What a thread's place in the tile gives is formed anew where it is used: the row statistics, the scores and P take 80 of
        // the 88 registers, and a value that is spilled comes back through the shared memory that the products keep busy.
        struct Place {
            uint32_t h, qq, row, lane_addr;
            __device__ __forceinline__ Place()
            {
                uint32_t t;
                asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
                h = t >> 8; qq = (t >> 7) & 1u; row = t & 127u; lane_addr = (t & 96u) << 16;
            }
            __device__ __forceinline__ uint32_t column() const { return h * 64 + qq * 32; }   // of S^T / dP^T in region A; bf16 pairs of P^T: h * 64 + qq * 16
        };
        int kt = 0;
        for (int t = 0; units.take(t); ++t) {
            const int count = slots[t & 1].count, end = kt + count;
            for (; kt < end; ++kt) {
                const int s = stage_of(kt);
                mbar_wait(&bars[V2_QFULL + s], phase_of(kt), ab);
                // the 32 row statistics of this thread's query columns go into registers before the wait for S^T: while the
                // products stream their operands, a shared-memory load inside the arithmetic below waits a few hundred cycles
                float4 nlr[8];
                uint32_t kw = 0xffffffffu;   // which of its 32 query columns the thread's key row keeps
                bool drop = false;           // some thread of the warp drops some
                const int tile = tiles[kt & 3];
                uint32_t from;               // tensor-memory address of the thread's columns of S^T
                {
                    const Place at;
                    from = T_A + at.lane_addr + at.column();
                    const float4 *sNL = reinterpret_cast<const float4 *>(smem + L::oLSE + s * 512 + at.column() * 4);
#pragma unroll
                    for (int q = 0; q < 8; ++q) nlr[q] = sNL[q];
                    // a mask finer than the tile: the keep bits of this thread's key row and its 32 query columns
                    if constexpr (FINE) {
                        const int jg = slots[t & 1].tile * TK + (int)at.row, ig0 = (tile & 0x3fffffff) * TQ + (int)at.column();
                        kw = ig0 < n && jg < n ? fine_word(a.fine, a.mask_heads, slots[t & 1].bh, false, jg, ig0) : 0u;
                    }
                }
                mbar_wait(&bars[V2_S], kt & 1, ab);
                tcgen05_fence_after();
                uint32_t ppack[16];   // P as bf16 pairs: what dV uses, and what dS is formed from
                {
                    uint32_t sv[32];
                    tmem_ld32(from, sv);
                    if (tile < 0) {
                        const Place at;
                        const int jg = slots[t & 1].tile * TK + (int)at.row, ig0 = (tile & 0x3fffffff) * TQ + (int)at.column(), left = n - ig0;
                        if (left < 32) kw &= left > 0 ? 0xffffffffu >> (32 - left) : 0u;
                        if (jg >= n) kw = 0u;
                        if (causal && jg > ig0) kw &= jg - ig0 < 32 ? 0xffffffffu << (jg - ig0) : 0u;
                    }
                    if (FINE || tile < 0) drop = __any_sync(0xffffffffu, kw != 0xffffffffu);
                    tmem_wait_ld();
                    tcgen05_fence_before();
                    warp_arrive(&bars[V2_SLD], lane);   // region A may take dP^T
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 nl = nlr[q];
                        float p0, p1;
                        p_pair(sv[q * 4 + 0], sv[q * 4 + 1], a.sl2, nl.x, nl.y, p0, p1);
                        ppack[q * 2 + 0] = pack_bf16(p0, p1);
                        p_pair(sv[q * 4 + 2], sv[q * 4 + 3], a.sl2, nl.z, nl.w, p0, p1);
                        ppack[q * 2 + 1] = pack_bf16(p0, p1);
                    }
                    if (drop) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) ppack[e] &= (kw & (1u << (2 * e)) ? 0xffffu : 0u) | (kw & (2u << (2 * e)) ? 0xffff0000u : 0u);
                    }
                }
                float4 dsr[8];   // -scale * D of the same columns, again ahead of the wait
                const Place at;
                {
                    const float4 *sDs = reinterpret_cast<const float4 *>(smem + L::oD + s * 512 + at.column() * 4);
#pragma unroll
                    for (int q = 0; q < 8; ++q) dsr[q] = sDs[q];
                }
                const uint32_t from2 = T_A2 + at.lane_addr + at.column();
                // P^T goes into region B before dP^T is awaited: a tensor-memory store issued while products run takes
                // several hundred cycles, which now pass during that wait.  Its first 32 columns per half held dQ^T of the
                // previous tile; the reducers release them after their first load
                mbar_wait(&bars[V2_DQREL], (kt - 1) & 1, ab);
                tcgen05_fence_after();
                tmem_st16(T_B + at.lane_addr + at.h * 64 + at.qq * 16, ppack);
                mbar_wait(&bars[V2_DP], kt & 1, ab);
                tcgen05_fence_after();
                {
                    uint32_t dv[32];
                    tmem_ld32(from2, dv);
                    tmem_wait_ld();
                    tcgen05_fence_before();
                    warp_arrive(&bars[V2_DPLD], lane);   // region A may take the next S^T
                    tmem_wait_st();
                    tcgen05_fence_before();
                    warp_arrive(&bars[V2_P + at.h], lane);
                    uint8_t *slab = smem + L::odS + (L::NdS == 2 ? (kt & 1) * 2 * SLAB : 0) + at.h * SLAB;
                    // One buffer: dS^T(k) goes over dS^T(k-1), which the dK and dQ^T products of tile k-1 read.  Both have completed:
                    // the reducers release their columns (awaited above) only after dQ^T(k-1), the later of the two in the other
                    // thread's issue order, has landed.  Two buffers: dK(k-2) was issued before dQ^T(k-1)
#pragma unroll
                    for (int g = 0; g < 4; ++g) {    // 8 query columns = one 16-byte chunk
                        float ds[8];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t pk = ppack[g * 4 + e];   // bf16 -> fp32 is a 16-bit shift
                            const float4 dsc = dsr[g * 2 + e / 2];
                            ds_pair(pk, dv[g * 8 + 2 * e], dv[g * 8 + 2 * e + 1], a.scale, e & 1 ? dsc.z : dsc.x, e & 1 ? dsc.w : dsc.y, ds[2 * e], ds[2 * e + 1]);
                        }
                        if (drop) {   // stale tail entries of the row vectors may be anything: select, do not multiply
#pragma unroll
                            for (int e = 0; e < 8; ++e) ds[e] = (ppack[g * 4 + e / 2] & (e & 1 ? 0xffff0000u : 0xffffu)) != 0u ? ds[e] : 0.f;
                        }
                        *reinterpret_cast<uint4 *>(slab + sw128_offset(at.row, at.qq * 32 + g * 8)) =
                            make_uint4(pack_bf16(ds[0], ds[1]), pack_bf16(ds[2], ds[3]), pack_bf16(ds[4], ds[5]),
                                       pack_bf16(ds[6], ds[7]));
                    }
                }
                fence_proxy_async_smem();
                warp_arrive(&bars[V2_DS], lane);
            }
            // -------------------------------------------------------- epilogue: dV_j, dK_j (32 columns per warpgroup)
            const size_t bh = slots[t & 1].bh;
            const Place at;
            const int jg = slots[t & 1].tile * TK + (int)at.row;
            warp_arrive(&bars[V2_WE + (t & 1)], lane);
            if (count > 0) {
                // dV and dK of the last tile have completed when its stage is released (dQ^T, queued after them, is the
                // reducers' business and reads neither accumulator)
                mbar_wait(&bars[V2_QEMPTY + stage_of(kt - 1)], phase_of(kt - 1), ab);
                tcgen05_fence_after();
            }
            const uint32_t cq = at.column();       // d = 64: the upper two warpgroups have no columns
            if (cq < HD) {
                const int jc = jg < n ? jg : 0;
                const bool wide = (((uintptr_t)a.dK | (uintptr_t)a.dV) & 31) == 0;
#pragma unroll
                for (int which = 0; which < 2; ++which) {
                    __nv_bfloat16 *po = (which == 0 ? a.dV : a.dK) + (bh * n + jc) * HD + cq;
#pragma unroll
                    for (int e0 = 0; e0 < 32; e0 += 16) {
                        uint32_t v[16], y[8];
                        tmem_ld16((which == 0 ? T_dV : T_dK) + at.lane_addr + cq + e0, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int u = 0; u < 8; ++u)   // without a query tile nothing has been accumulated
                            y[u] = count > 0 ? pack_bf16(__uint_as_float(v[2 * u]), __uint_as_float(v[2 * u + 1])) : 0u;
                        if (jg < n) store32(po + e0, y, wide);
                    }
                }
                tcgen05_fence_before();
            }
        }
    }
    tmem_leave(tm, 512, warp, ab);
}

// fp32 accumulator -> bf16 dQ
__global__ void __launch_bounds__(256) dq_convert_kernel(const float4 *__restrict__ acc, uint2 *__restrict__ out, size_t n4)
{
    chain_release();
    chain_wait();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        const float4 v = acc[i];
        out[i] = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
    }
}

template <int HD, bool WITH_DQ>
attn_status launch_bwd(const Problem &p)
{
    using L = BwdSmem<HD>;
    CUtensorMap mQ, mK, mV, mdO;
    const uint64_t BH = (uint64_t)p.BH;
    if (!make_tmap_bf16_3d(&mQ, p.Q, HD, p.n, BH, 128) || !make_tmap_bf16_3d(&mK, p.K, HD, p.n, BH, 128) ||
        !make_tmap_bf16_3d(&mV, p.V, HD, p.n, BH, 128) || !make_tmap_bf16_3d(&mdO, p.dO, HD, p.n, BH, 128))
        return ATTN_ERR_LAUNCH;
    BwdArgs a{};
    a.nLSE2 = p.nLSE2; a.nDs = p.D; a.dQ_acc = p.dQ_acc;
    a.dK = (__nv_bfloat16 *)p.dK; a.dV = (__nv_bfloat16 *)p.dV;
    a.n = p.n; a.BH = (int)p.BH; a.ns = p.stat_stride;
    a.mask_kind = p.mask_kind; a.block = p.block; a.nb = p.nb; a.mask_heads = p.mask_heads; a.fine = p.fine;
    a.col_ptr = p.col_ptr; a.row_idx = p.row_idx;
    a.scale = p.scale; a.sl2 = p.scale * 1.4426950408889634f;
    a.status = p.status;
    a.group = bwd_head_group(p);
    if (bwd_preprocess_launch(p, WITH_DQ) != ATTN_OK) return ATTN_ERR_LAUNCH;
    const dim3 grid((unsigned)((p.n + TK - 1) / TK * a.group), (unsigned)(p.BH / a.group));
    bool ok;
    launch_begin(WITH_DQ ? "tc_bwd_fused" : "tc_bwd_dkdv", p.stream);
    if (WITH_DQ) {
        constexpr uint32_t bytes = HD == 64 ? ((L::kBytes + 1023u) & ~1023u) + SLAB : L::kBytes;
        auto kernel = p.fine.mode ? tc_bwd_fused_kernel<HD, true> : tc_bwd_fused_kernel<HD, false>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
            return ATTN_ERR_LAUNCH;
        ok = launch_chained(kernel, grid, kThreadsFused, bytes, p.stream, mQ, mK, mV, mdO, a);
    } else {
        auto kernel = p.split ? tc_bwd_dkdv_kernel<HD, true> : tc_bwd_dkdv_kernel<HD, false>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DkdvSmem<HD>::kBytes) != cudaSuccess)
            return ATTN_ERR_LAUNCH;
        ok = launch_chained(kernel, grid, kThreadsDkdv, DkdvSmem<HD>::kBytes, p.stream, mQ, mK, mV, mdO, a);
    }
    launch_end(p.stream);
    if (!ok) return ATTN_ERR_LAUNCH;
    if (!WITH_DQ) return tc_bwd_dq(p);   // deterministic path: dQ without atomics, from its own kernel
    return bwd_dq_convert_launch(p);
}

}  // namespace

// Heads are launched in groups (key tile major inside a group).  The fp32 dQ accumulators of the heads that run
// at the same time should stay in L2 between the reductions of one key tile and the next: otherwise every reduced
// sector is fetched from and written back to device memory (measured on the block-sparse workload with n = 32768:
// 13 times the compulsory traffic with 8 heads in flight).  So the group is the largest of 8, 4, 2, 1 that divides
// the head count and whose accumulators take at most kAccBudget bytes.
int bwd_head_group(const Problem &p)
{
    constexpr size_t kAccBudget = 40u << 20;
    for (int g = 8; g > 1; g >>= 1)
        if (p.BH % g == 0 && (size_t)g * p.n * p.d * sizeof(float) <= kAccBudget) return g;
    return 1;
}

namespace {
template <int HD>
attn_status preprocess_launch_t(const Problem &p, bool clear_acc)
{
    const size_t rows = (size_t)p.BH * p.n, acc_elems = rows * HD;
    constexpr size_t rpw = 32 / (HD / 8);
    size_t blocks = ((rows + rpw - 1) / rpw + 7) / 8;
    if (blocks > (size_t)sm_count() * 8) blocks = (size_t)sm_count() * 8;
    launch_begin("tc_bwd_preprocess", p.stream);
    const bool ok = launch_chained(p.stat_stride == p.n ? tc_preprocess_kernel<HD, false> : tc_preprocess_kernel<HD, true>, (unsigned)blocks, 256, 0,
                                   p.stream, (const __nv_bfloat16 *)p.O, (const __nv_bfloat16 *)p.dO, p.LSE, p.D, p.nLSE2, rows, p.n,
                                   p.stat_stride, p.scale, clear_acc ? (uint4 *)p.dQ_acc : nullptr, acc_elems / 4, p.clear, p.status);
    launch_end(p.stream);
    return ok ? ATTN_OK : ATTN_ERR_LAUNCH;
}
}  // namespace

attn_status bwd_preprocess_launch(const Problem &p, bool clear_acc)
{
    if (p.d == 64) return preprocess_launch_t<64>(p, clear_acc);
    if (p.d == 128) return preprocess_launch_t<128>(p, clear_acc);
    if (p.d == 256) return preprocess_launch_t<256>(p, clear_acc);
    return ATTN_ERR_TILE;
}

attn_status bwd_dq_convert_launch(const Problem &p)
{
    if (!p.dQ) return ATTN_OK;   // the caller reads the fp32 accumulator itself
    const size_t n4 = (size_t)p.BH * p.n * p.d / 4;
    const size_t cap = (size_t)sm_count() * 16;
    const unsigned blocks = (unsigned)((n4 + 255) / 256 < cap ? (n4 + 255) / 256 : cap);
    launch_begin("bwd_dq_convert", p.stream);
    const bool ok = launch_chained(dq_convert_kernel, blocks, 256, 0, p.stream, (const float4 *)p.dQ_acc, (uint2 *)p.dQ, n4);
    launch_end(p.stream);
    return ok ? ATTN_OK : ATTN_ERR_LAUNCH;
}

size_t bwd_smem_bytes(int d) { return d == 64 ? BwdSmem<64>::kBytes : d == 128 ? BwdSmem<128>::kBytes : 0; }

attn_status tc_bwd(const Problem &p)
{
    if (p.cfg.tile_q == 64 || p.d == 256) return tc_bwd64(p);
    if (p.d == 64) return p.atomics ? launch_bwd<64, true>(p) : launch_bwd<64, false>(p);
    if (p.d == 128) return p.atomics ? launch_bwd<128, true>(p) : launch_bwd<128, false>(p);
    return ATTN_ERR_TILE;
}

}  // namespace attn
