// dQ without atomics (the query-stationary half of the backward whose results repeat bit for bit), bf16, d = 64 / 128.
//
// This is the loop order the paper prints for its large-cache phase 2: the outer loop is
// over query row blocks i (here: one CTA per block of 128 queries, whose dQ_i tile stays
// in tensor memory), the inner loop over the kept key blocks j.  Per (i, j):
//
//   S  = Q_i K_j^T                       tcgen05.mma, K-major smem operands, two S buffers
//   dP = dO_i V_j^T                      same, one buffer
//   dS = scale * exp2(S scale log2e - LSE_i log2e) o (dP - D_i)     256 threads, lane = query
//        -> bf16, written over S in tensor memory
//   dQ_i += dS K_j                       A = dS from tensor memory, B = K_j MN-major smem
//
// S and dP are recomputed here (the key-stationary kernel computes them too), which is
// the price of summing dQ in a fixed order: 7 products instead of 5 per tile pair.
// Roles: warps 0-15 = four warpgroups, warpgroup g owning key columns 32 g .. 32 g + 31 of every
// tile (no barrier couples them, so their exp, dS and tensor-memory phases interleave freely);
// warp 16 lane 0 issues S and dP, warp 17 lane 0 issues dQ, warp 18 runs TMA and the schedule.  Tensor memory: S0 128, S1 128, dP 128,
// dQ d columns.
//
// A CTA takes the query tiles of CTAs that have not started yet (cluster launch control): Q, dO and the first products of the next
// one come while dQ of this one is written out.  24 heads, n = 3000, d = 64: 119 -> 113 us; 32 heads, n = 4096, d = 128, causal:
// 207 -> 203; 16 heads, n = 2047, d = 128, causal (two terms): 57.6 -> 55.8.
#include "attn_internal.h"
#include "tc_common.cuh"

namespace attn {
namespace {

using namespace tc;

constexpr int TQ = 128, TKD = 128;
constexpr int kSoftmaxThreads = 512;
constexpr int kThreads = kSoftmaxThreads + 96;   // + two MMA-issuing warps and the TMA warp
constexpr uint32_t SLAB = 128 * 128;

struct DqArgs {
    __nv_bfloat16 *dQ;
    const float *nLSE2, *nDs;
    int n, BH;
    int ns;                    // rows of nLSE2 and nDs per head (n, or n rounded up to a multiple of 4)
    int mask_kind, block, nb, mask_heads;
    const int *row_ptr, *col_idx;
    FineMask fine;
    float scale;
    uint32_t *status;
};

template <int HD>
struct DqSmem {
    static constexpr int NSTK = 3, NSTV = 2;   // K_j is needed first (S) and released last (dQ): three stages; V_j: two
    static constexpr uint32_t kSlabs = HD / 64;
    static constexpr uint32_t kTile = kSlabs * SLAB;     // one [128][HD] bf16 tile
    static constexpr uint32_t oQ = 0;
    static constexpr uint32_t odO = oQ + kTile;
    static constexpr uint32_t oK = odO + kTile;          // NSTK stages
    static constexpr uint32_t oV = oK + NSTK * kTile;    // NSTV stages
    static constexpr uint32_t oBar = oV + NSTV * kTile;
    static constexpr uint32_t oWork = oBar + 32 * 8;     // two slots of DqWork, the answer of the scheduler
    static constexpr uint32_t oMisc = oWork + 2 * 32 + 16;
    static constexpr uint32_t kUsed = oMisc + 16;
    static constexpr uint32_t kBytes = kUsed < 117 * 1024 ? 117 * 1024 : kUsed;   // one CTA per SM (512 TMEM columns)
    static_assert(kUsed <= 227 * 1024, "shared memory budget");
};

enum { DB_Q = 0, DB_KFULL = 1, DB_KEMPTY = 4, DB_VFULL = 7, DB_VEMPTY = 9, DB_S = 11, DB_DP = 13, DB_DQ = 14, DB_QEMPTY = 15,
       DB_CLC = 16, DB_WF = 17, DB_DPFREE = 19, DB_DS = 20, DB_WE = 22, DB_COUNT = 24 };

// One unit of work: a query tile of one head and the key tiles that it visits
struct DqWork {
    int tile, bh, count; // tile = -1: there is no more work
    int pad;
    const int *cols;     // key blocks of a mask with lists
    int pad2[2];
};
static_assert(sizeof(DqWork) == 32, "two slots in shared memory");

__device__ __forceinline__ float ex2_fast(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// SPLIT: dS enters its product as two bf16 terms, x = hi + lo up to 2^-17, for calls whose dS must not be rounded to one (bf16
// storage whose length is no multiple of 8): a thread writes the rests over the other half of the 32 columns
// of S that it has read.  16 heads, n = 2047, causal: 58 us at d = 128, 48 us at d = 64.
template <int HD, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
tc_bwd_dq_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
                 const __grid_constant__ CUtensorMap mV, const __grid_constant__ CUtensorMap mdO, const DqArgs a)
{
    using L = DqSmem<HD>;
    constexpr int NSTK = L::NSTK, NSTV = L::NSTV;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::oBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(smem + L::oMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + L::oMisc + 4);
    const Abort ab{abort_flag, a.status};

    volatile DqWork *slots = reinterpret_cast<volatile DqWork *>(smem + L::oWork);
    constexpr int kWarps = kSoftmaxThreads / 32;

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int n = a.n;
    const bool lists = mask_is_block(a.mask_kind), causal = mask_is_causal(a.mask_kind);
    const int sub = lists ? a.block / TKD : 1;

    if ((smem_u32(smem) & 1023u) != 0) {
        chain_wait();
        if (tid == 0) atomicExch(a.status, 9u);
        return;
    }
    if (tid == 0) {
        *abort_flag = 0;
        for (int b = 0; b < DB_COUNT; ++b)   // DPFREE, DS: one arrival per warp; WE: both issuers and the dS warps
            mbar_init(&bars[b], b >= DB_WE ? 2 + kWarps : b >= DB_DPFREE ? kWarps : 1);
        fence_barrier_init();
        prefetch_tensormap(&mQ); prefetch_tensormap(&mK); prefetch_tensormap(&mV); prefetch_tensormap(&mdO);
    }
    chain_wait();
    if (warp == 0) tmem_alloc(tmem_base_s, 512);
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    chain_release();
    const uint32_t tm = *tmem_base_s;
    const uint32_t T_dP = tm + 256, T_dQ = tm + 384;

    // the units of work of this CTA as the loading warp publishes them
    const UnitQueue<DqWork, UnitIo<>> units{slots, &bars[DB_WF], &bars[DB_WE], &bars[DB_CLC], smem + L::oWork + 2 * sizeof(DqWork), {ab}};
    auto key_tile = [&](const int *cols, int e) { return !lists ? e : sub == 1 ? cols[e] : cols[e / sub] * sub + e % sub; };

    // In every role k counts the key tiles of all units of work so far (a wait for what belongs to a tile before the first returns
    // at once): the barriers run on, and the loads and first products of the next unit come while dQ of this one is written out.
    if (warp == 18) {
        // ------------------------------------------------------------ TMA producer, and the schedule
        const int nt = (n + TQ - 1) / TQ;
        int bx = blockIdx.x, by = blockIdx.y;
        int k = 0, nq = 0;
        bool more = true;
        for (int t = 0; more; ++t) {
            const int it = nt - 1 - bx, bh = by, i0 = it * TQ;    // heaviest causal tiles first
            const int last_i = min(i0 + TQ, n) - 1;
            const int *cols = nullptr;
            int count;
            if (lists) {
                // the lists ascend: what lies beyond n or (block mask AND causal) begins after the last query is at their end
                const long mh = a.mask_heads == 1 ? 0 : bh;
                const int *rp = a.row_ptr + mh * 2 * a.nb + 2 * (i0 / a.block);
                const int first = rp[0], raw = (rp[1] - first) * sub, limit = causal ? last_i : n - 1;
                cols = a.col_idx + mh * (long)a.nb * a.nb + first;
                count = 0;
                for (int e = lane; e < raw; e += 32) count += key_tile(cols, e) * TKD <= limit;
                count = __reduce_add_sync(0xffffffffu, count);
            } else {
                count = causal ? last_i / TKD + 1 : (n + TKD - 1) / TKD;
            }
            auto load_unit = [&]() -> bool {   // false: there is no further unit, or the kernel is giving up
                volatile DqWork *to = units.claim(t);
                if (!to) return false;
                to->tile = it; to->bh = bh; to->count = count; to->cols = cols;
                units.publish(t);
                if (count > 0) {
                    if (!mbar_wait(&bars[DB_QEMPTY], (nq - 1) & 1, ab)) return false;   // dP of the unit before
                    ++nq;
                    mbar_expect_tx(&bars[DB_Q], 2 * L::kTile);
#pragma unroll
                    for (uint32_t sl = 0; sl < L::kSlabs; ++sl) {
                        tma_load_3d(smem + L::oQ + sl * SLAB, &mQ, &bars[DB_Q], sl * 64, i0, bh);
                        tma_load_3d(smem + L::odO + sl * SLAB, &mdO, &bars[DB_Q], sl * 64, i0, bh);
                    }
                } else {
                    units.ask();
                }
                for (int e = 0; e < count; ++e, ++k) {
                    const int jt = key_tile(cols, e), sk = k % NSTK, sv = k % NSTV;
                    if (e == max(count - 2, 0)) units.ask();
                    if (k >= NSTK && !mbar_wait(&bars[DB_KEMPTY + sk], ((k / NSTK) - 1) & 1, ab)) return false;
                    mbar_expect_tx(&bars[DB_KFULL + sk], L::kTile);
#pragma unroll
                    for (uint32_t sl = 0; sl < L::kSlabs; ++sl)
                        tma_load_3d(smem + L::oK + sk * L::kTile + sl * SLAB, &mK, &bars[DB_KFULL + sk], sl * 64, jt * TKD, bh);
                    if (k >= NSTV && !mbar_wait(&bars[DB_VEMPTY + sv], ((k / NSTV) - 1) & 1, ab)) return false;
                    mbar_expect_tx(&bars[DB_VFULL + sv], L::kTile);
#pragma unroll
                    for (uint32_t sl = 0; sl < L::kSlabs; ++sl)
                        tma_load_3d(smem + L::oV + sv * L::kTile + sl * SLAB, &mV, &bars[DB_VFULL + sv], sl * 64, jt * TKD, bh);
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
        // ------------------------------------------------------------ MMA issuer A: the products the warps wait for, S and dP,
        // one tile ahead.  (Two issuing threads: a thread that waits on a barrier or commits cannot keep the short
        // queue of the tensor pipe filled; B's dQ products are ordered against A's through barriers only.)
        if (lane == 0) {
            constexpr uint32_t idesc_s = idesc_bf16(128, 128, 0, 0);
            constexpr uint32_t kSlab = SLAB >> 4;
            const uint32_t kQ = desc_lo_kmajor(smem_u32(smem + L::oQ)), kdO = desc_lo_kmajor(smem_u32(smem + L::odO));
            int k = 0, nq = 0;
            for (int t = 0; units.take_alone(t); ++t) {
                const int end = k + slots[t & 1].count;
                mbar_arrive(&bars[DB_WE + (t & 1)]);
                if (k == end) continue;
                if (!mbar_wait(&bars[DB_Q], nq & 1, ab)) break;
                ++nq;
                for (; k < end; ++k) {
                    const int s = k % NSTK;
                    mbar_wait(&bars[DB_KFULL + s], (k / NSTK) & 1, ab);
                    // the buffer of S(k) held dS(k-2): the dQ product of tile k-2 (other thread) must have consumed it
                    if (k >= 2) mbar_wait(&bars[DB_KEMPTY + (k - 2) % NSTK], ((k - 2) / NSTK) & 1, ab);
                    tcgen05_fence_after();
                    const uint32_t kK = desc_lo_kmajor(smem_u32(smem + L::oK + s * L::kTile));
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        const uint32_t off = (kk / 4) * kSlab + (kk % 4) * 2;
                        mma_ss_lo(tm + (k & 1) * 128, kQ + off, kK + off, idesc_s, kk > 0);
                    }
                    mma_commit(&bars[DB_S + (k & 1)]);
                    // dP(k) once every thread has read dP(k-1) out of tensor memory
                    mbar_wait(&bars[DB_DPFREE], (k - 1) & 1, ab);
                    if (!mbar_wait(&bars[DB_VFULL + k % NSTV], (k / NSTV) & 1, ab)) break;
                    tcgen05_fence_after();
                    const uint32_t kV = desc_lo_kmajor(smem_u32(smem + L::oV + (k % NSTV) * L::kTile));
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        const uint32_t off = (kk / 4) * kSlab + (kk % 4) * 2;
                        mma_ss_lo(T_dP, kdO + off, kV + off, idesc_s, kk > 0);
                    }
                    mma_commit(&bars[DB_DP]);
                    mma_commit(&bars[DB_VEMPTY + k % NSTV]);
                }
                mma_commit(&bars[DB_QEMPTY]);
            }
        }
    } else if (warp == 17) {
        // ------------------------------------------------------------ MMA issuer B: dQ_i += dS K_j
        if (lane == 0) {
            constexpr uint32_t idesc_dq = idesc_bf16(128, HD, 0, 1);
            int k = 0;
            for (int t = 0; units.take_alone(t); ++t) {
                const int begin = k, end = k + slots[t & 1].count;
                mbar_arrive(&bars[DB_WE + (t & 1)]);
                for (; k < end; ++k) {
                    const int s = k % NSTK, b = k & 1;
                    if (!mbar_wait(&bars[DB_KFULL + s], (k / NSTK) & 1, ab)) break;
                    mbar_wait(&bars[DB_DS + b], (k >> 1) & 1, ab);   // of every warp: the first of a unit has been preceded by their reading dQ
                    tcgen05_fence_after();
                    const uint32_t mK_ = desc_lo_mnmajor(smem_u32(smem + L::oK + s * L::kTile), SLAB);
#pragma unroll
                    for (int kk = 0; kk < TKD / 16; ++kk) {
                        const uint32_t dS = tm + b * 128 + (kk / 2) * 32 + (kk % 2) * 8;
                        mma_ts_lo(T_dQ, dS, mK_ + kk * 128, idesc_dq, (k > begin) || (kk > 0));
                        if constexpr (SPLIT) mma_ts_lo(T_dQ, dS + 16, mK_ + kk * 128, idesc_dq, 1);
                    }
                    mma_commit(&bars[DB_KEMPTY + s]);
                }
                if (end > begin) mma_commit(&bars[DB_DQ]);
            }
        }
    } else {
        // ------------------------------------------------------------ dS warpgroups: wg splits the key columns
        const int wg = warp / 4;
        const int row = (warp % 4) * 32 + lane;           // tensor-memory lane = query row of the tile
        const uint32_t lane_addr = (uint32_t)((warp % 4) * 32) << 16;
        const float sl2 = a.scale * 1.4426950408889634f;
        const bool wide = ((uintptr_t)a.dQ & 31) == 0;
        int k = 0, nq = 0;
        for (int t = 0; units.take(t); ++t) {
            const int i0 = slots[t & 1].tile * TQ, bh = slots[t & 1].bh, count = slots[t & 1].count, begin = k;
            const int *cols = slots[t & 1].cols;
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[DB_WE + (t & 1)]);
            const int ig = i0 + row;
            const float nl = ig < n ? a.nLSE2[(size_t)bh * a.ns + ig] : -INFINITY;   // -inf: every probability of the row is 0
            const float dsi = ig < n ? a.nDs[(size_t)bh * a.ns + ig] : 0.f;
            for (; k < begin + count; ++k) {
                const int jt = key_tile(cols, k - begin);
                const int b = k & 1, j0 = jt * TKD + wg * 32;
                const uint32_t T_S = tm + b * 128;
                // a mask finer than the tile: the keep bits of this thread's query row and its 32 key columns
                uint32_t kw = 0xffffffffu;
                if (a.fine.mode) kw = (ig < n && j0 < n) ? fine_word(a.fine, a.mask_heads, bh, true, ig, j0) : 0u;
                const bool masked = (causal && jt * TKD + TKD - 1 > i0) || jt * TKD + TKD > n || a.fine.mode != 0;
                mbar_wait(&bars[DB_S + b], (k >> 1) & 1, ab);
                tcgen05_fence_after();
                float p[32];
                {
                    uint32_t sv0[32];
                    tmem_ld32(T_S + lane_addr + wg * 32, sv0);
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(p[e]), "=f"(p[e + 1]) : "l"(fma_pair(sv0[e], sv0[e + 1], sl2, nl, nl)));
                        p[e] = ex2_fast(p[e]);
                        p[e + 1] = ex2_fast(p[e + 1]);
                    }
                }
                if (masked) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        const int jg = j0 + e;
                        if (jg >= n || (causal && jg > ig) || !((kw >> e) & 1u)) p[e] = 0.f;
                    }
                }
                mbar_wait(&bars[DB_DP], k & 1, ab);
                tcgen05_fence_after();
                uint32_t dpack[16], drest[SPLIT ? 16 : 1];
                {
                    uint32_t dv0[32];
                    tmem_ld32(T_dP + lane_addr + wg * 32, dv0);
                    tmem_wait_ld();
                    tcgen05_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars[DB_DPFREE]);
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        float d0, d1;
                        mul_pair(fma_pair(dv0[e], dv0[e + 1], a.scale, dsi, dsi), __float_as_uint(p[e]), __float_as_uint(p[e + 1]), d0, d1);
                        dpack[e / 2] = pack_bf16(d0, d1);
                        if constexpr (SPLIT) drest[e / 2] = pack_bf16_rest(d0, d1, dpack[e / 2]);
                    }
                }
                // dS (bf16 pairs) over the first 16 of the 32 S columns this thread has read itself
                tmem_st16(T_S + lane_addr + wg * 32, dpack);
                if constexpr (SPLIT) tmem_st16(T_S + lane_addr + wg * 32 + 16, drest);
                tmem_wait_st();
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[DB_DS + b]);
            }
            // -------------------------------------------------------- epilogue: dQ_i (dS carried the scale)
            if (count > 0) {
                mbar_wait(&bars[DB_DQ], nq & 1, ab);
                ++nq;
                tcgen05_fence_after();
            }
            constexpr int OW = HD / 4;   // dQ columns per warpgroup: 32 or 16
            const int ic = ig < n ? ig : 0;
            __nv_bfloat16 *pq = a.dQ + ((size_t)bh * n + ic) * HD + wg * OW;
#pragma unroll
            for (int e0 = 0; e0 < OW; e0 += 16) {
                uint32_t v[16], y[8];
                tmem_ld16(T_dQ + lane_addr + wg * OW + e0, v);
                tmem_wait_ld();
#pragma unroll
                for (int u = 0; u < 8; ++u)   // without a key tile nothing has been accumulated
                    y[u] = count > 0 ? pack_bf16(__uint_as_float(v[2 * u]), __uint_as_float(v[2 * u + 1])) : 0u;
                if (ig < n) store32(pq + e0, y, wide);
            }
            tcgen05_fence_before();
        }
    }
    tmem_leave(tm, 512, warp, ab);
}

template <int HD>
attn_status launch_dq(const Problem &p)
{
    using L = DqSmem<HD>;
    CUtensorMap mQ, mK, mV, mdO;
    const uint64_t BH = (uint64_t)p.BH;
    if (!make_tmap_bf16_3d(&mQ, p.Q, HD, p.n, BH, 128) || !make_tmap_bf16_3d(&mK, p.K, HD, p.n, BH, 128) ||
        !make_tmap_bf16_3d(&mV, p.V, HD, p.n, BH, 128) || !make_tmap_bf16_3d(&mdO, p.dO, HD, p.n, BH, 128))
        return ATTN_ERR_LAUNCH;
    DqArgs a{};
    a.dQ = (__nv_bfloat16 *)p.dQ;
    a.nLSE2 = p.nLSE2; a.nDs = p.D;
    a.n = p.n; a.BH = (int)p.BH; a.ns = p.stat_stride;
    a.mask_kind = p.mask_kind; a.block = p.block; a.nb = p.nb; a.mask_heads = p.mask_heads; a.fine = p.fine;
    a.row_ptr = p.row_ptr; a.col_idx = p.col_idx;
    a.scale = p.scale;
    a.status = p.status;
    auto kernel = p.split ? tc_bwd_dq_kernel<HD, true> : tc_bwd_dq_kernel<HD, false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::kBytes) != cudaSuccess)
        return ATTN_ERR_LAUNCH;
    const dim3 grid((p.n + TQ - 1) / TQ, (unsigned)p.BH);
    launch_begin("tc_bwd_dq", p.stream);
    const bool ok = launch_chained(kernel, grid, kThreads, L::kBytes, p.stream, mQ, mK, mV, mdO, a);
    launch_end(p.stream);
    return ok ? ATTN_OK : ATTN_ERR_LAUNCH;
}

}  // namespace

// Requires p.D = -scale * rowsum(dO o O) and p.nLSE2 = -LSE log2(e), as the key-stationary launch leaves them.
attn_status tc_bwd_dq(const Problem &p)
{
    if (p.d == 64) return launch_dq<64>(p);
    if (p.d == 128) return launch_dq<128>(p);
    return ATTN_ERR_TILE;
}

}  // namespace attn
