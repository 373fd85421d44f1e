// Fused forward for bf16 on the 5th-generation tensor cores: O = softmax(scale Q K^T) V
// and LSE, never writing a score tile to device memory (Definition 3.1; large-cache
// tiling: one or two row blocks of 128 queries stay on chip, key/value blocks stream through).
//
// A CTA owns a tile of 128 queries (tensor-memory lane = query row), or two of them, and walks the
// kept key tiles j:
//
//   S   = Q_i K_j^T                  tcgen05.mma, operands K-major in shared memory
//   m, l running row maximum / row sum in the exp2 domain; the reference maximum is
//       only moved (and O rescaled in tensor memory) when the tile maximum exceeds it
//       by more than 2^8 -- the final LSE does not depend on which reference was used
//   P   = exp2(S * scale*log2e - m)  -> bf16, in tensor memory (columns of its own; d = 256 and the two-term kernels: over S)
//   O  += P V_j                      A = P from tensor memory, B = V_j MN-major
//
// Four kernels.  tc_fwd_flow_kernel (d = 64, 128): a thread holds a whole row of scores, S has buffers of its own that
// are free as soon as it has been copied out.  PAIR (no mask or causal, calls with enough tiles): two query tiles per CTA, a
// softmax warpgroup each.  Otherwise one query tile, the two softmax warpgroups take alternate key tiles, each with a partial
// accumulator of its own, and the two partial softmaxes are merged in the epilogue.  tc_fwd_pair_kernel and
// tc_fwd_rows_kernel: the same two shapes, a CTA per unit of work, for calls whose P must not be rounded to one bf16 term; its second term takes the
// tensor memory that the S buffers would need.  tc_fwd_kernel (d = 256; key tiles of 64): both warpgroups
// split the columns of every tile and exchange row maxima through shared memory, one accumulator of
// 256 columns.  The roles and the tensor-memory layout are described at each kernel.
#include <type_traits>

#include "attn_internal.h"
#include "tc_common.cuh"

namespace attn {
namespace {

using namespace tc;

constexpr int TQ = 128;
constexpr int kSoftmaxThreads = 256;
constexpr int kThreads = kSoftmaxThreads + 96;   // d = 256: two issuing warps and the loading warp
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.f;   // log2 units

struct FwdArgs {
    __nv_bfloat16 *O;
    float *LSE;
    int n, BH;
    int group;                      // heads per launch group (divides BH): blockIdx.x is query tile major inside a group
    int mask_kind, block, nb, mask_heads;
    const int *row_ptr, *col_idx;   // block-CSR of the mask
    FineMask fine;                  // a mask finer than the tiles (32- / 64-wide blocks, element bitmap)
    float scale;
    uint32_t *status;
};

template <int HD>
struct FwdCfg {                                                // d = 256
    static constexpr int TKF = 64;
    static constexpr int NST = 2;
    static constexpr uint32_t kQSlab = 128 * 128;              // [128 queries][64 bf16]
    static constexpr uint32_t kKSlab = TKF * 128;              // [TKF keys][64 bf16]
    static constexpr uint32_t kSlabs = HD / 64;
    static constexpr uint32_t kQTile = kSlabs * kQSlab;
    static constexpr uint32_t kKTile = kSlabs * kKSlab;
    static constexpr uint32_t oQ = 0;
    static constexpr uint32_t oK = oQ + kQTile;                // NST stages
    static constexpr uint32_t oV = oK + NST * kKTile;          // NST stages
    static constexpr uint32_t oX = oV + NST * kKTile;          // row-max exchange [2 buffers][2 wg][128]; row sums reuse buffer 0
    static constexpr uint32_t oBar = oX + 4 * 128 * 4;
    static constexpr uint32_t oMisc = oBar + 24 * 8;
    static constexpr uint32_t kUsed = oMisc + 64;
    static_assert(kUsed <= 227 * 1024, "shared memory budget");
    // at least 117 KB so that only one CTA (which allocates all 512 tensor-memory columns) fits per SM
    static constexpr uint32_t kBytes = kUsed < 117 * 1024 ? 117 * 1024 : kUsed;
};

// FB_KVEMPTY: O += P V of the tile that this stage held has completed; the loading thread takes it as the release of the stage, a
// softmax thread as the news that O holds the product.  When it asks, the completion before is known from S of its own tile, whose
// K came after that one, and the next one needs its P.  A barrier that completes with every tile's product could be two
// completions behind: of the product of tile k - 2 nothing but the release of its stage is known from S(k).
enum { FB_Q = 0, FB_KVFULL = 1, FB_KVEMPTY = 3, FB_S = 5, FB_P = 7 };

template <int TKF>
struct KeyIter {
    // Enumerates the key tiles (of TKF keys) a query tile `it` (128 queries) has to visit.
    int kind, n, sub, raw, last_i;
    const int *cols;
    __device__ KeyIter(const FwdArgs &a, int it, long bh) : kind(a.mask_kind), n(a.n), sub(1), raw(0), cols(nullptr)
    {
        last_i = min(it * TQ + TQ, n) - 1;
        const int ntk = (n + TKF - 1) / TKF;
        if (kind == ATTN_MASK_NONE) raw = ntk;
        else if (kind == ATTN_MASK_CAUSAL) {
            const int last_i = min(it * TQ + TQ, n) - 1;
            raw = last_i / TKF + 1;
        } else {
            sub = a.block / TKF;
            const int I = it * TQ / a.block;
            const long mh = a.mask_heads == 1 ? 0 : bh;
            const int *rp = a.row_ptr + mh * 2 * a.nb + 2 * I;
            cols = a.col_idx + mh * (long)a.nb * a.nb + rp[0];
            raw = (rp[1] - rp[0]) * sub;
        }
    }
    __device__ int tile(int idx) const
    {
        int jt;
        if (mask_is_block(kind)) jt = cols[idx / sub] * sub + idx % sub;
        else jt = idx;
        // block mask AND causal: a key tile that begins after the last query of the tile keeps nothing
        if (kind == ATTN_MASK_BLOCK_SPARSE_CAUSAL && jt * TKF > last_i) return -1;
        return jt * TKF < n ? jt : -1;
    }
};

__device__ __forceinline__ float ex2_fast_f(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void named_bar_sync_f(int id, int count)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// one arrival per warp: every lane has finished (and fenced) its part
__device__ __forceinline__ void warp_arrive_f(uint64_t *bar, int lane)
{
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

// LSE of a row from its reference m (log2 units) and its sum l: m ln2 + ln l with one rounding of the size of the result.
// l = 2^e f: the logarithm of f < 2 is small, m + e is kept with what the addition loses, ln2 in two terms.  ex2.approx comes out
// 4.5e-8 too small on average (measured over [-10, 0]), which a sum does not average out; the logarithm gives it back.
// Relative error of the LSE, 32 heads, n = 2048, d = 128, causal: 3.67e-8 with m * kLn2 + logf(l), 2.75e-8 this way; n = 257, P as
// two terms: 3.56e-8 with the sum in 64 bits and no correction, 2.99e-8 this way, 3.13e-8 on the FMA kernels.
__device__ __forceinline__ float row_lse(float m, float l)
{
    if (!(l > 0.f)) return -INFINITY;
    const uint32_t bits = __float_as_uint(l);
    const float e = (float)((int)(bits >> 23) - 127), f = __uint_as_float((bits & 0x7fffffu) | 0x3f800000u);
    const float s = m + e, t = s - m, lost = (m - (s - t)) + (e - t);
    constexpr float kLn2Rest = (float)(0.69314718055994530942 - (double)kLn2);
    return fmaf(s, kLn2, fmaf(lost, kLn2, fmaf(s, kLn2Rest, logf(f) + 4.5e-8f)));
}

// x = exp2(v * s + n) of two scores; both are added to `sum`
__device__ __forceinline__ void exp_pair(uint32_t v0, uint32_t v1, uint64_t s2, uint64_t n2, uint64_t &sum, float &x0, float &x1)
{
    uint64_t x;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(v0), "r"(v1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(x) : "l"(x), "l"(s2), "l"(n2));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x));
    x0 = ex2_fast_f(x0);
    x1 = ex2_fast_f(x1);
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(x0), "f"(x1));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(sum) : "l"(sum), "l"(x));
}
__device__ __forceinline__ float sum_of(const uint64_t (&sum)[4])
{
    float a[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) asm("mov.b64 {%0, %1}, %2;" : "=f"(a[2 * e]), "=f"(a[2 * e + 1]) : "l"(sum[e]));
    return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}
// d = 256.  Bound by the exchange of row maxima between the warpgroups on every tile of 64 keys and the chain around it.  One issuing
// thread for S and one for P V, P reported by one arrival a warp instead of 256 a tile, packed exponentials: 8 heads, n = 4096, no
// mask: 258 -> 185 us.
template <int HD>
__global__ void __launch_bounds__(kThreads, 1)
tc_fwd_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
              const __grid_constant__ CUtensorMap mV, const FwdArgs a)
{
    using C = FwdCfg<HD>;
    constexpr int TKF = C::TKF, NST = C::NST;
    constexpr int CW = TKF / 2;      // key columns per warpgroup
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::oBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(smem + C::oMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + C::oMisc + 4);
    float *xmax = reinterpret_cast<float *>(smem + C::oX);            // [2][2][128]
    float *xsum = xmax;                                               // [2][128], reuses exchange buffer 0 in the epilogue
    const Abort ab{abort_flag, a.status};

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int nt = (a.n + TQ - 1) / TQ;
    const int it = nt - 1 - (int)blockIdx.x / a.group;    // heaviest causal tiles first
    const long bh = (long)blockIdx.y * a.group + blockIdx.x % a.group;
    const int i0 = it * TQ, n = a.n;

    if ((smem_u32(smem) & 1023u) != 0) {
        chain_wait();
        if (tid == 0) atomicExch(a.status, 9u);
        return;
    }
    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(&bars[FB_Q], 1);
        for (int s = 0; s < NST; ++s) { mbar_init(&bars[FB_KVFULL + s], 1); mbar_init(&bars[FB_KVEMPTY + s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&bars[FB_S + b], 1); mbar_init(&bars[FB_P + b], kSoftmaxThreads / 32); }
        fence_barrier_init();
        prefetch_tensormap(&mQ); prefetch_tensormap(&mK); prefetch_tensormap(&mV);
    }
    chain_wait();
    if (warp == 0) tmem_alloc(tmem_base_s, 512);
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    chain_release();
    if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) *a.status = 0u;
    const uint32_t tm = *tmem_base_s;
    const uint32_t T_O = tm + 256;
    const KeyIter<TKF> iter(a, it, bh);

    // number of valid key tiles (same in every role)
    int niter = 0;
    for (int idx = 0; idx < iter.raw; ++idx) niter += iter.tile(idx) >= 0;

    if (warp == 9) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            mbar_expect_tx(&bars[FB_Q], C::kQTile);
#pragma unroll
            for (uint32_t sl = 0; sl < C::kSlabs; ++sl)
                tma_load_3d(smem + C::oQ + sl * C::kQSlab, &mQ, &bars[FB_Q], sl * 64, i0, (int)bh);
            int k = 0;
            for (int idx = 0; idx < iter.raw; ++idx) {
                const int jt = iter.tile(idx);
                if (jt < 0) continue;
                const int s = k % NST;
                if (k >= NST && !mbar_reload(&bars[FB_KVFULL + s], &bars[FB_KVEMPTY + s], ((k / NST) - 1) & 1, ab)) break;
                uint64_t *bar = &bars[FB_KVFULL + s];
                mbar_expect_tx(bar, 2 * C::kKTile);
#pragma unroll
                for (uint32_t sl = 0; sl < C::kSlabs; ++sl) {
                    tma_load_3d(smem + C::oK + s * C::kKTile + sl * C::kKSlab, &mK, bar, sl * 64, jt * TKF, (int)bh);
                    tma_load_3d(smem + C::oV + s * C::kKTile + sl * C::kKSlab, &mV, bar, sl * 64, jt * TKF, (int)bh);
                }
                ++k;
            }
        }
    } else if (warp == 8) {
        // ------------------------------------------------------------ MMA issuer A: S = Q K^T, up to two tiles ahead
        if (lane == 0 && niter == 0) mbar_wait(&bars[FB_Q], 0, ab);   // let the Q load land before exit
        if (lane == 0 && niter > 0) {
            constexpr uint32_t idesc_s = idesc_bf16(128, TKF, 0, 0);
            const uint32_t kQ = desc_lo_kmajor(smem_u32(smem + C::oQ));
            mbar_wait(&bars[FB_Q], 0, ab);
            for (int k = 0; k < niter; ++k) {
                const int s = k % NST;
                // K of tile k goes where that of tile k - 2 was, so its load tells that O += P V of that tile, which read P from
                // this S buffer, has completed
                mbar_wait(&bars[FB_KVFULL + s], (k / NST) & 1, ab);
                tcgen05_fence_after();
                const uint32_t kK = desc_lo_kmajor(smem_u32(smem + C::oK + s * C::kKTile));
#pragma unroll
                for (int kk = 0; kk < HD / 16; ++kk)
                    mma_ss_lo(tm + (k & 1) * 128, kQ + (kk / 4) * (C::kQSlab >> 4) + (kk % 4) * 2,
                              kK + (kk / 4) * (C::kKSlab >> 4) + (kk % 4) * 2, idesc_s, kk > 0);
                mma_commit(&bars[FB_S + (k & 1)]);
            }
        }
    } else if (warp == 10) {
        // ------------------------------------------------------------ MMA issuer B: O += P V
        if (lane == 0) {
            constexpr uint32_t idesc_o = idesc_bf16(128, HD, 0, 1);
            for (int k = 0; k < niter; ++k) {
                const int s = k % NST, b = k & 1;
                mbar_wait(&bars[FB_P + b], (k >> 1) & 1, ab);
                tcgen05_fence_after();
                const uint32_t mV_ = desc_lo_mnmajor(smem_u32(smem + C::oV + s * C::kKTile), C::kKSlab);
#pragma unroll
                for (int kk = 0; kk < TKF / 16; ++kk)
                    mma_ts_lo(T_O, tm + b * 128 + kk * 8, mV_ + kk * 128, idesc_o, (k > 0) || (kk > 0));
                mma_commit(&bars[FB_KVEMPTY + s]);
            }
        }
    } else {
        // ------------------------------------------------------------ softmax warpgroups
        const int wg = warp / 4;
        const int row = (warp % 4) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp % 4) * 32) << 16;
        const int ig = i0 + row;
        const float sl2 = a.scale * kLog2e;
        float m_ref = -INFINITY, l_part = 0.f;
        int k = 0;
        for (int idx = 0; idx < iter.raw; ++idx) {
            const int jt = iter.tile(idx);
            if (jt < 0) continue;
            const int b = k & 1, j0 = jt * TKF;
            // a mask finer than the tile: the keep bits of this thread's query row and its 32 key columns, fetched
            // before the wait for S
            uint32_t kw = 0xffffffffu;
            if (a.fine.mode) kw = (ig < n && j0 + wg * CW < n) ? fine_word(a.fine, a.mask_heads, bh, true, ig, j0 + wg * CW) : 0u;
            mbar_wait(&bars[FB_S + b], (k >> 1) & 1, ab);
            tcgen05_fence_after();
            const uint32_t T_S = tm + b * 128;
            float sv[CW];
#pragma unroll
            for (int c = 0; c < CW; c += 32) {
                uint32_t v[32];
                tmem_ld32(T_S + lane_addr + wg * CW + c, v);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) sv[c + e] = __uint_as_float(v[e]);   // raw scores; scale * log2e enters below
            }
            const bool need_mask = (mask_is_causal(a.mask_kind) && j0 + TKF - 1 > i0) || j0 + TKF > n || a.fine.mode != 0;
            float mx = -INFINITY;
            if (need_mask) {
                const bool causal = mask_is_causal(a.mask_kind);
#pragma unroll
                static_assert(CW == 32, "one keep word per thread and tile");
#pragma unroll
                for (int e = 0; e < CW; ++e) {
                    const int jg = j0 + wg * CW + e;
                    if (jg >= n || (causal && jg > ig) || !((kw >> e) & 1u)) sv[e] = -INFINITY;
                }
            }
#pragma unroll
            for (int e = 0; e < CW; ++e) mx = fmaxf(mx, sv[e]);
            float *xm = xmax + b * 256;
            xm[wg * 128 + row] = mx;
            named_bar_sync_f(1, kSoftmaxThreads);   // also: every S read of this tile is done
            const float m_tile = fmaxf(xm[row], xm[128 + row]) * sl2;   // scale > 0: the maximum commutes with it
            const bool need = m_tile > m_ref + kRescaleThreshold || (m_ref == -INFINITY && m_tile != -INFINITY);
            if (__any_sync(0xffffffffu, need)) {
                const float m_new = need ? fmaxf(m_ref, m_tile) : m_ref;
                const float alpha = (need && m_ref != -INFINITY) ? ex2_fast_f(m_ref - m_new) : 1.f;
                if (k > 0) {
                    mbar_wait(&bars[FB_KVEMPTY + (k - 1) % NST], ((k - 1) / NST) & 1, ab);   // O += P V of the previous tile has landed
                    tcgen05_fence_after();
#pragma unroll
                    for (int c = 0; c < HD / 2; c += 32) {
                        uint32_t v[32];
                        tmem_ld32(T_O + lane_addr + wg * (HD / 2) + c, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * alpha);
                        tmem_st32(T_O + lane_addr + wg * (HD / 2) + c, v);
                    }
                }
                l_part *= alpha;
                m_ref = m_new;
            }
            const float noff = m_ref == -INFINITY ? 0.f : -m_ref;
            uint32_t pp[CW / 2];
            uint64_t s2, n2, sum[4] = {0ull, 0ull, 0ull, 0ull};
            asm("mov.b64 %0, {%1, %1};" : "=l"(s2) : "f"(sl2));
            asm("mov.b64 %0, {%1, %1};" : "=l"(n2) : "f"(noff));
#pragma unroll
            for (int e = 0; e < CW; e += 2) {
                float p0, p1;
                exp_pair(__float_as_uint(sv[e]), __float_as_uint(sv[e + 1]), s2, n2, sum[(e / 2) & 3], p0, p1);
                pp[e / 2] = pack_bf16(p0, p1);
            }
            l_part += sum_of(sum);
            tmem_st16(T_S + lane_addr + wg * (CW / 2), pp);
            tmem_wait_st();
            tcgen05_fence_before();
            warp_arrive_f(&bars[FB_P + b], lane);
            ++k;
        }
        // ------------------------------------------------------------ epilogue
        named_bar_sync_f(1, kSoftmaxThreads);   // everyone is done with the row-max exchange buffers
        xsum[wg * 128 + row] = l_part;
        named_bar_sync_f(1, kSoftmaxThreads);
        const float l_tot = xsum[row] + xsum[128 + row];
        if (k > 0) {
            mbar_wait(&bars[FB_KVEMPTY + (k - 1) % NST], ((k - 1) / NST) & 1, ab);   // the last product
            tcgen05_fence_after();
        }
        const float inv = l_tot > 0.f ? 1.f / l_tot : 0.f;
        const int ic = ig < n ? ig : 0;
        __nv_bfloat16 *po = a.O + ((size_t)bh * n + ic) * HD + wg * (HD / 2);
#pragma unroll
        for (int c = 0; c < HD / 2; c += 32) {
            uint32_t v[32];
            if (k > 0) {
                tmem_ld32(T_O + lane_addr + wg * (HD / 2) + c, v);
                tmem_wait_ld();
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = 0u;
            }
            if (ig < n) {
#pragma unroll
                for (int e = 0; e < 32; e += 8) {
                    uint4 o;
                    o.x = pack_bf16(__uint_as_float(v[e]) * inv, __uint_as_float(v[e + 1]) * inv);
                    o.y = pack_bf16(__uint_as_float(v[e + 2]) * inv, __uint_as_float(v[e + 3]) * inv);
                    o.z = pack_bf16(__uint_as_float(v[e + 4]) * inv, __uint_as_float(v[e + 5]) * inv);
                    o.w = pack_bf16(__uint_as_float(v[e + 6]) * inv, __uint_as_float(v[e + 7]) * inv);
                    *reinterpret_cast<uint4 *>(po + c + e) = o;
                }
            }
        }
        if (wg == 0 && ig < n) a.LSE[(size_t)bh * n + ig] = row_lse(m_ref, l_tot);
    }
    tmem_leave(tm, 512, warp, ab);
}

// The work of a softmax thread on its row of 128 scores.  While one warpgroup waits for its products the other one's warps are
// alone on their schedulers, so the length of this instruction sequence, not a pipe, is what it takes: three-operand maxima
// and packed multiply-adds and additions (the roundings of the scalar ones) save 190 of about 700 instructions (forward of
// 32 heads, n = 8192, d = 128, pairs of query tiles: 585 -> 563 us at that point).
__device__ __forceinline__ float max3(float x, float y, float z)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
    return r;
}
__device__ __forceinline__ float row_max(const uint32_t (&v)[128])
{
    float m[8];   // eight independent chains
#pragma unroll
    for (int e = 0; e < 8; ++e) m[e] = fmaxf(__uint_as_float(v[e]), __uint_as_float(v[e + 8]));
#pragma unroll
    for (int c = 16; c < 128; c += 16)
#pragma unroll
        for (int e = 0; e < 8; ++e) m[e] = max3(m[e], __uint_as_float(v[c + e]), __uint_as_float(v[c + e + 8]));
    return fmaxf(max3(max3(m[0], m[1], m[2]), m[3], m[4]), max3(m[5], m[6], m[7]));
}
// P = exp2(v * sl2 + noff) as two bf16 terms: pairs of leading terms over the first 64 columns of S (every thread overwrites
// only its own lane, whose scores it already holds), what they lose over the other 64; returns the sum of the row of P before
// rounding.
//
// The first 96 keys of P are handed over (`early`, one arrival per warp) as soon as they are stored: the tensor core, idle by
// then, forms their part of O += P V under the exponentials of the rest.
__device__ __forceinline__ float exp_row_split(const uint32_t (&v)[128], float sl2, float noff, uint32_t to, uint64_t *early, uint64_t *last, int lane)
{
    uint64_t s2, n2, sum[4] = {0ull, 0ull, 0ull, 0ull};
    asm("mov.b64 %0, {%1, %1};" : "=l"(s2) : "f"(sl2));
    asm("mov.b64 %0, {%1, %1};" : "=l"(n2) : "f"(noff));
#pragma unroll
    for (int c = 0; c < 128; c += 32) {
        uint32_t pp[16], pl[16];
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
            float x0, x1;
            exp_pair(v[c + e], v[c + e + 1], s2, n2, sum[(e / 2) & 3], x0, x1);
            pp[e / 2] = pack_bf16(x0, x1);
            pl[e / 2] = pack_bf16_rest(x0, x1, pp[e / 2]);
        }
        tmem_st16(to + c / 2, pp);
        tmem_st16(to + 64 + c / 2, pl);
        if (c >= 64) {
            tmem_wait_st();
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(c == 64 ? early : last);
        }
    }
    return sum_of(sum);
}

// ---------------------------------------------------------------------------------------
// d = 64 and 128, P as two bf16 terms: the two softmax warpgroups take ALTERNATE key tiles.  Warpgroup w owns the S buffer w and
// an accumulator O_w of its own (tensor memory: S_0 128, S_1 128, O_0 d, O_1 d columns), and a thread owns a
// whole row of its tile: the row maximum needs no exchange, and while one warpgroup is loading, taking the
// maximum or storing P, the other one keeps the MUFU pipe busy with its exponentials.  Each warpgroup runs its
// own online softmax (m_w, l_w, O_w) over its tiles; the two partial results are merged once at the end:
// O = (2^(m_0 - m) O_0 + 2^(m_1 - m) O_1) / (2^(m_0 - m) l_0 + 2^(m_1 - m) l_1), m = max(m_0, m_1).
// Issue order of the single issuing thread: S(0), S(1), then per tile k: O_{k&1} += P(k) V(k), S(k+2).
// The issuing thread waits for P alone and commits S alone (why: tc_fwd_pair_kernel).  K(k+2) and V(k+2) report to the barrier of
// P(k), which it waits for before S(k+2); the loading thread takes S(k) complete as the release of their stages: K(k+2) goes
// where K(k) was, and O += P(k-2) V was issued before S(k), so V needs four stages.
template <int HD>
struct RowsCfg {
    static constexpr int NK = 2, NV = 4;
    static constexpr uint32_t kSlab = 128 * 128, kSlabs = HD / 64, kTile = kSlabs * kSlab;
    static constexpr uint32_t oQ = 0;
    static constexpr uint32_t oK = oQ + kTile;
    static constexpr uint32_t oV = oK + NK * kTile;
    static constexpr uint32_t oX = oV + NV * kTile;            // merge of the two partial softmaxes
    static constexpr uint32_t oBar = oX + 4 * 128 * 4;
    static constexpr uint32_t oMisc = oBar + 12 * 8;
    static constexpr uint32_t kUsed = oMisc + 64;
    static_assert(kUsed <= 227 * 1024 && 256 + 2 * HD <= 512, "layout of the row-per-thread forward");
    static constexpr uint32_t kBytes = kUsed < 117 * 1024 ? 117 * 1024 : kUsed;   // one CTA per SM: all of tensor memory
};
enum { F2_Q = 0, F2_K1 = 1, F2_V01 = 2, F2_S = 3, F2_PE = 5, F2_P = 7, F2_O = 9 };

// 384 threads: warps 0-7 softmax, warp 8 MMA issuer, warp 9 TMA producer, warps 10-11 only complete that warpgroup.
// Three warps per scheduler cap the launch at 168 registers; after launch the last warpgroup gives registers up and
// the softmax warpgroups take them (256 x 224 + 128 x 40 = 62,464 of the 384 x 168 = 64,512 the block holds), so
// that a thread can keep its whole row of 128 scores.
constexpr int kThreadsRows = kSoftmaxThreads + 128;
// P enters its product as two bf16 terms (columns 0-63 and 64-127 of S).
template <int HD, bool FINE>
__global__ void __launch_bounds__(kThreadsRows, 1)
tc_fwd_rows_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
                   const __grid_constant__ CUtensorMap mV, const FwdArgs a)
{
    using C = RowsCfg<HD>;
    constexpr int TKF = 128, NK = C::NK, NV = C::NV;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::oBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(smem + C::oMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + C::oMisc + 4);
    float *xm = reinterpret_cast<float *>(smem + C::oX);   // [2 warpgroups][128 rows] reference maxima
    float *xl = xm + 256;                                  // [2][128] row sums
    const Abort ab{abort_flag, a.status};

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int nt = (a.n + TQ - 1) / TQ;
    const int it = nt - 1 - (int)blockIdx.x / a.group;    // heaviest causal tiles first
    const long bh = (long)blockIdx.y * a.group + blockIdx.x % a.group;
    const int i0 = it * TQ, n = a.n;

    if ((smem_u32(smem) & 1023u) != 0) {
        chain_wait();
        if (tid == 0) atomicExch(a.status, 9u);
        return;
    }
    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(&bars[F2_Q], 1);
        mbar_init(&bars[F2_K1], 1);
        mbar_init(&bars[F2_V01], 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars[F2_S + b], 1);
            mbar_init(&bars[F2_PE + b], 4);
            mbar_init(&bars[F2_P + b], 5);   // four warps and the loading thread
            mbar_init(&bars[F2_O + b], 1);
        }
        fence_barrier_init();
        prefetch_tensormap(&mQ); prefetch_tensormap(&mK); prefetch_tensormap(&mV);
    }
    chain_wait();
    if (warp == 0) tmem_alloc(tmem_base_s, 512);
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    chain_release();
    if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) *a.status = 0u;
    const uint32_t tm = *tmem_base_s;
    const KeyIter<TKF> iter(a, it, bh);

    int niter = 0;   // number of valid key tiles (same in every role)
    for (int idx = 0; idx < iter.raw; ++idx) niter += iter.tile(idx) >= 0;

    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
      if (warp == 9) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            auto load = [&](uint32_t to, const CUtensorMap *m, uint64_t *bar, int row) {
#pragma unroll
                for (uint32_t sl = 0; sl < C::kSlabs; ++sl) tma_load_3d(smem + to + sl * C::kSlab, m, bar, sl * 64, row, (int)bh);
            };
            mbar_expect_tx(&bars[F2_Q], (niter > 0 ? 2 : 1) * C::kTile);
            load(C::oQ, &mQ, &bars[F2_Q], i0);
            int k = 0;
            bool go = true;
            for (int idx = 0; idx < iter.raw; ++idx) {
                const int jt = iter.tile(idx);
                if (jt < 0) continue;
                uint64_t *bar_k = k == 0 ? &bars[F2_Q] : &bars[F2_K1], *bar_v = &bars[F2_V01];
                if (k == 0) mbar_expect_tx(bar_v, (niter > 1 ? 2 : 1) * C::kTile);
                if (k == 1) mbar_expect_tx(bar_k, C::kTile);
                if (k >= 2) {
                    // S(k-2) is the newest completion its barrier can have here (S(k) needs the loads below)
                    if (!(go = mbar_wait(&bars[F2_S + (k & 1)], ((k - 2) >> 1) & 1, ab))) break;
                    bar_k = bar_v = &bars[F2_P + (k & 1)];
                    mbar_expect_tx(bar_k, 2 * C::kTile);
                }
                load(C::oK + k % NK * C::kTile, &mK, bar_k, jt * TKF);
                load(C::oV + k % NV * C::kTile, &mV, bar_v, jt * TKF);
                ++k;
            }
            // the last two tiles have nothing to load behind them
            for (int q = max(niter - 2, 0); q < niter && go; ++q) {
                go = mbar_wait(&bars[F2_S + (q & 1)], (q >> 1) & 1, ab);
                if (go) mbar_arrive(&bars[F2_P + (q & 1)]);
            }
        }
      } else if (warp == 8) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0 && niter == 0) mbar_wait(&bars[F2_Q], 0, ab);   // let the Q load land before exit
        if (lane == 0 && niter > 0) {
            constexpr uint32_t idesc_s = idesc_bf16(128, TKF, 0, 0);
            constexpr uint32_t idesc_o = idesc_bf16(128, HD, 0, 1);
            const uint32_t kQ = desc_lo_kmajor(smem_u32(smem + C::oQ));
            auto issue_S = [&](int k) {   // K of tile k is there
                const uint32_t kK = desc_lo_kmajor(smem_u32(smem + C::oK + (k % NK) * C::kTile));
#pragma unroll
                for (int kk = 0; kk < HD / 16; ++kk) {
                    const uint32_t off = (kk / 4) * (C::kSlab >> 4) + (kk % 4) * 2;
                    mma_ss_lo(tm + (k & 1) * 128, kQ + off, kK + off, idesc_s, kk > 0);
                }
                mma_commit(&bars[F2_S + (k & 1)]);
            };
            mbar_wait(&bars[F2_Q], 0, ab);
            tcgen05_fence_after();
            issue_S(0);
            if (niter > 1) {
                mbar_wait(&bars[F2_K1], 0, ab);
                tcgen05_fence_after();
                issue_S(1);
            }
            mbar_wait(&bars[F2_V01], 0, ab);
            for (int k = 0; k < niter; ++k) {
                const int b = k & 1;
                const uint32_t mV_ = desc_lo_mnmajor(smem_u32(smem + C::oV + (k % NV) * C::kTile), C::kSlab);
                const uint32_t tO = tm + 256 + b * HD, tP = tm + b * 128;
                mbar_wait(&bars[F2_PE + b], (k >> 1) & 1, ab);   // the first 96 keys, then the rest (and K, V of tile k + 2)
                tcgen05_fence_after();
                bool landed = true;
#pragma unroll
                for (int kk = 0; kk < TKF / 16; ++kk) {
                    if (kk == 6) {
                        landed = mbar_wait(&bars[F2_P + b], (k >> 1) & 1, ab);
                        tcgen05_fence_after();
                    }
                    mma_ts_lo(tO, tP + kk * 8, mV_ + kk * 128, idesc_o, (k > 1) || (kk > 0));
                    mma_ts_lo(tO, tP + 64 + kk * 8, mV_ + kk * 128, idesc_o, 1);
                }
                // the products execute in issue order: S(k+2) overwrites buffer b after P(k) has been consumed, and
                // its completion tells warpgroup b that O_b holds the product of tile k as well
                if (!landed) break;
                if (k + 2 < niter) issue_S(k + 2);
                else mma_commit(&bars[F2_O + b]);   // the last product of each warpgroup, for the epilogue
            }
        }
      }
    } else {
        // ------------------------------------------------------------ softmax warpgroup w: tiles k = w, w + 2, ...
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        const int w = warp / 4;
        const int row = (warp % 4) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp % 4) * 32) << 16;
        const int ig = i0 + row;
        const float sl2 = a.scale * kLog2e;
        const uint32_t T_S = tm + w * 128, T_O = tm + 256 + w * HD;
        float m_ref = -INFINITY, l_run = 0.f;
        int k = 0, cnt = 0;
        for (int idx = 0; idx < iter.raw; ++idx) {
            const int jt = iter.tile(idx);
            if (jt < 0) continue;
            if ((k++ & 1) != w) continue;
            const int j0 = jt * TKF;
            const bool causal = mask_is_causal(a.mask_kind);
            const bool need_mask = (causal && j0 + TKF - 1 > i0) || j0 + TKF > n || FINE;
            // a mask finer than the tile: the keep bits of this thread's query row, all four words in flight before the wait for S
            uint32_t kws[TKF / 32];
            if constexpr (FINE) {
#pragma unroll
                for (int q = 0; q < TKF / 32; ++q)
                    kws[q] = (ig < n && j0 + q * 32 < n) ? fine_word(a.fine, a.mask_heads, bh, true, ig, j0 + q * 32) : 0u;
            }
            const bool here = mbar_wait(&bars[F2_S + w], cnt & 1, ab);
            tcgen05_fence_after();
            // the whole row of raw scores in registers: four loads in flight, one wait
            uint32_t v[TKF];
#pragma unroll
            for (int c = 0; c < TKF; c += 32) tmem_ld32(T_S + lane_addr + c, *reinterpret_cast<uint32_t(*)[32]>(&v[c]));
            tmem_wait_ld();
            if (need_mask) {
                const bool edge = (causal && j0 + TKF - 1 > i0) || j0 + TKF > n;   // entries dropped by position as well
#pragma unroll
                for (int q = 0; q < TKF / 32; ++q) {
                    // a word that keeps all or nothing (the rule with 32- and 64-wide blocks) needs no test per entry
                    uint32_t kw = 0xffffffffu;
                    if constexpr (FINE) kw = kws[q];
                    if (FINE && !edge && kw == 0xffffffffu) continue;
                    if (FINE && kw == 0u) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[q * 32 + e] = 0xff800000u;   // -inf
                        continue;
                    }
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        const int jg = j0 + q * 32 + e;
                        if (jg >= n || (causal && jg > ig) || !((kw >> e) & 1u)) v[q * 32 + e] = 0xff800000u;
                    }
                }
            }
            const float m_tile = row_max(v) * sl2;   // scale > 0: the maximum commutes with it
            const bool need = m_tile > m_ref + kRescaleThreshold || (m_ref == -INFINITY && m_tile != -INFINITY);
            if (__any_sync(0xffffffffu, need)) {
                const float m_new = need ? fmaxf(m_ref, m_tile) : m_ref;
                const float alpha = (need && m_ref != -INFINITY) ? ex2_fast_f(m_ref - m_new) : 1.f;
                if (cnt > 0) {   // O_w += P V of this warpgroup's previous tile was issued before this tile's S: it has landed
#pragma unroll
                    for (int c = 0; c < HD; c += 16) {
                        uint32_t o[16];
                        tmem_ld16(T_O + lane_addr + c, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                        tmem_st16(T_O + lane_addr + c, o);
                    }
                }
                l_run *= alpha;
                m_ref = m_new;
            }
            const float noff = m_ref == -INFINITY ? 0.f : -m_ref;
            // P = exp2(S * scale * log2e - m_ref) as bf16 pairs over the first 64 columns of S (every thread
            // overwrites only its own lane, whose scores it already holds)
            l_run += exp_row_split(v, sl2, noff, T_S + lane_addr, &bars[F2_PE + w], &bars[F2_P + w], here ? lane : -1);
            ++cnt;
        }
        // ------------------------------------------------------------ epilogue: merge the two partial softmaxes
        xm[w * 128 + row] = m_ref;
        xl[w * 128 + row] = l_run;
        named_bar_sync_f(1, kSoftmaxThreads);
        const float m0 = xm[row], m1 = xm[128 + row], l0 = xl[row], l1 = xl[128 + row];
        const float m_all = fmaxf(m0, m1);
        const float a0 = m0 == -INFINITY ? 0.f : ex2_fast_f(m0 - m_all), a1 = m1 == -INFINITY ? 0.f : ex2_fast_f(m1 - m_all);
        const float l_tot = a0 * l0 + a1 * l1;
        const float inv = l_tot > 0.f ? 1.f / l_tot : 0.f;
        const float c0 = a0 * inv, c1 = a1 * inv;
        const int cnt0 = (niter + 1) / 2, cnt1 = niter / 2;
        if (cnt0 > 0) mbar_wait(&bars[F2_O], 0, ab);
        if (cnt1 > 0) mbar_wait(&bars[F2_O + 1], 0, ab);
        tcgen05_fence_after();
        const int ic = ig < n ? ig : 0;
        __nv_bfloat16 *po = a.O + ((size_t)bh * n + ic) * HD + w * (HD / 2);
#pragma unroll
        for (int c = 0; c < HD / 2; c += 32) {
            uint32_t v0[32], v1[32];
            if (cnt0 > 0) tmem_ld32(tm + 256 + lane_addr + w * (HD / 2) + c, v0);
            if (cnt1 > 0) tmem_ld32(tm + 256 + HD + lane_addr + w * (HD / 2) + c, v1);
            tmem_wait_ld();
            float o[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                // a partial accumulator that never received a product holds stale bits: select, do not multiply
                const float x0 = cnt0 > 0 ? __uint_as_float(v0[e]) * c0 : 0.f;
                const float x1 = cnt1 > 0 ? __uint_as_float(v1[e]) * c1 : 0.f;
                o[e] = x0 + x1;
            }
            if (ig < n) {
#pragma unroll
                for (int e = 0; e < 32; e += 8)
                    *reinterpret_cast<uint4 *>(po + c + e) = make_uint4(pack_bf16(o[e], o[e + 1]), pack_bf16(o[e + 2], o[e + 3]),
                                                                        pack_bf16(o[e + 4], o[e + 5]), pack_bf16(o[e + 6], o[e + 7]));
            }
        }
        if (w == 0 && ig < n) a.LSE[(size_t)bh * n + ig] = row_lse(m_all, l_tot);
    }
    tmem_leave(tm, 512, warp, ab);
}

// ---------------------------------------------------------------------------------------
// The same with 256 queries per CTA, for masks without lists.  Warpgroup w owns the query tile w and walks every key tile.  Tensor
// memory as above (S_0, S_1, O_0, O_1); nothing is merged at the end.  Issue order: S_0(0), S_1(0), then per key tile k:
// O_0 += P_0 V, S_0(k+1), O_1 += P_1 V, S_1(k+1).
//
// What bounds these kernels is the issuing thread.  While S = Q K^T streams both operands from shared memory, whose port that
// saturates, a barrier operation of this thread takes 110 to 200 cycles, done or not: with loads, releases and P on barriers of
// their own it spent 1,200 of a 3,990-cycle period (two tiles, d = 128) on them and was never idle.  Here it waits for nothing
// but P and commits nothing but S.  The loads of K(k+1) and V(k+1) report to the barrier of P_0(k), which the thread waits for
// anyway before S_0(k+1); the loading thread takes S_0(k) complete as the release of the stages they go to: S_1(k-1) and
// O_1 += P_1(k-2) V were issued before it, so two K stages and three V stages suffice.  S_0(k) is the newest completion its
// barrier can have there, so the parity wait cannot be a phase behind.
template <int HD>
struct PairCfg {
    static constexpr int NK = 2, NV = 3;                       // stages
    static constexpr uint32_t kSlab = 128 * 128, kSlabs = HD / 64, kTile = kSlabs * kSlab;
    static constexpr uint32_t oQ = 0;                          // two query tiles
    static constexpr uint32_t oK = oQ + 2 * kTile;
    static constexpr uint32_t oV = oK + NK * kTile;
    static constexpr uint32_t oBar = oV + NV * kTile;
    static constexpr uint32_t oMisc = oBar + 12 * 8;
    static constexpr uint32_t kUsed = oMisc + 64;
    static_assert(kUsed <= 227 * 1024, "shared memory budget");
    static constexpr uint32_t kBytes = kUsed < 117 * 1024 ? 117 * 1024 : kUsed;   // one CTA per SM: all of tensor memory
};
enum { F3_Q = 0, F3_V0 = 1, F3_S = 2, F3_PE = 4, F3_P = 6, F3_O = 8 };

template <int HD>
__global__ void __launch_bounds__(kThreadsRows, 1)
tc_fwd_pair_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
                   const __grid_constant__ CUtensorMap mV, const FwdArgs a)
{
    using C = PairCfg<HD>;
    constexpr int TKF = 128, NK = C::NK, NV = C::NV;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::oBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(smem + C::oMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + C::oMisc + 4);
    const Abort ab{abort_flag, a.status};

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int n = a.n;
    const int i0 = ((n + 255) / 256 - 1 - (int)blockIdx.x / a.group) * 256;   // heaviest causal tiles first
    const long bh = (long)blockIdx.y * a.group + blockIdx.x % a.group;
    const bool causal = mask_is_causal(a.mask_kind);

    if ((smem_u32(smem) & 1023u) != 0) {
        chain_wait();
        if (tid == 0) atomicExch(a.status, 9u);
        return;
    }
    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(&bars[F3_Q], 1);
        mbar_init(&bars[F3_V0], 1);
        for (int w = 0; w < 2; ++w) {
            mbar_init(&bars[F3_S + w], 1);
            mbar_init(&bars[F3_PE + w], 4);
            mbar_init(&bars[F3_P + w], w == 0 ? 5 : 4);   // four warps, P_0 also the loading thread
            mbar_init(&bars[F3_O + w], 1);
        }
        fence_barrier_init();
        prefetch_tensormap(&mQ); prefetch_tensormap(&mK); prefetch_tensormap(&mV);
    }
    chain_wait();
    if (warp == 0) tmem_alloc(tmem_base_s, 512);
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    chain_release();
    if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) *a.status = 0u;
    const uint32_t tm = *tmem_base_s;

    // key tiles of query tile w (the second one may lie beyond n)
    auto count = [&](int w) {
        const int first = i0 + w * TQ;
        if (first >= n) return 0;
        return causal ? (min(first + TQ, n) - 1) / TKF + 1 : (n + TKF - 1) / TKF;
    };
    const int n0 = count(0), n1 = count(1), most = max(n0, n1);   // n0 > 0

    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
      if (warp == 9) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            auto load = [&](uint32_t to, const CUtensorMap *m, uint64_t *bar, int row) {
#pragma unroll
                for (uint32_t sl = 0; sl < C::kSlabs; ++sl) tma_load_3d(smem + to + sl * C::kSlab, m, bar, sl * 64, row, (int)bh);
            };
            mbar_expect_tx(&bars[F3_Q], (n1 > 0 ? 3 : 2) * C::kTile);
            load(C::oQ, &mQ, &bars[F3_Q], i0);
            load(C::oK, &mK, &bars[F3_Q], 0);
            if (n1 > 0) load(C::oQ + C::kTile, &mQ, &bars[F3_Q], i0 + TQ);
            mbar_expect_tx(&bars[F3_V0], C::kTile);
            load(C::oV, &mV, &bars[F3_V0], 0);
            for (int k = 0; k < n0; ++k) {
                // the loads before have landed (P_0(k-1), known from S_0(k) unless the CTA is giving up)
                if (!mbar_wait(&bars[F3_P], (k - 1) & 1, ab) || !mbar_wait(&bars[F3_S], k & 1, ab)) break;
                if (k + 1 < most) {
                    mbar_expect_tx(&bars[F3_P], 2 * C::kTile);
                    load(C::oK + (k + 1) % NK * C::kTile, &mK, &bars[F3_P], (k + 1) * TKF);
                    load(C::oV + (k + 1) % NV * C::kTile, &mV, &bars[F3_P], (k + 1) * TKF);
                } else {
                    mbar_arrive(&bars[F3_P]);
                }
            }
        }
      } else if (warp == 8) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc_s = idesc_bf16(128, TKF, 0, 0);
            constexpr uint32_t idesc_o = idesc_bf16(128, HD, 0, 1);
            const uint32_t kQ = desc_lo_kmajor(smem_u32(smem + C::oQ));
            auto issue_S = [&](int w, int k) {   // K of tile k is there: waited for with P_0(k-1), V with it
                const uint32_t kK = desc_lo_kmajor(smem_u32(smem + C::oK + (k % NK) * C::kTile));
#pragma unroll
                for (int kk = 0; kk < HD / 16; ++kk) {
                    const uint32_t off = (kk / 4) * (C::kSlab >> 4) + (kk % 4) * 2;
                    mma_ss_lo(tm + w * 128, kQ + w * (C::kTile >> 4) + off, kK + off, idesc_s, kk > 0);
                }
                mma_commit(&bars[F3_S + w]);
            };
            auto issue_O = [&](int w, int k) {
                const uint32_t mV_ = desc_lo_mnmajor(smem_u32(smem + C::oV + (k % NV) * C::kTile), C::kSlab);
                const uint32_t tO = tm + 256 + w * HD, tP = tm + w * 128;
                mbar_wait(&bars[F3_PE + w], k & 1, ab);   // the first 96 keys, then the rest
                tcgen05_fence_after();
#pragma unroll
                for (int kk = 0; kk < TKF / 16; ++kk) {
                    if (kk == 6) {
                        mbar_wait(&bars[F3_P + w], k & 1, ab);
                        tcgen05_fence_after();
                    }
                    mma_ts_lo(tO, tP + kk * 8, mV_ + kk * 128, idesc_o, (k > 0) || (kk > 0));
                    mma_ts_lo(tO, tP + 64 + kk * 8, mV_ + kk * 128, idesc_o, 1);
                }
            };
            mbar_wait(&bars[F3_Q], 0, ab);
            tcgen05_fence_after();
            issue_S(0, 0);
            if (n1 > 0) issue_S(1, 0);
            mbar_wait(&bars[F3_V0], 0, ab);
            for (int k = 0; k < most; ++k) {
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    const int mine = w == 0 ? n0 : n1;
                    if (k >= mine) continue;
                    // the products execute in issue order: S_w(k+1) overwrites P_w(k) after it has been consumed, and its
                    // completion tells warpgroup w that O_w holds the product of tile k as well
                    issue_O(w, k);
                    if (k + 1 < mine) issue_S(w, k + 1);
                    else mma_commit(&bars[F3_O + w]);
                }
            }
        }
      }
    } else {
        // ------------------------------------------------------------ softmax warpgroup w: query tile w
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        const int w = warp / 4;
        const int row = (warp % 4) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp % 4) * 32) << 16;
        const int iw = i0 + w * TQ, ig = iw + row, mine = w == 0 ? n0 : n1;
        const float sl2 = a.scale * kLog2e;
        const uint32_t T_S = tm + w * 128, T_O = tm + 256 + w * HD;
        float m_ref = -INFINITY, l_run = 0.f;
        for (int k = 0; k < mine; ++k) {
            const int j0 = k * TKF;
            const bool here = mbar_wait(&bars[F3_S + w], k & 1, ab);
            tcgen05_fence_after();
            uint32_t v[TKF];   // the whole row of raw scores in registers: four loads in flight, one wait
#pragma unroll
            for (int c = 0; c < TKF; c += 32) tmem_ld32(T_S + lane_addr + c, *reinterpret_cast<uint32_t(*)[32]>(&v[c]));
            tmem_wait_ld();
            if ((causal && j0 + TKF - 1 > iw) || j0 + TKF > n) {
                const int keep = min(n, causal ? ig + 1 : n) - j0;   // the row keeps its first `keep` entries of the tile
#pragma unroll
                for (int e = 0; e < TKF; ++e)
                    if (e >= keep) v[e] = 0xff800000u;   // -inf
            }
            const float m_tile = row_max(v) * sl2;   // scale > 0: the maximum commutes with it
            const bool need = m_tile > m_ref + kRescaleThreshold || (m_ref == -INFINITY && m_tile != -INFINITY);
            const float m_new = need ? fmaxf(m_ref, m_tile) : m_ref;
            if (__any_sync(0xffffffffu, need)) {
                const float alpha = (need && m_ref != -INFINITY) ? ex2_fast_f(m_ref - m_new) : 1.f;
                if (k > 0) {   // O_w += P V of the previous tile was issued before this tile's S_w: it has landed
#pragma unroll
                    for (int c = 0; c < HD; c += 32) {
                        uint32_t o[32];
                        tmem_ld32(T_O + lane_addr + c, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                        tmem_st32(T_O + lane_addr + c, o);
                    }
                }
                l_run *= alpha;
                m_ref = m_new;
            }
            const float noff = m_ref == -INFINITY ? 0.f : -m_ref;
            l_run += exp_row_split(v, sl2, noff, T_S + lane_addr, &bars[F3_PE + w], &bars[F3_P + w], here ? lane : -1);
        }
        // ------------------------------------------------------------ epilogue
        if (mine > 0) {
            const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
            mbar_wait(&bars[F3_O + w], 0, ab);
            tcgen05_fence_after();
            const int ic = ig < n ? ig : 0;
            __nv_bfloat16 *po = a.O + ((size_t)bh * n + ic) * HD;
#pragma unroll
            for (int c = 0; c < HD; c += 32) {
                uint32_t o[32];
                tmem_ld32(T_O + lane_addr + c, o);
                tmem_wait_ld();
                if (ig < n) {
#pragma unroll
                    for (int e = 0; e < 32; e += 8) {
                        float x[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) x[u] = __uint_as_float(o[e + u]) * inv;
                        *reinterpret_cast<uint4 *>(po + c + e) = make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]),
                                                                            pack_bf16(x[4], x[5]), pack_bf16(x[6], x[7]));
                    }
                }
            }
            if (ig < n) a.LSE[(size_t)bh * n + ig] = row_lse(m_ref, l_run);
        }
    }
    tmem_leave(tm, 512, warp, ab);
}

// ---------------------------------------------------------------------------------------
// d = 64 and 128, P as one bf16 term.  PAIR: two query tiles, warpgroup w owns tile w and walks every key tile; otherwise one
// query tile whose key tiles the warpgroups take in turn (as in tc_fwd_rows_kernel, merged at the end).
//
// S = Q K^T goes into a buffer X that no P is written to (tensor memory, d = 128: X 128 columns, P_0, P_1 64 each, O_0, O_1 128
// each; d = 64: two buffers X).  The warpgroup copies its row into registers and gives X back, so that the next S is formed
// under its exponentials, and P goes to columns of its own, free once the product before has read them.  With P over S (the
// kernels above) S of the next tile waits for P and its product: a chain of 3,290 cycles a tile and warpgroup, period of
// two tiles 3,800; here a warpgroup's chain is 2,100 (wait seen 130, copy and maximum 550, exponentials 1,420) and the
// period 3,030.  Bound now, d = 128: the one X (S 690, seen and copied 400, given back and seen 150 to 300, for each of two
// warpgroups); d = 64: the warpgroup's own chain, the MUFU pipe 70 % busy.
// Two issuing threads: A forms S, B adds P V; nothing orders their products but the barriers of X and P.
// 32 heads, n = 8192, d = 128, causal: 566 -> 525 us; block-sparse, 32 heads, n = 32768, 10 %: 1844 -> 1794 us; 24 heads,
// n = 3000, d = 64, one query tile: 109 -> 105 us; 64 heads, n = 2048, d = 64: 127 us both.
//
// A CTA stays on its SM and takes the block indices of CTAs that have not started yet (cluster launch control), in the order of
// the launch.  The loading warp publishes each unit of work in one of two slots; every role walks from one unit to the next by
// itself, with its barriers running on: Q of the next unit is loaded once the last S of this one has been formed, and its first
// S is there when a warpgroup has written its O.  With a CTA per unit 7.4 to 7.8 us a CTA passed outside its tiles (launch 0.7,
// set-up 0.6, lists and first loads 1.5 to 3.0, epilogue and the slower warpgroup 3.0 to 4.5), as long as five tiles take.
// 32 heads, n = 8192, d = 128, causal: 450 -> 432 us; 32 heads, n = 4096: 133 -> 121; block-sparse as above: 1794 -> 1605;
// block-sparse and causal, 16 heads, n = 8192, 20 %: 129 -> 84; window of 512 keys, 16 heads, n = 4096: 66 -> 64, and 51 with the
// keep words fetched a tile ahead and tested by one predicate an entry; 64 heads, n = 2048, d = 64: 127 -> 119 (a session at
// full clock, kernel alone).
//
// A row's largest probabilities are what the rounding of P to bf16 costs most, and the one that the reference was taken from is
// exactly 1.  Two partial softmaxes a row (one query tile) have two such entries, one softmax has one, and its O is one per cent further
// from 64 bits.  So the first kExactTiles tiles after the first one move the reference (up, by less than one unit beyond what the
// maximum asks for) to where their largest entry is a power of two.  Error of O, 32 heads, n = 4096, d = 128, causal, against
// the two partial softmaxes': 1.010 times without, 0.994 with two exact tiles (1.000 with one, emulated).  It costs
// two rescalings of O per query tile (32 heads, n = 8192, d = 128, causal: 574 -> 584 us with 16 columns at a time, 573 with 32).
constexpr unsigned kExactTiles = 2;   // PAIR
template <int HD, bool PAIR>
struct FlowCfg {
    static constexpr int NQ = PAIR ? 2 : 1;                    // query tiles
    static constexpr int NK = PAIR ? 2 : 3, NV = 3;            // stages
    static constexpr int NX = HD == 64 ? 2 : 1;                // S buffers
    static constexpr uint32_t kSlab = 128 * 128, kSlabs = HD / 64, kTile = kSlabs * kSlab;
    static constexpr uint32_t oQ = 0;
    static constexpr uint32_t oK = oQ + NQ * kTile;
    static constexpr uint32_t oV = oK + NK * kTile;
    static constexpr uint32_t oX = oV + NV * kTile;            // merge of the two partial softmaxes (one query tile)
    static constexpr uint32_t oBar = oX + (PAIR ? 0 : 4 * 128 * 4);
    static constexpr uint32_t oWork = oBar + 32 * 8;           // two slots of FlowWork, the answer of the scheduler
    static constexpr uint32_t oMisc = oWork + 2 * 32 + 16;
    static constexpr uint32_t kUsed = oMisc + 16;
    static_assert(kUsed <= 227 * 1024, "shared memory budget");
    static constexpr uint32_t kBytes = kUsed < 117 * 1024 ? 117 * 1024 : kUsed;   // one CTA per SM: all of tensor memory
    static constexpr uint32_t tP = NX * 128, tO = tP + 128;    // tensor-memory columns
    static_assert(tO + 2 * HD == 512, "tensor memory");
};
enum { F4_QF = 0, F4_QE = 2, F4_KF = 4, F4_KE = 7, F4_VF = 10, F4_VE = 13, F4_S = 16, F4_O = 18, F4_CLC = 20, F4_WF = 21, F4_WE = 23,
       F4_XF = 25, F4_PE = 27, F4_P = 29, F4_COUNT = 31 };

// One unit of work: a query tile (or two) of one head
struct FlowWork {
    int tile, bh;      // query tile (or two) of that many rows; -1: there is no more work
    int n0, n1;        // items of the warpgroups
    const int *cols;   // key blocks of a mask with lists
    int pad[2];
};
static_assert(sizeof(FlowWork) == 32, "two slots in shared memory");

// P = exp2(v * sl2 + noff) as bf16 pairs into columns of its own; returns the sum of the row of P before rounding.  `free` waits
// until the columns may be written, by when 64 keys are ready.  The first 96 keys are handed over (`early`, one arrival per
// warp) as soon as they are stored: their part of O += P V is formed under the exponentials of the rest.
template <typename Free>
__device__ __forceinline__ float exp_row(const uint32_t (&v)[128], float sl2, float noff, uint32_t to, uint64_t *early, uint64_t *last, int lane, Free &&free)
{
    uint64_t s2, n2, sum[4] = {0ull, 0ull, 0ull, 0ull};
    asm("mov.b64 %0, {%1, %1};" : "=l"(s2) : "f"(sl2));
    asm("mov.b64 %0, {%1, %1};" : "=l"(n2) : "f"(noff));
    auto pair = [&](int c) {
        float x0, x1;
        exp_pair(v[c], v[c + 1], s2, n2, sum[(c / 2) & 3], x0, x1);
        return pack_bf16(x0, x1);
    };
    {
        uint32_t pp[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) pp[e] = pair(2 * e);
        free();
        tmem_st32(to, pp);
    }
#pragma unroll
    for (int c = 64; c < 128; c += 32) {
        uint32_t pp[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) pp[e] = pair(c + 2 * e);
        tmem_st16(to + c / 2, pp);
        tmem_wait_st();
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(c == 64 ? early : last);
    }
    return sum_of(sum);
}

template <int HD, bool PAIR, bool FINE>
__global__ void __launch_bounds__(kThreadsRows, 1)
tc_fwd_flow_kernel(const __grid_constant__ CUtensorMap mQ, const __grid_constant__ CUtensorMap mK,
                   const __grid_constant__ CUtensorMap mV, const FwdArgs a)
{
    using C = FlowCfg<HD, PAIR>;
    constexpr int TKF = 128, NK = C::NK, NV = C::NV, NX = C::NX, QROWS = C::NQ * TQ;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::oBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(smem + C::oMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + C::oMisc + 4);
    volatile FlowWork *slots = reinterpret_cast<volatile FlowWork *>(smem + C::oWork);
    float *xm = reinterpret_cast<float *>(smem + C::oX);   // !PAIR: [2 warpgroups][128 rows] reference maxima
    float *xl = xm + 256;                                  // [2][128] row sums
    const Abort ab{abort_flag, a.status};

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int n = a.n;
    const bool causal = mask_is_causal(a.mask_kind), lists = mask_is_block(a.mask_kind);
    const int sub = lists ? a.block / TKF : 1;

    if ((smem_u32(smem) & 1023u) != 0) {
        chain_wait();
        if (tid == 0) atomicExch(a.status, 9u);
        return;
    }
    if (tid == 0) {
        *abort_flag = 0;
        for (int b = 0; b < F4_COUNT; ++b)   // XF, PE, P: the four warps of a warpgroup; WE: both issuers and eight warps
            mbar_init(&bars[b], b >= F4_XF ? 4 : b >= F4_WE ? 10 : 1);
        fence_barrier_init();
        prefetch_tensormap(&mQ); prefetch_tensormap(&mK); prefetch_tensormap(&mV);
    }
    chain_wait();
    if (warp == 0) tmem_alloc(tmem_base_s, 512);
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    chain_release();
    if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) *a.status = 0u;
    const uint32_t tm = *tmem_base_s;

    // Items of a unit of work in the order in which their S is formed.  PAIR: (query tile w, key tile k) = (0, 0), (1, 0), (0, 1),
    // ..., then what one query tile has left; otherwise item k is key tile k of warpgroup k % 2.
    struct Order {
        int both, items, tiles;
        bool zero;   // the rest belongs to warpgroup 0
        __device__ Order(int n0, int n1) : both(min(n0, n1)), items(n0 + n1), tiles(PAIR ? max(n0, n1) : n0 + n1), zero(n0 > n1) {}
        __device__ int item(int w, int c) const { return c < both ? 2 * c + w : both + c; }   // c-th item of warpgroup w
        __device__ int group(int i) const { return i < 2 * both ? i & 1 : zero ? 0 : 1; }
        __device__ int nth(int i) const { return i < 2 * both ? i >> 1 : i - both; }          // its index there
        __device__ int tile(int i) const { return PAIR ? nth(i) : i; }
        __device__ bool begins(int i) const { return !PAIR || i >= 2 * both || (i & 1) == 0; }  // the first item of its key tile
        __device__ bool ends(int i) const { return !PAIR || i >= 2 * both || (i & 1) != 0; }    // the last one
    };
    // the t-th unit of work of this CTA as the loading warp has published it
    const UnitQueue<FlowWork, UnitIo<kSoftmaxThreads>> units{slots, &bars[F4_WF], &bars[F4_WE], &bars[F4_CLC], smem + C::oWork + 2 * sizeof(FlowWork), {ab}};
    auto unit = [&](int t) {
        const volatile FlowWork &v = slots[t & 1];
        return FlowWork{v.tile, v.bh, v.n0, v.n1, v.cols, {}};
    };

    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
      if (warp == 9) {
        // ------------------------------------------------------------ TMA producer, and the schedule
        auto load = [&](uint32_t to, const CUtensorMap *m, uint64_t *bar, int row, int bh) {
            mbar_expect_tx(bar, C::kTile);
#pragma unroll
            for (uint32_t sl = 0; sl < C::kSlabs; ++sl) tma_load_3d(smem + to + sl * C::kSlab, m, bar, sl * 64, row, bh);
        };
        int bx = blockIdx.x, by = blockIdx.y;
        int kt = 0;                // key tiles loaded so far
        int nq0 = 0, nq1 = 0;      // loads of each Q buffer so far
        bool more = true;
        for (int t = 0; more; ++t) {
            const int tile = (n + QROWS - 1) / QROWS - 1 - bx / a.group, i0 = tile * QROWS;   // heaviest causal tiles first
            const int bh = by * a.group + bx % a.group;
            int n0, n1;
            const int *cols = nullptr;
            if constexpr (PAIR) {
                auto count = [&](int w) {   // key tiles of query tile w (the second one may lie beyond n)
                    const int first = i0 + w * TQ;
                    if (first >= n) return 0;
                    return causal ? (min(first + TQ, n) - 1) / TKF + 1 : (n + TKF - 1) / TKF;
                };
                n0 = count(0), n1 = count(1);
            } else {
                int kept = 0;
                const int last_i = min(i0 + TQ, n) - 1;
                if (lists) {
                    // the lists ascend, so what lies beyond n or (block mask AND causal) begins after the last query is at their end
                    const long mh = a.mask_heads == 1 ? 0 : bh;
                    const int *rp = a.row_ptr + mh * 2 * a.nb + 2 * (i0 / a.block);
                    const int first = rp[0], raw = (rp[1] - first) * sub, limit = causal ? last_i : n - 1;
                    cols = a.col_idx + mh * (long)a.nb * a.nb + first;
                    for (int e = lane; e < raw; e += 32) kept += (cols[e / sub] * sub + e % sub) * TKF <= limit;
                    kept = __reduce_add_sync(0xffffffffu, kept);
                } else {
                    kept = causal ? last_i / TKF + 1 : (n + TKF - 1) / TKF;
                }
                n0 = (kept + 1) / 2, n1 = kept / 2;
            }
            const Order o(n0, n1);
            auto load_unit = [&]() -> bool {   // false: there is no further unit, or the kernel is giving up
                volatile FlowWork *f = units.claim(t);
                if (!f) return false;
                f->tile = tile; f->bh = bh; f->n0 = n0; f->n1 = n1; f->cols = cols;
                units.publish(t);
                if (o.items > 0) {
                    if (nq0 > 0 && !mbar_wait(&bars[F4_QE], (nq0 - 1) & 1, ab)) return false;
                    load(C::oQ, &mQ, &bars[F4_QF], i0, bh);
                    ++nq0;
                }
                int jt = lists && o.tiles > 0 ? cols[0] * sub : 0;
                for (int k = 0; k < o.tiles; ++k, ++kt) {
                    const int sk = kt % NK, sv = kt % NV;
                    const int here = jt;
                    if (k + 1 < o.tiles) jt = lists ? cols[(k + 1) / sub] * sub + (k + 1) % sub : k + 1;
                    if (k == max(o.tiles - 2, 0)) units.ask();
                    if (kt >= NK && !mbar_wait(&bars[F4_KE + sk], (kt / NK - 1) & 1, ab)) return false;
                    load(C::oK + sk * C::kTile, &mK, &bars[F4_KF + sk], here * TKF, bh);
                    if (PAIR && k == 0 && n1 > 0) {
                        if (nq1 > 0 && !mbar_wait(&bars[F4_QE + 1], (nq1 - 1) & 1, ab)) return false;
                        load(C::oQ + C::kTile, &mQ, &bars[F4_QF + 1], i0 + TQ, bh);
                        ++nq1;
                    }
                    if (kt >= NV && !mbar_wait(&bars[F4_VE + sv], (kt / NV - 1) & 1, ab)) return false;
                    load(C::oV + sv * C::kTile, &mV, &bars[F4_VF + sv], here * TKF, bh);
                }
                if (o.tiles == 0) units.ask();
                return units.next(t, bx, by);
            };
            if (lane == 0) more = load_unit();
            __syncwarp();
            more = __shfl_sync(0xffffffffu, (int)more, 0) != 0;
            bx = __shfl_sync(0xffffffffu, bx, 0);
            by = __shfl_sync(0xffffffffu, by, 0);
        }
      } else if (warp == 8) {
        // ------------------------------------------------------------ MMA issuer A: S = Q K^T
        if (lane == 0) {
            constexpr uint32_t idesc_s = idesc_bf16(128, TKF, 0, 0);
            const uint32_t kQ = desc_lo_kmajor(smem_u32(smem + C::oQ));
            int g = 0, kt0 = 0, last_w = -1;   // items and key tiles before this unit of work; warpgroup of the item before
            int nq0 = 0, nq1 = 0;
            for (int t = 0; units.take_alone(t); ++t) {
                const FlowWork f = unit(t);
                mbar_arrive(&bars[F4_WE + (t & 1)]);
                const Order o(f.n0, f.n1);
                for (int i = 0; i < o.items; ++i, ++g) {
                    const int w = o.group(i), k = kt0 + o.tile(i), x = g % NX;
                    const int q = PAIR ? w : 0;
                    if (i == 0 || (PAIR && i == 1 && w == 1)) {
                        if (!mbar_wait(&bars[F4_QF + q], (q == 0 ? nq0 : nq1) & 1, ab)) break;
                        if (q == 0) ++nq0; else ++nq1;
                    }
                    if (o.begins(i) && !mbar_wait(&bars[F4_KF + k % NK], (k / NK) & 1, ab)) break;
                    if (g >= NX) mbar_wait(&bars[F4_XF + x], (g / NX - 1) & 1, ab);
                    // two items of one warpgroup in a row: the barrier of its S may not complete a second time before it has seen the first
                    if (NX > 1 && w == last_w) mbar_wait(&bars[F4_XF + (g - 1) % NX], ((g - 1) / NX) & 1, ab);
                    last_w = w;
                    tcgen05_fence_after();
                    const uint32_t kK = desc_lo_kmajor(smem_u32(smem + C::oK + (k % NK) * C::kTile));
                    const uint32_t kQw = kQ + q * (C::kTile >> 4);
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        const uint32_t off = (kk / 4) * (C::kSlab >> 4) + (kk % 4) * 2;
                        mma_ss_lo(tm + x * 128, kQw + off, kK + off, idesc_s, kk > 0);
                    }
                    mma_commit(&bars[F4_S + w]);
                    if (o.ends(i)) mma_commit(&bars[F4_KE + k % NK]);
                    if (PAIR ? o.nth(i) + 1 == (w == 0 ? f.n0 : f.n1) : i + 1 == o.items) mma_commit(&bars[F4_QE + q]);
                }
                kt0 += o.tiles;
            }
        }
      } else if (warp == 10) {
        // ------------------------------------------------------------ MMA issuer B: O += P V
        if (lane == 0) {
            constexpr uint32_t idesc_o = idesc_bf16(128, HD, 0, 1);
            int kt0 = 0, c0 = 0, c1 = 0;   // key tiles and items of each warpgroup before this unit of work
            for (int t = 0; units.take_alone(t); ++t) {
                const FlowWork f = unit(t);
                mbar_arrive(&bars[F4_WE + (t & 1)]);
                const Order o(f.n0, f.n1);
                for (int i = 0; i < o.items; ++i) {
                    const int w = o.group(i), c = o.nth(i), k = kt0 + o.tile(i);
                    const uint32_t parity = (c + (w == 0 ? c0 : c1)) & 1;
                    const uint32_t mV_ = desc_lo_mnmajor(smem_u32(smem + C::oV + (k % NV) * C::kTile), C::kSlab);
                    const uint32_t tO = tm + C::tO + w * HD, tP = tm + C::tP + w * 64;
                    if (o.begins(i) && !mbar_wait(&bars[F4_VF + k % NV], (k / NV) & 1, ab)) break;
                    mbar_wait(&bars[F4_PE + w], parity, ab);   // the first 96 keys, then the rest
                    tcgen05_fence_after();
#pragma unroll
                    for (int kk = 0; kk < TKF / 16; ++kk) {
                        if (kk == 6) {
                            mbar_wait(&bars[F4_P + w], parity, ab);
                            tcgen05_fence_after();
                        }
                        mma_ts_lo(tO, tP + kk * 8, mV_ + kk * 128, idesc_o, (c > 0) || (kk > 0));
                    }
                    if (o.ends(i)) mma_commit(&bars[F4_VE + k % NV]);
                    mma_commit(&bars[F4_O + w]);
                }
                kt0 += o.tiles;
                c0 += f.n0;
                c1 += f.n1;
            }
        }
      }
    } else {
        // ------------------------------------------------------------ softmax warpgroup w
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        const int w = warp / 4;
        const int row = (warp % 4) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp % 4) * 32) << 16;
        const float sl2 = a.scale * kLog2e;
        const uint32_t T_P = tm + C::tP + w * 64 + lane_addr, T_O = tm + C::tO + w * HD + lane_addr;
        const bool wide = ((uintptr_t)a.O & 31) == 0;
        int g0 = 0, c0 = 0;   // items of both warpgroups and of this one before this unit of work
        // one query tile: the warpgroups meet at a named barrier for the merge, so all their warps take a unit or none does
        bool more = PAIR ? units.take(0) : units.take_together(0);
        for (int t = 0; more; ++t) {
            const FlowWork f = unit(t);
            warp_arrive_f(&bars[F4_WE + (t & 1)], lane);
            const Order o(f.n0, f.n1);
            const int iw = f.tile * QROWS + (PAIR ? w * TQ : 0), ig = iw + row, mine = w == 0 ? f.n0 : f.n1;
            const long bh = f.bh;
            float m_ref = -INFINITY, l_run = 0.f;
            // key tiles of this warpgroup's next two items and the keep bits of the next one are fetched ahead
            auto tile_at = [&](int c) {
                if (PAIR || !lists) return PAIR ? c : o.item(w, c);
                const int i = min(o.item(w, c), o.items - 1);
                return sub == 1 ? f.cols[i] : f.cols[i / sub] * sub + i % sub;
            };
            auto keep_words = [&](int j0, uint32_t (&to)[TKF / 32]) {
                const int last = min(n - 1, causal ? ig : n - 1);   // of the keys that the row may keep by position
#pragma unroll
                for (int q = 0; q < TKF / 32; ++q) {
                    const int left = last - (j0 + q * 32);
                    to[q] = ig < n && left >= 0 ? fine_word(a.fine, a.mask_heads, bh, true, ig, j0 + q * 32) & (0xffffffffu >> (31 - min(left, 31))) : 0u;
                }
            };
            int jt = mine > 0 ? tile_at(0) : 0, jt1 = mine > 1 ? tile_at(1) : 0;
            uint32_t kws[TKF / 32], kws1[TKF / 32];
            if constexpr (FINE) {
                if (mine > 0) keep_words(jt * TKF, kws);
            }
            for (int c = 0; c < mine; ++c) {
                const int x = (g0 + o.item(w, c)) % NX;
                const int j0 = jt * TKF;
                const bool edge = (causal && j0 + TKF - 1 > iw) || j0 + TKF > n;   // entries dropped by position
                jt = jt1;
                if (c + 2 < mine) jt1 = tile_at(c + 2);
                if constexpr (FINE) {
                    if (c + 1 < mine) keep_words(jt * TKF, kws1);
                }
                mbar_wait(&bars[F4_S + w], (c0 + c) & 1, ab);
                tcgen05_fence_after();
                uint32_t v[TKF];   // the whole row of raw scores in registers: four loads in flight, one wait
#pragma unroll
                for (int e = 0; e < TKF; e += 32) tmem_ld32(tm + x * 128 + lane_addr + e, *reinterpret_cast<uint32_t(*)[32]>(&v[e]));
                tmem_wait_ld();
                tcgen05_fence_before();
                warp_arrive_f(&bars[F4_XF + x], lane);   // the buffer may take the next S
                if constexpr (FINE) {
#pragma unroll
                    for (int q = 0; q < TKF / 32; ++q) {
                        if (__all_sync(0xffffffffu, kws[q] == 0xffffffffu)) continue;
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (!(kws[q] & (1u << e))) v[q * 32 + e] = 0xff800000u;   // -inf
                    }
                } else if (edge) {
                    const int keep = min(n, causal ? ig + 1 : n) - j0;   // the row keeps its first `keep` entries of the tile
#pragma unroll
                    for (int e = 0; e < TKF; ++e)
                        if (e >= keep) v[e] = 0xff800000u;   // -inf
                }
                const float m_tile = row_max(v) * sl2;   // scale > 0: the maximum commutes with it
                bool need = m_tile > m_ref + kRescaleThreshold || (m_ref == -INFINITY && m_tile != -INFINITY);
                float m_new = need ? fmaxf(m_ref, m_tile) : m_ref;
                if (PAIR && c - 1u < kExactTiles && m_ref != -INFINITY && m_tile != -INFINITY) {
                    // the next reference from which the tile's maximum is a whole number of powers of two away, by less than one
                    // unit up also where the sum is rounded (references of 2^24 and more)
                    m_new = m_tile > m_ref ? m_tile : fminf(fmaxf(m_tile + ceilf(m_ref - m_tile), m_ref), m_ref + 1.f);
                    need = true;
                }
                // O_w += P V of this warpgroup's previous item: it reads P_w and adds to O_w
                bool landed = c == 0;
                auto wait_landed = [&] {
                    if (!landed) {
                        mbar_wait(&bars[F4_O + w], (c0 + c - 1) & 1, ab);
                        tcgen05_fence_after();
                        landed = true;
                    }
                };
                if (__any_sync(0xffffffffu, need)) {
                    const float alpha = (need && m_ref != -INFINITY) ? ex2_fast_f(m_ref - m_new) : 1.f;
                    if (c > 0) {
                        wait_landed();
#pragma unroll
                        for (int e0 = 0; e0 < HD; e0 += 32) {
                            uint32_t ov[32];
                            tmem_ld32(T_O + e0, ov);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; ++e) ov[e] = __float_as_uint(__uint_as_float(ov[e]) * alpha);
                            tmem_st32(T_O + e0, ov);
                        }
                    }
                    l_run *= alpha;
                    m_ref = m_new;
                }
                const float noff = m_ref == -INFINITY ? 0.f : -m_ref;
                l_run += exp_row(v, sl2, noff, T_P, &bars[F4_PE + w], &bars[F4_P + w], lane, wait_landed);
                if constexpr (FINE) {
#pragma unroll
                    for (int q = 0; q < TKF / 32; ++q) kws[q] = kws1[q];
                }
            }
            g0 += o.items;
            c0 += mine;
            // -------------------------------------------------------- epilogue, while S of the next unit of work is formed
            const int ic = ig < n ? ig : 0;
            if constexpr (PAIR) {
                if (mine > 0) {
                    const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
                    mbar_wait(&bars[F4_O + w], (c0 - 1) & 1, ab);
                    tcgen05_fence_after();
                    __nv_bfloat16 *po = a.O + ((size_t)bh * n + ic) * HD;
#pragma unroll
                    for (int e0 = 0; e0 < HD; e0 += 32) {
                        uint32_t ov[32];
                        tmem_ld32(T_O + e0, ov);
                        tmem_wait_ld();
                        if (ig < n) {
#pragma unroll
                            for (int e = 0; e < 32; e += 16) {
                                uint32_t y[8];
#pragma unroll
                                for (int u = 0; u < 8; ++u)
                                    y[u] = pack_bf16(__uint_as_float(ov[e + 2 * u]) * inv, __uint_as_float(ov[e + 2 * u + 1]) * inv);
                                store32(po + e0 + e, y, wide);
                            }
                        }
                    }
                    if (ig < n) a.LSE[(size_t)bh * n + ig] = row_lse(m_ref, l_run);
                }
                more = units.take(t + 1);
            } else {
                // merge the two partial softmaxes
                xm[w * 128 + row] = m_ref;
                xl[w * 128 + row] = l_run;
                named_bar_sync_f(1, kSoftmaxThreads);
                const float m0 = xm[row], m1 = xm[128 + row], l0 = xl[row], l1 = xl[128 + row];
                const float m_all = fmaxf(m0, m1);
                const float a0 = m0 == -INFINITY ? 0.f : ex2_fast_f(m0 - m_all), a1 = m1 == -INFINITY ? 0.f : ex2_fast_f(m1 - m_all);
                const float l_tot = a0 * l0 + a1 * l1;
                const float inv = l_tot > 0.f ? 1.f / l_tot : 0.f;
                const float s0 = a0 * inv, s1 = a1 * inv;
                // the other warpgroup's last product as well: that warpgroup has come this far, so it has seen the one before
                // complete, and the barrier is at most one completion behind
                const int c_0 = w == 0 ? c0 : g0 - c0, c_1 = w == 0 ? g0 - c0 : c0;
                if (f.n0 > 0) mbar_wait(&bars[F4_O], (c_0 - 1) & 1, ab);
                if (f.n1 > 0) mbar_wait(&bars[F4_O + 1], (c_1 - 1) & 1, ab);
                tcgen05_fence_after();
                __nv_bfloat16 *po = a.O + ((size_t)bh * n + ic) * HD + w * (HD / 2);
#pragma unroll
                for (int e0 = 0; e0 < HD / 2; e0 += 16) {
                    uint32_t v0[16], v1[16], z[8];
                    tmem_ld16(tm + C::tO + lane_addr + w * (HD / 2) + e0, v0);
                    tmem_ld16(tm + C::tO + HD + lane_addr + w * (HD / 2) + e0, v1);
                    tmem_wait_ld();
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        // a partial accumulator that never received a product holds stale bits: select, do not multiply
                        float y[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float x1 = f.n1 > 0 ? __uint_as_float(v1[2 * u + e]) * s1 : 0.f;
                            y[e] = f.n0 > 0 ? fmaf(__uint_as_float(v0[2 * u + e]), s0, x1) : x1;
                        }
                        z[u] = pack_bf16(y[0], y[1]);
                    }
                    if (ig < n) store32(po + e0, z, wide);
                }
                if (w == 0 && ig < n) a.LSE[(size_t)bh * n + ig] = row_lse(m_all, l_tot);
                // both accumulators and the exchange buffers have been read: P of the next unit of work may be handed over
                tcgen05_fence_before();
                more = units.take_together(t + 1);
            }
        }
    }
    tmem_leave(tm, 512, warp, ab);
}

// Heads that are launched together.  Under a causal mask the query tiles of a group start longest first; head after head the
// last head's longest tile starts when the grid is nearly done (d = 128, 32 heads, n = 8192 461 us so, 426 us in groups; 16 heads,
// n = 4096 95 and 66).  The group's K and V should stay in L2 while its tiles run.
int fwd_head_group(const Problem &p)
{
    constexpr size_t kBudget = 40u << 20;
    if (!mask_is_causal(p.mask_kind)) return 1;
    for (int g = 32; g > 1; g >>= 1)
        if (p.BH % g == 0 && (size_t)g * p.n * p.d * 4 <= kBudget) return g;
    return 1;
}

// 256 queries per CTA or 128.  A pair of query tiles shares its key tiles, but takes 1.7 (d = 128) to 1.9 times (d = 64, two
// terms) as long as one of them: it pays where the SMs have several units each, not where the halves of the pairs would fill a
// last wave that the pairs leave half empty.  The line: pairs that occupy half of the SMs, under a causal mask an average share
// of the SMs that exceeds the longest row 1.7 times, BH (T + 1) / 2 / 148 >= 1.7 for T tiles.  It was drawn with kernels of a CTA
// per unit; the kernels as they are, pairs / single tiles in us (calls back to back):
//   chosen for pairs    causal d = 128: 32 heads, n = 8192 439 / 536; 32 heads, n = 4096 122 / 136; 12 heads, n = 8192 211 / 186
//                       causal d = 64: 64 heads, n = 8192 760 / 831; 24 heads, n = 3000 67 / 59
//                       no mask: d = 128, 32 heads, n = 4096 231 / 238; d = 64, 64 heads, n = 2048 115 / 117; 6 heads, n = 8192 223 / 174
//                       two terms, d = 128: 32 heads, n = 8191, causal 776 / 822; 12 heads, n = 4095, no mask 207 / 159
//   chosen for single   causal d = 128: 16 heads, n = 2048 35 / 26; 40 heads, n = 1000 23 / 28; no mask, 16 heads, n = 1000 22 / 16
// Over 1,361 such points (d = 64 and 128, both masks, 1 to 128 heads, n = 512 to 16384) the choice is 1.5 to 2.5 % slower than the
// better one on average, 2.0 to 4.4 % with two terms, and at most 41 %.
// Not where results have to be repeatable: the two shapes differ in the last bits, and a head's result must not depend on how
// many others are in the call (24 heads, n = 3000, d = 64, no mask: 91 us, 97 so).
bool pair_pays(const Problem &p)
{
    if (p.cfg.deterministic) return false;
    const long tiles = (p.n + 127) / 128, sms = sm_count();
    if (p.mask_kind == ATTN_MASK_CAUSAL) return p.BH * (tiles + 1) * 10 >= sms * 34;
    return p.mask_kind == ATTN_MASK_NONE && (tiles + 1) / 2 * p.BH >= sms / 2;
}

template <int HD>
attn_status launch_fwd(const Problem &p)
{
    constexpr uint32_t TKF = HD == 256 ? 64 : 128;
    CUtensorMap mQ, mK, mV;
    const uint64_t BH = (uint64_t)p.BH;
    if (!make_tmap_bf16_3d(&mQ, p.Q, HD, p.n, BH, 128) || !make_tmap_bf16_3d(&mK, p.K, HD, p.n, BH, TKF) ||
        !make_tmap_bf16_3d(&mV, p.V, HD, p.n, BH, TKF))
        return ATTN_ERR_LAUNCH;
    FwdArgs a{};
    a.O = (__nv_bfloat16 *)p.Oout; a.LSE = p.LSEout;
    a.n = p.n; a.BH = (int)p.BH;
    a.mask_kind = p.mask_kind; a.block = p.block; a.nb = p.nb; a.mask_heads = p.mask_heads; a.fine = p.fine;
    a.row_ptr = p.row_ptr; a.col_idx = p.col_idx;
    a.scale = p.scale;
    a.status = p.status;
    a.group = fwd_head_group(p);
    if constexpr (HD != 256) {
        const bool pair = pair_pays(p);
        if (pair || !p.split) {
            void (*kernel)(CUtensorMap, CUtensorMap, CUtensorMap, FwdArgs) =
                p.split ? tc_fwd_pair_kernel<HD> : pair ? tc_fwd_flow_kernel<HD, true, false>
                : p.fine.mode ? tc_fwd_flow_kernel<HD, false, true> : tc_fwd_flow_kernel<HD, false, false>;
            const uint32_t bytes = p.split ? PairCfg<HD>::kBytes : pair ? FlowCfg<HD, true>::kBytes : FlowCfg<HD, false>::kBytes;
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return ATTN_ERR_LAUNCH;
            const int rows = pair ? 256 : 128;
            launch_begin("tc_fwd", p.stream);
            const bool ok = launch_chained(kernel, dim3((p.n + rows - 1) / rows * a.group, (unsigned)p.BH / a.group), kThreadsRows, bytes, p.stream, mQ, mK, mV, a);
            launch_end(p.stream);
            return ok ? ATTN_OK : ATTN_ERR_LAUNCH;
        }
    }
    void (*kernel)(CUtensorMap, CUtensorMap, CUtensorMap, FwdArgs);
    using C = typename std::conditional<HD == 256, FwdCfg<HD>, RowsCfg<HD>>::type;
    const uint32_t bytes = C::kBytes;
    if constexpr (HD == 256) kernel = tc_fwd_kernel<HD>;
    else kernel = p.fine.mode ? tc_fwd_rows_kernel<HD, true> : tc_fwd_rows_kernel<HD, false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
        return ATTN_ERR_LAUNCH;
    const dim3 grid((p.n + TQ - 1) / TQ * a.group, (unsigned)p.BH / a.group);
    launch_begin("tc_fwd", p.stream);
    const bool ok = launch_chained(kernel, grid, HD == 256 ? kThreads : kThreadsRows, bytes, p.stream, mQ, mK, mV, a);
    launch_end(p.stream);
    return ok ? ATTN_OK : ATTN_ERR_LAUNCH;
}

}  // namespace

size_t fwd_smem_bytes(int d)
{
    return d == 64 ? FlowCfg<64, false>::kUsed : d == 128 ? FlowCfg<128, false>::kUsed : d == 256 ? FwdCfg<256>::kUsed : 0;
}

attn_status tc_fwd(const Problem &p)
{
    if (p.d == 64) return launch_fwd<64>(p);
    if (p.d == 128) return launch_fwd<128>(p);
    if (p.d == 256) return launch_fwd<256>(p);
    return ATTN_ERR_TILE;
}

}  // namespace attn
