// Tensor-core backward of the softmax branch over the retained tokens (Section 4.2: the logit
// gradient is p (dp - <do, o>); k, v gradients exist only for retained tokens), bf16 storage,
// sm_100a.  With p_ij = exp(scale q_i.k_j - lse_i) over the retained keys j <= i:
//   dv_j = sum_i p_ij do_i,   dp_ij = do_i.v_j,   ds_ij = scale p_ij (dp_ij - D_i),
//   dq_i = sum_j ds_ij k_j,   dk_j = sum_i ds_ij q_i           (D_i = <do_i, o_i>)
// Two kernels, both recomputing p from the saved log-sum-exp:
//   * query side: one CTA per 128 queries walks the compacted K/V in tiles of 64 keys
//     (S = Q K^T and dP = dO V^T into TMEM, ds rows by two threads per query, dQ += dS K);
//   * key side: one CTA per 128 retained keys walks the query tiles that can see them
//     (S^T = K Q^T and dP^T = V dO^T, rows by two threads per key, dV += P^T dO, dK += dS^T Q).
// Every operand is fp16 (q, k, v convert exactly; p, ds, do are computed values that need more
// than bf16's 8 significant bits to keep the gradients within tolerance); accumulation is fp32.
#include "common.cuh"
#include "natsl_internal.h"
#include "tc_common.cuh"

namespace natsl {

namespace {

using namespace tc;

// Two threads per row (query or key), 32 of a tile's 64 columns and half of the result's each: the chain from a tile's
// logits to its operands and the epilogue are half as long as with one.  Measured at 64 columns and two CTAs per SM: 2000
// cycles per tile of a CTA on the query side, 2900 on the key side, of which the MMAs (N = 64: 50 cycles each) take
// 1200 and 1600; launch to first tile 4600, epilogue 4700 before its stores went through shared memory.
constexpr int kRowsB = 256;          // row threads: warps 0-3 columns 0-31 of a tile, warps 4-7 columns 32-63
constexpr int kMmaWarpB = 8, kTmaWarpB = 9;
constexpr int kThreadsB = kRowsB + 64;
constexpr int kMiscB = 2048;
constexpr float kLog2e = 1.4426950408889634f;

struct MiscB {
    uint64_t barQ, full[3], empty[3], barS, barDP, barSfree, barP, barAcc;
    uint32_t tmem_base;
    int abort_flag, wait_kcycles;   // in this order: the waits read the limit as abort_flag[1]
    uint32_t kept[4];               // query side: which of the CTA's own tokens are retained
    alignas(16) float lse[3][64], dsum[3][64];   // key side: per query of the tile in a stage (copied with it)
};
static_assert(sizeof(MiscB) <= kMiscB, "misc page too small");

// ==========================================================================================
// Query side
// ==========================================================================================
template <int D> struct QLayout {
    static constexpr int KB = D / 64;
    static constexpr int kQ = KB * 128 * 128;             // 128 queries x D fp16
    static constexpr int kKV = KB * 64 * 128;             // 64 keys x D fp16
    static constexpr int kStages = 3;
    static constexpr int oQ = 0, oDO = kQ, oK = 2 * kQ, oV = oK + kStages * kKV, oDS = oV + kStages * kKV;
    static constexpr int oMisc = oDS + 128 * 128;
    static constexpr int kTotal = oMisc + kMiscB;
    static constexpr int kTmem = D == 64 ? 256 : 512;     // S 64 + dP 64 + dQ D
};

// kG softmax heads per linear head (Section 4.3, grouped heads): a CTA's head is then one slice of D
// columns of rows of kG D columns -- the x coordinate of every copy and the column offset of every
// store --, the lists of retained tokens are the linear head's, lse and Dsm are [B,H,kG,L].
template <int D, int kG>
__global__ void __launch_bounds__(kThreadsB, D == 64 ? 2 : 1)
softmax_bwd_dq_tc_kernel(const __grid_constant__ CUtensorMap map_q,    // Qh  [B*H*L][D] fp16, box 128
                         const __grid_constant__ CUtensorMap map_do,   // dO16 [B*H*L][D] fp16, box 128
                         const __grid_constant__ CUtensorMap map_k,    // k16 [B*H*cap][D], box 64
                         const __grid_constant__ CUtensorMap map_v,    // v16 [B*H*cap][D], box 64
                         int cap, const int32_t *__restrict__ sm_idx,
                         const int32_t *__restrict__ sm_chunk_prefix, const float *__restrict__ lse,
                         const float *__restrict__ Dsm, float scale_sm, float *__restrict__ dq_sm,
                         int32_t *status, int L, int H, int wait_kcycles) {
    using SL = QLayout<D>;
    constexpr int KB = SL::KB;
    extern __shared__ __align__(1024) uint8_t smem[];
    MiscB &ms = *reinterpret_cast<MiscB *>(smem + SL::oMisc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NP = (L + 127) / 128, NC = L / kC;
    const int p = NP - 1 - (int)blockIdx.x;
    const int bhg = blockIdx.y, bh = bhg / kG, x0 = (bhg % kG) * D, b = bh / H, h = bh % H;
    const int32_t *pre = sm_chunk_prefix + (size_t)bh * (NC + 1);
    const int n_full = min(pre[2 * p], cap), n_end = min(pre[min(2 * p + 2, NC)], cap);
    const int T = (n_end + 63) / 64;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicMin(status, (int)NATSL_ERR_CUDA);
        return;
    }
    if (tid == 0) {
        mbar_init(&ms.barQ, 1);
        for (int s = 0; s < SL::kStages; ++s) { mbar_init(&ms.full[s], 1); mbar_init(&ms.empty[s], 1); }
        mbar_init(&ms.barS, 1);
        mbar_init(&ms.barSfree, kRowsB);
        mbar_init(&ms.barP, kRowsB);
        mbar_init(&ms.barAcc, 1);
        ms.abort_flag = 0;
        ms.wait_kcycles = wait_kcycles;
        fence_mbar_init();
    }
    if (tid < 4) ms.kept[tid] = 0u;
    if (warp == kMmaWarpB) tmem_alloc(&ms.tmem_base, SL::kTmem);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = ms.tmem_base;
    const uint32_t tS = tmem, tDP = tmem + 64, tDQ = tmem + 128;
    volatile int *abort_flag = &ms.abort_flag;

    if (warp == kTmaWarpB) {
        if (lane == 0 && T > 0) {      // nothing is loaded for a tile that sees no retained key
            mbar_arrive_expect_tx(&ms.barQ, 2 * SL::kQ);
            for (int kb = 0; kb < KB; ++kb) {
                tma_load_2d(smem + SL::oQ + kb * 16384, &map_q, &ms.barQ, x0 + kb * 64, bh * L + p * 128);
                tma_load_2d(smem + SL::oDO + kb * 16384, &map_do, &ms.barQ, x0 + kb * 64, bh * L + p * 128);
            }
            int t = 0;
            for (; t < T; ++t) {
                const int s = t % SL::kStages;
                if (!mbar_wait(&ms.empty[s], ((t / SL::kStages) & 1) ^ 1, abort_flag)) break;
                mbar_arrive_expect_tx(&ms.full[s], 2 * SL::kKV);
                for (int kb = 0; kb < KB; ++kb) {
                    tma_load_2d(smem + SL::oK + s * SL::kKV + kb * 8192, &map_k, &ms.full[s], x0 + kb * 64,
                                bh * cap + t * 64);
                    tma_load_2d(smem + SL::oV + s * SL::kKV + kb * 8192, &map_v, &ms.full[s], x0 + kb * 64,
                                bh * cap + t * 64);
                }
            }
            for (int u = max(0, t - SL::kStages); u < t; ++u)    // no copy in flight at retirement
                mbar_wait_drain(&ms.full[u % SL::kStages], (u / SL::kStages) & 1);
            mbar_wait_drain(&ms.barQ, 0);
        }
    } else if (warp == kMmaWarpB) {
        const int Tu = (int)uniform((uint32_t)T);
        if (Tu > 0) {
            constexpr uint32_t id_s = make_idesc(kFmtF16, 128, 64, false, false);
            constexpr uint32_t id_dq = make_idesc(kFmtF16, 128, D, false, true);
            const uint32_t tm = uniform(tmem), sm = smem_u32(smem), aQ = sm + SL::oQ, aDO = sm + SL::oDO, aDS = sm + SL::oDS;
            auto issue_s = [&](int t) {
                const uint32_t aK = sm + SL::oK + (t % SL::kStages) * SL::kKV, aV = sm + SL::oV + (t % SL::kStages) * SL::kKV;
                if (!elect_one()) return;
#pragma unroll
                for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                    for (int k16 = 0; k16 < 4; ++k16) {
                        mma_ss(tm, desc_kmajor(aQ + kb * 16384 + k16 * 32),
                               desc_kmajor(aK + kb * 8192 + k16 * 32), id_s, (kb | k16) != 0);
                        mma_ss(tm + 64, desc_kmajor(aDO + kb * 16384 + k16 * 32),
                               desc_kmajor(aV + kb * 8192 + k16 * 32), id_s, (kb | k16) != 0);
                    }
                mma_commit(&ms.barS);
            };
            bool ok = wait_all(&ms.barQ, 0, abort_flag) && wait_all(&ms.full[0], 0, abort_flag);
            if (ok) {
                tc_fence_after_sync();
                issue_s(0);
            }
            for (int t = 0; ok && t < Tu; ++t) {
                // S and dP of the next tile go into the same TMEM columns as soon as the row threads
                // have read this tile's out of them (barSfree), i.e. while they still compute dS.
                if (t + 1 < Tu) {
                    ok = wait_all(&ms.full[(t + 1) % SL::kStages], ((t + 1) / SL::kStages) & 1, abort_flag) &&
                         wait_all(&ms.barSfree, t & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after_sync();
                    issue_s(t + 1);
                }
                ok = wait_all(&ms.barP, t & 1, abort_flag);
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t aK = sm + SL::oK + (t % SL::kStages) * SL::kKV;
                if (elect_one()) {
#pragma unroll
                    for (int k16 = 0; k16 < 4; ++k16)
                        mma_ss(tm + 128, desc_kmajor(aDS + k16 * 32), desc_mnmajor(aK + k16 * 2048, 8192), id_dq, (t | k16) != 0);
                    mma_commit(&ms.barAcc);
                    mma_commit(&ms.empty[t % SL::kStages]);     // K/V stage t is free after dQ(t)
                }
            }
        }
    } else {
        const int wq = warp & 3, half = warp >> 2, r = wq * 32 + lane, i_abs = p * 128 + r;
        const bool row_ok = i_abs < L;
        const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
        const float sl2 = scale_sm * kLog2e;
        float lse2 = row_ok ? lse[(size_t)bhg * L + i_abs] * kLog2e : 0.f;
        if (lse2 == -INFINITY) lse2 = 0.f;                  // no key: every logit is masked below
        const float Di = row_ok ? Dsm[(size_t)bhg * L + i_abs] : 0.f;
        bool ok = true;
        // The compacted keys are in position order, so row i sees exactly the first `cnt` of them: all earlier ones
        // plus a population count of the CTA's own.
        if (half == 0 && n_full + r < n_end) {
            const int rel = sm_idx[(size_t)bh * L + n_full + r] - p * 128;
            atomicOr(&ms.kept[(rel >> 5) & 3], 1u << (rel & 31));
        }
        named_barrier_sync(1, kRowsB);
        int cnt = n_full + __popc(ms.kept[wq] & ((2u << lane) - 1u));
        for (int e = 0; e < wq; ++e) cnt += __popc(ms.kept[e]);
        if (!row_ok) cnt = 0;
        const uint64_t sl22 = pack2(sl2, sl2), nl2 = pack2(-lse2, -lse2), sm2 = pack2(scale_sm, scale_sm);
        for (int t = 0; t < T; ++t) {
            ok = mbar_wait(&ms.barS, t & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
            uint32_t dk[16];                                // ds as packed fp16 pairs
            const int vis = cnt - t * 64 - 32 * half;       // keys of this thread's 32 that the row sees
            const bool all_vis = __all_sync(0xffffffffu, vis >= 32);
            {
                uint32_t sv[32], dv[32];
                tmem_ld32(tS + lane_base + 32 * half, sv);
                tmem_ld32(tDP + lane_base + 32 * half, dv);
                tmem_wait_ld();
                tc_fence_before_sync();
                mbar_arrive(&ms.barSfree);
                if (!all_vis) {                             // mask the logit (exp2(-inf) = 0): no branch per element
#pragma unroll
                    for (int c = 0; c < 32; ++c) sv[c] = c < vis ? sv[c] : 0xff800000u;
                }
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                    const float2 e = unpack2(fma2(pack2(__uint_as_float(sv[c]), __uint_as_float(sv[c + 1])), sl22, nl2));
                    const uint64_t pr = mul2(pack2(ex2_ftz(e.x), ex2_ftz(e.y)), sm2);
                    const float2 ds = unpack2(mul2(pr, pack2(__uint_as_float(dv[c]) - Di, __uint_as_float(dv[c + 1]) - Di)));
                    dk[c >> 1] = pack_half2(ds.x, ds.y);
                }
            }
            if (t > 0) {
                ok = mbar_wait(&ms.barAcc, (t - 1) & 1, abort_flag);   // dS buffer consumed
                if (!ok) break;
            }
#pragma unroll
            for (int pc = 0; pc < 4; ++pc)
                *reinterpret_cast<uint4 *>(smem + SL::oDS + sw128_offset(r, 4 * half + pc)) = make_uint4(dk[4 * pc], dk[4 * pc + 1], dk[4 * pc + 2], dk[4 * pc + 3]);
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&ms.barP);
        }
        if (ok && T > 0) {
            ok = mbar_wait(&ms.barAcc, (T - 1) & 1, abort_flag);
            tc_fence_after_sync();
        }
        if (ok) {
            const float gi = grad_scale(status).y;          // dO and Dsm arrive times the gradient scale
            float *dst = dq_sm + (((size_t)b * L + p * 128 + wq * 32) * H + h) * (D * kG) + x0;
#pragma unroll
            for (int cbi = 0; cbi < D / 64; ++cbi) {
                const int cb = half * (D / 64) + cbi;
                uint32_t x[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) x[c] = 0u;
                if (T > 0) {
                    tmem_ld32(tDQ + lane_base + cb * 32, x);
                    tmem_wait_ld();
                }
                // (the Q and dO tiles have been read)
                store_rows32(smem + warp * 4096, x, gi, dst + cb * 32, (size_t)H * (D * kG), L - p * 128 - wq * 32, lane);
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarpB) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, SL::kTmem);
    }
    if (tid == 0 && ms.abort_flag) atomicMin(status, (int)NATSL_ERR_TIMEOUT);
}

// ==========================================================================================
// Key side
// ==========================================================================================
// dS^T goes to the multiplier through TMEM, over the dP^T it was formed from, which leaves shared memory for a third
// query tile in flight at two CTAs per SM (D = 64).  With two, a tile's copy could start only when the product
// two tiles back had released its place and was a serial part of the chain: 2700 cycles per tile.
template <int D> struct KLayout {
    static constexpr int KB = D / 64;
    static constexpr int kKV = KB * 128 * 128;            // 128 keys x D fp16
    static constexpr int kQ = KB * 64 * 128;              // 64 queries x D fp16
    static constexpr int kStages = 3;
    static constexpr int oK = 0, oV = kKV, oQ = 2 * kKV, oDO = oQ + kStages * kQ, oP = oDO + kStages * kQ;
    static constexpr int oMisc = oP + 128 * 128;
    static constexpr int kTotal = oMisc + kMiscB;
    static constexpr int kTmem = D == 64 ? 256 : 512;     // S^T 64 + dP^T 64 + dV D + dK D
};

// All (batch, head) pairs of a key tile before the next tile: a CTA of the earliest keys runs over every query tile and
// was, with the tiles of a pair in sequence, the tail of the launch (24 k tiles of 64 columns: 355 -> 234 us).
// Two CTAs per SM at D = 64, where shared memory and TMEM allow it: left to itself the compiler takes 176 registers,
// which leaves one, and the kernel, a chain of waits, then runs with four row warps per SM.
template <int D, bool kMask, int kG>   // kMask: also the per-key sums of the mask gradient (dmask); kG: as above
__global__ void __launch_bounds__(kThreadsB, D == 64 ? 2 : 1)
softmax_bwd_dkv_tc_kernel(const __grid_constant__ CUtensorMap map_q,    // Qh [B*H*L][D], box 64
                          const __grid_constant__ CUtensorMap map_do,   // dO16, box 64
                          const __grid_constant__ CUtensorMap map_k,    // k16 [B*H*cap][D], box 128
                          const __grid_constant__ CUtensorMap map_v,    // v16, box 128
                          int cap, const int32_t *__restrict__ sm_idx,
                          const int32_t *__restrict__ sm_chunk_prefix,
                          const float *__restrict__ lse, const float *__restrict__ Dsm,
                          float scale_sm, float *__restrict__ dk_sm, float *__restrict__ dv_sm,
                          float *__restrict__ dmask,     // [B*H*cap]: sum_i p_ij (dp_ij - D_i) per key j
                          int32_t *status, int L, int H, int wait_kcycles) {
    using SL = KLayout<D>;
    constexpr int KB = SL::KB;
    extern __shared__ __align__(1024) uint8_t smem[];
    MiscB &ms = *reinterpret_cast<MiscB *>(smem + SL::oMisc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NC = L / kC;
    const int kt = blockIdx.y, bhg = blockIdx.x, bh = bhg / kG, x0 = (bhg % kG) * D;    // earliest keys first: the most queries
    const int n_sm = min(sm_chunk_prefix[(size_t)bh * (NC + 1) + NC], cap);
    if (kt * 128 >= n_sm) return;                        // uniform: no retained key in this tile
    const int first_pos = sm_idx[(size_t)bh * L + kt * 128];
    const int qt0 = first_pos / 64;                       // first query tile that sees a key of the tile
    const int T = NC - qt0;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicMin(status, (int)NATSL_ERR_CUDA);
        return;
    }
    if (tid == 0) {
        mbar_init(&ms.barQ, 1);
        for (int s = 0; s < SL::kStages; ++s) { mbar_init(&ms.full[s], 1); mbar_init(&ms.empty[s], 1 + kRowsB); }
        mbar_init(&ms.barS, 1);
        mbar_init(&ms.barDP, 1);
        mbar_init(&ms.barSfree, kRowsB);
        mbar_init(&ms.barP, kRowsB);
        mbar_init(&ms.barAcc, 1);
        ms.abort_flag = 0;
        ms.wait_kcycles = wait_kcycles;
        fence_mbar_init();
    }
    if (warp == kMmaWarpB) tmem_alloc(&ms.tmem_base, SL::kTmem);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = ms.tmem_base;
    const uint32_t tS = tmem, tDP = tmem + 64, tDV = tmem + 128, tDK = tmem + 128 + D;
    volatile int *abort_flag = &ms.abort_flag;

    if (warp == kTmaWarpB) {
        if (lane == 0) {
            mbar_arrive_expect_tx(&ms.barQ, 2 * SL::kKV);
            for (int kb = 0; kb < KB; ++kb) {
                tma_load_2d(smem + SL::oK + kb * 16384, &map_k, &ms.barQ, x0 + kb * 64, bh * cap + kt * 128);
                tma_load_2d(smem + SL::oV + kb * 16384, &map_v, &ms.barQ, x0 + kb * 64, bh * cap + kt * 128);
            }
            int t = 0;
            for (; t < T; ++t) {
                const int s = t % SL::kStages;
                if (!mbar_wait(&ms.empty[s], ((t / SL::kStages) & 1) ^ 1, abort_flag)) break;
                mbar_arrive_expect_tx(&ms.full[s], 2 * SL::kQ + 512);
                bulk_load_1d(ms.lse[s], lse + (size_t)bhg * L + (qt0 + t) * 64, 256, &ms.full[s]);
                bulk_load_1d(ms.dsum[s], Dsm + (size_t)bhg * L + (qt0 + t) * 64, 256, &ms.full[s]);
                for (int kb = 0; kb < KB; ++kb) {
                    tma_load_2d(smem + SL::oQ + s * SL::kQ + kb * 8192, &map_q, &ms.full[s], x0 + kb * 64,
                                bh * L + (qt0 + t) * 64);
                    tma_load_2d(smem + SL::oDO + s * SL::kQ + kb * 8192, &map_do, &ms.full[s], x0 + kb * 64,
                                bh * L + (qt0 + t) * 64);
                }
            }
            for (int u = max(0, t - SL::kStages); u < t; ++u)
                mbar_wait_drain(&ms.full[u % SL::kStages], (u / SL::kStages) & 1);
            mbar_wait_drain(&ms.barQ, 0);
        }
    } else if (warp == kMmaWarpB) {
        constexpr uint32_t id_s = make_idesc(kFmtF16, 128, 64, false, false);
        constexpr uint32_t id_acc = make_idesc(kFmtF16, 128, D, false, true);
        const int Tu = (int)uniform((uint32_t)T);
        const uint32_t tm = uniform(tmem), sm = smem_u32(smem), aK = sm + SL::oK, aV = sm + SL::oV, aP = sm + SL::oP;
        auto stage = [&](int o, int t) { return sm + o + (t % SL::kStages) * SL::kQ; };
        auto issue_logits = [&](uint32_t dst, uint32_t a, uint32_t b, uint64_t *bar) {
            if (!elect_one()) return;
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16)
                    mma_ss(dst, desc_kmajor(a + kb * 16384 + k16 * 32), desc_kmajor(b + kb * 8192 + k16 * 32), id_s, (kb | k16) != 0);
            mma_commit(bar);
        };
        bool ok = wait_all(&ms.barQ, 0, abort_flag) && wait_all(&ms.full[0], 0, abort_flag);
        if (ok) {
            tc_fence_after_sync();
            issue_logits(tm, aK, stage(SL::oQ, 0), &ms.barS);
            issue_logits(tm + 64, aV, stage(SL::oDO, 0), &ms.barDP);
        }
        for (int t = 0; ok && t < Tu; ++t) {
            // S^T of the next query tile goes into the same TMEM columns as soon as the row threads have read
            // this tile's out of them; dP^T of the next one behind this tile's products, which read dS^T there.
            if (t + 1 < Tu) {
                ok = wait_all(&ms.full[(t + 1) % SL::kStages], ((t + 1) / SL::kStages) & 1, abort_flag) &&
                     wait_all(&ms.barSfree, t & 1, abort_flag);
                if (!ok) break;
                tc_fence_after_sync();
                issue_logits(tm, aK, stage(SL::oQ, t + 1), &ms.barS);
            }
            ok = wait_all(&ms.barP, t & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t aQ = stage(SL::oQ, t), aDO = stage(SL::oDO, t);
            if (elect_one()) {
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16) {
                    mma_ss(tm + 128, desc_kmajor(aP + k16 * 32), desc_mnmajor(aDO + k16 * 2048, 8192), id_acc, (t | k16) != 0);
                    mma_ts(tm + 128 + D, tm + 64 + (k16 >> 1) * 32 + (k16 & 1) * 8, desc_mnmajor(aQ + k16 * 2048, 8192), id_acc,
                           (t | k16) != 0);
                }
                mma_commit(&ms.barAcc);
                mma_commit(&ms.empty[t % SL::kStages]);
            }
            if (t + 1 < Tu) issue_logits(tm + 64, aV, stage(SL::oDO, t + 1), &ms.barDP);
        }
    } else {
        const int wq = warp & 3, half = warp >> 2, r = wq * 32 + lane, j = kt * 128 + r;    // this thread's retained key
        const bool key_ok = j < n_sm;
        const int pos_j = key_ok ? sm_idx[(size_t)bh * L + j] : 0x7fffffff;
        const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
        const float sl2 = scale_sm * kLog2e;
        float msum = 0.f;                                   // mask gradient of this key, over all queries
        bool ok = true;
        for (int t = 0; t < T; ++t) {
            const int i0 = (qt0 + t) * 64 + 32 * half;      // this thread's 32 queries
            // per-query log-sum-exp and D of this tile, copied with the stage (the logits were formed from it, so it
            // is full; released below)
            const int sg = t % SL::kStages;
            float *lse_t = ms.lse[sg] + 32 * half;
            const float *dsum = ms.dsum[sg] + 32 * half;
            ok = mbar_wait(&ms.full[sg], (t / SL::kStages) & 1, abort_flag) && mbar_wait(&ms.barS, t & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
            const uint64_t sl22 = pack2(sl2, sl2), nl2 = pack2(-kLog2e, -kLog2e), sm2 = pack2(scale_sm, scale_sm);
            const int vis = pos_j - i0;                     // queries vis .. of the tile see this key
            const bool all_vis = __all_sync(0xffffffffu, vis <= 0);
            if (!all_vis) {     // a query without any key has lse = -inf, which must not meet a masked logit's -inf
                if (lse_t[lane] == -INFINITY) lse_t[lane] = 0.f;
                __syncwarp();
            }
            float x[32];                                    // logits, then probabilities
            tmem_ld32(tS + lane_base + 32 * half, reinterpret_cast<uint32_t (&)[32]>(x[0]));
            tmem_wait_ld();
            tc_fence_before_sync();
            mbar_arrive(&ms.barSfree);
            if (!all_vis) {                                 // mask the logit (exp2(-inf) = 0): no branch per element
#pragma unroll
                for (int c = 0; c < 32; ++c) x[c] = vis <= c ? x[c] : -INFINITY;
            }
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
                const uint64_t l2 = *reinterpret_cast<const uint64_t *>(&lse_t[c]);
                const float2 e = unpack2(fma2(pack2(x[c], x[c + 1]), sl22, mul2(l2, nl2)));
                x[c] = ex2_ftz(e.x);
                x[c + 1] = ex2_ftz(e.y);
            }
            // dP^T of this tile was issued behind the previous tile's products: they have read P and dS by now
            ok = mbar_wait(&ms.barDP, t & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
#pragma unroll
            for (int pc = 0; pc < 4; ++pc)
                *reinterpret_cast<uint4 *>(smem + SL::oP + sw128_offset(r, 4 * half + pc)) =
                    make_uint4(pack_half2(x[8 * pc], x[8 * pc + 1]), pack_half2(x[8 * pc + 2], x[8 * pc + 3]),
                               pack_half2(x[8 * pc + 4], x[8 * pc + 5]), pack_half2(x[8 * pc + 6], x[8 * pc + 7]));
            uint32_t dk[16];
            {
                uint32_t dv[32];
                tmem_ld32(tDP + lane_base + 32 * half, dv);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                    const float2 d2 = *reinterpret_cast<const float2 *>(&dsum[c]);
                    const uint64_t dm = mul2(pack2(x[c], x[c + 1]), pack2(__uint_as_float(dv[c]) - d2.x, __uint_as_float(dv[c + 1]) - d2.y));
                    if (kMask) {                            // dM_ij (Section 4.2)
                        const float2 m = unpack2(dm);
                        msum += m.x + m.y;
                    }
                    const float2 ds = unpack2(mul2(dm, sm2));
                    dk[c >> 1] = pack_half2(ds.x, ds.y);
                }
            }
            tmem_st16(tDP + lane_base + 32 * half, dk);     // dS^T over this thread's own dP^T
            tmem_wait_st();
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&ms.barP);
            mbar_arrive(&ms.empty[sg]);        // (the stage's release also waits for the MMAs' commit)
        }
        if (ok) {
            ok = mbar_wait(&ms.barAcc, (T - 1) & 1, abort_flag);
            tc_fence_after_sync();
        }
        if (kMask) {
            if (half == 1) (&ms.lse[0][0])[r] = msum;       // (every row thread is past its last tile)
            named_barrier_sync(1, kRowsB);
        }
        if (ok) {      // the TMEM loads are warp-wide: only the stores depend on the key being real
            const float gi = grad_scale(status).y;          // dO and Dsm arrive times the gradient scale
            if (kMask && half == 0 && key_ok) dmask[(size_t)bhg * cap + j] = gi * (msum + (&ms.lse[0][0])[r]);
#pragma unroll
            for (int cbi = 0; cbi < D / 64; ++cbi) {
                const int cb = half * (D / 64) + cbi;
                const size_t at = ((size_t)bh * cap + kt * 128 + wq * 32) * (D * kG) + x0 + cb * 32;
                const int rows = n_sm - kt * 128 - wq * 32;
                uint32_t x[32];
                tmem_ld32(tDV + lane_base + cb * 32, x);
                tmem_wait_ld();
                store_rows32(smem + warp * 4096, x, gi, dv_sm + at, D * kG, rows, lane);   // (K and V have been read)
                tmem_ld32(tDK + lane_base + cb * 32, x);
                tmem_wait_ld();
                store_rows32(smem + warp * 4096, x, gi, dk_sm + at, D * kG, rows, lane);
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarpB) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, SL::kTmem);
    }
    if (tid == 0 && ms.abort_flag) atomicMin(status, (int)NATSL_ERR_TIMEOUT);
}

// q (bf16, [B,L,H,d]) -> fp16 [B,H,L,d]; 8 values per thread.  norm_eps >= 0: each of the `groups` slices
// of a row RMS-normalised on the way (Section 4.3: the softmax operation's q; a slice's pieces sit in
// neighbouring lanes).
template <int D>
__global__ void __launch_bounds__(256)
to_f16_bhld_kernel(const __nv_bfloat16 *__restrict__ q, __half *__restrict__ qh, int B, int L, int H,
                   int groups, float norm_eps) {
    constexpr int kPieces = D / 8;
    const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;
    const size_t total = (size_t)B * L * H * kPieces;
    if (idx >= total) return;
    const int pc = idx % kPieces;
    const size_t row = idx / kPieces;          // (b, l, h)
    const int h = row % H;
    const size_t bl = row / H;
    const int l = bl % L, b = bl / L;
    const uint4 u = reinterpret_cast<const uint4 *>(q)[idx];
    const uint32_t wv[4] = {u.x, u.y, u.z, u.w};
    uint32_t o[4];
    float rq = 1.f;
    if (norm_eps >= 0.f) {         // (the grid covers whole rows, so all lanes of a row are here)
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float lo = __uint_as_float(wv[i] << 16), hi = __uint_as_float(wv[i] & 0xffff0000u);
            ss = fmaf(lo, lo, fmaf(hi, hi, ss));
        }
        const int lanes = kPieces / groups;
        const unsigned row_mask = ((1u << kPieces) - 1u) << ((threadIdx.x & 31) & ~(kPieces - 1));
        for (int off = 1; off < lanes; off <<= 1) ss += __shfl_xor_sync(row_mask, ss, off);
        rq = rsqrtf(ss * groups / D + norm_eps);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        o[i] = pack_half2(__uint_as_float(wv[i] << 16) * rq, __uint_as_float(wv[i] & 0xffff0000u) * rq);
    reinterpret_cast<uint4 *>(qh)[(((size_t)b * H + h) * L + l) * kPieces + pc] =
        make_uint4(o[0], o[1], o[2], o[3]);
}

}  // namespace

cudaError_t launch_to_f16_bhld(const void *x, void *xh, Shape s, HeadGroups hg, cudaStream_t st) {
    const size_t pieces = (size_t)s.B * s.L * s.H * (s.d / 8);
    auto kernel = s.d == 128 ? to_f16_bhld_kernel<128> : to_f16_bhld_kernel<64>;
    kernel<<<(unsigned)((pieces + 255) / 256), 256, 0, st>>>((const __nv_bfloat16 *)x, (__half *)xh, s.B, s.L, s.H, hg.G,
                                                             hg.norm_eps);
    count_launch();
    return cudaGetLastError();
}

template <int D, int G>      // D: columns of a softmax head, G of them per linear head (s.d = D G)
static cudaError_t softmax_bwd_tc_impl(const void *Qh, const void *dO16, const void *k16,
                                       const void *v16, int cap, const int32_t *sm_idx,
                                       const int32_t *pre, const float *lse, const float *Dsm,
                                       float scale_sm, float *dq_sm, float *dk_sm, float *dv_sm,
                                       float *dmask, int32_t *status, Shape s,
                                       cudaStream_t st, cudaStream_t st_kv, cudaEvent_t after_dq) {
    const uint64_t BH = (uint64_t)s.B * s.H;
    constexpr int DL = D * G;
    cudaError_t e;
    CUtensorMap mq128, mdo128, mk64, mv64, mq64, mdo64, mk128, mv128;
    if (!tch::make_map_2d(&mq128, Qh, BH * s.L, DL, 128) || !tch::make_map_2d(&mdo128, dO16, BH * s.L, DL, 128) ||
        !tch::make_map_2d(&mk64, k16, BH * cap, DL, 64) || !tch::make_map_2d(&mv64, v16, BH * cap, DL, 64) ||
        !tch::make_map_2d(&mq64, Qh, BH * s.L, DL, 64) || !tch::make_map_2d(&mdo64, dO16, BH * s.L, DL, 64) ||
        !tch::make_map_2d(&mk128, k16, BH * cap, DL, 128) || !tch::make_map_2d(&mv128, v16, BH * cap, DL, 128))
        return cudaErrorInvalidValue;
    e = allow_smem(softmax_bwd_dq_tc_kernel<D, G>, QLayout<D>::kTotal);
    if (e != cudaSuccess) return e;
    auto dkv = dmask ? softmax_bwd_dkv_tc_kernel<D, true, G> : softmax_bwd_dkv_tc_kernel<D, false, G>;
    e = allow_smem(dkv, KLayout<D>::kTotal);
    if (e != cudaSuccess) return e;
    dim3 gq((s.L + 127) / 128, s.B * s.H * G);
    softmax_bwd_dq_tc_kernel<D, G><<<gq, kThreadsB, QLayout<D>::kTotal, st>>>(
        mq128, mdo128, mk64, mv64, cap, sm_idx, pre, lse, Dsm, scale_sm, dq_sm, status, s.L, s.H, debug_wait_kcycles());
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (after_dq && (e = cudaEventRecord(after_dq, st)) != cudaSuccess) return e;
    dim3 gk(s.B * s.H * G, (s.L + 127) / 128);
    dkv<<<gk, kThreadsB, KLayout<D>::kTotal, st_kv>>>(
        mq64, mdo64, mk128, mv128, cap, sm_idx, pre, lse, Dsm, scale_sm, dk_sm, dv_sm, dmask, status, s.L, s.H, debug_wait_kcycles());
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_softmax_bwd_tc(const void *Qh, const void *dO16, const void *k16,
                                  const void *v16, int cap, const int32_t *sm_idx,
                                  const int32_t *sm_chunk_prefix, const float *lse, const float *Dsm,
                                  float scale_sm, float *dq_sm, float *dk_sm, float *dv_sm,
                                  float *dmask, int32_t *status, Shape s,
                                  cudaStream_t st, cudaStream_t st_kv, cudaEvent_t after_dq, HeadGroups hg) {
    if (hg.G == 2 && s.d == 128)
        return softmax_bwd_tc_impl<64, 2>(Qh, dO16, k16, v16, cap, sm_idx, sm_chunk_prefix, lse, Dsm, scale_sm,
                                          dq_sm, dk_sm, dv_sm, dmask, status, s, st, st_kv, after_dq);
    if (hg.G > 1) return cudaErrorInvalidValue;
    if (s.d == 128)
        return softmax_bwd_tc_impl<128, 1>(Qh, dO16, k16, v16, cap, sm_idx, sm_chunk_prefix, lse, Dsm, scale_sm,
                                           dq_sm, dk_sm, dv_sm, dmask, status, s, st, st_kv, after_dq);
    return softmax_bwd_tc_impl<64, 1>(Qh, dO16, k16, v16, cap, sm_idx, sm_chunk_prefix, lse, Dsm, scale_sm,
                                      dq_sm, dk_sm, dv_sm, dmask, status, s, st, st_kv, after_dq);
}

}  // namespace natsl
