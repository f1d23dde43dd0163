// Tensor-core reverse scan of the chunkwise Gated DeltaNet backward (bf16 storage, sm_100a).
//
// With the notation of gdn_tc.cu and, per chunk, S0 = entry state, dS1 = gradient w.r.t. the exit
// state, dO = gradient of the linear read-out:
//   dU~ = P^T dO + diag(gamma_C / gamma) K dS1
//   dS0 = (scale_la diag(gamma) Q)^T dO + gamma_C dS1 - W^T dU~
// One CTA per (batch, head) walks the chunks backwards.  As in the forward scan the head dimension
// sits on the MMA's M axis: value column r of dS (row r of dS^T, TMEM lane r) belongs to the two
// threads (r, half 0 / 1) of warps q and q + 4, the fp32 gradient state lives in their registers,
// and the operands a thread produces (dS1, dU~ as fp16) are written to its own TMEM lane:
//   X1 = dO^T P            X2 = dS1^T K^T                       (both [d, 64 tokens])
//   dU~^T = X1 + X2 diag(gamma_C / gamma)        -> fp16 operand, in TMEM and to global
//   Y  = (diag(scale_la gamma) dO)^T Q - dU~^T W                ([d, d], second product negated)
//   dS0^T = gamma_C dS1^T + Y
// dO and scale_la gamma dO arrive as fp16 tiles [B,H,L,d]; P, W^T and the fp16 q, k copies are the
// forward's own intermediates.  dU~ and the chunk-exit gradients dS1 leave as the fp16 operands they are, in
// 16-byte pieces whose stores are contiguous over a warp (as fp32 rows they took 96 narrow stores per thread and
// chunk), in units of the gradient scale, for the chunk kernel.
#include "common.cuh"
#include "natsl_internal.h"
#include "tc_common.cuh"

namespace natsl {

namespace {

using namespace tc;

constexpr int kRsRowThreads = 256;
constexpr int kRsThreads = 320;
constexpr int kRsStages = 2;
constexpr int kRsMisc = 1024;
constexpr int kRsDecaySlots = 4;

template <int D> struct RsLayout {
    static constexpr int KB = D / 64;
    static constexpr int kT = KB * 8192;                   // a 64-token x D fp16 tile
    static constexpr int oDO = 0, oDOg = kT, oQ = 2 * kT, oK = 3 * kT, oW = 4 * kT;   // W^T: D rows x 64
    static constexpr int oP = oW + D * 128;
    static constexpr int kStage = oP + 8192;
    static constexpr int kG = 512;
    static constexpr int kTx = kStage + kG;
    static constexpr int oG = kRsStages * kStage;
    static constexpr int oMisc = oG + kRsDecaySlots * kG;
    static constexpr int kTotal = oMisc + kRsMisc;
    // TMEM columns: X1 [64], X2 [64] (X2's columns are then reused for the fp16 dU~ operand),
    // Y [D], A = fp16 dS1 operand [D/2 packed].
    static constexpr int cX1 = 0, cX2 = 64, cY = 128, cA = 128 + D;
    static constexpr int kTmemCols = D == 128 ? 512 : 256;
};

struct RsMisc {
    uint64_t full[kRsStages], empty[kRsStages], barA, barX, barB, barY;
    uint32_t tmem_base;
    int abort_flag, wait_kcycles;   // in this order: the waits read the limit as abort_flag[1]
};
static_assert(sizeof(RsMisc) <= kRsMisc, "misc page too small");

template <int D, bool kBlock>      // kBlock: block-level routing (softmax blocks were not committed)
__global__ void __launch_bounds__(kRsThreads, 1)
gdn_rscan_tc_kernel(const __grid_constant__ CUtensorMap map_do,    // dO (fp16) [B*H*L][D], box 64
                    const __grid_constant__ CUtensorMap map_dog,   // scale_la gamma dO (fp16), box 64
                    const __grid_constant__ CUtensorMap map_qh, const __grid_constant__ CUtensorMap map_kh,
                    const __grid_constant__ CUtensorMap map_wt,    // W^T [B*H*NC*D][64], box D
                    const __grid_constant__ CUtensorMap map_ph,    // P [B*H*NC*64][64], box 64
                    const float *__restrict__ Gd, __half *__restrict__ dU16, __half *__restrict__ dS16,
                    const float *__restrict__ dstate_out, float *__restrict__ dstate_in,
                    const uint8_t *__restrict__ block_route, int32_t *status, int L, int H, int wait_kcycles) {
    using SL = RsLayout<D>;
    constexpr int KB = SL::KB;
    constexpr int kHalfCols = D / 2;
    extern __shared__ __align__(1024) uint8_t smem[];
    RsMisc &ms = *reinterpret_cast<RsMisc *>(smem + SL::oMisc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NC = L / kC;
    const int bh = blockIdx.x, b = bh / H, h = bh % H;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicMin(status, (int)NATSL_ERR_CUDA);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < kRsStages; ++s) { mbar_init(&ms.full[s], 1); mbar_init(&ms.empty[s], 1); }
        mbar_init(&ms.barA, kRsRowThreads);
        mbar_init(&ms.barB, kRsRowThreads);
        mbar_init(&ms.barX, 1);
        mbar_init(&ms.barY, 1);
        ms.abort_flag = 0;
        ms.wait_kcycles = wait_kcycles;
        fence_mbar_init();
    }
    if (warp == 8) tmem_alloc(&ms.tmem_base, SL::kTmemCols);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = ms.tmem_base;
    volatile int *abort_flag = &ms.abort_flag;

    if (warp == 9) {
        if (lane == 0) {
            int n = 0;                                      // n-th chunk processed = chunk NC - 1 - n
            for (; n < NC; ++n) {
                const int c = NC - 1 - n, s = n % kRsStages;
                if (!mbar_wait(&ms.empty[s], ((n / kRsStages) & 1) ^ 1, abort_flag)) break;
                uint8_t *st = smem + s * SL::kStage;
                mbar_arrive_expect_tx(&ms.full[s], SL::kTx);
                for (int kb = 0; kb < KB; ++kb) {
                    tma_load_2d(st + SL::oDO + kb * 8192, &map_do, &ms.full[s], kb * 64, bh * L + c * 64);
                    tma_load_2d(st + SL::oDOg + kb * 8192, &map_dog, &ms.full[s], kb * 64, bh * L + c * 64);
                    tma_load_2d(st + SL::oQ + kb * 8192, &map_qh, &ms.full[s], kb * 64, bh * L + c * 64);
                    tma_load_2d(st + SL::oK + kb * 8192, &map_kh, &ms.full[s], kb * 64, bh * L + c * 64);
                }
                tma_load_2d(st + SL::oW, &map_wt, &ms.full[s], 0, (bh * NC + c) * D);
                tma_load_2d(st + SL::oP, &map_ph, &ms.full[s], 0, (bh * NC + c) * 64);
                bulk_load_1d(smem + SL::oG + (n % kRsDecaySlots) * SL::kG, Gd + ((size_t)bh * NC + c) * 128,
                             SL::kG, &ms.full[s]);
            }
            for (int u = max(0, n - kRsStages); u < n; ++u)      // no copy in flight at retirement
                mbar_wait_drain(&ms.full[u % kRsStages], (u / kRsStages) & 1);
        }
    } else if (warp == 8) {
        constexpr uint32_t id_x1 = make_idesc(kFmtF16, 128, 64, true, true);    // A = dO (MN), B = P (MN)
        constexpr uint32_t id_x2 = make_idesc(kFmtF16, 128, 64, false, false);  // A = dS1 (TMEM), B = K
        constexpr uint32_t id_y1 = make_idesc(kFmtF16, 128, D, true, true);     // A = dOg (MN), B = Q (MN)
        constexpr uint32_t id_y2 = make_idesc(kFmtF16, 128, D, false, false, true);   // -dU~ (TMEM) x W^T
        const uint32_t tm = uniform(tmem), sm = smem_u32(smem);
        for (int n = 0; n < NC; ++n) {
            const int s = n % kRsStages;
            const uint32_t st = sm + s * SL::kStage;
            if (!wait_all(&ms.full[s], (n / kRsStages) & 1, abort_flag)) break;
            tc_fence_after_sync();
            // X1 does not involve the gradient state and its columns are free (every row thread
            // read them before its barB arrival of the previous chunk): issue it ahead.
            if (elect_one()) {
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16)
                    mma_ss(tm + SL::cX1, desc_mnmajor(st + SL::oDO + k16 * 2048, 8192),
                           desc_mnmajor(st + SL::oP + k16 * 2048, 0), id_x1, k16 != 0);
            }
            // barA: the row threads have consumed the previous chunk's Y and written dS1.
            if (!wait_all(&ms.barA, n & 1, abort_flag)) break;
            tc_fence_after_sync();
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk)
                    mma_ts(tm + SL::cX2, tm + SL::cA + kk * 8,
                           desc_kmajor(st + SL::oK + (kk >> 2) * 8192 + (kk & 3) * 32), id_x2, kk != 0);
                mma_commit(&ms.barX);
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16)
                    mma_ss(tm + SL::cY, desc_mnmajor(st + SL::oDOg + k16 * 2048, 8192),
                           desc_mnmajor(st + SL::oQ + k16 * 2048, 8192), id_y1, k16 != 0);
            }
            if (!wait_all(&ms.barB, n & 1, abort_flag)) break;
            tc_fence_after_sync();
            if (elect_one()) {
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16)
                    mma_ts(tm + SL::cY, tm + SL::cX2 + (k16 >> 1) * 32 + (k16 & 1) * 8,
                           desc_kmajor(st + SL::oW + k16 * 32), id_y2, true);
                mma_commit(&ms.barY);
                mma_commit(&ms.empty[s]);
            }
        }
    } else {
        const int q = warp & 3, half = warp >> 2;
        const int r = q * 32 + lane;
        const bool active = r < D;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const int col0 = half * kHalfCols, tk0 = half * 32;
        // The read-out gradients arrive times the power of two gsc.x (grad_scale): the gradient
        // state is carried in those units, and what leaves the kernel is multiplied by gsc.y = 1 / gsc.x.
        const float2 gsc = grad_scale(status);
        float G[kHalfCols];                                 // dS^T row r, key columns col0..
#pragma unroll
        for (int x = 0; x < kHalfCols; ++x)     // gradient arriving at the final state, if any
            G[x] = active && dstate_out ? gsc.x * dstate_out[((size_t)bh * D + col0 + x) * D + r] : 0.f;
        bool ok = true;
        for (int n = 0; n < NC && ok; ++n) {
            const int c = NC - 1 - n, s = n % kRsStages;
            const float *e1 = reinterpret_cast<const float *>(smem + SL::oG + (n % kRsDecaySlots) * SL::kG);
            const float *e2 = e1 + 64;
            // block-level routing: the update K~^T U~ of a softmax block never reached the state,
            // so the exit-state gradient does not flow into its dU~ (it still decays into dS0)
            const float commit = kBlock && block_route[((size_t)b * L + (size_t)c * 64) * H + h] ? 0.f : 1.f;
            // ---- dS1 (exit-state gradient of chunk c): fp16 operand into TMEM, then (behind the
            // arrival, off the chain) the copy the chunk kernel reads ----
            uint32_t pk[kHalfCols / 2];
            {
#pragma unroll
                for (int x = 0; x < kHalfCols / 2; ++x) pk[x] = pack_half2(G[2 * x], G[2 * x + 1]);
                if (kHalfCols == 64)
                    tmem_st32(tmem + SL::cA + half * (kHalfCols / 2) + lane_base,
                              reinterpret_cast<const uint32_t (&)[32]>(pk));
                else
                    tmem_st16(tmem + SL::cA + half * (kHalfCols / 2) + lane_base,
                              reinterpret_cast<const uint32_t (&)[16]>(pk));
                tmem_wait_st();
            }
            tc_fence_before_sync();
            mbar_arrive(&ms.barA);
            if (active) {
                uint4 *dst = reinterpret_cast<uint4 *>(dS16) + (((size_t)bh * NC + c) * (D / 8) + col0 / 8) * D + r;
#pragma unroll
                for (int x = 0; x < kHalfCols / 8; ++x)
                    dst[(size_t)x * D] = make_uint4(pk[4 * x], pk[4 * x + 1], pk[4 * x + 2], pk[4 * x + 3]);
            }
            ok = mbar_wait(&ms.full[s], (n / kRsStages) & 1, abort_flag);   // decay factors of the chunk
            if (!ok) break;
            {
                const float gC = e1[63];
#pragma unroll
                for (int x = 0; x < kHalfCols; ++x) G[x] *= gC;
            }
            // ---- dU~ for this thread's 32 tokens ----
            ok = mbar_wait(&ms.barX, n & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
            uint32_t dpk[16];
            {
                float du[32];
                uint32_t x1[32], x2[32];
                tmem_ld32(tmem + SL::cX1 + tk0 + lane_base, x1);
                tmem_ld32(tmem + SL::cX2 + tk0 + lane_base, x2);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    du[j] = fmaf(kBlock ? commit * e2[tk0 + j] : e2[tk0 + j], __uint_as_float(x2[j]),
                                 __uint_as_float(x1[j]));
#pragma unroll
                for (int x = 0; x < 16; ++x) dpk[x] = pack_half2(du[2 * x], du[2 * x + 1]);
                // into this thread's own X2 columns: 16 packed columns per 32 tokens
                tmem_st16(tmem + SL::cX2 + tk0 + lane_base, dpk);
                tmem_wait_st();
            }
            tc_fence_before_sync();
            mbar_arrive(&ms.barB);
            if (active) {                                   // the copy, behind the arrival
                uint4 *dst = reinterpret_cast<uint4 *>(dU16) + (((size_t)bh * NC + c) * 8 + tk0 / 8) * D + r;
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    dst[(size_t)x * D] = make_uint4(dpk[4 * x], dpk[4 * x + 1], dpk[4 * x + 2], dpk[4 * x + 3]);
            }
            // ---- dS0 = gamma_C dS1 + Y ----
            ok = mbar_wait(&ms.barY, n & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
#pragma unroll
            for (int cb = 0; cb < kHalfCols / 32; ++cb) {
                uint32_t y[32];
                tmem_ld32(tmem + SL::cY + col0 + cb * 32 + lane_base, y);
                tmem_wait_ld();
#pragma unroll
                for (int x = 0; x < 32; ++x) G[cb * 32 + x] += __uint_as_float(y[x]);
            }
            tc_fence_before_sync();
        }
        if (ok && active && dstate_in) {                    // what is left is the gradient of the initial state
#pragma unroll
            for (int x = 0; x < kHalfCols; ++x) dstate_in[((size_t)bh * D + col0 + x) * D + r] = gsc.y * G[x];
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, SL::kTmemCols);
    }
    if (tid == 0 && ms.abort_flag) atomicMin(status, (int)NATSL_ERR_TIMEOUT);
}

// ------------------------------------------------------------------------------------------
// 64 x 64 x 64 products on warp-level MMAs
// ------------------------------------------------------------------------------------------
constexpr int kCkThreads = 256;
constexpr int kLdH = 72;                       // row stride of a staged 64x64 fp16 tile, elements
constexpr int kTileH = 64 * kLdH;

// acc (16 x 32 block at (row0, n0) of a 64 x 64 result) += A B over k = 0..63, fp16 tiles.
// AT: A is stored [k][m] (else [m][k]);  BNK: B is stored [n][k] (else [k][n]).
template <bool AT, bool BNK>
__device__ __forceinline__ void mma64(const __half *A, const __half *B, int row0, int n0, int lane,
                                      float (&acc)[4][4]) {
    const int l7 = lane & 7, m1 = (lane >> 3) & 1, m2 = lane >> 4;
    const uint32_t sa = smem_u32(A), sb = smem_u32(B);
#pragma unroll
    for (int k0 = 0; k0 < 64; k0 += 16) {
        uint32_t a[4], b[4];
        if (!AT) ldmatrix_x4(sa + 2 * ((row0 + l7 + 8 * m1) * kLdH + k0 + 8 * m2), a);
        else ldmatrix_x4_trans(sa + 2 * ((k0 + l7 + 8 * m2) * kLdH + row0 + 8 * m1), a);
#pragma unroll
        for (int np = 0; np < 2; ++np) {       // two 8-column tiles per load
            const int nb = n0 + 16 * np;
            if (BNK) ldmatrix_x4(sb + 2 * ((nb + l7 + 8 * m2) * kLdH + k0 + 8 * m1), b);
            else ldmatrix_x4_trans(sb + 2 * ((k0 + l7 + 8 * m1) * kLdH + nb + 8 * m2), b);
            mma_m16n8k16(acc[2 * np], a, b[0], b[1]);
            mma_m16n8k16(acc[2 * np + 1], a, b[2], b[3]);
        }
    }
}

// ------------------------------------------------------------------------------------------
// Backward of the softmax branch through a query's own block under block-level routing
// (Section 4.1: both operations compute the inner-chunk correlations; Section 4.2: ds = p (dp -
// <do, o>)).  A query in a linear block reads, besides the retained tokens of earlier softmax
// blocks (the kernels over the compacted K/V handle those), the causal part of its own block of
// 64 tokens.  One CTA per linear block adds that part, five 64 x 64 x 64 products on the
// warp-level tensor-core path (fp16 tiles, fp32 accumulation):
//   S = Q K^T, dP = dO V^T;  p_ij = exp(scale s_ij - lse_i), ds_ij = scale p_ij (dp_ij - D_i), j <= i
//   dq += dS K  (added to the query-side result of the compacted kernels)
//   dk  = dS^T Q,  dv = P^T dO  (written: the tokens of a linear block have no other
//                                 softmax-branch gradient)
// with lse_i and D_i = <do_i, o_i> of the whole softmax row.  Softmax heads of 64 KB columns: KB = 1 for
// d = 64 or kG = 2 heads per linear head of d = 128 (Section 4.3; the head is then a column slice of rows
// of 128 columns, lse / Dsm are [B,H,kG,L]), KB = 2 for d = 128 (two tiles per operand: the logit products
// add over them, the three results are formed half by half).  kNorm: q and k are RMS-normalised per softmax
// head as they are staged.
template <int KB> constexpr int own_smem() { return (4 * KB + 2) * kTileH * 2; }

template <int kG, bool kNorm, int KB>
__global__ void __launch_bounds__(kCkThreads, KB == 1 ? 3 : 2)
softmax_bwd_own_block_kernel(const __nv_bfloat16 *__restrict__ q, const __nv_bfloat16 *__restrict__ k,
                             const __nv_bfloat16 *__restrict__ v, float norm_eps, const __half *__restrict__ do16,
                             const float *__restrict__ lse, const float *__restrict__ Dsm,
                             const uint8_t *__restrict__ route, float scale_sm,
                             float *__restrict__ dq_sm, float *__restrict__ dk_x,
                             float *__restrict__ dv_x, const int32_t *gsc_status, int L, int H) {
    static_assert(KB == 1 || kG == 1, "grouped heads have 64 columns");
    constexpr int D = 64 * KB, DL = D * kG;
    const float ginv = grad_scale(gsc_status).y;   // do16 and Dsm arrive times the gradient scale
    extern __shared__ __align__(16) uint8_t smraw[];
    __half *sQ = reinterpret_cast<__half *>(smraw), *sK = sQ + KB * kTileH, *sV = sK + KB * kTileH,
           *sDO = sV + KB * kTileH, *sP = sDO + KB * kTileH, *sDS = sP + kTileH;      // KB tiles per operand
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int c = blockIdx.x, bhg = blockIdx.y, bh = bhg / kG, col0 = (bhg % kG) * D, b = bh / H, h = bh % H;
    const size_t ts = (size_t)H * DL;
    const size_t tok0 = (((size_t)b * L + (size_t)c * kC) * H + h) * DL + col0;
    if (route[((size_t)b * L + (size_t)c * kC) * H + h]) return;   // a softmax block: its tokens are retained ones
    {
        const int r0 = tid >> 4, c4 = (tid & 15) * 4;
        auto cv = [](uint32_t w) {                                  // bf16 pair -> fp16 pair (exact)
            return pack_half2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
        };
#pragma unroll
        for (int kb = 0; kb < KB; ++kb)
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int r = r0 + 16 * it, tl = kb * kTileH + r * kLdH + c4;
            const size_t off = tok0 + (size_t)r * ts + kb * 64 + c4;
            const uint2 xv = *reinterpret_cast<const uint2 *>(v + off);
            const size_t offh = ((size_t)bh * L + (size_t)c * kC + r) * DL + col0 + kb * 64 + c4;      // [B,H,L,DL]
            const uint2 xo = *reinterpret_cast<const uint2 *>(do16 + offh);
            const uint2 xq = *reinterpret_cast<const uint2 *>(q + off), xk = *reinterpret_cast<const uint2 *>(k + off);
            if (kNorm) {     // RMS over the softmax head's columns of the row, 16 lanes x 4 (64-column heads)
                auto f4 = [](uint2 w) {
                    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                                       __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
                };
                const float4 fq = f4(xq), fk = f4(xk);
                float sq = fmaf(fq.x, fq.x, fmaf(fq.y, fq.y, fmaf(fq.z, fq.z, fq.w * fq.w)));
                float sk = fmaf(fk.x, fk.x, fmaf(fk.y, fk.y, fmaf(fk.z, fk.z, fk.w * fk.w)));
                if (KB == 2) {       // (128-column heads: the other block's columns too)
                    const float4 gq = f4(*reinterpret_cast<const uint2 *>(q + off + (1 - 2 * kb) * 64));
                    const float4 gk = f4(*reinterpret_cast<const uint2 *>(k + off + (1 - 2 * kb) * 64));
                    sq += fmaf(gq.x, gq.x, fmaf(gq.y, gq.y, fmaf(gq.z, gq.z, gq.w * gq.w)));
                    sk += fmaf(gk.x, gk.x, fmaf(gk.y, gk.y, fmaf(gk.z, gk.z, gk.w * gk.w)));
                }
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) {
                    sq += __shfl_xor_sync(0xffffffffu, sq, o);
                    sk += __shfl_xor_sync(0xffffffffu, sk, o);
                }
                const float rq = rsqrtf(sq / D + norm_eps), rk = rsqrtf(sk / D + norm_eps);
                *reinterpret_cast<uint2 *>(sQ + tl) = make_uint2(pack_half2(fq.x * rq, fq.y * rq), pack_half2(fq.z * rq, fq.w * rq));
                *reinterpret_cast<uint2 *>(sK + tl) = make_uint2(pack_half2(fk.x * rk, fk.y * rk), pack_half2(fk.z * rk, fk.w * rk));
            } else {
                *reinterpret_cast<uint2 *>(sQ + tl) = make_uint2(cv(xq.x), cv(xq.y));
                *reinterpret_cast<uint2 *>(sK + tl) = make_uint2(cv(xk.x), cv(xk.y));
            }
            *reinterpret_cast<uint2 *>(sV + tl) = make_uint2(cv(xv.x), cv(xv.y));
            *reinterpret_cast<uint2 *>(sDO + tl) = xo;
        }
    }
    __syncthreads();
    const int row0 = 16 * (warp & 3), n0 = 32 * (warp >> 2);
    const int iA = row0 + g, iB = iA + 8;
    const size_t rowA = (size_t)bhg * L + (size_t)c * kC + iA;
    const float l2e = 1.4426950408889634f;
    const float lseA = lse[rowA] * l2e, lseB = lse[rowA + 8] * l2e, DA = Dsm[rowA], DB = Dsm[rowA + 8];
    // dq so far, this lane's groups of four columns: asked for before the products, added after them
    const size_t col4 = tok0 + (size_t)iA * ts + n0 + 8 * (t & 1) + 4 * (t >> 1);
    float4 dq_old[2][2];
    auto load_dq = [&](int kb) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
#pragma unroll
            for (int u = 0; u < 2; ++u)
                dq_old[hf][u] = *reinterpret_cast<const float4 *>(dq_sm + col4 + (size_t)(8 * hf) * ts + kb * 64 + 16 * u);
    };
    load_dq(0);
    float pr[4][4], acc[4][4];
    auto zero = [](float (&a)[4][4]) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) a[nt][e] = 0.f;
    };
    auto put = [&](__half *X, const float (&a)[4][4]) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            *reinterpret_cast<uint32_t *>(X + iA * kLdH + n0 + 8 * nt + 2 * t) = pack_half2(a[nt][0], a[nt][1]);
            *reinterpret_cast<uint32_t *>(X + iB * kLdH + n0 + 8 * nt + 2 * t) = pack_half2(a[nt][2], a[nt][3]);
        }
    };
    // p = exp(scale s - lse), causal inside the block (mask on the exponent: no branch per element)
    zero(pr);
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) mma64<false, true>(sQ + kb * kTileH, sK + kb * kTileH, row0, n0, lane, pr);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = n0 + 8 * nt + 2 * t + (e & 1), i = e < 2 ? iA : iB;
            pr[nt][e] = ex2_ftz(j <= i ? fmaf(pr[nt][e], scale_sm * l2e, -(e < 2 ? lseA : lseB)) : -INFINITY);
        }
    put(sP, pr);
    // ds = scale p (dp - D)
    zero(acc);
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) mma64<false, true>(sDO + kb * kTileH, sV + kb * kTileH, row0, n0, lane, acc);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[nt][e] = scale_sm * pr[nt][e] * (acc[nt][e] - (e < 2 ? DA : DB));
    put(sDS, acc);
    __syncthreads();
    // Rows leave in groups of four columns: the lanes of a pair swap halves of neighbouring 8-column tiles.
    auto out4 = [&](float *dst, float (&a)[4][4], const float4 (*add)[2], int kb) {
        const bool odd = t & 1;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float &x0 = a[2 * u][e], &x1 = a[2 * u + 1][e];
                const float r = __shfl_xor_sync(0xffffffffu, odd ? x0 : x1, 1);
                x0 = odd ? r : x0;
                x1 = odd ? x1 : r;
            }
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float4 y = add ? add[hf][u] : make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4 *>(dst + col4 + (size_t)(8 * hf) * ts + kb * 64 + 16 * u) =
                    make_float4(fmaf(ginv, a[2 * u][2 * hf], y.x), fmaf(ginv, a[2 * u][2 * hf + 1], y.y),
                                fmaf(ginv, a[2 * u + 1][2 * hf], y.z), fmaf(ginv, a[2 * u + 1][2 * hf + 1], y.w));
            }
    };
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) {
        zero(acc);
        mma64<false, false>(sDS, sK + kb * kTileH, row0, n0, lane, acc);          // dq += dS K
        out4(dq_sm, acc, dq_old, kb);
        if (kb + 1 < KB) load_dq(kb + 1);
        zero(acc);
        mma64<true, false>(sDS, sQ + kb * kTileH, row0, n0, lane, acc);           // dk = dS^T Q
        out4(dk_x, acc, nullptr, kb);
        zero(acc);
        mma64<true, false>(sP, sDO + kb * kTileH, row0, n0, lane, acc);           // dv = P^T dO
        out4(dv_x, acc, nullptr, kb);
    }
}

}  // namespace

template <int D>
static cudaError_t rscan_tc_impl(const GdnTcWs &ws, const GdnTcGrads &gr, const float *dstate_out, float *dstate_in,
                                 const uint8_t *block_route, int32_t *status, Shape s, cudaStream_t st) {
    const int NC = s.L / kC;
    const uint64_t BH = (uint64_t)s.B * s.H;
    CUtensorMap mdo, mdog, mqh, mkh, mwt, mph;
    if (!tch::make_map_2d(&mdo, gr.dO16, BH * s.L, D, 64) || !tch::make_map_2d(&mdog, gr.dOg16, BH * s.L, D, 64) ||
        !tch::make_map_2d(&mqh, ws.Qh, BH * s.L, D, 64) || !tch::make_map_2d(&mkh, ws.Kh, BH * s.L, D, 64) ||
        !tch::make_map_2d(&mwt, ws.Wt, BH * NC * D, 64, D) || !tch::make_map_2d(&mph, ws.Ph, BH * NC * 64, 64, 64))
        return cudaErrorInvalidValue;
    auto kernel = block_route ? gdn_rscan_tc_kernel<D, true> : gdn_rscan_tc_kernel<D, false>;
    cudaError_t e = allow_smem(kernel, RsLayout<D>::kTotal);
    if (e != cudaSuccess) return e;
    kernel<<<s.B * s.H, kRsThreads, RsLayout<D>::kTotal, st>>>(
        mdo, mdog, mqh, mkh, mwt, mph, ws.Gd, (__half *)gr.dU16, (__half *)gr.dS16, dstate_out, dstate_in, block_route,
        status, s.L, s.H, debug_wait_kcycles());
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_gdn_rscan_tc(const GdnTcWs &ws, const GdnTcGrads &gr, const float *dstate_out, float *dstate_in,
                                const uint8_t *block_route, int32_t *status, Shape s, cudaStream_t st) {
    if (s.d == 128) return rscan_tc_impl<128>(ws, gr, dstate_out, dstate_in, block_route, status, s, st);
    return rscan_tc_impl<64>(ws, gr, dstate_out, dstate_in, block_route, status, s, st);
}

// d score per block and head (Section 4.2), for the active operation only: a softmax block sums the
// mask gradients of its 64 keys (contiguous in the compacted order), a linear block takes the kappa
// sum of its chunk; the other entry is zero.  dscore [B, L/C, H, 2] = (linear, softmax).
namespace {
__global__ void __launch_bounds__(64)
dscore_kernel(const uint8_t *__restrict__ route, const int32_t *__restrict__ sm_chunk_prefix,
              const float *__restrict__ dmask, const float *__restrict__ kap_c,
              const float *__restrict__ kappa_tok, int cap, float *__restrict__ dscore, int L, int H, int G) {
    const int c = blockIdx.x, bh = blockIdx.y, b = bh / H, h = bh % H, NC = L / kC;
    float *dst = dscore + (((size_t)b * NC + c) * H + h) * 2;
    if (route[((size_t)b * L + (size_t)c * kC) * H + h]) {
        // (grouped heads: dmask is [B,H,G,cap]; the softmax heads of a group share the block's mask)
        const int row = sm_chunk_prefix[(size_t)bh * (NC + 1) + c] + (int)threadIdx.x;
        float x = 0.f;
        for (int gg = 0; gg < G; ++gg) x += row < cap ? dmask[((size_t)bh * G + gg) * cap + row] : 0.f;
        x = warp_sum(x);
        __shared__ float part[2];
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
        __syncthreads();
        if (threadIdx.x == 0) { dst[0] = 0.f; dst[1] = part[0] + part[1]; }
    } else if (kappa_tok) {
        float x = warp_sum(kappa_tok[(size_t)bh * L + (size_t)c * kC + threadIdx.x]);
        __shared__ float part2[2];
        if ((threadIdx.x & 31) == 0) part2[threadIdx.x >> 5] = x;
        __syncthreads();
        if (threadIdx.x == 0) { dst[0] = part2[0] + part2[1]; dst[1] = 0.f; }
    } else if (threadIdx.x == 0) {
        dst[0] = kap_c[(size_t)bh * NC + c];
        dst[1] = 0.f;
    }
}
}  // namespace

cudaError_t launch_dscore(const uint8_t *route, const int32_t *sm_chunk_prefix, const float *dmask,
                          const float *kap_c, const float *kappa_tok, int cap, float *dscore, Shape s,
                          cudaStream_t st, int G) {
    dim3 grid(s.L / kC, s.B * s.H);
    dscore_kernel<<<grid, 64, 0, st>>>(route, sm_chunk_prefix, dmask, kap_c, kappa_tok, cap, dscore, s.L, s.H,
                                       G > 1 ? G : 1);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_softmax_bwd_own_block(const void *q, const void *k, const void *v,
                                         const void *do16, const float *lse, const float *Dsm,
                                         const uint8_t *route, float scale_sm, float *dq_sm,
                                         float *dk_x, float *dv_x, const int32_t *gsc, Shape s,
                                         cudaStream_t st, HeadGroups hg) {
    const int G = hg.G;
    const bool qn = hg.norm_eps >= 0.f;
    if (!s.bf16 || !((s.d == 64 && G <= 1) || (s.d == 128 && G <= 2))) return cudaErrorInvalidValue;
    auto kernel = softmax_bwd_own_block_kernel<1, false, 1>;
    int smem = own_smem<1>();
    if (s.d == 64 && qn) kernel = softmax_bwd_own_block_kernel<1, true, 1>;
    if (s.d == 128 && G == 2) kernel = qn ? softmax_bwd_own_block_kernel<2, true, 1> : softmax_bwd_own_block_kernel<2, false, 1>;
    if (s.d == 128 && G <= 1) {
        kernel = qn ? softmax_bwd_own_block_kernel<1, true, 2> : softmax_bwd_own_block_kernel<1, false, 2>;
        smem = own_smem<2>();
    }
    cudaError_t e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(s.L / kC, s.B * s.H * (G == 2 ? 2 : 1));
    kernel<<<grid, kCkThreads, smem, st>>>(
        (const __nv_bfloat16 *)q, (const __nv_bfloat16 *)k, (const __nv_bfloat16 *)v, hg.norm_eps, (const __half *)do16,
        lse, Dsm, route, scale_sm, dq_sm, dk_x, dv_x, gsc, s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

}  // namespace natsl
