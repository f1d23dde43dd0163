// Tensor-core chunkwise Gated DeltaNet (Section 3, chunkwise equations, specialised to the gated
// delta rule of Section 4.3; decay applied on every token, state update only for linear tokens)
// for bf16 storage on sm_100a: a chunk-parallel "prepare" kernel and a sequential "scan" kernel.
//
// Notation per chunk of C = 64 tokens: beta~ = (1 - route) beta, G_i = inclusive cumulative log
// decay, gamma_i = exp(G_i), Gamma_ij = exp(G_i - G_j) (j <= i):
//   A_ij = beta~_i Gamma_ij (k_i.k_j) (j < i),  T = (I + A)^-1,
//   U = T diag(beta~) V,  W = T diag(beta~ gamma) K,  P_ij = scale_la Gamma_ij (q_i.k_j) (j <= i)
//   U~ = U - W S;  O = scale_la diag(gamma) Q S + P U~;  S <- gamma_C S + (diag(gamma_C/gamma) K)^T U~
// Block-level routing (Section 4.1: both operations compute the inner-chunk correlations) uses the
// same kernels with beta~ = beta for every token and the state update of a softmax block left
// out (S <- gamma_C S), so that its chunk sees the delta rule but the later ones do not.
//
// Precision.  q, k, v are exact bf16 inputs, but T, W, U~, P and S are computed quantities: an
// 8-bit significand on them puts the layer output 1.4-2e-2 x RMS off (the whole error budget), so
// every tensor-core operand here is fp16 (11-bit significand; the inputs convert exactly, all
// magnitudes are O(1) and decay factors only shrink them).  The 16x16 diagonal blocks of T are
// inverted in fp32, its blocks below the diagonal come from fp16 products with fp32 accumulation
// (their error stays at the level of the fp16 rounding T gets as an operand anyway), and U, which
// is only ever added to an accumulator, stays fp32.
//
// All products are laid out "transposed", with the head dimension on the MMA's M axis
// (M = 128 rows = TMEM lanes = one thread each) and the 64 tokens of a chunk on N or K, so that
// every operand a thread has to produce is one contiguous 128-byte row of a swizzled tile.
#include "common.cuh"
#include "natsl_internal.h"
#include "tc_common.cuh"

namespace natsl {

namespace {

using namespace tc;

constexpr int kRowThreads = 128;

// bf16 -> fp16, 8 values in place
__device__ __forceinline__ uint4 bf16x8_to_f16x8(uint4 u) {
    const uint32_t wv[4] = {u.x, u.y, u.z, u.w};
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        o[i] = pack_half2(__uint_as_float(wv[i] << 16), __uint_as_float(wv[i] & 0xffff0000u));
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// ss + sum of the squares of 8 bf16 values; 8 bf16 values times f as fp16
__device__ __forceinline__ float square_sum8(uint4 a, float ss) {
    const uint32_t wd[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float lo = __uint_as_float(wd[e] << 16), hi = __uint_as_float(wd[e] & 0xffff0000u);
        ss = fmaf(lo, lo, fmaf(hi, hi, ss));
    }
    return ss;
}
__device__ __forceinline__ uint4 scale_f16x8(uint4 a, float f) {
    const uint32_t wd[4] = {a.x, a.y, a.z, a.w};
    uint32_t o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        o[e] = pack_half2(__uint_as_float(wd[e] << 16) * f, __uint_as_float(wd[e] & 0xffff0000u) * f);
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// ==========================================================================================
// Prepare: one CTA per chunk of one (batch, head).  One MMA group with M = 128 stacks [Q ; K] on
// the rows against K: TMEM rows 0-63 then hold Q K^T (-> P) and rows 64-127 K K^T (-> A).  Warps 0-1
// (rows 0-63) compute the gates, P and the decay factors; warps 2-3 (rows 64-127) build A, form
// T = (I + A)^-1 blockwise (16x16 diagonal blocks by substitution through warp shuffles, the rest as
// a handful of warp-level MMAs), and write the fp16 operands T beta~ and T beta~ gamma; then all
// 128 threads (one head-dimension row each) take W^T out of TMEM.  Warp 4 issues TMA and MMAs.
// What bounds it is what it moves, so it hands on as little as the scan can work from: T beta~, W^T, P and the decay
// factors (33 KB a chunk of 128 columns; the scan reads q, k, v itself and forms U on its tensor cores), and W^T, P, T beta~
// leave through shared memory as whole tiles: five CTAs per SM, 124 us before, 79 then for 4096 chunks of 128 columns.  What
// it does per chunk is a chain, so nothing sits on it that need not: the tiles are multiplied as they come (bf16; the
// normalisation's factors go on the results), k becomes the fp16 operand of W while the other warps invert: 70 us.
// kTrain: the forward of a training step also writes the fp16 copies of q and k and U, T, the cumulative decays.
// ==========================================================================================
constexpr int kPrepThreads = 160;
constexpr int kPrepMisc = 2048;

template <int D, bool kTrain> struct PrepLayout {
    static constexpr int KB = D / 64;
    static constexpr int oV = 0;                           // kTrain: V, KB sub-tiles of 64 tokens x 64
    static constexpr int oQK = kTrain ? KB * 8192 : 0;     // per 64-column block: [Q 8 KB][K 8 KB]
    static constexpr int oX = oQK + KB * 16384;            // d = 64 only: A^T, then the T operands
    static constexpr int kX = D == 64 ? 16384 : 0;
    static constexpr int oP = oX + kX;                     // not kTrain: P's tile (there P leaves by plain stores: four CTAs fit)
    static constexpr int oMisc = oP + (kTrain ? 0 : 8192);
    static constexpr int kTotal = oMisc + kPrepMisc;
    static constexpr int kLoadBytes = KB * (kTrain ? 24576 : 16384);
    static constexpr int kTmemCols = kTrain ? 128 : 64;    // [Q ; K] K^T, then (U^T and) W^T
    static constexpr int kCtas = kTrain ? 4 : 5;
};

struct PrepMisc {
    uint64_t barLoad, barConv, barM, barXfree, barT, barUW;
    uint32_t tmem_base;
    int abort_flag, wait_kcycles;   // in this order: the waits read the limit as abort_flag[1]
    alignas(16) float G[64], bt[64], btg[64], rn[128], wsum[2];   // cumulative log decay, beta~, beta~ gamma (read in pairs)
};
static_assert(sizeof(PrepMisc) <= kPrepMisc, "misc page too small");

template <int D, bool kTrain>
__global__ void __launch_bounds__(kPrepThreads, PrepLayout<D, kTrain>::kCtas)
gdn_prepare_tc_kernel(const __grid_constant__ CUtensorMap map_q,
                      const __grid_constant__ CUtensorMap map_k,
                      const __grid_constant__ CUtensorMap map_v,       // (kTrain, like map_qh, map_kh, map_u16)
                      const __grid_constant__ CUtensorMap map_qh,
                      const __grid_constant__ CUtensorMap map_kh,
                      const __grid_constant__ CUtensorMap map_u16,     // U^T fp16 and W^T [B*H*NC*D][64], box 64
                      const __grid_constant__ CUtensorMap map_wt,
                      const __grid_constant__ CUtensorMap map_tb,      // T beta~ and P [B*H*NC*64][64], box 64
                      const __grid_constant__ CUtensorMap map_ph, const float *__restrict__ g,
                      const float *__restrict__ beta, const uint8_t *__restrict__ route,
                      float scale_la, __half *__restrict__ Ph, float *__restrict__ Gd, float *__restrict__ Rn, GdnTcExport ex,
                      int32_t *status, int head_words, int L, int H, float norm_eps, int wait_kcycles) {
    using PL = PrepLayout<D, kTrain>;
    constexpr int KB = PL::KB;
    extern __shared__ __align__(1024) uint8_t smem[];
    PrepMisc &ms = *reinterpret_cast<PrepMisc *>(smem + PL::oMisc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NC = L / kC;
    // (chunk fastest: a head-fastest order, whole rows of [B,L,H,d] read by neighbouring CTAs, and L2
    // prefetches of the next wave's tiles were both measured slower)
    const int c = (int)(blockIdx.x % NC), bh = (int)(blockIdx.x / NC), b = bh / H, h = bh % H;
    const int tok0 = c * kC;
    const size_t chunk = (size_t)bh * NC + c;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicMin(status, (int)NATSL_ERR_CUDA);
        return;
    }
    if (tid == 0) {
        mbar_init(&ms.barLoad, 1);
        mbar_init(&ms.barConv, kRowThreads);
        mbar_init(&ms.barM, 1);
        mbar_init(&ms.barXfree, 1);
        mbar_init(&ms.barT, kRowThreads);
        mbar_init(&ms.barUW, 1);
        ms.abort_flag = 0;
        ms.wait_kcycles = wait_kcycles;
        fence_mbar_init();
    }
    if (warp == 4) tmem_alloc(&ms.tmem_base, PL::kTmemCols);
    // (what is set up above needs nothing of the kernel ahead, whose last CTAs may still run)
    grid_dependency_wait();
    // The forward's first kernel: clears the status page.
    if (blockIdx.x == 0 && tid < head_words) status[tid] = 0;
    __threadfence();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    // The compaction behind this kernel needs nothing of it and may start as soon as the last CTAs have (it fills the
    // multiprocessors as they drain); the scan waits for both.
    launch_dependents();
    const uint32_t tmem = ms.tmem_base, tW = tmem + (kTrain ? 64 : 0);
    volatile int *abort_flag = &ms.abort_flag;
    uint8_t *sV = smem + PL::oV, *sQK = smem + PL::oQK, *sP = smem + PL::oP;
    // The fp16 tiles of A and T during the inversion, and afterwards the two fp16 operands: in the two Q blocks
    // once K K^T / Q K^T and the q copy are done with them (d = 128), or in their own region (d = 64).
    uint8_t *xLo = D == 128 ? sQK : smem + PL::oX;
    uint8_t *xHi = D == 128 ? sQK + 16384 : smem + PL::oX + 8192;
    // A wait that runs out is recorded and the chain goes on, on whatever the tiles then hold: the row threads meet at
    // barriers, and a limit runs out for each thread by itself.  Every product is issued all the same, so the end can wait
    // for the last one.
    auto wait = [&](uint64_t *bar) { (void)mbar_wait(bar, 0, abort_flag); };
    auto wait_warp = [&](uint64_t *bar) { (void)wait_all(bar, 0, abort_flag); };

    if (warp == 4) {
        const bool leader = elect_one();
        const uint32_t tm = uniform(tmem), tWu = tm + (kTrain ? 64 : 0), sm = smem_u32(smem);
        const uint32_t aV = sm + PL::oV, aQK = sm + PL::oQK, aK = aQK + 8192, aTb = D == 128 ? aQK : sm + PL::oX,
                       aTg = aTb + (D == 128 ? 16384 : 8192);
        if (leader) {
            mbar_arrive_expect_tx(&ms.barLoad, PL::kLoadBytes);
            for (int kb = 0; kb < KB; ++kb) {
                tma_load_4d(sQK + kb * 16384 + 8192, &map_k, &ms.barLoad, kb * 64, h, tok0, b);
                tma_load_4d(sQK + kb * 16384, &map_q, &ms.barLoad, kb * 64, h, tok0, b);
                if (kTrain) tma_load_4d(sV + kb * 8192, &map_v, &ms.barLoad, kb * 64, h, tok0, b);
            }
        }
        // kTrain: the tiles as fp16; otherwise as they come (bf16, exactly; the normalisation's factors go on the results)
        wait_warp(kTrain ? &ms.barConv : &ms.barLoad);
        // ---- fp16 copies of q and k for the backward; [Q ; K] K^T ----
        if (kTrain && leader) {
            for (int kb = 0; kb < KB; ++kb) {
                tma_store_2d(&map_qh, sQK + kb * 16384, kb * 64, bh * L + tok0);
                tma_store_2d(&map_kh, sQK + kb * 16384 + 8192, kb * 64, bh * L + tok0);
            }
            tma_store_commit();
        }
        tc_fence_after_sync();
        if (elect_one()) {
            constexpr uint32_t idesc = make_idesc(kTrain ? kFmtF16 : kFmtBF16, 128, 64, false, false);
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16)
                    mma_ss(tm, desc_kmajor(aQK + kb * 16384 + k16 * 32),
                           desc_kmajor(aQK + kb * 16384 + 8192 + k16 * 32), idesc, (kb | k16) != 0);
            mma_commit(&ms.barM);
        }
        if (kTrain) {
            if (leader) tma_store_wait_read();            // the q copy has left its blocks
            wait_warp(&ms.barM);                          // and the MMAs have read them
            if (leader) mbar_arrive(&ms.barXfree);
        }
        wait_warp(&ms.barT);
        // ---- T beta~ leaves; U^T = V^T (T beta~)^T,  W^T = K^T (T beta~ gamma)^T ----
        tc_fence_after_sync();
        if (elect_one()) {
            constexpr uint32_t idesc = make_idesc(kFmtF16, 128, 64, true, false);
            if (D == 128 || !kTrain) {
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16) {
                    if (kTrain) mma_ss(tm, desc_mnmajor(aV + k16 * 2048, 8192), desc_kmajor(aTb + k16 * 32), idesc, k16 != 0);
                    // (d = 64: rows 64-127 of M are of no interest, K again)
                    mma_ss(tWu, desc_mnmajor(aK + k16 * 2048, D == 128 ? 16384 : 0), desc_kmajor(aTg + k16 * 32), idesc, k16 != 0);
                }
            } else {
                // d = 64: rows 0-63 of M are V^T, rows 64-127 are K^T (16 KB further on);
                // N = 128 = [T beta~ ; T beta~ gamma] (adjacent).
                constexpr uint32_t idesc2 = make_idesc(kFmtF16, 128, 128, true, false);
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16)
                    mma_ss(tm, desc_mnmajor(aV + k16 * 2048, 16384), desc_kmajor(aTb + k16 * 32), idesc2, k16 != 0);
            }
            mma_commit(&ms.barUW);
        }
        if (leader) {
            tma_store_2d(&map_tb, xLo, 0, (int)chunk * 64);
            tma_store_commit();
            tma_store_wait_all();
        }
    } else {
        const int r = tid, i = r & 63;
        const bool solver = r >= 64;                       // rows 64-127: K K^T
        const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
        // ---- gates (warps 0-1): beta~, inclusive cumulative log decay within the chunk ----
        if (!solver) {
            const size_t t = ((size_t)b * L + tok0 + i) * H + h;
            float G = g[t];
            const float btv = route && route[t] ? 0.f : beta[t];   // route == nullptr: beta~ = beta
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float y = __shfl_up_sync(0xffffffffu, G, o);
                if (lane >= o) G += y;
            }
            if (lane == 31) ms.wsum[warp] = G;
            named_barrier_sync(1, 64);
            if (warp == 1) G += ms.wsum[0];
            ms.G[i] = G;
            ms.bt[i] = btv;
            ms.btg[i] = btv * exp_ftz(G);
        }
        wait(&ms.barLoad);
        if (!kTrain) {
            // Factors of q's and k's rows (1 without the normalisation), while the products of the tiles run.
            float rn = 1.f;
            if (norm_eps >= 0.f) {
                const uint8_t *rowp = sQK + (solver ? 8192 : 0) + i * 128;
                float ss = 0.f;
#pragma unroll
                for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                    for (int c = 0; c < 8; ++c) ss = square_sum8(*reinterpret_cast<const uint4 *>(rowp + kb * 16384 + ((c ^ (i & 7)) << 4)), ss);
                rn = rsqrtf(ss + norm_eps);
                Rn[chunk * 128 + r] = rn;                      // (the scan scales the rows likewise)
            }
            ms.rn[r] = rn;
            named_barrier_sync(3, kRowThreads);
        } else
        // ---- training step: tiles to fp16, in place ----
        if (norm_eps >= 0.f) {
            // L2-normalised q and k for the linear operation (Section 4.3): thread r owns row r of
            // [Q ; K] (all KB blocks of it), takes its 16-byte pieces in an order that spreads the warp
            // over the banks, and scales while it converts.  V is converted as below.
            static_assert(PL::oV == 0 && PL::oQK == (kTrain ? KB * 8192 : 0), "V tile first, [Q ; K] blocks behind it");
            for (int idx = r; kTrain && idx < KB * 8192 / 16; idx += kRowThreads) {
                uint4 *pp = reinterpret_cast<uint4 *>(smem) + idx;
                *pp = bf16x8_to_f16x8(*pp);
            }
            uint8_t *rowp = sQK + (solver ? 8192 : 0) + i * 128;
            float ss = 0.f;
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    ss = square_sum8(*reinterpret_cast<const uint4 *>(rowp + kb * 16384 + ((c ^ (i & 7)) << 4)), ss);
                }
            const float rn = rsqrtf(ss + norm_eps);
            Rn[chunk * 128 + r] = rn;                          // (q's rows, k's rows: the scan scales them likewise)
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    uint4 *pp = reinterpret_cast<uint4 *>(rowp + kb * 16384 + ((c ^ (i & 7)) << 4));
                    *pp = scale_f16x8(*pp, rn);
                }
        } else {
            for (int idx = r; idx < PL::kLoadBytes / 16; idx += kRowThreads) {
                uint4 *pp = reinterpret_cast<uint4 *>(smem) + idx;   // V and [Q ; K] are contiguous
                *pp = bf16x8_to_f16x8(*pp);
            }
        }
        if (kTrain) {
            fence_proxy_async_smem();
            mbar_arrive(&ms.barConv);
        }
        wait(kTrain ? &ms.barXfree : &ms.barM);
        {   // ---- warps 0-1: P; warps 2-3: T ----
            tc_fence_after_sync();
            const float G = ms.G[i];
            if (!solver) {
                // ---- decay factors for the scan, P (lower triangle).  A real loop over 8-column
                // pieces: straight-line code that runs once per CTA is bound by instruction fetch. ----
                float *gd = Gd + chunk * 128;
                gd[i] = exp_ftz(G);
                gd[64 + i] = exp_ftz(ms.G[63] - G);
                if (ex.Gcum) ex.Gcum[(size_t)bh * L + tok0 + i] = G;
                const float fq = kTrain ? scale_la : scale_la * ms.rn[i];
                uint4 *prow = reinterpret_cast<uint4 *>(Ph + (chunk * 64 + i) * 64);
#pragma unroll 1
                for (int pc = 0; pc < 8; ++pc) {
                    uint32_t d8[8];
                    tmem_ld8(tmem + lane_base + 8 * pc, d8);
                    tmem_wait_ld();
                    float x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int j = 8 * pc + e;
                        // the mask goes on the exponent (exp(-inf) = 0): a conditional around the whole
                        // expression compiles to one divergent branch per element
                        x[e] = fq * exp_ftz(j <= i ? G - ms.G[j] : -INFINITY) * __uint_as_float(d8[e]);
                        if (!kTrain) x[e] *= ms.rn[64 + j];
                    }
                    const uint4 pw = make_uint4(pack_half2(x[0], x[1]), pack_half2(x[2], x[3]),
                                                pack_half2(x[4], x[5]), pack_half2(x[6], x[7]));
                    if (kTrain) prow[pc] = pw;
                    else *reinterpret_cast<uint4 *>(sP + sw128_offset(i, pc)) = pw;
                }
                tc_fence_before_sync();
                if (!kTrain) {
                    fence_proxy_async_smem();
                    named_barrier_sync(1, 64);
                    if (tid == 0) {
                        tma_store_2d(&map_ph, sP, 0, (int)chunk * 64);
                        tma_store_commit();
                    }
                    // k as the fp16 operand of W, while the other two warps invert
#pragma unroll
                    for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const int row = (i >> 3) + 8 * e;
                            uint4 *pp = reinterpret_cast<uint4 *>(sQK + kb * 16384 + 8192) + row * 8 + (i & 7);
                            *pp = scale_f16x8(*pp, ms.rn[64 + row]);
                        }
                    fence_proxy_async_smem();
                }
                mbar_arrive(&ms.barT);
            } else {
                // ---- T = (I + A)^-1 with 16x16 blocks (T_bb = (I + A_bb)^-1 in fp32 registers; below the
                // diagonal T_10 = -T_11 A_10 T_00, T_32 likewise, then the 32x32 block
                // T_[23][01] = -T_[23][23] A_[23][01] T_[01][01], all as warp-level fp16 MMAs) ----
                const int sw = warp - 2;                   // solver warp: block rows 2 sw and 2 sw + 1
                const int bk = i >> 4, il = i & 15;        // this thread's block row, its row inside it
                const int g8 = lane >> 2, t4 = lane & 3;   // fragment coordinates
                const float btv = kTrain ? ms.bt[i] : ms.bt[i] * ms.rn[r];
                const uint32_t aA = smem_u32(xLo), aT = smem_u32(xHi);
                // A_ij = beta~_i Gamma_ij (k_i.k_j), j < i: blocks left of the diagonal as fp16 rows of
                // the A tile (xLo), the row of the diagonal block in registers.
                float ablk[16];
#pragma unroll
                for (int jb = 0; jb < 4; ++jb) {
                    uint32_t dd[16];                       // 16 columns at a time: all 64 would not fit the registers
                    if (jb <= 2 * sw + 1) {                // (warp-uniform)
                        tmem_ld16(tmem + lane_base + 16 * jb, dd);
                        tmem_wait_ld();
                    }
                    if (jb <= bk) {
                        float a[16];
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj) {
                            const int j = 16 * jb + jj;
                            a[jj] = btv * exp_ftz(j < i ? G - ms.G[j] : -INFINITY) * __uint_as_float(dd[jj]);
                            if (!kTrain) a[jj] *= ms.rn[64 + j];
                        }
                        if (jb < bk) {
#pragma unroll
                            for (int hp = 0; hp < 2; ++hp)
                                *reinterpret_cast<uint4 *>(xLo + sw128_offset(i, 2 * jb + hp)) = make_uint4(
                                    pack_half2(a[8 * hp], a[8 * hp + 1]), pack_half2(a[8 * hp + 2], a[8 * hp + 3]),
                                    pack_half2(a[8 * hp + 4], a[8 * hp + 5]), pack_half2(a[8 * hp + 6], a[8 * hp + 7]));
                        } else {
#pragma unroll
                            for (int jj = 0; jj < 16; ++jj) ablk[jj] = a[jj];
                        }
                    }
                }
                tc_fence_before_sync();
                // Row il of the diagonal block's inverse: t_j = [j = il] - sum_{m > j} t_m A_mj, from the
                // right; A_mj sits in the registers of the thread that owns row m of the block.
                float td[16];
                {
                    float sacc[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) sacc[j] = 0.f;
                    const int grp = lane & 16;
#pragma unroll
                    for (int m = 15; m >= 0; --m) {
                        td[m] = (m == il ? 1.f : 0.f) - sacc[m];
#pragma unroll
                        for (int j = 0; j < m; ++j)
                            sacc[j] = fmaf(td[m], __shfl_sync(0xffffffffu, ablk[j], grp + m), sacc[j]);
                    }
                }
#pragma unroll
                for (int hp = 0; hp < 2; ++hp)              // fp16 copy for the products: T tile (xHi)
                    *reinterpret_cast<uint4 *>(xHi + sw128_offset(i, 2 * bk + hp)) = make_uint4(
                        pack_half2(td[8 * hp], td[8 * hp + 1]), pack_half2(td[8 * hp + 2], td[8 * hp + 3]),
                        pack_half2(td[8 * hp + 4], td[8 * hp + 5]), pack_half2(td[8 * hp + 6], td[8 * hp + 7]));
                __syncwarp();
                // Address this lane supplies to a 16x16 ldmatrix.x4 whose corner is (row0, 16-byte piece pc0).
                const int lrow = (lane & 7) + ((lane >> 3) & 1) * 8, lpc = lane >> 4;
                auto frag_addr = [&](uint32_t base, int row0, int pc0) {
                    return base + sw128_offset(row0 + lrow, pc0 + lpc);
                };
                auto pack_a = [](const float (&lo)[4], const float (&hi)[4], uint32_t (&o)[4]) {
                    o[0] = pack_half2(lo[0], lo[1]); o[1] = pack_half2(lo[2], lo[3]);
                    o[2] = pack_half2(hi[0], hi[1]); o[3] = pack_half2(hi[2], hi[3]);
                };
                const int b0 = 2 * sw, b1 = b0 + 1, br = 2 + sw;
                float t10[2][4] = {};                       // this warp's T_{b1,b0} (sign applied below)
                {
                    uint32_t fa[4], fb[4], xa[4];
                    float x[2][4] = {};
                    ldmatrix_x4(frag_addr(aT, 16 * b1, 2 * b1), fa);            // T_{b1,b1}
                    ldmatrix_x4_trans(frag_addr(aA, 16 * b1, 2 * b0), fb);      // A_{b1,b0}
                    mma_m16n8k16(x[0], fa, fb[0], fb[1]);
                    mma_m16n8k16(x[1], fa, fb[2], fb[3]);
                    pack_a(x[0], x[1], xa);
                    ldmatrix_x4_trans(frag_addr(aT, 16 * b0, 2 * b0), fb);      // T_{b0,b0}
                    mma_m16n8k16(t10[0], xa, fb[0], fb[1]);
                    mma_m16n8k16(t10[1], xa, fb[2], fb[3]);
                }
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) t10[nt][e] = -t10[nt][e];
                    *reinterpret_cast<uint32_t *>(xHi + sw128_offset(16 * b1 + g8, 2 * b0 + nt) + 4 * t4) =
                        pack_half2(t10[nt][0], t10[nt][1]);
                    *reinterpret_cast<uint32_t *>(xHi + sw128_offset(16 * b1 + g8 + 8, 2 * b0 + nt) + 4 * t4) =
                        pack_half2(t10[nt][2], t10[nt][3]);
                }
                named_barrier_sync(2, 64);                  // both warps' A rows and T blocks are in place
                float r2[4][4] = {};                        // block row br of T_[23][01]
                {
                    uint32_t fa[4], fb[4], fc[4], ya[2][4];
                    float y[4][4] = {};                     // T_{br,[23]} A_[23][01]
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks) {
                        if (ks <= sw) {                     // T_23 = 0
                            ldmatrix_x4(frag_addr(aT, 16 * br, 2 * (2 + ks)), fa);
                            ldmatrix_x4_trans(frag_addr(aA, 16 * (2 + ks), 0), fb);
                            ldmatrix_x4_trans(frag_addr(aA, 16 * (2 + ks), 2), fc);
                            mma_m16n8k16(y[0], fa, fb[0], fb[1]);
                            mma_m16n8k16(y[1], fa, fb[2], fb[3]);
                            mma_m16n8k16(y[2], fa, fc[0], fc[1]);
                            mma_m16n8k16(y[3], fa, fc[2], fc[3]);
                        }
                    }
                    pack_a(y[0], y[1], ya[0]);
                    pack_a(y[2], y[3], ya[1]);
                    ldmatrix_x4_trans(frag_addr(aT, 0, 0), fb);                 // T_00
                    mma_m16n8k16(r2[0], ya[0], fb[0], fb[1]);
                    mma_m16n8k16(r2[1], ya[0], fb[2], fb[3]);
                    ldmatrix_x4_trans(frag_addr(aT, 16, 0), fb);                // T_10
                    mma_m16n8k16(r2[0], ya[1], fb[0], fb[1]);
                    mma_m16n8k16(r2[1], ya[1], fb[2], fb[3]);
                    ldmatrix_x4_trans(frag_addr(aT, 16, 2), fb);                // T_11 (T_01 = 0)
                    mma_m16n8k16(r2[2], ya[1], fb[0], fb[1]);
                    mma_m16n8k16(r2[3], ya[1], fb[2], fb[3]);
                }
                named_barrier_sync(2, 64);                  // both tiles have been read: reuse them
                // ---- operands T diag(beta~) (xLo) and T diag(beta~ gamma) (xHi), fp16 K-major rows ----
                __half *T16 = ex.T16 ? reinterpret_cast<__half *>(ex.T16) + chunk * 4096 : nullptr;   // [8][64][8]
                auto put2 = [&](int row, int col, float v0, float v1) {
                    const float2 fb = *reinterpret_cast<const float2 *>(&ms.bt[col]);
                    const float2 fg = *reinterpret_cast<const float2 *>(&ms.btg[col]);
                    const uint32_t off = sw128_offset(row, col >> 3) + (col & 7) * 2;
                    *reinterpret_cast<uint32_t *>(xLo + off) = pack_half2(v0 * fb.x, v1 * fb.y);
                    *reinterpret_cast<uint32_t *>(xHi + off) = pack_half2(v0 * fg.x, v1 * fg.y);
                    if (T16) *reinterpret_cast<uint32_t *>(T16 + ((col >> 3) * 64 + row) * 8 + (col & 7)) = pack_half2(v0, v1);
                };
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    put2(16 * b1 + g8, 16 * b0 + 8 * nt + 2 * t4, t10[nt][0], t10[nt][1]);
                    put2(16 * b1 + g8 + 8, 16 * b0 + 8 * nt + 2 * t4, t10[nt][2], t10[nt][3]);
                }
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    put2(16 * br + g8, 8 * nt + 2 * t4, -r2[nt][0], -r2[nt][1]);
                    put2(16 * br + g8 + 8, 8 * nt + 2 * t4, -r2[nt][2], -r2[nt][3]);
                }
#pragma unroll
                for (int hp = 0; hp < 2; ++hp) {            // own row of the diagonal block
                    float xb[8], xg[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        xb[e] = td[8 * hp + e] * ms.bt[16 * bk + 8 * hp + e];
                        xg[e] = td[8 * hp + e] * ms.btg[16 * bk + 8 * hp + e];
                    }
                    *reinterpret_cast<uint4 *>(xLo + sw128_offset(i, 2 * bk + hp)) =
                        make_uint4(pack_half2(xb[0], xb[1]), pack_half2(xb[2], xb[3]),
                                   pack_half2(xb[4], xb[5]), pack_half2(xb[6], xb[7]));
                    *reinterpret_cast<uint4 *>(xHi + sw128_offset(i, 2 * bk + hp)) =
                        make_uint4(pack_half2(xg[0], xg[1]), pack_half2(xg[2], xg[3]),
                                   pack_half2(xg[4], xg[5]), pack_half2(xg[6], xg[7]));
                    if (T16)
                        *reinterpret_cast<uint4 *>(T16 + ((2 * bk + hp) * 64 + i) * 8) =
                            make_uint4(pack_half2(td[8 * hp], td[8 * hp + 1]), pack_half2(td[8 * hp + 2], td[8 * hp + 3]),
                                       pack_half2(td[8 * hp + 4], td[8 * hp + 5]), pack_half2(td[8 * hp + 6], td[8 * hp + 7]));
                }
                for (int pc = 2 * bk + 2; pc < 8; ++pc) {   // right of the diagonal block: zero
                    *reinterpret_cast<uint4 *>(xLo + sw128_offset(i, pc)) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(xHi + sw128_offset(i, pc)) = make_uint4(0, 0, 0, 0);
                    if (T16) *reinterpret_cast<uint4 *>(T16 + (pc * 64 + i) * 8) = make_uint4(0, 0, 0, 0);
                }
                fence_proxy_async_smem();
                mbar_arrive(&ms.barT);
            }
            wait(&ms.barUW);
        }
        {   // ---- (U^T and) W^T as fp16 tiles, over V and K; thread r <-> head-dimension row ----
            tc_fence_after_sync();
            auto stage = [&](uint32_t from, uint8_t *tile, int row) {
                uint32_t x[2][32];
                tmem_ld32(from + lane_base, x[0]);
                tmem_ld32(from + lane_base + 32, x[1]);
                tmem_wait_ld();
#pragma unroll
                for (int pc = 0; pc < 8; ++pc) {
                    const uint32_t *xx = &x[pc >> 2][(8 * pc) & 31];
                    *reinterpret_cast<uint4 *>(tile + sw128_offset(row, pc)) =
                        make_uint4(pack_half2(__uint_as_float(xx[0]), __uint_as_float(xx[1])),
                                   pack_half2(__uint_as_float(xx[2]), __uint_as_float(xx[3])),
                                   pack_half2(__uint_as_float(xx[4]), __uint_as_float(xx[5])),
                                   pack_half2(__uint_as_float(xx[6]), __uint_as_float(xx[7])));
                }
            };
            uint8_t *sK = sQK + 8192;                          // a 64-row block of W^T per K block
            if (D == 128) {
                if (kTrain) stage(tmem, sV + (r >> 6) * 8192, i);
                stage(tW, sK + (r >> 6) * 16384, i);
            } else if (kTrain) {                               // (warp-uniform: rows 0-63 U^T, rows 64-127 W^T)
                if (r < 64) stage(tmem, sV, i);
                else stage(tW, sK, i);
            } else if (r < 64) {
                stage(tW, sK, i);
            }
            fence_proxy_async_smem();
        }
        named_barrier_sync(3, kRowThreads);
        if (tid == 0) {
            for (int kb = 0; kb < KB; ++kb) {
                if (kTrain) tma_store_2d(&map_u16, sV + kb * 8192, 0, (int)(chunk * D) + kb * 64);
                tma_store_2d(&map_wt, sQK + 8192 + kb * 16384, 0, (int)(chunk * D) + kb * 64);
            }
            tma_store_commit();
            tma_store_wait_all();
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 4) {
        if (*abort_flag) {          // no copy, no product in flight when the CTA gives its memories back
            mbar_wait_drain(&ms.barLoad, 0);
            mbar_wait_drain(&ms.barUW, 0);
        }
        tc_fence_after_sync();
        tmem_dealloc(tmem, PL::kTmemCols);
    }
    if (tid == 0 && ms.abort_flag) atomicMin(status, (int)NATSL_ERR_TIMEOUT);
}

// ==========================================================================================
// Scan: one CTA per (batch, head) -- or per segment of its chunks, see ScanSegments --, sequential
// over chunks.  Value column r of the state (row r of
// S^T, TMEM lane r) belongs to the two threads (r, half 0) and (r, half 1) of warps q and q + 4,
// which split every row between them; warps 8 and 11 issue MMAs, warp 9 issues TMA, warps 12-15 turn the q, k and v tiles
// into fp16.  The fp32 state
// lives in the registers of its two threads (half a row each); per chunk c:
//   (0) [ahead of the chunk]                                 MMA: X = U^T = V^T (T beta~)^T
//   (a) S_c (fp16 operand, in two parts) -> TMEM;            MMA: X -= S^T W^T, QS = S^T Q^T
//   (b) X = U~^T  -> operands U~ diag(gamma_C/gamma) and U~;
//                                      MMA: dS = (U~ diag(gamma_C/gamma))^T-rows x K,  X = U~^T P^T
//   (c) [for chunk c-1, half behind the MMAs of (a), half behind those of (b)]  o_la^T = scale_la diag(gamma) QS + X
//   next chunk: S_{c+1} = gamma_C S_c + dS
// QS and X are double-buffered in TMEM so that (c) of chunk c-1 runs behind the MMAs of chunk c; its X buffer is then
// that of (0) of chunk c+1.  (U from the prepare kernel in fp32, and q and k from it in fp16, were 64 of the 88 KB that a
// chunk took through HBM and back: the prepare kernel bounds the call.)
// What bounds a chunk is the chain (a), (b): the row threads' conversions, each behind a product whose latency is its
// issue and 150 cycles.  One lane issuing from its own loop took 80 to 100 cycles an instruction (see elect_one in
// tc_common.cuh), and the warp that issues the chain must not wait for anything else, hence the second one; the
// converting warps cost 15 % of the chunk by their shared-memory traffic.  64 chunks of 128 columns: 121 us with U, q, k
// prepared and one issuing lane; 156 with the conversions here, 127 with uniform issue, two parts and two issuing warps.
// The read-out leaves the kernel as fp16 in the orientation the row threads hold it in, one tile
// per chunk in 16-byte pieces of 8 tokens: o_laT [B,H,L/C,8 pieces,d,8 tokens], row r of piece p at
// slot r ^ p.  A thread then stores four 16-byte pieces per chunk and a warp's store is 512
// contiguous bytes, where token-major rows took one narrow store per token (the load/store unit's
// instruction rate, not its bytes, bounded that version).  The softmax kernel's epilogue copies the
// 16 KB tile into shared memory as it is and reads it transposed; the slot permutation keeps
// those reads free of bank conflicts.  Warp 10 publishes the per-chunk completion counters for a kernel that
// consumes o_laT beside this one: the release fence costs a few thousand cycles and must not sit
// on the row threads' chain.
// Registers: 512 threads start with 128; the row threads' two warpgroups go up to 176, the other two down to 80, which
// is the same sum.
// ==========================================================================================
constexpr int kScanRowThreads = 256;
constexpr int kScanThreads = 512;
constexpr int kScanConvThreads = 128;
constexpr int kScanStages = 3, kScanVStages = 2;
constexpr int kScanMisc = 1024;
constexpr int kDecaySlots = 8;                             // ring of per-chunk decay factors

template <int D> struct ScanLayout {
    static constexpr int KB = D / 64;
    static constexpr int kW = D * 128;                     // W^T tile: D rows x 64 tokens (fp16)
    static constexpr int kQ = KB * 8192;                   // Q tile: 64 tokens x D
    static constexpr int kK = KB * 8192;
    static constexpr int kP = 8192;
    static constexpr int kG = 512;                         // gamma_i and gamma_C / gamma_i, 64 each; likewise Rn
    static constexpr int oW = 0, oQ = oW + kW, oK = oQ + kQ, oP = oK + kK;
    static constexpr int kStage = oP + kP;
    static constexpr int kV = KB * 8192, kVStage = kV + 8192;   // V tile, T beta~
    static constexpr int oV = kScanStages * kStage;
    static constexpr int oG = oV + kScanVStages * kVStage;      // ring of decay factors, ring of q's and k's row factors
    static constexpr int oR = oG + kDecaySlots * kG;
    static constexpr int oMisc = oR + kDecaySlots * kG;
    static constexpr int kTotal = oMisc + kScanMisc;
    static constexpr int kTmemCols = 512;
    // TMEM columns.  dS: fp32 state increment [D].  U: the fp16 operands of each thread's 32 tokens (U~ | U~
    // diag(gamma_C/gamma), 16 + 16 packed columns).  A: the fp16 state operand [D/2 packed].  QS, X: double-buffered
    // fp32 [64] each; X is U, then U~, then P U~ of its chunk.
    static constexpr int cS = 0, cU = D, cA = D + 64, cQS = cA + D / 2, cX = cQS + 128;
    static_assert(cX + 128 <= 512, "TMEM budget");
    static constexpr int kParts = D / 64;                  // parts of 32 columns in which a thread's half row is handed over
    static_assert(kTotal <= 227 * 1024, "shared memory");
};

struct ScanMisc {
    uint64_t full[kScanStages], empty[kScanStages], conv[kScanStages], fullV[kScanVStages], emptyV[kScanVStages],
        convV[kScanVStages], barA[2], barU, barWS, barB, barB2, barSU, barD3[2], barE;
    uint32_t tmem_base;
    int abort_flag, wait_kcycles;   // in this order: the waits read the limit as abort_flag[1]
    int emit_count;                 // row warps x chunks whose read-out rows have been stored
};
static_assert(sizeof(ScanMisc) <= kScanMisc, "misc page too small");

template <int D, bool kBlock>      // kBlock: block-level routing (softmax blocks are not committed)
__global__ void __launch_bounds__(kScanThreads, 1)
gdn_scan_tc_kernel(const __grid_constant__ CUtensorMap map_wt,
                   const __grid_constant__ CUtensorMap map_q,      // the layer's q, k, v [B,L,H,D] bf16, box 64 x 64
                   const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v,
                   const __grid_constant__ CUtensorMap map_ph, const __grid_constant__ CUtensorMap map_tb,
                   const float *__restrict__ Gd, const float *__restrict__ Rn, float scale_la,
                   const float *__restrict__ state_in, float *__restrict__ state_out,
                   __half *__restrict__ o_la16, float *__restrict__ o_la32, int32_t *emit_flags,
                   GdnTcExport ex, ScanSegments sg,
                   const uint8_t *__restrict__ block_route, int32_t *status, int L, int H, int wait_kcycles) {
    using SL = ScanLayout<D>;
    constexpr int KB = SL::KB;
    constexpr int kHalfCols = D / 2;                       // state columns per thread
    extern __shared__ __align__(1024) uint8_t smem[];
    ScanMisc &ms = *reinterpret_cast<ScanMisc *>(smem + SL::oMisc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NC = L / kC;
    // Which (batch, head), which segment of its chunks, and which of the two segment runs (see
    // ScanSegments): c below counts the chunks of the segment, c0 + c is the chunk's index.
    // (Everything of it is the same for all threads; little of it stays alive, for the row threads have no registers to
    // spare: with a few words spilled a call of five chunks took 3 us longer.)
    int bh = blockIdx.x, slot = blockIdx.x, c0 = 0, ncs = NC;
    bool var = false;
    if (sg.mode != 0) {
        const int runs = sg.mode == 1 ? 2 * sg.nseg - 3 : sg.nseg;                    // CTAs per (batch, head)
        bh = blockIdx.x / runs;
        const int run = blockIdx.x - bh * runs;
        var = sg.mode == 1 && run >= sg.nseg - 1;
        const int seg = var ? run - (sg.nseg - 2) : run;
        slot = bh * sg.nseg + seg;
        c0 = seg * sg.ncs;
        ncs = seg == sg.nseg - 1 ? NC - c0 : sg.ncs;
    }
    const int b = bh / H, h = bh - b * H;
    const bool emit_out = sg.mode != 1, zero_u = var;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicMin(status, (int)NATSL_ERR_CUDA);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < kScanStages; ++s) {
            mbar_init(&ms.full[s], 1); mbar_init(&ms.empty[s], 1); mbar_init(&ms.conv[s], kScanConvThreads);
        }
        for (int s = 0; s < kScanVStages; ++s) {
            mbar_init(&ms.fullV[s], 1); mbar_init(&ms.emptyV[s], 1); mbar_init(&ms.convV[s], kScanConvThreads);
        }
        mbar_init(&ms.barE, kScanRowWarps);
        for (int s = 0; s < 2; ++s) mbar_init(&ms.barA[s], kScanRowThreads);
        mbar_init(&ms.barB, kScanRowThreads);
        mbar_init(&ms.barB2, kScanRowThreads);
        mbar_init(&ms.barU, 1);
        mbar_init(&ms.barWS, 1);
        mbar_init(&ms.barSU, 1);
        for (int s = 0; s < 2; ++s) mbar_init(&ms.barD3[s], 1);
        ms.abort_flag = 0;
        ms.wait_kcycles = wait_kcycles;
        ms.emit_count = 0;
        fence_mbar_init();
    }
    if (warp == 8) tmem_alloc(&ms.tmem_base, SL::kTmemCols);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = ms.tmem_base;
    volatile int *abort_flag = &ms.abort_flag;
    // Everything before this kernel in the stream has ended from here on.  A kernel launched behind this one as a
    // programmatic dependent (the softmax branch) may start as soon as every CTA of this grid is here; it reads o_la
    // chunk by chunk behind emit_flags.
    grid_dependency_wait();
    launch_dependents();

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        if (warp == 9) {
            if (lane == 0) {
                int c = 0, nv = 0;
                bool ok = true;
                const uint32_t tx = SL::kW + SL::kK + SL::kG + (emit_out ? SL::kQ + SL::kP : 0) + (Rn ? SL::kG : 0);
                for (; c < ncs; ++c) {
                    const int s = c % kScanStages, sv = c % kScanVStages, tok = (c0 + c) * 64;
                    const size_t chunk = (size_t)bh * NC + c0 + c;
                    if (!zero_u) {
                        ok = mbar_wait(&ms.emptyV[sv], ((c / kScanVStages) & 1) ^ 1, abort_flag);
                        if (!ok) break;
                        uint8_t *sp = smem + SL::oV + sv * SL::kVStage;
                        mbar_arrive_expect_tx(&ms.fullV[sv], SL::kVStage);
                        for (int kb = 0; kb < KB; ++kb) tma_load_4d(sp + kb * 8192, &map_v, &ms.fullV[sv], kb * 64, h, tok, b);
                        tma_load_2d(sp + SL::kV, &map_tb, &ms.fullV[sv], 0, (int)chunk * 64);
                        nv = c + 1;
                    }
                    ok = mbar_wait(&ms.empty[s], ((c / kScanStages) & 1) ^ 1, abort_flag);
                    if (!ok) break;
                    uint8_t *st = smem + s * SL::kStage;
                    mbar_arrive_expect_tx(&ms.full[s], tx);
                    tma_load_2d(st + SL::oW, &map_wt, &ms.full[s], 0, (int)(chunk * D));
                    for (int kb = 0; kb < KB; ++kb) {
                        if (emit_out) tma_load_4d(st + SL::oQ + kb * 8192, &map_q, &ms.full[s], kb * 64, h, tok, b);
                        tma_load_4d(st + SL::oK + kb * 8192, &map_k, &ms.full[s], kb * 64, h, tok, b);
                    }
                    if (emit_out) tma_load_2d(st + SL::oP, &map_ph, &ms.full[s], 0, (int)chunk * 64);
                    // A decay slot is reused kDecaySlots chunks later, i.e. only after the stages of the
                    // chunks up to c + kDecaySlots - kScanStages have been released, which every row
                    // thread's work on chunk c precedes.
                    bulk_load_1d(smem + SL::oG + (c % kDecaySlots) * SL::kG, Gd + chunk * 128, SL::kG, &ms.full[s]);
                    if (Rn) bulk_load_1d(smem + SL::oR + (c % kDecaySlots) * SL::kG, Rn + chunk * 128, SL::kG, &ms.full[s]);
                }
                // No copy may be in flight when the CTA retires: the copies issued last are waited for
                // here, with a bound of their own and whatever the abort flag says.
                for (int u = max(0, c - kScanStages); u < c; ++u)
                    mbar_wait_drain(&ms.full[u % kScanStages], (u / kScanStages) & 1);
                for (int u = max(0, nv - kScanVStages); u < nv; ++u)
                    mbar_wait_drain(&ms.fullV[u % kScanVStages], (u / kScanVStages) & 1);
            }
        } else if (warp >= 12) {
            // ---- q, k, v tiles to fp16 in place (as given, exactly; normalised, times the row's factor) ----
            const int t = tid - 12 * 32;
            auto convert = [&](uint8_t *tile, const float *rn) {
                uint4 *pp = reinterpret_cast<uint4 *>(tile);
#pragma unroll 4
                for (int i = 0; i < KB * 8192 / 16 / kScanConvThreads; ++i) {
                    const int idx = t + i * kScanConvThreads;
                    const uint4 a = pp[idx];
                    pp[idx] = rn ? scale_f16x8(a, rn[(idx >> 3) & 63]) : bf16x8_to_f16x8(a);
                }
            };
            for (int c = 0; c < ncs; ++c) {
                const int s = c % kScanStages, sv = c % kScanVStages;
                if (!zero_u) {
                    if (!mbar_wait(&ms.fullV[sv], (c / kScanVStages) & 1, abort_flag)) break;
                    convert(smem + SL::oV + sv * SL::kVStage, nullptr);
                    fence_proxy_async_smem();
                    mbar_arrive(&ms.convV[sv]);
                }
                if (!mbar_wait(&ms.full[s], (c / kScanStages) & 1, abort_flag)) break;
                const float *rn = Rn ? reinterpret_cast<const float *>(smem + SL::oR + (c % kDecaySlots) * SL::kG) : nullptr;
                if (emit_out) convert(smem + s * SL::kStage + SL::oQ, rn);
                convert(smem + s * SL::kStage + SL::oK, rn ? rn + 64 : nullptr);
                fence_proxy_async_smem();
                mbar_arrive(&ms.conv[s]);
            }
        } else if (warp == 8) {
            constexpr uint32_t id_ws = make_idesc(kFmtF16, 128, 64, false, true, true);    // A = -S^T, B = W^T (MN-major)
            constexpr uint32_t id_qs = make_idesc(kFmtF16, 128, 64, false, false);   // B = Q
            constexpr uint32_t id_su = make_idesc(kFmtF16, 128, D, false, true);     // B = K (MN-major)
            constexpr uint32_t id_pu = make_idesc(kFmtF16, 128, 64, false, false);   // B = P
            const uint32_t tm = uniform(tmem), sm = smem_u32(smem);
            bool ok = true;
            for (int c = 0; c < ncs && ok; ++c) {
                const int s = c % kScanStages;
                const uint32_t st = sm + s * SL::kStage, tX = tm + SL::cX + 64 * (c & 1);
                if (!wait_all(&ms.conv[s], (c / kScanStages) & 1, abort_flag)) break;      // (and so the stage's copies)
                if (!zero_u && !wait_all(&ms.barU, c & 1, abort_flag)) break;
                // (the state's columns arrive in parts of 32 of each half of the row)
#pragma unroll
                for (int pt = 0; pt < SL::kParts; ++pt) {
                    ok = ok && wait_all(&ms.barA[pt], c & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after_sync();
                    if (elect_one()) {
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4) {
                            const int kk = D == 128 ? (k4 >> 1) * 4 + pt * 2 + (k4 & 1) : k4;
                            mma_ts(tX, tm + SL::cA + kk * 8, desc_mnmajor(st + SL::oW + kk * 2048, 0), id_ws, !zero_u || (pt | k4) != 0);
                        }
                        if (pt == SL::kParts - 1) mma_commit(&ms.barWS);
                    }
                }
                if (!ok) break;
                if (emit_out && elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        mma_ts(tm + SL::cQS + 64 * (c & 1), tm + SL::cA + kk * 8,
                               desc_kmajor(st + SL::oQ + (kk >> 2) * 8192 + (kk & 3) * 32), id_qs, kk != 0);
                }
                if (!wait_all(&ms.barB, c & 1, abort_flag)) break;
                tc_fence_after_sync();
                // The state update first: it is on the chain between the chunks.  The output product
                // behind it still reads its operand from the U columns after barSU has fired; the
                // row threads write those again behind the next chunk's W S product, issued behind it by
                // this thread, and MMAs of one thread execute in issue order.
                if (elect_one()) {
#pragma unroll
                    for (int k16 = 0; k16 < 4; ++k16)
                        mma_ts(tm + SL::cS, tm + SL::cU + (k16 >> 1) * 32 + 16 + (k16 & 1) * 8,
                               desc_mnmajor(st + SL::oK + k16 * 2048, 8192), id_su, k16 != 0);
                    mma_commit(&ms.barSU);
                }
                if (!wait_all(&ms.barB2, c & 1, abort_flag)) break;
                tc_fence_after_sync();
                if (elect_one()) {
                    if (emit_out) {
#pragma unroll
                        for (int k16 = 0; k16 < 4; ++k16)
                            mma_ts(tX, tm + SL::cU + (k16 >> 1) * 32 + (k16 & 1) * 8, desc_kmajor(st + SL::oP + k16 * 32), id_pu, k16 != 0);
                        mma_commit(&ms.barD3[c & 1]);
                    }
                    mma_commit(&ms.empty[s]);
                }
            }
        } else if (warp == 11) {
            // X of a chunk = U^T, ahead of it: once the read-out of the chunk two before has left the buffer
            constexpr uint32_t id_u = make_idesc(kFmtF16, 128, 64, true, false);     // A = V^T (MN-major), B = T beta~
            const uint32_t tm = uniform(tmem), sm = smem_u32(smem);
            for (int c = 0; c < ncs && !zero_u; ++c) {
                const int sv = c % kScanVStages;
                const uint32_t sp = sm + SL::oV + sv * SL::kVStage, tX = tm + SL::cX + 64 * (c & 1);
                if (!wait_all(&ms.convV[sv], (c / kScanVStages) & 1, abort_flag)) break;        // (and so the copies)
                // (the second chunk's, and without read-outs: once W S of the chunk before has run.  Either way no barrier here
                // can get two phases ahead of who waits for it: what completes its next phase needs this product first.)
                if (c > 0 && !(emit_out && c > 1 ? wait_all(&ms.barE, c & 1, abort_flag) : wait_all(&ms.barWS, (c - 1) & 1, abort_flag))) break;
                tc_fence_after_sync();
                if (elect_one()) {
#pragma unroll
                    for (int k16 = 0; k16 < 4; ++k16)              // (d = 64: rows 64-127 are of no interest, V again)
                        mma_ss(tX, desc_mnmajor(sp + k16 * 2048, D == 128 ? 8192 : 0), desc_kmajor(sp + SL::kV + k16 * 32), id_u, k16 != 0);
                    mma_commit(&ms.emptyV[sv]);
                    mma_commit(&ms.barU);
                }
            }
        } else if (warp == 10) {
            // Publisher: raises the per-chunk counters once all eight row warps have stored a chunk's
            // rows.  The row warps count in shared memory (after a block-scope fence); the gpu-scope
            // fence here then covers their stores, as in the usual "barrier, one thread fences and
            // sets the flag" hand-over.  Several chunks are published behind one fence when it lags.
            if (lane == 0 && emit_flags && emit_out) {
                volatile int *cnt = &ms.emit_count;
                const long long limit = wait_limit(abort_flag);
                long long t0 = clock64();
                int published = 0;
                while (published < ncs) {
                    const int done = *cnt / kScanRowWarps;
                    if (done > published) {
                        __threadfence();
                        for (int c = published; c < done; ++c)
                            red_release_add(emit_flags + (size_t)bh * NC + c0 + c, kScanRowWarps);
                        published = done;
                        t0 = clock64();
                    } else {
                        if (*abort_flag) break;
                        if (clock64() - t0 > limit) { *abort_flag = 1; break; }
                        __nanosleep(128);
                    }
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
        const int q = warp & 3, half = warp >> 2;
        const int r = q * 32 + lane;                      // value column / TMEM lane
        const bool active = r < D;                        // d = 64: rows 64-127 are zero padding
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const int col0 = half * kHalfCols;                // this thread's state columns (key dim)
        const int tk0 = half * 32;                        // ... and its tokens of every chunk
        float S[kHalfCols];                               // fp32 state at the entry of the current chunk
        const float *s_in = zero_u                    ? nullptr
                            : c0 == 0 && state_in     ? state_in + (size_t)bh * D * D
                            : c0 > 0 && sg.mode == 2  ? sg.start + (size_t)slot * D * D
                                                      : nullptr;
        if (s_in && active) {
#pragma unroll
            for (int x = 0; x < kHalfCols; ++x) S[x] = s_in[(size_t)(col0 + x) * D + r];
        } else {
#pragma unroll
            for (int x = 0; x < kHalfCols; ++x) S[x] = zero_u && active && col0 + x == r ? 1.f : 0.f;
        }
        // (c): output rows of chunk c (its QS / X buffers and decay slot are still intact), 16 of this thread's 32 tokens
        auto emit = [&](int c, int part) -> bool {
            const float *e1 = reinterpret_cast<const float *>(smem + SL::oG + (c % kDecaySlots) * SL::kG) + tk0 + 16 * part;
            if (part == 0) {                               // (q S ran ahead of it)
                if (!mbar_wait(&ms.barD3[c & 1], (c >> 1) & 1, abort_flag)) return false;
                tc_fence_after_sync();
            }
            uint32_t x[16], y[16];
            tmem_ld16(tmem + SL::cQS + 64 * (c & 1) + tk0 + 16 * part + lane_base, x);
            tmem_ld16(tmem + SL::cX + 64 * (c & 1) + tk0 + 16 * part + lane_base, y);
            tmem_wait_ld();
            tc_fence_before_sync();
            if (part == 1) {                               // this warp has read both buffers
                __syncwarp();
                if (lane == 0) mbar_arrive(&ms.barE);
            }
            float o[16];
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
                const float4 f = *reinterpret_cast<const float4 *>(e1 + i);
                o[i] = fmaf(scale_la * f.x, __uint_as_float(x[i]), __uint_as_float(y[i]));
                o[i + 1] = fmaf(scale_la * f.y, __uint_as_float(x[i + 1]), __uint_as_float(y[i + 1]));
                o[i + 2] = fmaf(scale_la * f.z, __uint_as_float(x[i + 2]), __uint_as_float(y[i + 2]));
                o[i + 3] = fmaf(scale_la * f.w, __uint_as_float(x[i + 3]), __uint_as_float(y[i + 3]));
            }
            if (o_la32 && active) {                        // fp32 token-major copy (tests, backward)
                const size_t off = (((size_t)b * L + (size_t)(c0 + c) * 64 + tk0 + 16 * part) * H + h) * D + r;
#pragma unroll
                for (int i = 0; i < 16; ++i) o_la32[off + (size_t)i * H * D] = o[i];
            }
            if (active) {
                uint4 *dst = reinterpret_cast<uint4 *>(o_la16 + ((size_t)bh * NC + c0 + c) * D * 64);
#pragma unroll
                for (int x4 = 0; x4 < 2; ++x4) {
                    const int pc = tk0 / 8 + 2 * part + x4;
                    dst[pc * D + (r ^ pc)] = make_uint4(pack_half2(o[8 * x4], o[8 * x4 + 1]), pack_half2(o[8 * x4 + 2], o[8 * x4 + 3]),
                                                        pack_half2(o[8 * x4 + 4], o[8 * x4 + 5]), pack_half2(o[8 * x4 + 6], o[8 * x4 + 7]));
                }
            }
            // this warp's rows of the chunk are stored: count it for the publisher
            if (part == 1 && emit_flags) {
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    atomicAdd(&ms.emit_count, 1);
                }
            }
            return true;
        };
        bool ok = true;
        for (int c = 0; c < ncs && ok; ++c) {
            const int s = c % kScanStages;
            const float *e2 = reinterpret_cast<const float *>(smem + SL::oG + (c % kDecaySlots) * SL::kG) + 64 + tk0;
            // Block-level routing: the delta rule runs over every block, but a softmax block's
            // update is not committed -- its state increment is multiplied by zero, so that the
            // state only decays across it (Section 4.3, the decay-always equation).
            const float commit =
                kBlock && block_route[((size_t)b * L + (size_t)(c0 + c) * 64) * H + h] ? 0.f : 1.f;
            // ---- (a) S_c = gamma_C S_{c-1} + dS_{c-1}, and as fp16 operand to TMEM: 32 columns at a time, so that their
            // products start while the next ones are worked on ----
            float gC = 1.f;
            if (c > 0) {
                gC = reinterpret_cast<const float *>(smem + SL::oG + ((c - 1) % kDecaySlots) * SL::kG)[63];
                ok = mbar_wait(&ms.barSU, (c - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after_sync();
            }
            uint32_t spk[kHalfCols / 2];
#pragma unroll
            for (int pt = 0; pt < SL::kParts; ++pt) {
                if (c > 0) {
                    uint32_t ds[32];
                    tmem_ld32(tmem + SL::cS + col0 + pt * 32 + lane_base, ds);
                    tmem_wait_ld();
#pragma unroll
                    for (int x = 0; x < 32; ++x) S[pt * 32 + x] = fmaf(S[pt * 32 + x], gC, __uint_as_float(ds[x]));
                }
#pragma unroll
                for (int x = 0; x < 16; ++x) spk[pt * 16 + x] = pack_half2(S[pt * 32 + 2 * x], S[pt * 32 + 2 * x + 1]);
                tmem_st16(tmem + SL::cA + half * (kHalfCols / 2) + pt * 16 + lane_base,
                          reinterpret_cast<const uint32_t (&)[16]>(spk[pt * 16]));
                tmem_wait_st();
                tc_fence_before_sync();
                mbar_arrive(&ms.barA[pt]);
            }
            // (exports for the backward go behind the arrivals, off the chain between the chunks)
            if (ex.S16 && active) {      // chunk-entry state: the operand itself, in pieces of keys
                uint4 *sc = reinterpret_cast<uint4 *>(ex.S16) + (((size_t)bh * NC + c0 + c) * (D / 8) + col0 / 8) * D + r;
#pragma unroll
                for (int x = 0; x < kHalfCols / 8; ++x)
                    sc[(size_t)x * D] = make_uint4(spk[4 * x], spk[4 * x + 1], spk[4 * x + 2], spk[4 * x + 3]);
            }
            // ---- behind the MMAs just released: the first half of the previous chunk's output ----
            ok = mbar_wait(&ms.full[s], (c / kScanStages) & 1, abort_flag);
            if (ok && c > 0 && emit_out) ok = emit(c - 1, 0);
            if (!ok) break;
            // ---- (b) U~ = U - W S for this thread's 32 tokens; the state update's operand first ----
            ok = mbar_wait(&ms.barWS, c & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
            uint32_t ux[32];
            tmem_ld32(tmem + SL::cX + 64 * (c & 1) + tk0 + lane_base, ux);
            tmem_wait_ld();
            uint32_t pk[16];
#pragma unroll
            for (int x = 0; x < 16; x += 2) {
                float4 f = *reinterpret_cast<const float4 *>(e2 + 2 * x);
                if (kBlock) { f.x *= commit; f.y *= commit; f.z *= commit; f.w *= commit; }
                pk[x] = pack_half2(__uint_as_float(ux[2 * x]) * f.x, __uint_as_float(ux[2 * x + 1]) * f.y);
                pk[x + 1] = pack_half2(__uint_as_float(ux[2 * x + 2]) * f.z, __uint_as_float(ux[2 * x + 3]) * f.w);
            }
            tmem_st16(tmem + SL::cU + tk0 + 16 + lane_base, pk);
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive(&ms.barB);
#pragma unroll
            for (int x = 0; x < 16; ++x) pk[x] = pack_half2(__uint_as_float(ux[2 * x]), __uint_as_float(ux[2 * x + 1]));
            tmem_st16(tmem + SL::cU + tk0 + lane_base, pk);
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive(&ms.barB2);
            if (ex.Ut16 && active) {     // U~: the operand itself, in pieces of tokens
                uint4 *ut = reinterpret_cast<uint4 *>(ex.Ut16) + (((size_t)bh * NC + c0 + c) * 8 + tk0 / 8) * D + r;
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    ut[(size_t)x * D] = make_uint4(pk[4 * x], pk[4 * x + 1], pk[4 * x + 2], pk[4 * x + 3]);
            }
            // ---- behind the MMAs just released: the rest of the previous chunk's output ----
            if (c > 0 && emit_out) ok = emit(c - 1, 1);
        }
        if (ok && emit_out) ok = emit(ncs - 1, 0) && emit(ncs - 1, 1);
        // where the state after the segment's last chunk goes
        float *final_state = sg.mode == 1 ? (zero_u ? sg.trans : sg.incr) + (size_t)slot * D * D
                             : state_out && c0 + ncs == NC ? state_out + (size_t)bh * D * D
                                                           : nullptr;
        if (ok && final_state) {
            ok = mbar_wait(&ms.barSU, (ncs - 1) & 1, abort_flag);
            if (ok) {
                tc_fence_after_sync();
                const float gC_last =
                    reinterpret_cast<const float *>(smem + SL::oG + ((ncs - 1) % kDecaySlots) * SL::kG)[63];
#pragma unroll
                for (int cb = 0; cb < kHalfCols / 32; ++cb) {
                    uint32_t ds[32];
                    tmem_ld32(tmem + SL::cS + col0 + cb * 32 + lane_base, ds);
                    tmem_wait_ld();
                    if (active) {
#pragma unroll
                        for (int x = 0; x < 32; ++x)
                            final_state[(size_t)(col0 + cb * 32 + x) * D + r] =
                                fmaf(S[cb * 32 + x], gC_last, __uint_as_float(ds[x]));
                    }
                }
            }
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

// start[1] = incr[0]; start[s+1] = M_s start[s] + B_s.  The value columns are independent: one CTA per (batch, head)
// and 16 of them.  The chain over the segments is serial, so what counts is the time of one step.  Four threads hold
// two rows of M_s in registers, a quarter each (the next segment's are fetched meanwhile); the state's columns come
// from shared memory, a row's four pieces rotated by the quarter that reads it (no bank conflicts), and packed fp32
// FMAs do the rest: a step is 1024 FMAs and 128 loads per thread.
// (With 4 columns per CTA every CTA of a pair read all of M_s, 33 MB per step for 16 pairs of 128 columns: 8 us a step.)
constexpr int kCombCols = 16;
template <int D>
__global__ void __launch_bounds__(2 * D)
scan_combine_kernel(const float *__restrict__ incr, const float *__restrict__ trans, float *__restrict__ start, int nseg) {
    constexpr int kP = D / 16;                         // 16-byte pieces of a row per thread
    __shared__ ulonglong2 Ss[2][D][4];                 // the state's 16 columns, double-buffered
    const int bh = blockIdx.y, v0 = blockIdx.x * kCombCols, r0 = (threadIdx.x >> 2) * 2, qt = threadIdx.x & 3;
    grid_dependency_wait();
    launch_dependents();
    float4 m[2][2][kP];                                // [buffer][row][piece 4 j + qt]
    auto fetch = [&](int sgi, float4 (&dst)[2][kP]) {
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            const float4 *src = reinterpret_cast<const float4 *>(trans + (((size_t)bh * nseg + sgi) * D + r0 + rr) * D) + qt;
#pragma unroll
            for (int j = 0; j < kP; ++j) dst[rr][j] = __ldg(src + 4 * j);
        }
    };
    const size_t row = (size_t)r0 * D + v0 + 4 * qt;   // this thread's results: two rows, four columns
    auto at = [&](const float *x, int sgi, int rr) {
        return reinterpret_cast<const float4 *>(x + ((size_t)bh * nseg + sgi) * D * D + row + rr * D);
    };
    float4 cur[2], inc[2];
    auto put = [&](int sgi) {                          // entry state of segment sgi
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            *const_cast<float4 *>(at(start, sgi, rr)) = cur[rr];
            ulonglong2 w;
            w.x = pack2(cur[rr].x, cur[rr].y);
            w.y = pack2(cur[rr].z, cur[rr].w);
            Ss[sgi & 1][r0 + rr][(qt + (r0 >> 2)) & 3] = w;
        }
    };
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) cur[rr] = *at(incr, 0, rr);
    if (nseg > 2) fetch(1, m[1]);
    auto step = [&](int sgi, float4 (&mm)[2][kP], float4 (&next)[2][kP]) {
        put(sgi);
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) inc[rr] = *at(incr, sgi, rr);
        if (sgi + 2 < nseg) fetch(sgi + 1, next);
        __syncthreads();
        uint64_t acc[2][8];
#pragma unroll
        for (int rr = 0; rr < 2; ++rr)
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[rr][e] = 0;
#pragma unroll
        for (int j = 0; j < kP; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int k = 16 * j + 4 * qt + e;     // (k >> 2) & 3 = qt
                uint64_t mv[2];
#pragma unroll
                for (int rr = 0; rr < 2; ++rr) {
                    const float x = e == 0 ? mm[rr][j].x : e == 1 ? mm[rr][j].y : e == 2 ? mm[rr][j].z : mm[rr][j].w;
                    mv[rr] = pack2(x, x);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const ulonglong2 sv = Ss[sgi & 1][k][(u + qt) & 3];
#pragma unroll
                    for (int rr = 0; rr < 2; ++rr) {
                        acc[rr][2 * u] = fma2(mv[rr], sv.x, acc[rr][2 * u]);
                        acc[rr][2 * u + 1] = fma2(mv[rr], sv.y, acc[rr][2 * u + 1]);
                    }
                }
            }
        // sums over the four quarters; each lane keeps its four columns
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            uint64_t h[4], o[2];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint64_t keep = qt & 2 ? acc[rr][4 + e] : acc[rr][e], give = qt & 2 ? acc[rr][e] : acc[rr][4 + e];
                h[e] = add2(keep, __shfl_xor_sync(0xffffffffu, give, 2));
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint64_t keep = qt & 1 ? h[2 + e] : h[e], give = qt & 1 ? h[e] : h[2 + e];
                o[e] = add2(keep, __shfl_xor_sync(0xffffffffu, give, 1));
            }
            const float2 a = unpack2(o[0]), b2 = unpack2(o[1]);
            cur[rr] = make_float4(a.x + inc[rr].x, a.y + inc[rr].y, b2.x + inc[rr].z, b2.y + inc[rr].w);
        }
    };
    for (int sgi = 1; sgi + 1 < nseg; sgi += 2) {
        step(sgi, m[1], m[0]);
        if (sgi + 2 < nseg) step(sgi + 1, m[0], m[1]);
    }
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) *const_cast<float4 *>(at(start, nseg - 1, rr)) = cur[rr];
}

}  // namespace

cudaError_t launch_scan_combine(const ScanSegments &sg, Shape s, cudaStream_t st, bool pdl) {
    dim3 grid(s.d / kCombCols, s.B * s.H);
    auto kernel = s.d == 128 ? scan_combine_kernel<128> : scan_combine_kernel<64>;
    cudaError_t e = launch_kernel(kernel, grid, dim3(2 * s.d), 0, st, pdl, sg.incr, sg.trans, sg.start, sg.nseg);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

template <int D, bool kTrain>
static cudaError_t prepare_tc_impl(const void *q, const void *k, const void *v, const float *g,
                                   const float *beta, const uint8_t *route, float scale_la,
                                   const GdnTcWs &ws, const GdnTcExport &ex, int32_t *status,
                                   float norm_eps, int head_words, Shape s, cudaStream_t st, bool pdl) {
    using PL = PrepLayout<D, kTrain>;
    const int NC = s.L / kC;
    const uint64_t BH = (uint64_t)s.B * s.H;
    CUtensorMap mq, mk, mwt, mtb, mph;
    if (!tch::make_map_blhd(&mq, q, s.B, s.L, s.H, D, 64) ||
        !tch::make_map_blhd(&mk, k, s.B, s.L, s.H, D, 64) ||
        !tch::make_map_2d(&mwt, ws.Wt, BH * NC * D, 64, 64) ||
        !tch::make_map_2d(&mtb, ws.Tb, BH * NC * 64, 64, 64) ||
        !tch::make_map_2d(&mph, ws.Ph, BH * NC * 64, 64, 64))
        return cudaErrorInvalidValue;
    CUtensorMap mv = mq, mqh = mq, mkh = mq, mu = mq;          // (placeholders: only a training step's are used)
    if (kTrain && (!tch::make_map_blhd(&mv, v, s.B, s.L, s.H, D, 64) || !tch::make_map_2d(&mqh, ws.Qh, BH * s.L, D, 64) ||
                   !tch::make_map_2d(&mkh, ws.Kh, BH * s.L, D, 64) || !tch::make_map_2d(&mu, ex.U16, BH * NC * D, 64, 64)))
        return cudaErrorInvalidValue;
    auto kernel = gdn_prepare_tc_kernel<D, kTrain>;
    cudaError_t e = allow_smem(kernel, PL::kTotal);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)NC * (unsigned)BH);
    count_launch();
    return launch_kernel(kernel, grid, dim3(kPrepThreads), PL::kTotal, st, pdl, mq, mk, mv, mqh, mkh, mu, mwt, mtb, mph, g, beta,
                         route, scale_la, (__half *)ws.Ph, ws.Gd, ws.Rn, ex, status, head_words, s.L, s.H, norm_eps,
                         debug_wait_kcycles());
}

template <int D>
static cudaError_t scan_tc_impl(const void *q, const void *k, const void *v, const GdnTcWs &ws, float scale_la, const float *state_in,
                                float *state_out, const ScanOut &out, const GdnTcExport &ex,
                                const ScanSegments &sg, const uint8_t *block_route, int32_t *status,
                                Shape s, cudaStream_t st, bool pdl, bool normed) {
    const int NC = s.L / kC;
    const uint64_t BH = (uint64_t)s.B * s.H;
    CUtensorMap mwt, mq, mk, mv, mph, mtb;
    if (!tch::make_map_2d(&mwt, ws.Wt, BH * NC * D, 64, D) ||
        !tch::make_map_blhd(&mq, q, s.B, s.L, s.H, D, 64) ||
        !tch::make_map_blhd(&mk, k, s.B, s.L, s.H, D, 64) ||
        !tch::make_map_blhd(&mv, v, s.B, s.L, s.H, D, 64) ||
        !tch::make_map_2d(&mph, ws.Ph, BH * NC * 64, 64, 64) ||
        !tch::make_map_2d(&mtb, ws.Tb, BH * NC * 64, 64, 64))
        return cudaErrorInvalidValue;
    auto kernel = block_route ? gdn_scan_tc_kernel<D, true> : gdn_scan_tc_kernel<D, false>;
    cudaError_t e = allow_smem(kernel,
                                         ScanLayout<D>::kTotal);
    if (e != cudaSuccess) return e;
    const int ctas = s.B * s.H * (sg.mode == 0 ? 1 : sg.mode == 1 ? 2 * sg.nseg - 3 : sg.nseg);
    count_launch();
    return launch_kernel(kernel, dim3(ctas), dim3(kScanThreads), ScanLayout<D>::kTotal, st, pdl, mwt, mq, mk, mv, mph, mtb,
                         ws.Gd, normed ? ws.Rn : nullptr, scale_la, state_in, state_out, (__half *)out.o_la16, out.o_la32,
                         out.emit_flags, ex, sg, block_route, status, s.L, s.H, debug_wait_kcycles());
}

cudaError_t launch_gdn_prepare_tc(const void *q, const void *k, const void *v, const float *g,
                                  const float *beta, const uint8_t *route, float scale_la,
                                  const GdnTcWs &ws, const GdnTcExport &ex, int32_t *status, Shape s,
                                  cudaStream_t st, int head_words, float norm_eps, bool pdl) {
#define RUN(D, TR) return prepare_tc_impl<D, TR>(q, k, v, g, beta, route, scale_la, ws, ex, status, norm_eps, head_words, s, st, pdl)
    if (s.d == 128) {
        if (ex.U16) RUN(128, true);
        RUN(128, false);
    }
    if (ex.U16) RUN(64, true);
    RUN(64, false);
#undef RUN
}

cudaError_t launch_gdn_scan_tc(const void *q, const void *k, const void *v, const GdnTcWs &ws, float scale_la, const float *state_in,
                               float *state_out, const ScanOut &out, const GdnTcExport &ex,
                               const ScanSegments &sg, const uint8_t *block_route, int32_t *status,
                               Shape s, cudaStream_t st, bool pdl, bool normed) {
    if (s.d == 128)
        return scan_tc_impl<128>(q, k, v, ws, scale_la, state_in, state_out, out, ex, sg, block_route, status, s, st, pdl, normed);
    return scan_tc_impl<64>(q, k, v, ws, scale_la, state_in, state_out, out, ex, sg, block_route, status, s, st, pdl, normed);
}

}  // namespace natsl
