// Tensor-core softmax branch over the retained tokens (Section 4.1, O_nla with mask M^nla) with
// the RMS-norm / weighted combination (Section 4.3, Norm equation) as its epilogue, for bf16
// storage on sm_100a.
//
// One CTA owns 128 consecutive queries of one (batch, head) and walks the compacted K/V of that
// head in tiles of 64 retained tokens: logits = Q K^T as a bf16 tcgen05 MMA into TMEM (q and k
// are exact bf16 inputs), online softmax in registers (one thread per query row), probabilities
// written as fp16 into the TMEM columns their logits came from and P V as an fp16 MMA with A in
// TMEM (V is gathered as fp16: the bf16 inputs convert exactly, and an 11-bit probability keeps the
// branch output within ~2e-3 of its RMS where an 8-bit one would not).  At 128 columns the logits are
// double-buffered in TMEM, so that the probabilities of tile t + 1 never wait for the product of tile
// t; at 64 a CTA has one logit tile and the SM a third CTA (see SmLayout).  K and V
// tiles arrive by TMA into two-stage rings.
// Epilogue: o_la arrives as the scan leaves it, fp16 and transposed per chunk (o_laT, one 16 KB tile
// per chunk: [8 pieces][d][8 tokens], row r of piece p at slot r ^ p); the CTA's two tiles come in
// by bulk copies (into the Q tile, free once the last Q K^T has run) while the last K/V tile is still
// being processed, and each warp reads its 32 queries out of them transposed, in the layout it reads the accumulator in,
// normalises the rows of both branches, combines them and writes them into a swizzled
// shared-memory tile that one bulk tensor store sends out.
// The kernel may run beside the scan that produces o_la (launched behind it as a programmatic
// dependent): nothing before the epilogue needs o_la, and the epilogue's load waits, bounded, for
// the per-chunk counters the scan raises (emit_flags); CTAs are then ordered by query tile first,
// so that the tiles whose chunks the scan finishes first are also scheduled first.
// Warp roles: four softmax/epilogue warps (thread r <-> query row r <-> TMEM lane r), a warp that issues the
// MMAs and one that issues the TMA loads.
// What it costs: with two key tiles of 128 columns a CTA lives 15 thousand cycles, of which 3500 pass before the first
// logits, 1100 a tile and, before its epilogue read o_laT and the accumulator in the matrix layout (ldmatrix, stmatrix,
// 16x256b), 8 thousand behind the last; now 4500.  88 us before, 75 now for 4 x 4096 tokens and 16 heads by itself, 343 and 298
// for one sequence of 32768.  With 64-column heads in the paper's mode an own-block tile takes twice as long as a retained one
// (its keys are normalised and its values converted first), and waiting for instructions is a seventh of the stalls.
// Block-level routing (template flag): after the retained tiles, one more tile per linear block of
// the CTA's two, holding that block's own 64 tokens (Section 4.1, inner-chunk correlations).
// Grouped softmax heads (template count kG; Section 4.3, several softmax heads under one linear head's
// mask): the kG softmax heads of linear head h are the kG column slices of D columns of its q, k, v.
// A CTA then serves one softmax head: its Q, K, V tiles are the slice's columns of the same tensors
// ([B,L,H,kG D] read as [B,L,H kG,D]), the retained-token lists, the counters and the weights are the
// linear head's, the softmax output is normalised over the slice and the linear read-out over its
// whole row of kG D columns, of which the CTA writes its slice.  With norm_eps >= 0 the logits are
// those of RMS-normalised q and k rows (Section 4.3), both as fp16: the K rows were normalised when
// they were gathered, the softmax threads normalise the Q tile in place before the first product.
#include "common.cuh"
#include "natsl_internal.h"
#include "route_slice.cuh"
#include "tc_common.cuh"

namespace natsl {

namespace {

using namespace tc;

constexpr int kBM = 128;        // queries per CTA
constexpr int kBN = 64;         // retained tokens per K/V tile
constexpr int kSoftmaxThreads = 128;                // one per query row
constexpr int kThreadsS = kSoftmaxThreads + 64;
constexpr int kMiscBytes = 1024;

template <int D> struct SmLayout {
    static constexpr int KB = D / 64;                    // 64-column blocks of the head dimension
    // What overlaps: at 64 columns three CTAs per SM, each one tile at a time (128 TMEM columns: O and one logit tile); at
    // 128 two CTAs, each with the next tile's logits ready (256 columns).  A CTA's tile is a chain, and a third of a CTA is
    // its fixed part, another chain, so independent CTAs fill the SM better than more tiles in flight in each.  Forward of
    // 96 pairs of 2048 tokens: 64.8 us with two warpgroups and three logit tiles in each of two CTAs, 53 now; with four
    // CTAs 54 (their 80 registers mean reading half the logits twice).
    static constexpr int kLogits = D == 64 ? 1 : 2;
    static constexpr int kCtas = D == 64 ? 3 : 2;
    static constexpr int kTmemCols = D == 64 ? 128 : 256;
    static constexpr int kStages = 2;                    // K/V tiles in flight
    static constexpr int kQBytes = KB * kBM * 128;
    static constexpr int kKStage = KB * kBN * 128;
    static constexpr int kVStage = KB * kBN * 128;
    static constexpr int oQ = 0;
    static constexpr int oK = oQ + kQBytes;
    static constexpr int oV = oK + kStages * kKStage;
    static constexpr int oMisc = oV + kStages * kVStage;
    static constexpr int kTotal = oMisc + kMiscBytes;
};

struct Misc {                    // lives in the last kMiscBytes of the CTA's shared memory
    uint64_t barQ, barQn, barKn[2], fullK[2], emptyK[2], fullV[2], emptyV[2], barS[2], barP[2], barO[2], barE;
    uint32_t tmem_base;
    int abort_flag, wait_kcycles;   // in this order: the waits read the limit as abort_flag[1]
    uint32_t kept[kBM / 32];        // which of the CTA's own tokens are retained
};
static_assert(sizeof(Misc) <= kMiscBytes, "misc page too small");

// Sum of squares of N 16-byte pieces of bf16 of one swizzled row, and the same pieces rewritten as fp16 times f.
template <int N> __device__ __forceinline__ float row_square_sum(const uint8_t *rowp, int p0, int x) {
    float ss = 0.f;
#pragma unroll
    for (int c = 0; c < N; ++c) {
        const uint4 a = *reinterpret_cast<const uint4 *>(rowp + (((p0 + c) ^ x) << 4));
        const uint32_t wd[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float lo = __uint_as_float(wd[e] << 16), hi = __uint_as_float(wd[e] & 0xffff0000u);
            ss = fmaf(lo, lo, fmaf(hi, hi, ss));
        }
    }
    return ss;
}
template <int N> __device__ __forceinline__ void row_to_fp16(uint8_t *rowp, int p0, int x, float f) {
#pragma unroll
    for (int c = 0; c < N; ++c) {
        uint4 *pp = reinterpret_cast<uint4 *>(rowp + (((p0 + c) ^ x) << 4));
        const uint4 a = *pp;
        const uint32_t wd[4] = {a.x, a.y, a.z, a.w};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            o[e] = pack_half2(__uint_as_float(wd[e] << 16) * f, __uint_as_float(wd[e] & 0xffff0000u) * f);
        *pp = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// kBlock: block-level routing (own-block tiles after the retained ones); kG: softmax heads per linear
// head; kNorm: RMS-normalised q and k (norm_eps is read only then)
template <int D, bool kBlock, int kG, bool kNorm>
__global__ void __launch_bounds__(kThreadsS, SmLayout<D>::kCtas)
softmax_combine_tc_kernel(const __grid_constant__ CUtensorMap map_q,
                          const __grid_constant__ CUtensorMap map_k,
                          const __grid_constant__ CUtensorMap map_v,
                          const __grid_constant__ CUtensorMap map_out,    // out [B,L,H,D] bf16, box 128 x 64, if has_out
                          const __grid_constant__ CUtensorMap map_kd,     // the layer's k, v [B,L,H,D] bf16, box
                          const __grid_constant__ CUtensorMap map_vd,     //   64 x 64: own-block tiles (block routing)
                          const uint8_t *__restrict__ block_route, int appending, int cap, int capv, const int32_t *__restrict__ sm_idx,
                          const int32_t *__restrict__ sm_chunk_prefix,
                          const __half *__restrict__ o_laT, const int32_t *emit_flags,
                          const float *__restrict__ w,
                          float scale_sm, float eps, float norm_eps, int has_out, float *__restrict__ o_nla,
                          float *__restrict__ lse, int32_t *sm_len, int len_cap, int32_t *status, int L, int H,
                          int wait_kcycles, int segs, int seg_tiles) {
    using SL = SmLayout<D>;
    constexpr int KB = SL::KB, kStages = SL::kStages, kLogits = SL::kLogits, kAhead = kLogits - 1;
    constexpr int DL = D * kG;                            // columns of the linear head
    // the two o_laT tiles of the epilogue land in the Q tile and, for grouped heads, the K ring behind it
    static_assert(2 * DL * 128 <= SL::kQBytes + (kG > 1 ? kStages * SL::kKStage : 0), "o_laT tiles do not fit");
    static_assert(kG == 1 || SL::oK == SL::oQ + SL::kQBytes, "K ring must follow the Q tile");
    extern __shared__ __align__(1024) uint8_t smem[];
    Misc &ms = *reinterpret_cast<Misc *>(smem + SL::oMisc);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kMmaWarp = kSoftmaxThreads / 32, kTmaWarp = kMmaWarp + 1;
    const int NP = (L + kBM - 1) / kBM, NC = L / kC;
    // grid = (B*H, NP).  Beside the scan: in the order in which the scan finishes the query tiles -- ascending, a
    // position of every one of its segments (segs of seg_tiles tiles each, the last one longer) before the next
    // position -- and all (batch, head) pairs of a tile before the next tile.  Otherwise: long rows first.
    int p = emit_flags ? (int)blockIdx.y : NP - 1 - (int)blockIdx.y;
    if (emit_flags && p < segs * seg_tiles) p = (p % segs) * seg_tiles + p / segs;
    // blockIdx.x = (batch, linear head, softmax head of the group); H counts linear heads
    const int bhg = blockIdx.x, bh = bhg / kG, sg = bhg % kG, b = bh / H, h = bh % H;
    const int hq = h * kG + sg;                           // head index in the [B,L,H kG,D] view

    // This grid starts before the scan has ended and takes from it what the counters cover, which the final state is
    // not.  It must not end before the scan: a kernel that waits for this one -- a decode step launched as its
    // programmatic dependent, or any kernel behind it in a captured graph -- takes it that everything ahead has ended.
    // One thread of the query tile that the scan finishes last is enough.
    auto end_behind_scan = [&]() {
        if (tid == 0 && blockIdx.x == 0 && blockIdx.y == gridDim.y - 1) grid_dependency_wait();
    };

    if ((smem_u32(smem) & 1023u) != 0) {              // operand tiles need 1024-byte alignment
        if (tid == 0) atomicMin(status, (int)NATSL_ERR_CUDA);
        end_behind_scan();
        return;
    }
    if (warp == kMmaWarp) {
        tmem_alloc(&ms.tmem_base, SL::kTmemCols);
        launch_dependents();                          // (behind the allocation: see there)
    }
    // The TMA warp sets the barriers up and requests the Q tile before anything else, and goes on to the key tiles as soon
    // as it knows how many there are: it needs nothing of what the other warps set up.
    if (warp == kTmaWarp && lane == 0) {
        mbar_init(&ms.barQ, 1);
        mbar_init(&ms.barQn, kSoftmaxThreads);       // normalised queries written (NATSL_QK_NORM)
        mbar_init(&ms.barKn[0], kSoftmaxThreads);    // ... and the keys of an own-block tile: one barrier per tile,
        mbar_init(&ms.barKn[1], kSoftmaxThreads);    //     each completing once
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&ms.fullK[s], 1); mbar_init(&ms.emptyK[s], 1);
            mbar_init(&ms.fullV[s], 1); mbar_init(&ms.emptyV[s], 1);
        }
        for (int s = 0; s < kLogits; ++s) { mbar_init(&ms.barS[s], 1); mbar_init(&ms.barP[s], kSoftmaxThreads); }
        for (int s = 0; s < 2; ++s) mbar_init(&ms.barO[s], 1);
        mbar_init(&ms.barE, 1);
        ms.abort_flag = 0;
        ms.wait_kcycles = wait_kcycles;
        fence_mbar_init();
        prefetch_tmap(&map_q); prefetch_tmap(&map_k); prefetch_tmap(&map_v);
        mbar_arrive_expect_tx(&ms.barQ, SL::kQBytes);
        for (int kb = 0; kb < KB; ++kb)
            tma_load_4d(smem + SL::oQ + kb * kBM * 128, &map_q, &ms.barQ, kb * 64, hq, p * kBM, b);
    }
    if (warp == kTmaWarp) {
        __syncwarp();
        named_barrier_arrive(4, kThreadsS);
    }
    const int c0 = 2 * p, c1 = min(2 * p + 2, NC);
    const int32_t *pre = sm_chunk_prefix + (size_t)bh * (NC + 1);
    const int n_full = min(pre[c0], cap);             // retained tokens before the CTA's chunks
    const int n_end = min(pre[c1], cap);              // ... up to the end of the CTA's chunks
    const int T = (n_end + kBN - 1) / kBN;
    // Block-level routing (Section 4.1, intra-chunk correlations of both operations): a query in a
    // linear block also reads the causal part of its own block, whose tokens are not among the
    // retained ones.  Each linear block of the CTA's two adds one tile, taken from the layer's
    // own k and v after the retained tiles (the softmax threads turn its V tile into fp16 in
    // place, exactly as the gather does for the retained rows).
    int nx = 0, xc0 = 0;                                // number of own-block tiles; block of the first
    if (kBlock)
        for (int e = 0; e < c1 - c0; ++e)
            if (block_route[((size_t)b * L + (size_t)(c0 + e) * kC) * H + h] == 0) {
                if (nx == 0) xc0 = e;
                ++nx;
            }
    const int T2 = kBlock ? T + nx : T;
    auto own_block = [&](int t) { return t == T ? xc0 : 1; };   // block (0 or 1) of own-block tile t >= T

    if (sg == 0 && tid == 0) {
        // Block-level routing: one decision per chunk, so a chunk keeps all of its tokens or none.
        if (kBlock)
            for (int e = c0; e < c1; ++e) {
                const int n = pre[e + 1] - pre[e];
                if (n != 0 && n != kC) atomicMin(status, (int)NATSL_ERR_ROUTE);
            }
        // The stored length never exceeds the rows the cache has (the gather stops there and the overflow is
        // reported), so a later decode step cannot be led past the head's rows.
        if (c1 == NC) {
            const int n = pre[NC];
            if (n > len_cap) atomicMin(status, (int)NATSL_ERR_CACHE_FULL);
            if (sm_len) sm_len[bh] = min(n, len_cap);
        }
    }
    if (tid < kBM / 32) ms.kept[tid] = 0u;
    tc_fence_before_sync();
    if (warp != kTmaWarp) named_barrier_sync(4, kThreadsS);
    tc_fence_after_sync();
    const uint32_t tmem = ms.tmem_base;                   // (not the TMA warp's business)
    const uint32_t tO = tmem + 64 * kLogits;            // (logits at 0, and 64 at 128 columns)
    auto tS = [&](int t) { return tmem + 64 * (t % kLogits); };
    volatile int *abort_flag = &ms.abort_flag;

    if (warp == kTmaWarp) {
        // ------------------------------ TMA producer ------------------------------
        if (lane == 0) {
            int nk = 0, nv = 0;                 // K / V tiles requested so far
            bool ok = true;
            if (T2 > 0) {                       // nothing is loaded for a tile that sees no key at all
                // K and V tiles have their own rings: a K tile is free as soon as its Q K^T has run
                // (early), a V tile only after its P V; K(u) is therefore requested before V(u-1).
                for (int u = 0; u <= T2 && ok; ++u) {
                    if (u < T2) {
                        const int s = u % kStages;
                        ok = mbar_wait(&ms.emptyK[s], ((u / kStages) & 1) ^ 1, abort_flag);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&ms.fullK[s], SL::kKStage);
                        for (int kb = 0; kb < KB; ++kb) {
                            uint8_t *dst = smem + SL::oK + s * SL::kKStage + kb * kBN * 128;
                            if (!kBlock || u < T) tma_load_2d(dst, &map_k, &ms.fullK[s], sg * D + kb * 64, bh * cap + u * kBN);
                            else tma_load_4d(dst, &map_kd, &ms.fullK[s], kb * 64, hq, (c0 + own_block(u)) * kC, b);
                        }
                        nk = u + 1;
                    }
                    if (u >= 1) {
                        const int t = u - 1, s = t % kStages;
                        ok = mbar_wait(&ms.emptyV[s], ((t / kStages) & 1) ^ 1, abort_flag);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&ms.fullV[s], SL::kVStage);
                        for (int kb = 0; kb < KB; ++kb) {
                            uint8_t *dst = smem + SL::oV + s * SL::kVStage + kb * kBN * 128;
                            if (!kBlock || t < T) tma_load_2d(dst, &map_v, &ms.fullV[s], sg * D + kb * 64, bh * capv + t * kBN);
                            else tma_load_4d(dst, &map_vd, &ms.fullV[s], kb * 64, hq, (c0 + own_block(t)) * kC, b);
                        }
                        nv = t + 1;
                    }
                }
            }
            mbar_wait_drain(&ms.barQ, 0);       // (the Q tile's copy, read or not, before its place is reused)
            // beside the scan: the tile's chunks of o_la are complete once all row warps of the scan
            // CTA have raised the chunk's counter
            if (emit_flags) {
                for (int c = c0; c < c1 && ok; ++c)
                    ok = wait_counter_ge(emit_flags + (size_t)bh * NC + c, kScanRowWarps, abort_flag);
                fence_proxy_async_all();
            }
            // the Q tile and the K ring are free once the last Q K^T has run
            if (T2 > 0 && ok) ok = mbar_wait(&ms.emptyK[(T2 - 1) % kStages], ((T2 - 1) / kStages) & 1, abort_flag);
            bool e_issued = false;
            if (ok) {                           // the o_laT tiles of the CTA's one or two chunks
                mbar_arrive_expect_tx(&ms.barE, (c1 - c0) * DL * 128);
                for (int e = 0; e < c1 - c0; ++e)
                    bulk_load_1d(smem + SL::oQ + e * (DL * 128), o_laT + ((size_t)bh * NC + c0 + e) * DL * 64,
                                 DL * 128, &ms.barE);
                e_issued = true;
            }
            // No copy may be in flight when the CTA retires, aborted or not: wait (with a bound of
            // their own) for the copies issued last.
            for (int u = max(0, nk - kStages); u < nk; ++u)
                mbar_wait_drain(&ms.fullK[u % kStages], (u / kStages) & 1);
            for (int u = max(0, nv - kStages); u < nv; ++u)
                mbar_wait_drain(&ms.fullV[u % kStages], (u / kStages) & 1);
            if (e_issued) mbar_wait_drain(&ms.barE, 0);
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------ MMA issuer ------------------------------
        // (as a warp, with uniform operands: see elect_one)
        const int Tu = (int)uniform((uint32_t)T), T2u = (int)uniform((uint32_t)T2);
        if (T2u > 0) {
            // logits: q and k as given are bf16; normalised ones are fp16 (see the softmax threads)
            constexpr uint32_t idesc_qk = make_idesc(kNorm ? kFmtF16 : kFmtBF16, kBM, kBN, false, false);
            constexpr uint32_t idesc_pv = make_idesc(kFmtF16, kBM, D, false, true);
            const uint32_t tm = uniform(tmem), tOu = tm + 64 * kLogits, sm = smem_u32(smem), aQ = sm + SL::oQ;
            auto tSu = [&](int t) { return tm + 64 * (t % kLogits); };
            // (normalisation with block-level routing: an own-block tile's keys arrive raw and are
            // normalised in place by the softmax threads first.  One single-phase barrier per own-block
            // tile, of which a CTA has at most two: with one barrier and a phase per tile, nothing kept the
            // softmax threads from completing the second phase before this warp had looked at the
            // first -- a parity wait then never returns.)
            auto own_keys_ready = [&](int t) {
                return !(kBlock && kNorm) || t < Tu || wait_all(&ms.barKn[t - Tu], 0, abort_flag);
            };
            // logits of tile t, as soon as its keys are there (and its TMEM columns free: MMAs run in issue order)
            auto next_qk = [&](int t) {
                if (t >= T2u) return true;
                if (!wait_all(&ms.fullK[t % kStages], (t / kStages) & 1, abort_flag) || !own_keys_ready(t)) return false;
                tc_fence_after_sync();
                const uint32_t aK = sm + SL::oK + (t % kStages) * SL::kKStage;
                if (elect_one()) {
#pragma unroll
                    for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                        for (int k16 = 0; k16 < 4; ++k16)
                            mma_ss(tSu(t), desc_kmajor(aQ + kb * kBM * 128 + k16 * 32),
                                   desc_kmajor(aK + kb * kBN * 128 + k16 * 32), idesc_qk, (kb | k16) != 0);
                    mma_commit(&ms.emptyK[t % kStages]);
                    mma_commit(&ms.barS[t % kLogits]);
                }
                return true;
            };
            bool ok = wait_all(&ms.barQ, 0, abort_flag) && (!kNorm || wait_all(&ms.barQn, 0, abort_flag));
            for (int t = 0; t < kAhead && ok; ++t) ok = next_qk(t);
            for (int t = 0; ok && t < T2u; ++t) {
                // (keys that the softmax threads still have to normalise must not hold up this tile's product)
                const bool late = kAhead > 0 && kBlock && kNorm && t + kAhead >= Tu;
                if (!late) ok = next_qk(t + kAhead);
                ok = ok && wait_all(&ms.barP[t % kLogits], (t / kLogits) & 1, abort_flag) &&
                     wait_all(&ms.fullV[t % kStages], (t / kStages) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t aV = sm + SL::oV + (t % kStages) * SL::kVStage;
                if (elect_one()) {
#pragma unroll
                    for (int k16 = 0; k16 < 4; ++k16)      // A = P(t): fp16 pairs in the first 32 columns of S(t)
                        mma_ts(tOu, tSu(t) + k16 * 8, desc_mnmajor(aV + k16 * 2048, kBN * 128), idesc_pv, (t | k16) != 0);
                    mma_commit(&ms.emptyV[t % kStages]);
                    mma_commit(&ms.barO[t & 1]);
                }
                if (late) ok = next_qk(t + kAhead);
            }
        }
    } else {
        // ------------------------------ softmax + epilogue ------------------------------
        const int q = warp;                             // quarter of the rows
        const int r = tid;                              // query row inside the tile, TMEM lane
        const int i_abs = p * kBM + r;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const float sl2 = scale_sm * 1.4426950408889634f;
        float m = -INFINITY, l = 0.f;                   // maximum (base 2) the row's sum is relative to; the sum
        bool ok = true;
        // Which of the CTA's own tokens are retained (sm_idx lists this call's retained tokens; when the call
        // appends to a cache, pre[0] were there before): the keys a row sees are then a population count.
        if (n_full + r < n_end) {
            const int rel = sm_idx[(size_t)bh * L + n_full + r - (appending ? pre[0] : 0)] - p * kBM;
            atomicOr(&ms.kept[(rel >> 5) & 3], 1u << (rel & 31));
        }
        if (kNorm && T2 > 0) {
            // RMS-normalised queries (Section 4.3): thread r rewrites row r (bf16, as loaded) as fp16 of the normalised
            // row, over the D columns of its softmax head;
            // the keys were normalised and stored as fp16 when they were gathered, so the logit product is
            // an fp16 MMA (bf16 keeps 8 bits: rounding the normalised keys to it alone costs 2.8e-2 of the
            // branch output's RMS).
            ok = mbar_wait(&ms.barQ, 0, abort_flag);
            uint8_t *rowp = smem + SL::oQ + r * 128;
            float ss = 0.f;
            if (ok)
#pragma unroll
                for (int kb = 0; kb < KB; ++kb) ss += row_square_sum<8>(rowp + kb * kBM * 128, 0, r & 7);
            if (ok) {
                const float rq = rsqrtf(ss / D + norm_eps);
#pragma unroll
                for (int kb = 0; kb < KB; ++kb) row_to_fp16<8>(rowp + kb * kBM * 128, 0, r & 7, rq);
                fence_proxy_async_smem();
                mbar_arrive(&ms.barQn);
            }
        }
        float2 wv = make_float2(0.5f, 0.5f);             // (w_nla, w_la) of this row
        if (w && i_abs < L) wv = __ldg(reinterpret_cast<const float2 *>(w + (((size_t)b * L + i_abs) * H + h) * 2));
        named_barrier_sync(1, kSoftmaxThreads);
        // The compacted keys are in position order, so row i sees exactly the first `cnt` of them:
        // all n_full earlier ones plus those of the CTA's own chunks at positions <= i.
        int cnt = n_full + __popc(ms.kept[q] & ((2u << lane) - 1u));
#pragma unroll
        for (int e = 0; e < kBM / 32 - 1; ++e) cnt += e < q ? __popc(ms.kept[e]) : 0;
        for (int t = 0; ok && t < T2; ++t) {
            if (kBlock && kNorm && t >= T) {
                // Keys of an own-block tile (block-level routing with normalisation): raw bf16 rows from the
                // layer's k; two threads per row rewrite it as fp16 of the RMS-normalised row.  (Every thread arrives for
                // itself: threads whose wait ran out leave the loop, so none may wait here for the others.)
                ok = mbar_wait(&ms.fullK[t % kStages], (t / kStages) & 1, abort_flag);
                if (!ok) break;
                uint8_t *rowp = smem + SL::oK + (t % kStages) * SL::kKStage + (r >> 1) * 128;
                float ss = 0.f;
#pragma unroll
                for (int kb = 0; kb < KB; ++kb) ss += row_square_sum<4>(rowp + kb * kBN * 128, 4 * (r & 1), (r >> 1) & 7);
                ss += __shfl_xor_sync(0xffffffffu, ss, 1);
                const float rk = rsqrtf(ss / D + norm_eps);
#pragma unroll
                for (int kb = 0; kb < KB; ++kb) row_to_fp16<4>(rowp + kb * kBN * 128, 4 * (r & 1), (r >> 1) & 7, rk);
                fence_proxy_async_smem();
                mbar_arrive(&ms.barKn[t - T]);
            }
            ok = mbar_wait(&ms.barS[t % kLogits], (t / kLogits) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
            // Keys of this tile the row sees: an own-block tile's 0 .. r % 64 if the row is in that block, else those
            // of the compacted order before `cnt`.
            const int vis = kBlock && t >= T ? ((r >> 6) == own_block(t) ? (r & 63) + 1 : 0) : cnt - t * kBN;
            const bool cut_off = !__all_sync(0xffffffffu, vis >= kBN);   // some row of the warp is cut off here
            // 32 raw logits at a time (the scale goes into the exponent's FMA)
            auto load_half = [&](int hf, float (&x)[32]) {
                tmem_ld32(tS(t) + lane_base + 32 * hf, reinterpret_cast<uint32_t (&)[32]>(x));
                tmem_wait_ld();
                if (cut_off) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) x[c] = c + 32 * hf < vis ? x[c] : -INFINITY;
                }
            };
            auto max_half = [&](const float (&x)[32]) {      // four independent chains
                float m4[4] = {x[0], x[1], x[2], x[3]};
#pragma unroll
                for (int c = 4; c < 28; c += 8)
#pragma unroll
                    for (int e = 0; e < 4; ++e) m4[e] = max3(m4[e], x[c + e], x[c + 4 + e]);
#pragma unroll
                for (int e = 0; e < 4; ++e) m4[e] = fmaxf(m4[e], x[28 + e]);
                return fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
            };
            float xa[32], xb[32];
            load_half(0, xa);
            float mx = max_half(xa);
            load_half(1, xb);
            // (scale_sm > 0, checked on the host: the maximum of the raw logits is the maximum logit)
            mx = fmaxf(mx, max_half(xb)) * sl2;
            // The running maximum only has to
            // bound the exponents, not equal the true maximum: it is raised (and O rescaled) only when a logit
            // exceeds it by more than 8 (base 2), so probabilities stay below 2^8 and, for inputs whose logits
            // vary little, the accumulator is never touched between the tiles.  lse = m + log2(l) holds for
            // any such m.
            const float m_old = m;
            m = (mx > m_old + 8.f || m_old == -INFINITY) ? fmaxf(m_old, mx) : m_old;
            const float m_use = m == -INFINITY ? 0.f : m;
            uint64_t ps[2] = {0ull, 0ull};
            uint32_t pk[32];                            // P(t), over the logits this thread has consumed
            const uint64_t sl22 = pack2(sl2, sl2), nm2 = pack2(-m_use, -m_use);
            auto exps = [&](int hf, const float (&x)[32]) {
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                    const float2 e = unpack2(fma2(pack2(x[c], x[c + 1]), sl22, nm2));
                    const float p0 = ex2_ftz(e.x), p1 = ex2_ftz(e.y);
                    ps[(c >> 1) & 1] = add2(ps[(c >> 1) & 1], pack2(p0, p1));
                    pk[16 * hf + (c >> 1)] = pack_half2(p0, p1);
                }
            };
            exps(1, xb);
            exps(0, xa);
            const float2 psf = unpack2(add2(ps[0], ps[1]));
            l = l * ex2_ftz(m_old - m_use) + (psf.x + psf.y);    // (m = -inf: l is 0)
            tmem_st32(tS(t) + lane_base, pk);
            if (t > 0 && __any_sync(0xffffffffu, m != m_old)) {
                // (the logits of tile t were issued behind the product of tile t - 2 at the latest, so the phase of this
                // barrier before tile t - 1's has completed and the parity is unambiguous)
                ok = mbar_wait(&ms.barO[(t - 1) & 1], ((t - 1) >> 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after_sync();
                const float corr = ex2_ftz(m_old - m_use);   // m = -inf -> 0; unchanged m -> 1
#pragma unroll 1
                for (int cb = 0; cb < D / 32; ++cb) {
                    uint32_t ov[32];
                    tmem_ld32(tO + lane_base + cb * 32, ov);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 32; ++c) ov[c] = __float_as_uint(__uint_as_float(ov[c]) * corr);
                    tmem_st32(tO + lane_base + cb * 32, ov);
                }
            }
            tmem_wait_st();
            if (kBlock && t >= T) {   // own-block tile: its V rows arrived as bf16; fp16 in place (exact)
                ok = mbar_wait(&ms.fullV[t % kStages], (t / kStages) & 1, abort_flag);
                if (!ok) break;
                uint4 *vt = reinterpret_cast<uint4 *>(smem + SL::oV + (t % kStages) * SL::kVStage);
                for (int i = r; i < SL::kVStage / 16; i += kSoftmaxThreads) {
                    const uint4 a = vt[i];
                    auto cv = [](uint32_t wd) {
                        return pack_half2(__uint_as_float(wd << 16), __uint_as_float(wd & 0xffff0000u));
                    };
                    vt[i] = make_uint4(cv(a.x), cv(a.y), cv(a.z), cv(a.w));
                }
                fence_proxy_async_smem();
            }
            tc_fence_before_sync();
            mbar_arrive(&ms.barP[t % kLogits]);
        }
        if (ok && T2 > 0) {
            ok = mbar_wait(&ms.barO[(T2 - 1) & 1], ((T2 - 1) >> 1) & 1, abort_flag);
            tc_fence_after_sync();
        }
        // ---- epilogue ----
        if (ok) ok = mbar_wait(&ms.barE, 0, abort_flag);        // the tile's rows of o_la have landed
        // o_laT tiles (fp16): chunk e of the CTA at oQ + e * D * 128; piece pc (tokens 8 pc ..) of
        // head-dimension row `row` at 16-byte slot pc * D + (row ^ pc): eight such rows are an 8 x 8 matrix, which ldmatrix
        // transposes on the way.  The accumulator is read in the layout that gives (lane l: tokens l / 4, + 8 and the
        // columns 2 (l % 4), + 1 of every 8), and `out` leaves that layout through stmatrix.
        // out tile (bf16): box kb (columns 64 kb ..) at oV + kb * 16 KB, row r, piece j at j ^ (r & 7).
        // (A thread reading its own token's column out of these tiles took a two-byte load per value, twice: the epilogue
        // was 8 of the 15 thousand cycles of a CTA with two key tiles.)
        const float inv = l > 0.f ? 1.f / l : 0.f;       // l = 0 (no visible key): o_nla = 0
        const uint32_t sm32 = smem_u32(smem);
        const int l8 = lane & 7, mi = lane >> 3, g8 = lane >> 2;
        constexpr int NB = D / 32;                       // 32-column blocks of the softmax head
        // this lane's share of 16 tokens (from tok0 on) x 32 columns (from col on) of o_la, fp16 pairs: [8-column block][token half]
        auto load_la = [&](int row0, int col, uint32_t (&la)[4][2]) {
            const int pc = ((row0 & 63) >> 3) + (mi & 1);
            const uint32_t tile = sm32 + SL::oQ + (row0 >> 6) * (DL * 128) + pc * (DL * 16);
#pragma unroll
            for (int c2 = 0; c2 < 2; ++c2) {
                uint32_t v[4];
                ldmatrix_x4_trans(tile + (((col + 16 * c2 + 8 * (mi >> 1) + l8) ^ pc) << 4), v);
                la[2 * c2][0] = v[0]; la[2 * c2][1] = v[1]; la[2 * c2 + 1][0] = v[2]; la[2 * c2 + 1][1] = v[3];
            }
        };
        auto quad_sum = [](float x) {
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            return x + __shfl_xor_sync(0xffffffffu, x, 2);
        };
#pragma unroll 1
        for (int hh = 0; hh < 2; ++hh) {                 // 16 of the warp's 32 tokens at a time
            const int row0 = 32 * q + 16 * hh;
            uint32_t o[NB][16], la[NB][4][2];
            float ssn[2] = {0.f, 0.f}, ssl[2] = {0.f, 0.f};        // squares: tokens row0 + g8, + 8
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
                if (T2 > 0) tmem_ld_16x32(tO + lane_base + ((uint32_t)(16 * hh) << 16) + 32 * nb, o[nb]);
                else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) o[nb][e] = 0u;
                }
            auto squares = [&](const uint32_t (&a)[4][2]) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int t8 = 0; t8 < 2; ++t8) {
                        const float2 y = __half22float2(*reinterpret_cast<const __half2 *>(&a[j][t8]));
                        ssl[t8] = fmaf(y.x, y.x, fmaf(y.y, y.y, ssl[t8]));
                    }
            };
            if (kG > 1) {        // the other softmax heads' columns of the linear row: mean square only
#pragma unroll 1
                for (int e = 0; e < (kG - 1) * NB; ++e) {
                    const int gg = e / NB;
                    load_la(row0, (gg < sg ? gg : gg + 1) * D + e % NB * 32, la[0]);
                    squares(la[0]);
                }
            }
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
                load_la(row0, sg * D + 32 * nb, la[nb]);
                squares(la[nb]);
            }
            if (T2 > 0) tmem_wait_ld();
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    ssn[(e >> 1) & 1] = fmaf(__uint_as_float(o[nb][e]), __uint_as_float(o[nb][e]), ssn[(e >> 1) & 1]);
            float iv[2], wn[2], wl[2];
#pragma unroll
            for (int t8 = 0; t8 < 2; ++t8) {
                const int src = 16 * hh + g8 + 8 * t8;     // the lane that holds the token's row
                iv[t8] = __shfl_sync(0xffffffffu, inv, src);
                // mean square of the normalised row = inv^2 * mean square of the accumulator row
                wn[t8] = __shfl_sync(0xffffffffu, wv.x, src) * rsqrtf(iv[t8] * iv[t8] * quad_sum(ssn[t8]) / D + eps) * iv[t8];   // applies to the raw accumulator
                wl[t8] = __shfl_sync(0xffffffffu, wv.y, src) * rsqrtf(quad_sum(ssl[t8]) / DL + eps);
            }
            if (has_out && ok) {
                const int r_st = row0 + 8 * (mi & 1) + l8;
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) {
                        uint32_t y[4];                     // [8-column block][token half]
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int cb = 2 * c2 + (j >> 1), t8 = j & 1;
                            const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&la[nb][cb][t8]));
                            y[j] = pack_bf162(fmaf(wn[t8], __uint_as_float(o[nb][4 * cb + 2 * t8]), wl[t8] * a.x),
                                              fmaf(wn[t8], __uint_as_float(o[nb][4 * cb + 2 * t8 + 1]), wl[t8] * a.y));
                        }
                        const int col = 32 * nb + 16 * c2 + 8 * (mi >> 1);
                        stmatrix_x4(sm32 + SL::oV + (col >> 6) * (kBM * 128) + sw128_offset(r_st, (col & 63) >> 3), y[0], y[1], y[2], y[3]);
                    }
            }
            if (o_nla && ok) {          // the raw branch output (fp32): a quad's pairs of columns are whole 32-byte sectors
#pragma unroll
                for (int t8 = 0; t8 < 2; ++t8) {
                    const int i = p * kBM + row0 + g8 + 8 * t8;
                    float *dst = o_nla + (((size_t)b * L + i) * H + h) * DL + sg * D + 2 * (lane & 3);
                    if (i < L)
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                            for (int cb = 0; cb < 4; ++cb)
                                *reinterpret_cast<float2 *>(dst + 32 * nb + 8 * cb) =
                                    make_float2(iv[t8] * __uint_as_float(o[nb][4 * cb + 2 * t8]), iv[t8] * __uint_as_float(o[nb][4 * cb + 2 * t8 + 1]));
                }
            }
        }
        if (ok && lse && i_abs < L)
            lse[(size_t)bhg * L + i_abs] = l > 0.f ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
        fence_proxy_async_smem();
        named_barrier_sync(1, kSoftmaxThreads);
        if (tid == 0 && ok) {
            if (has_out)
                for (int kb = 0; kb < KB; ++kb)
                    tma_store_4d(&map_out, smem + SL::oV + kb * (kBM * 128), kb * 64, hq, p * kBM, b);
            tma_store_commit();
            tma_store_wait_read();                      // shared memory may go once it has been read
        }
    }
    // ------------------------------ teardown ------------------------------
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, SL::kTmemCols);
    }
    if (tid == 0 && ms.abort_flag) atomicMin(status, (int)NATSL_ERR_TIMEOUT);
    end_behind_scan();
}

// Route compaction and gather of the retained K/V in one kernel (the softmax branch's half of the forward's
// set-up; grid = (slices of the chunks, B*H)).  A CTA lists its slice's retained tokens (see route_slice.cuh) and copies
// their K rows (bf16) and V rows (as fp16) into the compacted layouts [B,H,cap,d] / [B,H,capv,d] (optionally K as
// fp16 too, for the backward).  The fp16 rows behind the last one are zeroed up to the next multiple of 128, so
// that a K/V tile never multiplies a zero probability or a zero logit gradient with an uninitialised value.
// It also clears the scan's per-chunk counters of the call.  It needs nothing of the prepare kernel before it in
// the stream and is its programmatic dependent, so that it runs where that kernel's last wave leaves room; it only
// must not end before it, since the scan waits for this kernel.
struct RouteArgs {
    const uint8_t *route;
    int32_t *sm_idx, *prefix, *emit_flags;
    const int32_t *base_in;                          // [B,H] entries the cache already holds, or nullptr
};
template <int D>
__global__ void __launch_bounds__(kRouteThreads)
route_gather_kernel(const __nv_bfloat16 *__restrict__ k, const __nv_bfloat16 *__restrict__ v, const RouteArgs ra,
                    __nv_bfloat16 *__restrict__ k_sm, __nv_bfloat16 *__restrict__ v_sm,
                    __half *__restrict__ v16, __half *__restrict__ k16, int cap, int capv, int slice_chunks,
                    int groups, float norm_eps, int raw_k_sm, int L, int H) {
    // raw_k_sm (with the normalisation): k_sm is a cache that keeps the keys as given; the normalised
    // fp16 keys then go to k16 only
    constexpr int kVecPerRow = D * 2 / 16;
    constexpr int kRows = kRouteThreads / kVecPerRow;
    __shared__ RouteLists rl;
    const int bh = blockIdx.y, b = bh / H, h = bh % H, NC = L / kC;
    const int tid = threadIdx.x;
    launch_dependents();
    const int base0 = ra.base_in ? ra.base_in[bh] : 0;
    const RouteSlice sl = list_slice(rl, ra.route + (size_t)b * L * H + h, ra.prefix + (size_t)bh * (NC + 1), base0, slice_chunks, NC, H);
    for (int i = tid; i < sl.nc; i += kRouteThreads) ra.emit_flags[(size_t)bh * NC + sl.c_lo + i] = 0;
    // RMS-normalised keys of the softmax operation (Section 4.3), per softmax head = per slice of D / groups
    // columns, as fp16 (the softmax kernel's logit product is an fp16 MMA in this mode): the slice's pieces
    // sit in neighbouring lanes of the row's lanes.  bf16 pieces in, fp16 pieces out.
    const int piece = tid % kVecPerRow;
    auto rms_fp16 = [&](uint4 kk) {
        const uint32_t kw[4] = {kk.x, kk.y, kk.z, kk.w};
        float f[8], ss = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(kw[i] << 16);
            f[2 * i + 1] = __uint_as_float(kw[i] & 0xffff0000u);
            ss = fmaf(f[2 * i], f[2 * i], fmaf(f[2 * i + 1], f[2 * i + 1], ss));
        }
        const int lanes = kVecPerRow / groups;            // lanes per slice (a power of two)
        const unsigned row_mask = (kVecPerRow == 32 ? 0xffffffffu : ((1u << kVecPerRow) - 1u))
                                  << ((threadIdx.x & 31) & ~(kVecPerRow - 1));
        for (int o = 1; o < lanes; o <<= 1) ss += __shfl_xor_sync(row_mask, ss, o);
        const float rk = rsqrtf(ss * groups / D + norm_eps);
        return make_uint4(pack_half2(f[0] * rk, f[1] * rk), pack_half2(f[2] * rk, f[3] * rk),
                          pack_half2(f[4] * rk, f[5] * rk), pack_half2(f[6] * rk, f[7] * rk));
    };
    auto to_fp16 = [](uint4 x) {
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = pack_half2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
        return make_uint4(o[0], o[1], o[2], o[3]);
    };
    // ---- the slice's rows: one row per group of kVecPerRow threads, chunk by chunk of the list ----
    for_each_row<kVecPerRow>(rl, sl, [&](int row, int tok) {
        if (piece == 0) ra.sm_idx[(size_t)bh * L + row - base0] = tok;
        if (row >= cap) return;
        const size_t dst = ((size_t)bh * cap + row) * D, src = (((size_t)b * L + tok) * H + h) * D;
        uint4 *dv16 = reinterpret_cast<uint4 *>(v16 + ((size_t)bh * capv + row) * D) + piece;
        uint4 *dk16 = k16 ? reinterpret_cast<uint4 *>(k16 + ((size_t)bh * capv + row) * D) + piece : nullptr;
        uint4 kk = reinterpret_cast<const uint4 *>(k + src)[piece];
        const uint4 vv = reinterpret_cast<const uint4 *>(v + src)[piece];
        if (norm_eps >= 0.f && raw_k_sm) reinterpret_cast<uint4 *>(k_sm + dst)[piece] = kk;
        if (norm_eps >= 0.f) kk = rms_fp16(kk);
        if (!(norm_eps >= 0.f && raw_k_sm)) reinterpret_cast<uint4 *>(k_sm + dst)[piece] = kk;
        if (dk16) *dk16 = norm_eps >= 0.f ? kk : to_fp16(kk);      // (normalised: already fp16)
        if (v_sm) reinterpret_cast<uint4 *>(v_sm + dst)[piece] = vv;
        *dv16 = to_fp16(vv);
    });
    // ---- rows of earlier calls: only the fp16 copy of their V rows is made (and, with the normalisation, the
    // normalised copy of their keys, which the cache keeps as given) ----
    if (ra.base_in) {
        const int n_prev = min(base0, cap);
        for (int row = blockIdx.x * kRows + tid / kVecPerRow; row < n_prev; row += gridDim.x * kRows) {
            const size_t dst = ((size_t)bh * cap + row) * D, d16 = ((size_t)bh * capv + row) * D;
            reinterpret_cast<uint4 *>(v16 + d16)[piece] = to_fp16(reinterpret_cast<const uint4 *>(v_sm + dst)[piece]);
            if (k16 && norm_eps >= 0.f)
                reinterpret_cast<uint4 *>(k16 + d16)[piece] = rms_fp16(reinterpret_cast<const uint4 *>(k_sm + dst)[piece]);
        }
    }
    if (sl.c_lo + sl.nc == NC) {                           // zero rows behind the last one
        const int n = min(sl.base + sl.mine, cap), n_pad = min((n + 127) / 128 * 128, capv);
        for (int row = n + tid / kVecPerRow; row < n_pad; row += kRows) {
            const size_t d16 = ((size_t)bh * capv + row) * D;
            reinterpret_cast<uint4 *>(v16 + d16)[piece] = make_uint4(0u, 0u, 0u, 0u);
            if (k16) reinterpret_cast<uint4 *>(k16 + d16)[piece] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    if (tid == 0) grid_dependency_wait();
}

}  // namespace

template <int D, int G>      // D: columns of a softmax head; G of them per linear head (s.d = D G)
static cudaError_t softmax_tc_impl(const void *q, const void *k_sm, const void *v16, int32_t cap,
                                   int32_t capv, const int32_t *sm_idx, const int32_t *pre,
                                   const void *o_la16, const int32_t *emit_flags, const float *w,
                                   float scale_sm, float eps, float norm_eps, void *out, float *o_nla, float *lse,
                                   int32_t *sm_len, int len_cap, BlockRouting br, bool appending, int32_t *status, Shape s,
                                   cudaStream_t st, int segs, int seg_tiles) {
    using SL = SmLayout<D>;
    CUtensorMap mq, mk, mv, mout, mkd, mvd;
    // q, out, k, v [B,L,H,G D] are read as [B,L,H G,D]; the compacted K/V rows keep all G D columns
    if (!tch::make_map_blhd(&mq, q, s.B, s.L, s.H * G, D, kBM) ||
        !tch::make_map_2d(&mk, k_sm, (uint64_t)s.B * s.H * cap, D * G, kBN) ||
        !tch::make_map_2d(&mv, v16, (uint64_t)s.B * s.H * capv, D * G, kBN))
        return cudaErrorInvalidValue;
    mout = mq;                                             // placeholder when `out` is not asked for
    if (out && !tch::make_map_blhd(&mout, out, s.B, s.L, s.H * G, D, kBM)) return cudaErrorInvalidValue;
    mkd = mq;
    mvd = mq;
    if (br.route && (!tch::make_map_blhd(&mkd, br.k, s.B, s.L, s.H * G, D, kBN) ||
                     !tch::make_map_blhd(&mvd, br.v, s.B, s.L, s.H * G, D, kBN)))
        return cudaErrorInvalidValue;
    auto kernel = softmax_combine_tc_kernel<D, false, G, false>;
    if (norm_eps >= 0.f) kernel = softmax_combine_tc_kernel<D, false, G, true>;
    if (br.route) kernel = norm_eps >= 0.f ? softmax_combine_tc_kernel<D, true, G, true>
                                          : softmax_combine_tc_kernel<D, true, G, false>;
    cudaError_t e = allow_smem(kernel, SL::kTotal);
    if (e != cudaSuccess) return e;
    // With emit_flags the kernel is launched as a programmatic dependent of the kernel before it in
    // the stream (the scan): it may start once all of the scan's CTAs are resident, and finds o_la
    // through the flags.  A launch the runtime serialises instead finds every flag already raised.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s.B * s.H * G, (s.L + kBM - 1) / kBM);
    cfg.blockDim = dim3(kThreadsS);
    cfg.dynamicSmemBytes = SL::kTotal;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = emit_flags ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, kernel, mq, mk, mv, mout, mkd, mvd, br.route, appending ? 1 : 0,
                           (int)cap, (int)capv, sm_idx, pre, (const __half *)o_la16, emit_flags, w, scale_sm, eps,
                           norm_eps, out ? 1 : 0, o_nla, lse, sm_len, len_cap, status, s.L, s.H, debug_wait_kcycles(), segs, seg_tiles);
    count_launch();
    return e;
}

cudaError_t launch_softmax_combine_tc(const void *q, const void *k_sm, const void *v16, int32_t cap,
                                      int32_t capv, const int32_t *sm_idx,
                                      const int32_t *sm_chunk_prefix, const void *o_la16,
                                      const int32_t *emit_flags, const float *w, float scale_sm,
                                      float eps, void *out, float *o_nla, float *lse, int32_t *sm_len, int len_cap,
                                      BlockRouting br, bool appending, int32_t *status, Shape s, cudaStream_t st,
                                      HeadGroups hg, int segs, int seg_tiles) {
    if (hg.G == 2 && s.d == 128)
        return softmax_tc_impl<64, 2>(q, k_sm, v16, cap, capv, sm_idx, sm_chunk_prefix, o_la16, emit_flags,
                                      w, scale_sm, eps, hg.norm_eps, out, o_nla, lse, sm_len, len_cap, br, appending, status, s, st, segs,
                                         seg_tiles);
    if (hg.G > 1) return cudaErrorInvalidValue;
    if (s.d == 128)
        return softmax_tc_impl<128, 1>(q, k_sm, v16, cap, capv, sm_idx, sm_chunk_prefix, o_la16, emit_flags,
                                       w, scale_sm, eps, hg.norm_eps, out, o_nla, lse, sm_len, len_cap, br, appending, status, s, st, segs,
                                         seg_tiles);
    return softmax_tc_impl<64, 1>(q, k_sm, v16, cap, capv, sm_idx, sm_chunk_prefix, o_la16, emit_flags, w,
                                  scale_sm, eps, hg.norm_eps, out, o_nla, lse, sm_len, len_cap, br, appending, status, s, st, segs,
                                         seg_tiles);
}

template <int D>
static cudaError_t route_gather_impl(const void *k, const void *v, const RouteArgs &ra, void *k_sm, void *v_sm, void *v16,
                                     void *k16, int cap, int capv, Shape s, cudaStream_t st, bool pdl, HeadGroups hg, bool raw_k_sm) {
    const int NC = s.L / kC, BH = s.B * s.H, cps = slice_chunks_of(NC, BH, 4);
    dim3 grid((NC + cps - 1) / cps, BH);
    count_launch();
    return launch_kernel(route_gather_kernel<D>, grid, dim3(kRouteThreads), 0, st, pdl, (const __nv_bfloat16 *)k,
                         (const __nv_bfloat16 *)v, ra, (__nv_bfloat16 *)k_sm, (__nv_bfloat16 *)v_sm, (__half *)v16,
                         (__half *)k16, cap, capv, cps, hg.G, hg.norm_eps, raw_k_sm ? 1 : 0, s.L, s.H);
}

cudaError_t launch_route_gather_tc(const void *k, const void *v, const uint8_t *route, int32_t *sm_idx,
                                   int32_t *sm_chunk_prefix, const int32_t *base_in, void *k_sm, void *v_sm, void *v16,
                                   void *k16, int32_t cap, int32_t capv, int32_t *emit_flags, Shape s, cudaStream_t st,
                                   bool pdl, HeadGroups hg, bool raw_k_sm) {
    const RouteArgs ra{route, sm_idx, sm_chunk_prefix, emit_flags, base_in};
    if (s.d == 128) return route_gather_impl<128>(k, v, ra, k_sm, v_sm, v16, k16, cap, capv, s, st, pdl, hg, raw_k_sm);
    return route_gather_impl<64>(k, v, ra, k_sm, v_sm, v16, k16, cap, capv, s, st, pdl, hg, raw_k_sm);
}

}  // namespace natsl
