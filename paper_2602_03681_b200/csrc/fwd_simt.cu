// fp32 CUDA-core forward of the hybrid layer: the chunkwise Gated DeltaNet branch (prepare +
// scan), and the softmax branch over the retained tokens with the RMS-norm / weighted
// combination fused into its epilogue.  This is the exact-precision path (fp32 storage needs
// ~1e-6 relative error, which rules out bf16/tf32 tensor-core operands); it also accepts bf16
// storage and then serves as the in-library cross-check of the tensor-core kernels.
//
// Chunkwise form (Section 3, chunkwise equations, specialised to the gated delta rule of
// Section 4.3), per chunk of C = 64 tokens, beta~ = (1 - route) beta, G_i = inclusive
// cumulative log decay inside the chunk, gamma_i = exp(G_i), Gamma_ij = exp(G_i - G_j):
//   A_ij = beta~_i Gamma_ij (k_i.k_j) (j<i);  (I + A) W = diag(beta~ gamma) K;  (I + A) U = diag(beta~) V
//   P_ij = scale_la (q_i.k_j) Gamma_ij (j<=i)
//   U~ = U - W S;   O = scale_la diag(gamma) Q S + P U~;   S <- gamma_C S + (diag(gamma_C/gamma) K)^T U~
#include "common.cuh"
#include "natsl_internal.h"
#include "tc_common.cuh"

namespace natsl {

namespace {

constexpr int kThreads = 256;

// Small calls (few (batch, head) pairs, a few hundred tokens) are what this path is used for most, and there every
// kernel is a chain of latencies on a mostly idle chip: the kernels below cut their work finer when there is
// little of it, ask for their operands ahead of time by asynchronous copies, and are programmatic dependents of one another.

// 16 (or 4) bytes global -> shared, asynchronously; one group per commit.
__device__ __forceinline__ void copy16_async(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy4_async(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// R x N tile (row stride `ts` elements) into fp32 shared memory, rows of LD floats: asynchronously from fp32, through
// registers from bf16.
template <int R, int N, int LD, typename T>
__device__ __forceinline__ void load_tile(const T *__restrict__ src, size_t ts, float *dst) {
    static_assert(R * N % (4 * kThreads) == 0, "whole pieces per thread");
#pragma unroll 4
    for (int idx = threadIdx.x; idx < R * N / 4; idx += kThreads) {
        const int r = idx / (N / 4), c4 = (idx % (N / 4)) * 4;
        if constexpr (sizeof(T) == 4) copy16_async(dst + r * LD + c4, src + (size_t)r * ts + c4);
        else store4(dst + r * LD + c4, load4(src + (size_t)r * ts + c4));
    }
}
// Inclusive prefix sum of 64 values in shared memory by one warp.
__device__ __forceinline__ void prefix64(const float *x, float *y, int lane) {
    const float a = x[2 * lane], b = x[2 * lane + 1];
    float s = a + b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float z = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += z;
    }
    y[2 * lane + 1] = s;
    y[2 * lane] = s - b;
}
// acc (even and odd columns apart) += <a, b> over four columns
__device__ __forceinline__ void fma4(ulonglong2 a, ulonglong2 b, uint64_t &acc) {
    acc = tc::fma2(a.x, b.x, acc);
    acc = tc::fma2(a.y, b.y, acc);
}
__device__ __forceinline__ ulonglong2 lds4(const float *p) { return *reinterpret_cast<const ulonglong2 *>(p); }
// the first `n` (any number) of four values, zeros behind them
__device__ __forceinline__ ulonglong2 first_of(ulonglong2 a, int n) {
    const float2 lo = tc::unpack2(a.x), hi = tc::unpack2(a.y);
    return make_ulonglong2(tc::pack2(n > 0 ? lo.x : 0.f, n > 1 ? lo.y : 0.f), tc::pack2(n > 2 ? hi.x : 0.f, n > 3 ? hi.y : 0.f));
}
__device__ __forceinline__ float both(uint64_t a) { const float2 x = tc::unpack2(a); return x.x + x.y; }

// Sums of N values over W neighbouring lanes; lane w of them keeps values w N / W .. (the upper halves of the exchange
// travel while the lower ones are kept, so this takes N (1 - 1 / W) shuffles instead of N log2 W).
template <int N, int W>
__device__ __forceinline__ void sum_lanes(float (&x)[N]) {
    int n = N;
#pragma unroll
    for (int m = W / 2; m > 0; m >>= 1) {
        n /= 2;
        const bool up = threadIdx.x & m;
#pragma unroll
        for (int e = 0; e < N; ++e)
            if (e < n) {
                const float keep = up ? x[n + e] : x[e], give = up ? x[e] : x[n + e];
                x[e] = keep + __shfl_xor_sync(0xffffffffu, give, m);
            }
    }
}

// ------------------------------------------------------------------------------------------
// Prepare: state-independent per-chunk quantities.  grid = (kParts L/C, B*H): a chunk's right-hand sides (D columns of
// W, D of U) are cut into kParts, each CTA forms all of A and its share of P's rows.  Four parts when there are few
// chunks, one otherwise (A is then formed once).  K K^T and Q K^T: 4 x 4 outputs of each per thread, packed FMAs along
// the columns.  Substitution in blocks of 16 rows: one thread per column solves the block's rows (in registers), then
// all threads subtract its products from the rows below -- a loop that runs four times over one block's code.
// (One thread per column over all 64 rows was 2016 unrolled FMAs that run once: 40 KB of code, and its warps waited for
// instructions.  Eight chunks of 64 columns: 19.2 us by itself, 10.5 now.)
// ------------------------------------------------------------------------------------------
template <int D, int kParts> struct SimtPrep {
    static constexpr int LD = D + 4, LA = kC + 4;
    static constexpr int kCols = 2 * D / kParts, LX = kCols + 4;         // right-hand-side columns of a CTA
    static constexpr int kPRows = kC / kParts;                           // rows of P
    static constexpr int oK = 0, oQ = oK + kC * LD, oX = oQ + kPRows * LD, oA = oX + kC * LX, oG = oA + kC * LA;
    static constexpr int kBytes = (oG + 3 * kC) * 4;
};

template <typename T, int D, int kParts>
__global__ void __launch_bounds__(kThreads)
gdn_prepare_simt_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v,
                        const float *__restrict__ g, const float *__restrict__ beta,
                        const uint8_t *__restrict__ route, float scale_la, float *__restrict__ W,
                        float *__restrict__ U, float *__restrict__ P, float *__restrict__ Abar,
                        float *__restrict__ Gcum, int32_t *clear, int clear_words, int L, int H) {
    using SP = SimtPrep<D, kParts>;
    constexpr int LD = SP::LD, LA = SP::LA, LX = SP::LX, kCols = SP::kCols, kPE = SP::kPRows / 16;
    extern __shared__ __align__(16) float smem[];
    float *Ks = smem + SP::oK;              // [64][LD]
    float *Qs = smem + SP::oQ;              // [kPRows][LD]
    float *Xs = smem + SP::oX;              // [64][LX]: right-hand sides, then the solution
    float *At = smem + SP::oA;              // [64][LA]: column j of A
    float *Gs = smem + SP::oG;              // [64] inclusive cumulative log decay
    float *bts = Gs + kC, *raw = bts + kC;  // [64] beta~; [64] log decay

    const int c = blockIdx.x / kParts, part = blockIdx.x % kParts, bh = blockIdx.y, b = bh / H, h = bh % H;
    const int tid = threadIdx.x;
    const size_t ts = (size_t)H * D;
    const size_t tok0 = ((size_t)b * L + (size_t)c * kC) * H + h;  // index of the chunk's first token
    tc::grid_dependency_wait();
    // (the forward's first kernel: clears the status page, before any kernel behind this one can report into it)
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && tid < clear_words) clear[tid] = 0;
    __threadfence();
    tc::launch_dependents();

    const bool hasW = part * kCols < D, hasU = (part + 1) * kCols > D;   // (one part: both; several: one of them)
    load_tile<kC, D, LD>(k + tok0 * D, ts, Ks);
    load_tile<SP::kPRows, D, LD>(q + tok0 * D + (size_t)(part * SP::kPRows) * ts, ts, Qs);
    constexpr int kVCols = kParts == 1 ? D : kCols;
    if (hasU) load_tile<kC, kVCols, LX>(v + tok0 * D + (kParts == 1 ? 0 : part * kCols - D), ts, Xs + (kParts == 1 ? D : 0));
    if (tid < kC) {
        const size_t t = tok0 + (size_t)tid * H;
        bts[tid] = route && route[t] ? 0.f : beta[t];   // route == nullptr: beta~ = beta
        raw[tid] = g[t];
    }
    copies_wait();
    __syncthreads();
    if (tid < 32) prefix64(raw, Gs, tid);
    // A (strictly lower), Abar = A without the beta~ row factor (the backward needs it), and
    // P = scale_la (Q K^T) . Gamma, lower triangle including the diagonal.  Thread: rows ti + 16 e, columns tj + 16 e.
    {
        const int ti = tid >> 4, tj = tid & 15;
        uint64_t a[4][4], pq[kPE][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int ei = 0; ei < 4; ++ei) a[ei][e] = 0ull;
#pragma unroll
            for (int ei = 0; ei < kPE; ++ei) pq[ei][e] = 0ull;
        }
#pragma unroll 2
        for (int x = 0; x < D; x += 4) {
            ulonglong2 kj[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) kj[e] = lds4(Ks + (tj + 16 * e) * LD + x);
#pragma unroll
            for (int ei = 0; ei < 4; ++ei) {
                const ulonglong2 ki = lds4(Ks + (ti + 16 * ei) * LD + x);
#pragma unroll
                for (int e = 0; e <= ei; ++e) fma4(ki, kj[e], a[ei][e]);
            }
#pragma unroll
            for (int ei = 0; ei < kPE; ++ei) {
                const ulonglong2 qi = lds4(Qs + (ti + 16 * ei) * LD + x);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (kParts > 1 || e <= ei) fma4(qi, kj[e], pq[ei][e]);
            }
        }
        __syncthreads();                      // the cumulative decays are there
        const size_t cc = ((size_t)bh * (L / kC) + c) * kC * kC;
#pragma unroll
        for (int ei = 0; ei < 4; ++ei)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = ti + 16 * ei, j = tj + 16 * e;
                const float av = j < i ? __expf(Gs[i] - Gs[j]) * both(a[ei][e]) : 0.f;
                if (Abar && part == 0) Abar[cc + i * kC + j] = av;
                At[j * LA + i] = bts[i] * av;
            }
#pragma unroll
        for (int ei = 0; ei < kPE; ++ei)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = part * SP::kPRows + ti + 16 * ei, j = tj + 16 * e;
                P[cc + i * kC + j] = j <= i ? scale_la * __expf(Gs[i] - Gs[j]) * both(pq[ei][e]) : 0.f;
            }
        if (Gcum && part == 0 && tid < kC) Gcum[(size_t)bh * L + c * kC + tid] = Gs[tid];
    }
    // right-hand sides: beta~ gamma K, beta~ V
    constexpr int kTpc = kThreads / kCols;            // threads per column
    const int col = tid % kCols, sub = tid / kCols;
    const bool isW = kParts == 1 ? col < D : hasW;
    const int dcol = (part * kCols + col) % D;         // column of W or U
    for (int i = sub; i < kC; i += kTpc)
        Xs[i * LX + col] = bts[i] * (isW ? __expf(Gs[i]) * Ks[i * LD + dcol] : Xs[i * LX + col]);
    __syncthreads();
    float *dst = (isW ? W : U) + tok0 * D + dcol;
#pragma unroll 1
    for (int r0 = 0; r0 < kC; r0 += 16) {
        if (sub == 0) {
            float x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = Xs[(r0 + i) * LX + col];
#pragma unroll
            for (int j = 0; j < 15; ++j)
#pragma unroll
                for (int i4 = (j + 1) / 4; i4 < 4; ++i4) {
                    const float4 aj = *reinterpret_cast<const float4 *>(At + (r0 + j) * LA + r0 + 4 * i4);   // (zero for i <= j)
                    if (4 * i4 > j) x[4 * i4] = fmaf(-aj.x, x[j], x[4 * i4]);
                    if (4 * i4 + 1 > j) x[4 * i4 + 1] = fmaf(-aj.y, x[j], x[4 * i4 + 1]);
                    if (4 * i4 + 2 > j) x[4 * i4 + 2] = fmaf(-aj.z, x[j], x[4 * i4 + 2]);
                    if (4 * i4 + 3 > j) x[4 * i4 + 3] = fmaf(-aj.w, x[j], x[4 * i4 + 3]);
                }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                Xs[(r0 + i) * LX + col] = x[i];
                dst[(size_t)(r0 + i) * ts] = x[i];
            }
        }
        __syncthreads();
        if (r0 + 16 < kC) {
            float x[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) x[j] = Xs[(r0 + j) * LX + col];
            for (int i = r0 + 16 + 4 * sub; i < kC; i += 4 * kTpc) {
                float y[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) y[e] = Xs[(i + e) * LX + col];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float4 aj = *reinterpret_cast<const float4 *>(At + (r0 + j) * LA + i);
                    y[0] = fmaf(-aj.x, x[j], y[0]); y[1] = fmaf(-aj.y, x[j], y[1]);
                    y[2] = fmaf(-aj.z, x[j], y[2]); y[3] = fmaf(-aj.w, x[j], y[3]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) Xs[(i + e) * LX + col] = y[e];
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------------------------------
// Scan: sequential over chunks, one CTA per (batch, head, slice of NV value columns), grid = (D/NV, B*H).  NV = 8
// when slices of 32 would leave most of the chip idle: a chunk's step is a chain, and four times shorter for it;
// with many (batch, head) pairs the wider slice reads the chunk's operands a quarter as often.
// What bounds a step is latency, so the next chunk's operands travel while this one is worked on (K, P, U, g and, where
// they fit twice, W and Q from the step's start; else W and Q from its middle), and the products have as much reuse
// per load as 256 threads allow: 2 rows x 4 columns (U~ and q S; P U~) or 4 x 4 (state) per thread, the sum over the inner
// index split over neighbouring lanes.  Row lengths are such that the lanes' 16-byte loads fall on different banks.
// (Loading at the step's start and one row x two columns per thread: 33 us for 16 CTAs of four chunks, 13.8 now.)
// ------------------------------------------------------------------------------------------
template <int D, int NV> struct SimtScan {
    static constexpr int kPad = NV == 8 ? 16 : 4;        // rows 64 bytes apart for 4 x 4 lanes (row, quarter), 16 for 32 rows
    static constexpr int LD = D + kPad, LK = D + 4, LP = kC + kPad, LU = kC + kPad;
    static constexpr int kTwice = D == 64 ? 2 : 1;       // W and Q buffers
    static constexpr int oS = 0, oW = oS + NV * LD, oQ = oW + kTwice * kC * LD, oK = oQ + kTwice * kC * LD,
                         oP = oK + 2 * kC * LK, oU = oP + 2 * kC * LP, oUs = oU + 2 * kC * NV, oUt = oUs + kC * NV,
                         oG = oUt + NV * LU;
    static constexpr int kBytes = (oG + 5 * kC + 1) * 4;
    static_assert(kBytes <= 227 * 1024, "shared memory of a CTA");
};

template <typename T, int D, int NV>
__global__ void __launch_bounds__(kThreads)
gdn_scan_simt_kernel(const T *__restrict__ q, const T *__restrict__ k, const float *__restrict__ g,
                     const float *__restrict__ W, const float *__restrict__ U,
                     const float *__restrict__ P, float scale_la, const float *__restrict__ state_in,
                     float *__restrict__ state_out, float *__restrict__ chunk_states,
                     float *__restrict__ Ut, float *__restrict__ o_la,
                     const uint8_t *__restrict__ block_route, int L, int H) {
    using SS = SimtScan<D, NV>;
    constexpr int LD = SS::LD, LK = SS::LK, LP = SS::LP, LU = SS::LU;
    constexpr int kCg = NV / 4;                          // column groups: a thread's columns are cg + kCg {0 .. 3}
    constexpr int kW1 = kThreads / (32 * kCg);           // lanes that share a 2 x 4 tile
    constexpr int kRw = kW1 == 1 ? 2 : 1, kCl = kW1 == 1 ? 4 : 2;       // rows x columns a lane keeps of it
    static_assert(kW1 == 1 || kW1 == 4, "NV = 8 or 32");
    extern __shared__ __align__(16) float smem[];
    float *Ss = smem + SS::oS;                           // [NV][LD]: value columns of the state
    float *Us = smem + SS::oUs, *Uts = smem + SS::oUt;   // U~: [64][NV] and [NV][LU]
    float *raw = smem + SS::oG;                          // [2][64] log decay
    float *Gs = raw + 2 * kC;                            // [64] cumulative
    float *e1 = Gs + kC, *e2 = e1 + kC;                  // [64] scale_la gamma_i; [64] gamma_C / gamma_i
    volatile int *outside = reinterpret_cast<int *>(e2 + kC);        // whether U~ has an infinity or a NaN

    const int slice = blockIdx.x, bh = blockIdx.y, b = bh / H, h = bh % H, tid = threadIdx.x;
    const int NC = L / kC;
    const size_t ts = (size_t)H * D;
    const int c0 = slice * NV;
    tc::grid_dependency_wait();
    tc::launch_dependents();

    auto first_token = [&](int c) { return ((size_t)b * L + (size_t)c * kC) * H + h; };
    auto fetch_wq = [&](int c) {
        const size_t at = first_token(c) * D, o = (c % SS::kTwice) * kC * LD;
        load_tile<kC, D, LD>(W + at, ts, smem + SS::oW + o);
        load_tile<kC, D, LD>(q + at, ts, smem + SS::oQ + o);
    };
    auto fetch_rest = [&](int c) {
        const size_t tok0 = first_token(c);
        const int o = c & 1;
        load_tile<kC, D, LK>(k + tok0 * D, ts, smem + SS::oK + o * kC * LK);
        load_tile<kC, kC, LP>(P + ((size_t)bh * NC + c) * kC * kC, kC, smem + SS::oP + o * kC * LP);
        for (int idx = tid; idx < kC * kCg; idx += kThreads)
            copy16_async(smem + SS::oU + (o * kC + idx / kCg) * NV + idx % kCg * 4,
                         U + (tok0 + (size_t)(idx / kCg) * H) * D + c0 + idx % kCg * 4);
        if (tid < kC) copy4_async(raw + o * kC + tid, g + tok0 + (size_t)tid * H);
    };
    fetch_wq(0);
    fetch_rest(0);
    if (tid == 0) *outside = 0;
    for (int idx = tid; idx < D * NV; idx += kThreads) {
        const int a = idx / NV, cc = idx % NV;
        Ss[cc * LD + a] = state_in ? state_in[((size_t)bh * D + a) * D + c0 + cc] : 0.f;
    }
    // 2 x 4 tiles: rows rp and rp + 32, columns cg + kCg {0 .. 3}; lane w1 of the tile's keeps, of the sums, row
    // r and the kCl columns from cc0 on (or, alone, all of it)
    const int w1 = tid % kW1, cg = tid / kW1 % kCg, rp = tid / (kW1 * kCg);
    const int r0 = kW1 == 1 ? rp : rp + 32 * (w1 >> 1), cc0 = kW1 == 1 ? 0 : 2 * (w1 & 1);
    for (int c = 0; c < NC; ++c) {
        const size_t tok0 = first_token(c);
        const float *Ws = smem + SS::oW + (c % SS::kTwice) * kC * LD, *Qs = smem + SS::oQ + (c % SS::kTwice) * kC * LD;
        const float *Ks = smem + SS::oK + (c & 1) * kC * LK, *Ps = smem + SS::oP + (c & 1) * kC * LP;
        const float *Uin = smem + SS::oU + (c & 1) * kC * NV;
        copies_wait();
        __syncthreads();
        if (c + 1 < NC) {
            if (SS::kTwice == 2) fetch_wq(c + 1);
            fetch_rest(c + 1);
        }
        if (chunk_states) {  // state at chunk entry, [B,H,NC,D,D]
            for (int idx = tid; idx < D * NV; idx += kThreads) {
                const int a = idx / NV, cc = idx % NV;
                chunk_states[(((size_t)bh * NC + c) * D + a) * D + c0 + cc] = Ss[cc * LD + a];
            }
        }
        if (tid < 32) {
            prefix64(raw + (c & 1) * kC, Gs, tid);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = tid + 32 * u;
                e1[i] = scale_la * __expf(Gs[i]);
                e2[i] = __expf(Gs[kC - 1] - Gs[i]);
            }
        }
        // U~ = U - W S, and q S while the state's columns pass by
        float qs[kRw * kCl];
        bool finite = true;                               // this thread's U~
        {
            uint64_t acc[2][4][2];                        // [row][column][W S, q S]
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[e][x][0] = acc[e][x][1] = 0ull;
#pragma unroll 4
            for (int a = 4 * w1; a < D; a += 4 * kW1) {
                ulonglong2 sv[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) sv[x] = lds4(Ss + (cg + kCg * x) * LD + a);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const ulonglong2 wv = lds4(Ws + (rp + 32 * e) * LD + a), qv = lds4(Qs + (rp + 32 * e) * LD + a);
#pragma unroll
                    for (int x = 0; x < 4; ++x) { fma4(wv, sv[x], acc[e][x][0]); fma4(qv, sv[x], acc[e][x][1]); }
                }
            }
            float sum[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) sum[e] = both(acc[e >> 3][(e >> 1) & 3][e & 1]);
            sum_lanes<16, kW1>(sum);
#pragma unroll
            for (int e = 0; e < kRw; ++e)
#pragma unroll
                for (int x = 0; x < kCl; ++x) {
                    const int r = r0 + 32 * e, cc = cg + kCg * (cc0 + x);
                    const float u = Uin[r * NV + cc] - sum[2 * (kCl * e + x)];
                    finite &= fabsf(u) < INFINITY;
                    qs[kCl * e + x] = sum[2 * (kCl * e + x) + 1];
                    Us[r * NV + cc] = u;
                    Uts[cc * LU + r] = u;
                    if (Ut) Ut[(tok0 + (size_t)r * H) * D + c0 + cc] = u;
                }
        }
        if (!finite) *outside = 1;                        // (once and for all: the state takes it along)
        __syncthreads();
        const bool again = *outside;
        if (SS::kTwice == 1 && c + 1 < NC) fetch_wq(c + 1);
        // O = scale_la gamma_r q_r S + sum_{j<=r} P_rj U~_j.  P is zero above the diagonal, but zero times an infinity or a
        // NaN is not: where there is one among U~, the sums are formed again, of the tokens up to each row's own only.
        {
            uint64_t acc[2][4];
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[e][x] = 0ull;
#pragma unroll 4
            for (int j = 4 * w1; j < kC; j += 4 * kW1) {
                const ulonglong2 p1 = lds4(Ps + (rp + 32) * LP + j), p0 = lds4(Ps + rp * LP + j);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const ulonglong2 uv = lds4(Uts + (cg + kCg * x) * LU + j);
                    if (j < 32) fma4(p0, uv, acc[0][x]);
                    fma4(p1, uv, acc[1][x]);
                }
            }
            if (again) {
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int x = 0; x < 4; ++x) acc[e][x] = 0ull;
#pragma unroll 1
                for (int j = 4 * w1; j < kC; j += 4 * kW1) {
                    const ulonglong2 p1 = lds4(Ps + (rp + 32) * LP + j), p0 = lds4(Ps + rp * LP + j);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const ulonglong2 uv = lds4(Uts + (cg + kCg * x) * LU + j);
                        if (j < 32) fma4(p0, first_of(uv, rp + 1 - j), acc[0][x]);
                        fma4(p1, first_of(uv, rp + 33 - j), acc[1][x]);
                    }
                }
            }
            float sum[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) sum[e] = both(acc[e >> 2][e & 3]);
            sum_lanes<8, kW1>(sum);
#pragma unroll
            for (int e = 0; e < kRw; ++e)
#pragma unroll
                for (int x = 0; x < kCl; ++x) {
                    const int r = r0 + 32 * e;
                    o_la[(tok0 + (size_t)r * H) * D + c0 + cg + kCg * (cc0 + x)] = fmaf(e1[r], qs[kCl * e + x], sum[kCl * e + x]);
                }
        }
        // S <- gamma_C S + (diag(gamma_C / gamma) K)^T U~  (nobody reads S any more); 4 keys x 4 columns per tile
        {
            constexpr int kTiles = D * NV / 16, kW3 = kThreads / kTiles, kKeep = 16 / kW3;
            const int w3 = tid % kW3, tile = tid / kW3, c4 = tile % kCg * 4, a4 = tile / kCg * 4;
            float acc[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] = 0.f;
            // block-level routing: a softmax block's update is not committed, the state only decays
            if (!(block_route && block_route[tok0])) {
#pragma unroll 4
                for (int j = w3; j < kC; j += kW3) {
                    const float4 kv = *reinterpret_cast<const float4 *>(Ks + j * LK + a4);
                    const float4 uv = *reinterpret_cast<const float4 *>(Us + j * NV + c4);
                    const float f = e2[j];
                    const float ka[4] = {kv.x * f, kv.y * f, kv.z * f, kv.w * f}, uu[4] = {uv.x, uv.y, uv.z, uv.w};
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[e] = fmaf(ka[e & 3], uu[e >> 2], acc[e]);
                }
                sum_lanes<16, kW3>(acc);
            }
            const float gC = __expf(Gs[kC - 1]);
#pragma unroll
            for (int e = 0; e < kKeep; ++e) {
                const int at = w3 * kKeep + e;
                float *sp = Ss + (c4 + (at >> 2)) * LD + a4 + (at & 3);
                *sp = fmaf(gC, *sp, acc[e]);
            }
        }
    }
    __syncthreads();
    if (state_out) {
        for (int idx = tid; idx < D * NV; idx += kThreads) {
            const int a = idx / NV, cc = idx % NV;
            state_out[((size_t)bh * D + a) * D + c0 + cc] = Ss[cc * LD + a];
        }
    }
}

// ------------------------------------------------------------------------------------------
// Softmax branch over the retained tokens (Section 4.1, O_nla with mask M^nla) with the
// combination (Section 4.3, Norm equation) as epilogue.  grid = (L/(16 kR), B*H*G): 64 query rows per CTA, or 16 when
// blocks of 64 would leave most of the chip idle.  A half warp owns kR rows: lane kk of it the logits of keys kk and kk + 16 of
// a 32-key tile, and D / 16 columns of the rows' sums; probabilities pass between its lanes through shared memory.  The next
// tile's keys and values travel while this one is worked on.  A programmatic dependent of the scan: the tiles
// are worked on beside it, the epilogue waits for it.
// (A row's logits over 32 lanes and a shuffle per probability kept the shuffle unit, not the FMAs, busy: 72 us for
// 16 pairs of 1024 tokens of 64 columns by itself, 48.5 now; 485 -> 315 at 4096 tokens.)
// G softmax heads per linear head (Section 4.3, grouped heads): softmax head (h, sg) works on the
// columns [sg D, (sg+1) D) of q, k, v rows of DL = G D columns; lists, weights and the linear read-out
// are those of linear head h; the softmax output is normalised over its D columns, the linear
// read-out over all DL, and the CTA writes its D columns of `out`.  lse is [B,H,G,L].
// ------------------------------------------------------------------------------------------
template <int D, int kR> struct SimtSoft {
    static constexpr int kRows = 16 * kR, LD = D + 4, LPr = 32 + 4;
    static constexpr int oQ = 0, oK = oQ + kRows * LD, oV = oK + 2 * 32 * LD, oP = oV + 2 * 32 * D, oPos = oP + kRows * LPr;
    static constexpr int kBytes = (oPos + 64) * 4;
};
__device__ __forceinline__ float half_warp_sum(float x) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

template <typename T, int D, int G, int kR>
__global__ void __launch_bounds__(kThreads)
softmax_combine_simt_kernel(const T *__restrict__ q, const T *__restrict__ k_sm,
                            const T *__restrict__ v_sm, int cap, const int32_t *__restrict__ sm_idx,
                            const int32_t *__restrict__ sm_chunk_prefix,
                            const float *o_la, const float *__restrict__ w,
                            float scale_sm, float eps, T *__restrict__ out,
                            float *__restrict__ o_nla, float *__restrict__ lse,
                            const uint8_t *__restrict__ block_route, const T *__restrict__ k_tok,
                            const T *__restrict__ v_tok, int L, int H) {
    using SS = SimtSoft<D, kR>;
    constexpr int kRows = SS::kRows, LD = SS::LD, LPr = SS::LPr, DL = D * G;
    constexpr int VW = D >= 64 ? 4 : 2, NU = D / (16 * VW);          // a lane's columns: VW kk + 16 VW u ..
    extern __shared__ __align__(16) float smem[];
    float *Qs = smem + SS::oQ;             // [kRows][LD]
    float *Pr = smem + SS::oP;             // [kRows][LPr]
    int *pos = reinterpret_cast<int *>(smem + SS::oPos);  // [2][32]

    const int c = blockIdx.x * kRows / kC, row0 = blockIdx.x * kRows % kC;        // chunk, first row inside it
    const int bhg = blockIdx.y, bh = bhg / G, sg = bhg % G, b = bh / H, h = bh % H;
    const int NC = L / kC, tid = threadIdx.x, kk = tid & 15, rg = tid >> 4;       // this thread's rows: rg + 16 e
    const size_t ts = (size_t)H * DL;
    const size_t tok0 = ((size_t)b * L + (size_t)c * kC) * H + h;
    tc::launch_dependents();
    const int n_end = min(sm_chunk_prefix[(size_t)bh * (NC + 1) + c + 1], cap);
    const int col0 = sg * D;                             // first column of this softmax head
    for (int idx = tid; idx < kRows * D / 4; idx += kThreads) {
        const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
        store4(Qs + r * LD + c4, load4(q + tok0 * DL + (size_t)(row0 + r) * ts + col0 + c4));
    }
    const T *kb = k_sm + (size_t)bh * cap * DL + col0, *vb = v_sm + (size_t)bh * cap * DL + col0;
    // Block-level routing: a query in a linear block also reads the causal part of its own block
    // (two more tiles of 32 keys, taken from the layer's own k and v).
    const int n_ret = (n_end + 31) / 32 * 32;
    const int n_all = n_ret + (block_route && block_route[tok0] == 0 ? kC : 0);
    auto fetch = [&](int j0) {
        const bool own = j0 >= n_ret;
        float *Kt = smem + SS::oK + (j0 / 32 & 1) * 32 * LD, *Vt = smem + SS::oV + (j0 / 32 & 1) * 32 * D;
#pragma unroll 2
        for (int idx = tid; idx < 32 * D / 4; idx += kThreads) {
            const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
            if (!own && j0 + r >= n_end) {
                store4(Kt + r * LD + c4, make_float4(0.f, 0.f, 0.f, 0.f));
                store4(Vt + r * D + c4, make_float4(0.f, 0.f, 0.f, 0.f));
                continue;
            }
            const T *ks = own ? k_tok + (tok0 + (size_t)(j0 - n_ret + r) * H) * DL + col0 + c4 : kb + (size_t)(j0 + r) * DL + c4;
            const T *vs = own ? v_tok + (tok0 + (size_t)(j0 - n_ret + r) * H) * DL + col0 + c4 : vb + (size_t)(j0 + r) * DL + c4;
            if constexpr (sizeof(T) == 4) {
                copy16_async(Kt + r * LD + c4, ks);
                copy16_async(Vt + r * D + c4, vs);
            } else {
                store4(Kt + r * LD + c4, load4(ks));
                store4(Vt + r * D + c4, load4(vs));
            }
        }
        if (tid < 32) {
            int *pp = pos + (j0 / 32 & 1) * 32 + tid;
            if (!own && j0 + tid < n_end)
                copy4_async(reinterpret_cast<float *>(pp), reinterpret_cast<const float *>(sm_idx + (size_t)bh * L + j0 + tid));
            else
                *pp = own ? c * kC + (j0 - n_ret) + tid : 0x7fffffff;
        }
    };
    float m[kR], z[kR], acc[kR][NU * VW];
#pragma unroll
    for (int e = 0; e < kR; ++e) {
        m[e] = -INFINITY; z[e] = 0.f;
#pragma unroll
        for (int x = 0; x < NU * VW; ++x) acc[e][x] = 0.f;
    }
    if (n_all > 0) fetch(0);
    for (int j0 = 0; j0 < n_all; j0 += 32) {
        const float *Kt = smem + SS::oK + (j0 / 32 & 1) * 32 * LD, *Vt = smem + SS::oV + (j0 / 32 & 1) * 32 * D;
        copies_wait();
        __syncthreads();
        if (j0 + 32 < n_all) fetch(j0 + 32);
        const int pos0 = pos[(j0 / 32 & 1) * 32 + kk], pos1 = pos[(j0 / 32 & 1) * 32 + kk + 16];
        uint64_t sa[kR][2];
#pragma unroll
        for (int e = 0; e < kR; ++e) sa[e][0] = sa[e][1] = 0ull;
#pragma unroll 4
        for (int x = 0; x < D; x += 4) {
            const ulonglong2 k0 = lds4(Kt + kk * LD + x), k1 = lds4(Kt + (kk + 16) * LD + x);
#pragma unroll
            for (int e = 0; e < kR; ++e) {
                const ulonglong2 qx = lds4(Qs + (rg + 16 * e) * LD + x);
                fma4(qx, k0, sa[e][0]);
                fma4(qx, k1, sa[e][1]);
            }
        }
#pragma unroll
        for (int e = 0; e < kR; ++e) {
            const int i = c * kC + row0 + rg + 16 * e;
            const float s0 = pos0 <= i ? both(sa[e][0]) * scale_sm : -INFINITY, s1 = pos1 <= i ? both(sa[e][1]) * scale_sm : -INFINITY;
            float mx = fmaxf(s0, s1);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float m_new = fmaxf(m[e], mx), m_use = m_new == -INFINITY ? 0.f : m_new;
            const float p0 = pos0 <= i ? __expf(s0 - m_use) : 0.f, p1 = pos1 <= i ? __expf(s1 - m_use) : 0.f;
            const float corr = __expf(m[e] - m_use);     // exp(-inf) = 0 on the first tile
            z[e] = z[e] * corr + (p0 + p1);              // (this lane's keys; summed over the lanes at the end)
            m[e] = m_new;
            Pr[(rg + 16 * e) * LPr + kk] = p0;
            Pr[(rg + 16 * e) * LPr + kk + 16] = p1;
#pragma unroll
            for (int x = 0; x < NU * VW; ++x) acc[e][x] *= corr;
        }
        __syncwarp();                                    // (a row's lanes are in one warp)
#pragma unroll 2
        for (int j = 0; j < 32; j += 4) {
            float4 pv[kR];
#pragma unroll
            for (int e = 0; e < kR; ++e) pv[e] = *reinterpret_cast<const float4 *>(Pr + (rg + 16 * e) * LPr + j);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                float vx[NU * VW];
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    const float *vp = Vt + (j + jj) * D + VW * kk + 16 * VW * u;
                    if constexpr (VW == 4) {
                        const float4 y = *reinterpret_cast<const float4 *>(vp);
                        vx[4 * u] = y.x; vx[4 * u + 1] = y.y; vx[4 * u + 2] = y.z; vx[4 * u + 3] = y.w;
                    } else {
                        const float2 y = *reinterpret_cast<const float2 *>(vp);
                        vx[2 * u] = y.x; vx[2 * u + 1] = y.y;
                    }
                }
#pragma unroll
                for (int e = 0; e < kR; ++e) {
                    const float pe = jj == 0 ? pv[e].x : jj == 1 ? pv[e].y : jj == 2 ? pv[e].z : pv[e].w;
#pragma unroll
                    for (int x = 0; x < NU * VW; ++x) acc[e][x] = fmaf(pe, vx[x], acc[e][x]);
                }
            }
        }
        __syncwarp();                                    // the probabilities have been read
    }
    // epilogue: normalise both branches and combine.  Up to here the kernel has needed only what lies ahead of the scan,
    // and every CTA of the scan had waited for that before this kernel could start.
    tc::grid_dependency_wait();
#pragma unroll
    for (int e = 0; e < kR; ++e) {
        const int i = c * kC + row0 + rg + 16 * e;
        const size_t t = tok0 + (size_t)(row0 + rg + 16 * e) * H;
        z[e] = half_warp_sum(z[e]);
        const float inv = z[e] > 0.f ? 1.f / z[e] : 0.f;
        float ol[NU * VW], ssn = 0.f, ssl = 0.f;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const float *op = o_la + t * DL + col0 + VW * kk + 16 * VW * u;
            if constexpr (VW == 4) {
                const float4 y = __ldcg(reinterpret_cast<const float4 *>(op));
                ol[4 * u] = y.x; ol[4 * u + 1] = y.y; ol[4 * u + 2] = y.z; ol[4 * u + 3] = y.w;
            } else {
                const float2 y = __ldcg(reinterpret_cast<const float2 *>(op));
                ol[2 * u] = y.x; ol[2 * u + 1] = y.y;
            }
        }
#pragma unroll
        for (int x = 0; x < NU * VW; ++x) {
            acc[e][x] *= inv;
            ssn = fmaf(acc[e][x], acc[e][x], ssn);
            ssl = fmaf(ol[x], ol[x], ssl);
        }
        if (G > 1)        // the linear read-out is normalised over its whole row
            for (int x = 0; x < DL / 16; ++x) {
                if ((16 * x) / D == sg) continue;
                const float y = __ldcg(o_la + t * DL + kk + 16 * x);
                ssl = fmaf(y, y, ssl);
            }
        ssn = half_warp_sum(ssn);
        ssl = half_warp_sum(ssl);
        const float fn = rsqrtf(ssn / D + eps), fl = rsqrtf(ssl / DL + eps);
        const float wn = w ? w[t * 2] : 0.5f, wl = w ? w[t * 2 + 1] : 0.5f;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const size_t at = t * DL + col0 + VW * kk + 16 * VW * u;
            const float *on = &acc[e][VW * u], *la = &ol[VW * u];
            auto y = [&](int x) { return wn * on[x] * fn + wl * la[x] * fl; };
            if constexpr (VW == 4) {
                if (out) store4(out + at, make_float4(y(0), y(1), y(2), y(3)));
                if (o_nla) store4(o_nla + at, make_float4(on[0], on[1], on[2], on[3]));
            } else {
#pragma unroll
                for (int x = 0; x < VW; ++x) {
                    if (out) out[at + x] = from_f32<T>(y(x));
                    if (o_nla) o_nla[at + x] = on[x];
                }
            }
        }
        if (lse && kk == 0) lse[(size_t)bhg * L + i] = z[e] > 0.f ? m[e] + __logf(z[e]) : -INFINITY;
    }
}

// Per-operation normalisation of q and k for fp32 storage (Section 4.3): one warp per row of d
// columns writes the L2-normalised row (linear operation) and the row with each of its G slices
// RMS-normalised (softmax operation).  The tensor-core path does both inside its kernels instead.
// (qk_norm_f32_kernel, below the vector helpers.)

// Backward of that normalisation, in place on fp32 gradients, one warp per row.  On entry dq holds the
// gradient with respect to the L2-normalised q (linear operation) and dq_sm the one with respect to the
// slice-wise RMS-normalised q (softmax operation); dk holds, for a linear token, the gradient with
// respect to the L2-normalised k and, for a retained token, the one with respect to the RMS-normalised k
// (a token's k reaches only the operation the token was routed to).  x^ = x r, r = (sum x^2 + e)^-1/2:
// dx = r (g - x^ <x^, g>);  x~ = x r, r = (mean x^2 + e)^-1/2 over a slice of ds columns:
// dx = r (g - x~ <x~, g> / ds).
// (One warp per row; a lane owns D / 32 neighbouring columns, moved as one vector.  A slice is an aligned
// group of 32 / G lanes, so one xor butterfly yields a slice's sum on the way to the row's.)
template <int N> __device__ __forceinline__ void load_vec(const float *p, float (&x)[N]) {
    if (N == 4) { const float4 v = *reinterpret_cast<const float4 *>(p); x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
    else { const float2 v = *reinterpret_cast<const float2 *>(p); x[0] = v.x; x[1] = v.y; }
}
template <int N> __device__ __forceinline__ void load_vec(const __nv_bfloat16 *p, float (&x)[N]) {
    if (N == 4) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        x[0] = __uint_as_float(v.x << 16); x[1] = __uint_as_float(v.x & 0xffff0000u);
        x[2] = __uint_as_float(v.y << 16); x[3] = __uint_as_float(v.y & 0xffff0000u);
    } else {
        const uint32_t v = *reinterpret_cast<const uint32_t *>(p);
        x[0] = __uint_as_float(v << 16); x[1] = __uint_as_float(v & 0xffff0000u);
    }
}
template <int N> __device__ __forceinline__ void store_vec(float *p, const float (&x)[N]) {
    if (N == 4) *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
    else *reinterpret_cast<float2 *>(p) = make_float2(x[0], x[1]);
}
template <int N> __device__ __forceinline__ void store_vec(__nv_bfloat16 *p, const float (&x)[N]) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(x[0], x[1]);
    if (N == 4) {
        __nv_bfloat162 hi = __floats2bfloat162_rn(x[2], x[3]);
        *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
    } else {
        *reinterpret_cast<uint32_t *>(p) = *reinterpret_cast<uint32_t *>(&lo);
    }
}

// The forward normalisation with the same layout (d = 64 or 128, a slice an aligned group of 32 / G lanes).
template <int D>
__global__ void __launch_bounds__(256)
qk_norm_f32_kernel(const float *__restrict__ q, const float *__restrict__ k, float *__restrict__ q_la,
                   float *__restrict__ k_la, float *__restrict__ q_sm, float *__restrict__ k_sm,
                   size_t rows, int G, float norm_eps) {
    constexpr int N = D / 32;
    const size_t row = (size_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= rows) return;
    const int lps = 32 / G;
    const float inv_ds = (float)G / D;
    const size_t at = row * D + (size_t)lane * N;
    float x[2][N];
    load_vec<N>(q + at, x[0]);
    load_vec<N>(k + at, x[1]);
#pragma unroll
    for (int which = 0; which < 2; ++which) {
        float ss = 0.f, ss_s = 0.f;
#pragma unroll
        for (int j = 0; j < N; ++j) ss = fmaf(x[which][j], x[which][j], ss);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            if (o == lps) ss_s = ss;
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
        }
        if (lps == 32) ss_s = ss;
        const float rl = rsqrtf(ss + norm_eps), rs = rsqrtf(fmaf(ss_s, inv_ds, norm_eps));
        float y[N];
#pragma unroll
        for (int j = 0; j < N; ++j) y[j] = x[which][j] * rl;
        store_vec<N>((which ? k_la : q_la) + at, y);
#pragma unroll
        for (int j = 0; j < N; ++j) y[j] = x[which][j] * rs;
        store_vec<N>((which ? k_sm : q_sm) + at, y);
    }
}

template <typename T, int D>
__global__ void __launch_bounds__(256)
qk_norm_bwd_f32_kernel(const T *__restrict__ q, const T *__restrict__ k,
                       const uint8_t *__restrict__ route, const float *dq_la,
                       const float *__restrict__ dq_sm, const float *dk_in, const float *dv_in,
                       T *dq, T *dk, T *dv, size_t rows, int G, float norm_eps,
                       const float *__restrict__ dk_sm) {
    constexpr int N = D / 32;
    const size_t row = (size_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= rows) return;
    const int lps = 32 / G;                                  // lanes per slice
    const float inv_ds = (float)G / D;
    const bool retained = route[row] != 0;
    const size_t at = row * D + (size_t)lane * N;
    if (dv_in) {
        float t[N];
        load_vec<N>(dv_in + at, t);
        store_vec<N>(dv + at, t);
    }
#pragma unroll
    for (int which = 0; which < 2; ++which) {
        const float *sm_in = which == 0 ? dq_sm : dk_sm;   // separate softmax-operation gradient, if any
        const bool l2_part = sm_in || !retained, rms_part = sm_in || retained;
        float x[N], g[N], gs[N], out[N];
        load_vec<N>((which ? k : q) + at, x);
        load_vec<N>((which ? dk_in : dq_la) + at, g);
        if (sm_in) load_vec<N>(sm_in + at, gs);
        float ss = 0.f, xg = 0.f, xs = 0.f;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            if (!sm_in) gs[j] = g[j];
            ss = fmaf(x[j], x[j], ss);
            xg = fmaf(x[j], g[j], xg);
            xs = fmaf(x[j], gs[j], xs);
        }
        float ss_s = 0.f, xs_s = 0.f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            if (o == lps) { ss_s = ss; xs_s = xs; }
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
            xg += __shfl_xor_sync(0xffffffffu, xg, o);
            xs += __shfl_xor_sync(0xffffffffu, xs, o);
        }
        if (lps == 32) { ss_s = ss; xs_s = xs; }
        const float rl = rsqrtf(ss + norm_eps), dot = rl * xg;
        const float rs = rsqrtf(fmaf(ss_s, inv_ds, norm_eps)), m = rs * xs_s * inv_ds;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            out[j] = l2_part ? rl * (g[j] - x[j] * rl * dot) : 0.f;
            if (rms_part) out[j] += rs * (gs[j] - x[j] * rs * m);
        }
        store_vec<N>((which ? dk : dq) + at, out);
    }
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
    return allow_smem(kernel, (int)bytes);
}

}  // namespace


// Chunks up to which the prepare kernel cuts a chunk into four, by head size: with more the four-fold A takes more than the
// finer split of the rest gains.  128 columns: as many as are resident at once (78 KB, two CTAs per SM: 296 CTAs).  64
// columns (49 KB, four per SM): three CTAs per SM, the fourth only shares their issue slots.  Whole call with four parts
// against one, us: 8 chunks of 64 columns 21.9 / 26.5, 70 39.4 / 43.4, 74 (pairs of two chunks) 36.9 / 35.5, 80 43.2 / 55.1, 84
// 60.0 / 60.2, 96 47.9 / 51.9 and 55.8 / 69.4, 98 62.0 / 77.1, 112 58.7 / 58.0 and 56.0 / 54.3, 128 65.7 / 65.4, 160 73.3 /
// 67.1, 192 99.5 / 85.0; of 128 columns 8 chunks 30.6 / 40.1, 70 94.4 / 97.8, 72 86.7 / 90.0, 74 50.8 / 54.5, 80 117.0 /
// 111.0, 96 98.8 / 92.2, 128 133.6 / 121.6.
template <int D> constexpr int kFewChunks = D == 64 ? 3 * 148 / 4 : 2 * 148 / 4;

#define NATSL_DISPATCH(FN, ...)                                                   \
    do {                                                                          \
        if (s.bf16) {                                                             \
            if (s.d == 128) return FN<__nv_bfloat16, 128>(__VA_ARGS__);           \
            return FN<__nv_bfloat16, 64>(__VA_ARGS__);                            \
        }                                                                         \
        if (s.d == 128) return FN<float, 128>(__VA_ARGS__);                       \
        return FN<float, 64>(__VA_ARGS__);                                        \
    } while (0)

template <typename T, int D>
static cudaError_t prepare_impl(const void *q, const void *k, const void *v, const float *g,
                                const float *beta, const uint8_t *route, float scale_la, float *W,
                                float *U, float *P, float *Abar, float *Gcum, Shape s,
                                cudaStream_t st, int32_t *clear, int clear_words) {
    const bool few = s.L / kC * s.B * s.H <= kFewChunks<D>;     // (see the kernel)
    const size_t smem = few ? SimtPrep<D, 4>::kBytes : SimtPrep<D, 1>::kBytes;
    auto kernel = few ? gdn_prepare_simt_kernel<T, D, 4> : gdn_prepare_simt_kernel<T, D, 1>;
    cudaError_t e = set_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(s.L / kC * (few ? 4 : 1), s.B * s.H);
    count_launch();
    return launch_kernel(kernel, grid, dim3(kThreads), smem, st, true, (const T *)q, (const T *)k,
                         (const T *)v, g, beta, route, scale_la, W, U, P, Abar, Gcum, clear, clear_words, s.L, s.H);
}

cudaError_t launch_gdn_prepare_simt(const void *q, const void *k, const void *v, const float *g,
                                    const float *beta, const uint8_t *route, float scale_la,
                                    float *W, float *U, float *P, float *Abar, float *Gcum, Shape s,
                                    cudaStream_t st, int32_t *clear, int clear_words) {
    NATSL_DISPATCH(prepare_impl, q, k, v, g, beta, route, scale_la, W, U, P, Abar, Gcum, s, st, clear, clear_words);
}

template <typename T, int D>
static cudaError_t scan_impl(const void *q, const void *k, const float *g, const float *W,
                             const float *U, const float *P, float scale_la, const float *state_in,
                             float *state_out, float *chunk_states, float *Ut, float *o_la,
                             const uint8_t *block_route, Shape s, cudaStream_t st, bool pdl) {
    const bool narrow = s.B * s.H * (D / 32) < 148;     // (see the kernel)
    const size_t smem = narrow ? SimtScan<D, 8>::kBytes : SimtScan<D, 32>::kBytes;
    auto kernel = narrow ? gdn_scan_simt_kernel<T, D, 8> : gdn_scan_simt_kernel<T, D, 32>;
    cudaError_t e = allow_smem(kernel, smem, true);      // (softmax CTAs fit beside 64-column scans: 115 -> 108 us at 16 pairs of 1024)
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_kernel(kernel, dim3(D / (narrow ? 8 : 32), s.B * s.H), dim3(kThreads), smem, st, pdl, (const T *)q,
                         (const T *)k, g, W, U, P, scale_la, state_in, state_out, chunk_states, Ut, o_la, block_route, s.L,
                         s.H);
}

cudaError_t launch_gdn_scan_simt(const void *q, const void *k, const float *g, const float *W,
                                 const float *U, const float *P, float scale_la,
                                 const float *state_in, float *state_out, float *chunk_states,
                                 float *Ut, float *o_la, const uint8_t *block_route, Shape s,
                                 cudaStream_t st, bool pdl) {
    NATSL_DISPATCH(scan_impl, q, k, g, W, U, P, scale_la, state_in, state_out, chunk_states, Ut, o_la,
                   block_route, s, st, pdl);
}

template <typename T, int D, int G = 1>
static cudaError_t softmax_impl(const void *q, const void *k_sm, const void *v_sm, int32_t cap,
                                const int32_t *sm_idx, const int32_t *pre, const float *o_la,
                                const float *w, float scale_sm, float eps, void *out, float *o_nla,
                                float *lse, BlockRouting br, Shape s, cudaStream_t st) {
    const bool few = (s.L / kC) * s.B * s.H * G < 148;   // (see the kernel)
    const int rows = few ? 16 : 64;
    const size_t smem = few ? SimtSoft<D, 1>::kBytes : SimtSoft<D, 4>::kBytes;
    auto kernel = few ? softmax_combine_simt_kernel<T, D, G, 1> : softmax_combine_simt_kernel<T, D, G, 4>;
    cudaError_t e = set_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_kernel(kernel, dim3(s.L / rows, s.B * s.H * G), dim3(kThreads), smem, st, true, (const T *)q,
                         (const T *)k_sm, (const T *)v_sm, cap, sm_idx, pre, o_la, w, scale_sm, eps, (T *)out, o_nla, lse,
                         br.route, (const T *)br.k, (const T *)br.v, s.L, s.H);
}

cudaError_t launch_softmax_combine_simt(const void *q, const void *k_sm, const void *v_sm,
                                        int32_t cap, const int32_t *sm_idx,
                                        const int32_t *sm_chunk_prefix, const float *o_la,
                                        const float *w, float scale_sm, float eps, void *out,
                                        float *o_nla, float *lse, BlockRouting br, Shape s,
                                        cudaStream_t st, int G) {
    if (G > 1) {      // grouped softmax heads: fp32 storage, d / G in {32, 64}
        if (s.bf16) return cudaErrorInvalidValue;
#define NATSL_GROUPED(DS, GG)                                                                           \
        if (s.d == DS * GG && G == GG)                                                                  \
            return softmax_impl<float, DS, GG>(q, k_sm, v_sm, cap, sm_idx, sm_chunk_prefix, o_la, w,    \
                                               scale_sm, eps, out, o_nla, lse, br, s, st)
        NATSL_GROUPED(32, 2);
        NATSL_GROUPED(64, 2);
        NATSL_GROUPED(32, 4);
#undef NATSL_GROUPED
        return cudaErrorInvalidValue;
    }
    NATSL_DISPATCH(softmax_impl, q, k_sm, v_sm, cap, sm_idx, sm_chunk_prefix, o_la, w, scale_sm, eps,
                   out, o_nla, lse, br, s, st);
}

cudaError_t launch_qk_norm_f32(const float *q, const float *k, float *q_la, float *k_la, float *q_sm, float *k_sm,
                               size_t rows, int d, int G, float norm_eps, cudaStream_t st) {
    const unsigned blocks = (unsigned)((rows + 7) / 8);
    if ((d != 64 && d != 128) || G < 1 || 32 % G != 0) return cudaErrorInvalidValue;
    auto kernel = d == 128 ? qk_norm_f32_kernel<128> : qk_norm_f32_kernel<64>;
    kernel<<<blocks, 256, 0, st>>>(q, k, q_la, k_la, q_sm, k_sm, rows, G, norm_eps);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_qk_norm_bwd_f32(const void *q, const void *k, bool bf16, const uint8_t *route,
                                   const float *dq_la, const float *dq_sm, const float *dk_in,
                                   const float *dv_in, void *dq, void *dk, void *dv, size_t rows, int d, int G,
                                   float norm_eps, cudaStream_t st, const float *dk_sm) {
    const unsigned blocks = (unsigned)((rows + 7) / 8);
    if ((d != 64 && d != 128) || G < 1 || 32 % G != 0) return cudaErrorInvalidValue;
#define NATSL_NB(TT, DD)                                                                                      \
    qk_norm_bwd_f32_kernel<TT, DD><<<blocks, 256, 0, st>>>((const TT *)q, (const TT *)k, route, dq_la, dq_sm,  \
                                                          dk_in, dv_in, (TT *)dq, (TT *)dk, (TT *)dv, rows, G, \
                                                          norm_eps, dk_sm)
    if (bf16) { if (d == 128) NATSL_NB(__nv_bfloat16, 128); else NATSL_NB(__nv_bfloat16, 64); }
    else { if (d == 128) NATSL_NB(float, 128); else NATSL_NB(float, 64); }
#undef NATSL_NB
    count_launch();
    return cudaGetLastError();
}

}  // namespace natsl
