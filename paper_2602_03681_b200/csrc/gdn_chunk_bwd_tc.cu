// Chunk-parallel part of the Gated DeltaNet backward on tensor cores (bf16 storage): everything that follows the
// reverse scan, one CTA per chunk, for 64- and 128-column heads.
//   dQg = dO S0^T        dW = -dU~ S0^T        dK~ = U~ dS1^T        N = dO U~^T
//   dKb = T^T dW         dVb = T^T dU~         M = -(dKb W^T + dVb U^T)          (T = (I + A)^-1)
//   Ns = scale_la (N . Gamma) [j <= i]    Mg = M . Gamma [j < i]    Ms = diag(beta~) Mg
//   dq = scale_la gamma dQg + Ns K + dq_softmax
//   dk = beta~ (gamma dKb + Mg K) + [(gamma_C/gamma) dK~ + Ms^T K + Ns^T Q]         (linear tokens)
//   dv = beta~ dVb                                                                  (linear tokens)
// and the per-token sums the gate gradients need.  With P = gamma dKb + Mg K and R the bracket of dk they are row
// dots with what is written anyway:
//   dG = <q, dq_lin> + beta~ <k, P> - <k, R>,   dbeta = <k, P> + <v, dVb>,   kappa = <k, (gamma_C/gamma) dK~>.
// What bounds it: an operand is 64 x D, the products are far below a tcgen05 tile in one dimension or chained
// through masks, so they are warp-level MMAs (a warp owns 32 rows and D / 4 columns) and the kernel lives off
// its operand traffic.  Everything is fp16 in HBM, as the forward's and the reverse scan's own MMA operands were, and
// arrives by asynchronous bulk or tensor copies in the layout the
// fragments are loaded from: token-major tiles with the 128-byte swizzle, or "pieces" (16-byte pieces of a
// transposed tile, all rows of a piece contiguous), so that every ldmatrix row set is free of bank conflicts and
// nothing is converted on the way.  Slots are reused as the chain goes on -- 112 KB at D = 128, two CTAs per SM.
// (Separate kernels for this chain -- state dot, three tile GEMMs with tf32 operands, two fused kernels --
// moved fp32 through HBM between them: 1090 us on 3840 chunks of 128 columns.)  The tf32 products they had at 128
// columns kept 11 significant bits of their operands, as fp16 does; against 64-bit gradients the errors of both agree
// within 2 % on every output, and dg, with the normalisation, is 4 to 6 times closer (tf32 operands are cut, not
// rounded).  What fp16 has less of is range: see put() and range() below.
// The three gradient operands are in units of the power of two gsc.x (grad_scale); results are multiplied by
// gsc.y where they are written.
#include "common.cuh"
#include "natsl_internal.h"
#include "tc_common.cuh"

namespace natsl {

namespace {

using namespace tc;

constexpr int kCbThreads = 256;

template <int D> struct CbLayout {
    static constexpr int kU = D * 128;                     // a 64 x D fp16 operand
    static constexpr int oA = 0, oB = kU, oC = 2 * kU, oE = 3 * kU;          // E: D x D state operand
    static constexpr int oK = oE + D * D * 2;
    static constexpr int oY = oK + kU, oT = oY + 8192;
    static constexpr int oF = oT + 8192;                   // D = 64: E holds one operand, so U needs a place
    static constexpr int oW = oE, oUt = D == 128 ? oE + kU : oF;
    static constexpr int oMisc = D == 128 ? oF : oF + kU;
    static constexpr int kMisc = 1024;
    static constexpr int kTotal = oMisc + kMisc;
    static constexpr int kCtas = D == 128 ? 2 : 3;
};

struct CbMisc {
    uint64_t bar[5];
    int abort_flag, wait_kcycles;   // in this order: the waits read the limit as abort_flag[1]
    float red[12];
    float fk, fv, fkv;              // dKb, dVb over what is stored of them (powers of two); fk / fv
    float G[64], bt[64];
};
static_assert(sizeof(CbMisc) <= 1024, "misc page too small");

// One row of 16-byte pieces of a fragment load.  sw: 64-column tiles with the 128-byte swizzle, 128-byte rows;
// pm: pieces, all R rows of a piece contiguous.
__device__ __forceinline__ uint32_t sw_at(uint32_t base, int row, int piece) {
    return base + row * 128 + ((piece ^ (row & 7)) << 4);
}

// Fragment addresses of a lane (l7, m1, m2: row within an 8 x 8 matrix, and which of the four matrices of a load);
// o: the operand's offset in shared memory, nb: the warp's first column.
struct Frag { uint32_t s; int m0, l7, m1, m2; };
struct ASw {                                  // A [m][k], swizzled 64-column tiles 8 KB apart
    Frag f; uint32_t o;
    __device__ __forceinline__ uint32_t operator()(int mt, int k0) const {
        return sw_at(f.s + o + (k0 >> 6) * 8192, f.m0 + 16 * mt + f.l7 + 8 * f.m1, ((k0 & 63) >> 3) + f.m2);
    }
};
struct ASwT {                                 // A stored [k][m], one swizzled 64-column tile
    Frag f; uint32_t o;
    __device__ __forceinline__ uint32_t operator()(int mt, int k0) const {
        return sw_at(f.s + o, k0 + f.l7 + 8 * f.m2, ((f.m0 + 16 * mt) >> 3) + f.m1);
    }
};
struct APmT {                                 // A stored [k][m] in pieces of m, R rows
    Frag f; uint32_t o; int R;
    __device__ __forceinline__ uint32_t operator()(int mt, int k0) const {
        return f.s + o + ((((f.m0 + 16 * mt) >> 3) + f.m1) * R + k0 + f.l7 + 8 * f.m2) * 16;
    }
};
struct BSwT {                                 // B stored [k][n], swizzled 64-column tiles
    Frag f; uint32_t o; int nb;
    __device__ __forceinline__ uint32_t operator()(int np, int k0) const {
        const int n = nb + 16 * np + 8 * f.m2;
        return sw_at(f.s + o + (n >> 6) * 8192, k0 + f.l7 + 8 * f.m1, (n & 63) >> 3);
    }
};
template <int D> struct BPmT {                // B stored [k][n] in pieces of n, D rows
    Frag f; uint32_t o; int nb;
    __device__ __forceinline__ uint32_t operator()(int np, int k0) const {
        return f.s + o + (((nb + 16 * np) / 8 + f.m2) * D + k0 + f.l7 + 8 * f.m1) * 16;
    }
};
template <int D> struct BPm {                 // B stored [n][k] in pieces of k, D rows
    Frag f; uint32_t o; int nb;
    __device__ __forceinline__ uint32_t operator()(int np, int k0) const {
        return f.s + o + ((k0 / 8 + f.m1) * D + nb + 16 * np + f.l7 + 8 * f.m2) * 16;
    }
};

// acc (32 x 8 NT block of a warp) += A B over k = 0 .. K - 1.  fa(mt, k0): this lane's address for the 16 x 16 block
// of A at row block mt; fb(np, k0): for the 16 x 16 block of B at column pair np.  AT: A stored [k][m];
// BT: B stored [k][n] (else [n][k]).
template <int NT, int K, bool AT, bool BT, typename FA, typename FB>
__device__ __forceinline__ void mma_block(FA fa, FB fb, float (&acc)[2][NT][4]) {
#pragma unroll 2
    for (int k0 = 0; k0 < K; k0 += 16) {
        uint32_t a[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            if (AT) ldmatrix_x4_trans(fa(mt, k0), a[mt]);
            else ldmatrix_x4(fa(mt, k0), a[mt]);
        }
#pragma unroll
        for (int np = 0; np < NT / 2; ++np) {
            uint32_t b[4];
            if (BT) ldmatrix_x4_trans(fb(np, k0), b);
            else ldmatrix_x4(fb(np, k0), b);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                mma_m16n8k16(acc[mt][2 * np], a[mt], b[0], b[1]);
                mma_m16n8k16(acc[mt][2 * np + 1], a[mt], b[2], b[3]);
            }
        }
    }
}
template <int NT> __device__ __forceinline__ void zero_acc(float (&acc)[2][NT][4]) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.f;
}

// Rows of a warp's block times a factor each; row0 = the lane's first row (rows row0 + 16 mt + 8 half).
template <int NT, typename F> __device__ __forceinline__ void scale_rows(float (&x)[2][NT][4], int row0, F f) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            const float fr = f(row0 + 16 * mt + 8 * hf);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) { x[mt][nt][2 * hf] *= fr; x[mt][nt][2 * hf + 1] *= fr; }
        }
}

struct CbArgs {
    const __half *Ut16, *dU16, *S16, *dS16, *T16;   // pieces (see natsl_internal.h), per chunk
    const __half *Qh;                                // [B,H,L,D]: the linear operation's q
    const __nv_bfloat16 *v;
    const float *Gcum, *beta, *dq_sm;                // dq_sm: added to dq (fp32, token-major) or nullptr
    const uint8_t *route;
    const float *dk_x, *dv_x;                        // kBlock: every token's softmax-branch dk, dv, added, or nullptr
    float scale_la;
    float *dg, *dbeta;
    const __nv_bfloat16 *q, *k;                      // kNorm: the rows that were normalised
    float norm_eps;
    int G;
    float *kap_c;                                    // [B,H,L/C] or nullptr: sum over the chunk of kappa = <dS1, K~^T U~>
    int32_t *status;
    int L, H, wait_kcycles;
};

// kBlock: block-level routing (every token takes part in the delta rule, a softmax block's update was not
// committed, every token's dk and dv have a softmax-branch part).
// kNorm (with kBlock): q and k were normalised by the forward, dq_sm and dk_x are gradients with respect to the
// softmax operation's copy, and the two row-local Jacobians are applied here, to the fp32 accumulators.  With x a row
// of q (or k), r_l = rsqrt(|x|^2 + eps), r_s = rsqrt(mean_slice x^2 + eps) and g, h the gradients of the two copies,
//   dx = r_l g + r_s h - x (r_l^3 <x, g> + r_s^3 mean_slice(x h)).
// (A kernel of its own for this read the five fp32 gradients back: 945 MB, 135 us on 3840 chunks of 128 columns.)
// TO: what dq, dk, dv are stored as.
template <int D, bool kBlock, bool kNorm, typename TO>
__global__ void __launch_bounds__(kCbThreads, CbLayout<D>::kCtas)
gdn_chunk_bwd_kernel(const __grid_constant__ CUtensorMap map_do,     // dO16 [B*H*L][D], box 64 x 64
                     const __grid_constant__ CUtensorMap map_kh, const __grid_constant__ CUtensorMap map_qh,
                     const __grid_constant__ CUtensorMap map_wt,     // W^T [B*H*NC*D][64], box D x 64
                     const __grid_constant__ CUtensorMap map_ut,     // U^T fp16, likewise
                     TO *__restrict__ dq, TO *__restrict__ dk, TO *__restrict__ dv, const CbArgs p) {
    using SL = CbLayout<D>;
    constexpr int KB = D / 64, NT = D / 32;
    extern __shared__ __align__(1024) uint8_t smem[];
    CbMisc &ms = *reinterpret_cast<CbMisc *>(smem + SL::oMisc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int NC = p.L / kC;
    const int c = blockIdx.x, bh = blockIdx.y, b = bh / p.H, h = bh % p.H;
    const size_t chunk = (size_t)bh * NC + c;
    const size_t ts = (size_t)p.H * D;                                               // token stride, elements
    const size_t tok0 = (((size_t)b * p.L + (size_t)c * kC) * p.H + h) * D;          // first token's row
    const float2 gsc = grad_scale(p.status);
    const bool committed = !kBlock || p.route[((size_t)b * p.L + (size_t)c * kC) * p.H + h] == 0;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicMin(p.status, (int)NATSL_ERR_CUDA);
        return;
    }
    // copies: 0: dO, U~   1: S0, K   2: dU~, T   3: W, U (where S0 was)   4: dS1, Q (where dV, W, U were)
    if (tid == 0) {
        for (int i = 0; i < 5; ++i) mbar_init(&ms.bar[i], 1);
        ms.abort_flag = 0;
        ms.wait_kcycles = p.wait_kcycles;
        ms.fk = ms.fv = ms.fkv = 1.f;
        fence_mbar_init();
        const int row = bh * p.L + c * kC;
        mbar_arrive_expect_tx(&ms.bar[0], 2 * SL::kU);
        for (int kb = 0; kb < KB; ++kb) tma_load_2d(smem + SL::oA + kb * 8192, &map_do, &ms.bar[0], kb * 64, row);
        bulk_load_1d(smem + SL::oB, p.Ut16 + chunk * D * 64, SL::kU, &ms.bar[0]);
        mbar_arrive_expect_tx(&ms.bar[1], D * D * 2 + SL::kU);
        bulk_load_1d(smem + SL::oE, p.S16 + chunk * D * D, D * D * 2, &ms.bar[1]);
        for (int kb = 0; kb < KB; ++kb) tma_load_2d(smem + SL::oK + kb * 8192, &map_kh, &ms.bar[1], kb * 64, row);
        mbar_arrive_expect_tx(&ms.bar[2], SL::kU + 8192);
        bulk_load_1d(smem + SL::oC, p.dU16 + chunk * D * 64, SL::kU, &ms.bar[2]);
        bulk_load_1d(smem + SL::oT, p.T16 + chunk * 4096, 8192, &ms.bar[2]);
    }
    if (tid < 64) {
        ms.G[tid] = p.Gcum[(size_t)bh * p.L + c * kC + tid];
        const size_t tk = ((size_t)b * p.L + (size_t)c * kC + tid) * p.H + h;
        ms.bt[tid] = !kBlock && p.route[tk] ? 0.f : p.beta[tk];
    }
    __syncthreads();
    // What comes later -- the operands that wait for their slots, and the rows that lanes read as fragments -- starts
    // towards L2 now: as plain loads and copies behind the MMAs they were most of the kernel's waits.
    if (tid == 32) {
        tma_prefetch_l2_2d(&map_wt, 0, (int)(chunk * D));
        tma_prefetch_l2_2d(&map_ut, 0, (int)(chunk * D));
        bulk_prefetch_l2(p.Qh + ((size_t)bh * p.L + c * kC) * D, SL::kU);
        bulk_prefetch_l2(p.dS16 + chunk * D * D, D * D * 2);
    }
    {                                   // (line by line: bulk prefetches of rows would queue up before the copies)
        const int ln = tid & 3;
        const size_t at = tok0 + (size_t)(tid >> 2) * ts;
        if (ln < D / 32) {
            if (p.dq_sm) prefetch_l2(p.dq_sm + at + 32 * ln);
            if (kBlock && p.dv_x) prefetch_l2(p.dv_x + at + 32 * ln);
            if (kBlock && p.dk_x) prefetch_l2(p.dk_x + at + 32 * ln);
        }
        if (ln < D / 64) {
            prefetch_l2(p.v + at + 64 * ln);
            if (kNorm) prefetch_l2(p.q + at + 64 * ln);
        } else if (kNorm && ln < D / 32) {
            prefetch_l2(p.k + at + 64 * ln - D);
        }
    }
    volatile int *abort_flag = &ms.abort_flag;
    // (a wait that runs out is recorded and the chain goes on: nothing below may leave a barrier short of threads)
    auto wait = [&](int i) { (void)mbar_wait(&ms.bar[i], 0, abort_flag); };

    // ---- this warp's block of every result: rows m0 .. m0 + 31, columns n0 .. (64-column results: j0 ..) ----
    const int m0 = 32 * (warp & 1), wc = warp >> 1, n0 = wc * (D / 4), j0 = wc * 16;
    const uint32_t s = smem_u32(smem);
    auto rowi = [&](int mt, int hf) { return m0 + 16 * mt + 8 * hf + g; };          // this lane's rows
    const Frag fr{s, m0, lane & 7, (lane >> 3) & 1, lane >> 4};
    auto a_sw = [&](uint32_t o) { return ASw{fr, o}; };
    auto a_swt = [&](uint32_t o) { return ASwT{fr, o}; };
    auto a_pmt = [&](uint32_t o, int R) { return APmT{fr, o, R}; };
    auto b_swt = [&](uint32_t o, int nb) { return BSwT{fr, o, nb}; };
    auto b_pmt = [&](uint32_t o, int nb) { return BPmT<D>{fr, o, nb}; };
    auto b_pm = [&](uint32_t o, int nb) { return BPm<D>{fr, o, nb}; };
    // acc -> swizzled token-major tile(s); whether one of this thread's values is out of fp16's range
    auto put = [&](uint32_t o, const float (&x)[2][NT][4], float f) -> bool {
        __half2 most = __half2half2(__ushort_as_half(0));
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const int n = n0 + 8 * nt, i = rowi(mt, hf);
                    const uint32_t w = pack_half2(f * x[mt][nt][2 * hf], f * x[mt][nt][2 * hf + 1]);
                    *reinterpret_cast<uint32_t *>(smem + o + (n >> 6) * 8192 + i * 128 + ((((n & 63) >> 3) ^ (i & 7)) << 4) + 4 * t) = w;
                    most = __hmax2(most, __habs2(*reinterpret_cast<const __half2 *>(&w)));
                }
        return __half_as_ushort(__hmax(__low2half(most), __high2half(most))) >= 0x7c00;
    };
    // row dots of x with a swizzled token-major tile, this lane's columns
    auto dot_sw = [&](uint32_t o, const float (&x)[2][NT][4], float (&d)[4]) {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                float a = 0.f;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const int n = n0 + 8 * nt, i = rowi(mt, hf);
                    const float2 y = __half22float2(*reinterpret_cast<const __half2 *>(
                        smem + o + (n >> 6) * 8192 + i * 128 + ((((n & 63) >> 3) ^ (i & 7)) << 4) + 4 * t));
                    a = fmaf(y.x, x[mt][nt][2 * hf], fmaf(y.y, x[mt][nt][2 * hf + 1], a));
                }
                d[2 * mt + hf] = a;
            }
    };
    // Results leave in groups of four columns: lanes of a pair swap halves of two neighbouring 8-column tiles, so that
    // tiles 2u and 2u + 1 of x hold columns cb + 16 u .. + 3 of a row.  (A lane's own pairs of columns took twice the
    // load and store instructions for half the bytes each, and every one of them touches 8 rows.)
    const int cb = n0 + 8 * (t & 1) + 4 * (t >> 1);
    auto regroup = [&](float (&x)[2][NT][4]) {
        const bool odd = t & 1;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int u = 0; u < NT; u += 2)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float r = __shfl_xor_sync(0xffffffffu, odd ? x[mt][u][e] : x[mt][u + 1][e], 1);
                    x[mt][u][e] = odd ? r : x[mt][u][e];
                    x[mt][u + 1][e] = odd ? x[mt][u + 1][e] : r;
                }
    };
    auto store = [&](TO *dst, float x0, float x1, float x2, float x3) {
        if constexpr (sizeof(TO) == 2) *reinterpret_cast<uint2 *>(dst) = make_uint2(pack_bf162(x0, x1), pack_bf162(x2, x3));
        else *reinterpret_cast<float4 *>(dst) = make_float4(x0, x1, x2, x3);
    };
    auto add4 = [](const float *add) { return add ? *reinterpret_cast<const float4 *>(add) : make_float4(0.f, 0.f, 0.f, 0.f); };
    auto bf4 = [](uint2 w) {
        return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                           __uint_as_float(w.y & 0xffff0000u));
    };
    // <y, x> over the four columns of tiles u, u + 1
    auto dot4 = [](float4 y, const float (&x)[NT][4], int u, int hf, float a) {
        return fmaf(y.x, x[u][2 * hf], fmaf(y.y, x[u][2 * hf + 1], fmaf(y.z, x[u + 1][2 * hf], fmaf(y.w, x[u + 1][2 * hf + 1], a))));
    };
    // kNorm: gradients of the two copies of a row of X -> gradient of the row, stored to dst.  x: g, regrouped,
    // times 1 / f; add: the softmax operation's gradient.  o: 4 KB for each half of the rows, free for the 4 warps
    // that share it (row dots of a row's 4 column blocks).
    auto norm_store = [&](TO *dst, const __nv_bfloat16 *X, const float *add, float (&x)[2][NT][4], float f, uint32_t o) {
        float *pt = reinterpret_cast<float *>(smem + o + (warp & 1) * 4096);
        uint2 w[2][2][NT / 2];
        float4 gs[2][2][NT / 2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const size_t at = tok0 + (size_t)rowi(mt, hf) * ts + cb;
#pragma unroll
                for (int u = 0; u < NT / 2; ++u) {
                    w[mt][hf][u] = *reinterpret_cast<const uint2 *>(X + at + 16 * u);
                    gs[mt][hf][u] = *reinterpret_cast<const float4 *>(add + at + 16 * u);
                }
            }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                float ss = 0.f, xg = 0.f, xs = 0.f;
#pragma unroll
                for (int u = 0; u < NT / 2; ++u) {
                    const float4 y = bf4(w[mt][hf][u]), z = gs[mt][hf][u];
                    ss = fmaf(y.x, y.x, fmaf(y.y, y.y, fmaf(y.z, y.z, fmaf(y.w, y.w, ss))));
                    xg = dot4(y, x[mt], 2 * u, hf, xg);
                    xs = fmaf(y.x, z.x, fmaf(y.y, z.y, fmaf(y.z, z.z, fmaf(y.w, z.w, xs))));
                }
#pragma unroll
                for (int m = 1; m < 4; m <<= 1) {
                    ss += __shfl_xor_sync(0xffffffffu, ss, m);
                    xg += __shfl_xor_sync(0xffffffffu, xg, m);
                    xs += __shfl_xor_sync(0xffffffffu, xs, m);
                }
                if (t == 0) {
                    const int i = rowi(mt, hf) & 31;
                    pt[i * 4 + wc] = ss;
                    pt[128 + i * 4 + wc] = f * xg;
                    pt[256 + i * 4 + wc] = xs;
                }
            }
        named_barrier_sync(2 + (warp & 1), 128);
        const bool two = p.G == 2;
        const float inv_ds = (two ? 2.f : 1.f) / D;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int i = rowi(mt, hf) & 31;
                const float4 a = *reinterpret_cast<const float4 *>(pt + i * 4);
                const float4 b4 = *reinterpret_cast<const float4 *>(pt + 128 + i * 4);
                const float4 e = *reinterpret_cast<const float4 *>(pt + 256 + i * 4);
                const float s0 = a.x + a.y, s1 = a.z + a.w, x0 = e.x + e.y, x1 = e.z + e.w;
                const float sl = two ? (wc < 2 ? s0 : s1) : s0 + s1, xl = two ? (wc < 2 ? x0 : x1) : x0 + x1;
                const float rl = rsqrtf(s0 + s1 + p.norm_eps), rs = rsqrtf(fmaf(sl, inv_ds, p.norm_eps));
                const float cx = rl * rl * rl * ((b4.x + b4.y) + (b4.z + b4.w)) + rs * rs * rs * (xl * inv_ds);
                const size_t at = tok0 + (size_t)rowi(mt, hf) * ts + cb;
                const float rf = rl * f;
#pragma unroll
                for (int u = 0; u < NT / 2; ++u) {
                    const float4 y = bf4(w[mt][hf][u]), z = gs[mt][hf][u];
                    store(dst + at + 16 * u, fmaf(-cx, y.x, fmaf(rf, x[mt][2 * u][2 * hf], rs * z.x)),
                          fmaf(-cx, y.y, fmaf(rf, x[mt][2 * u][2 * hf + 1], rs * z.y)),
                          fmaf(-cx, y.z, fmaf(rf, x[mt][2 * u + 1][2 * hf], rs * z.z)),
                          fmaf(-cx, y.w, fmaf(rf, x[mt][2 * u + 1][2 * hf + 1], rs * z.w)));
                }
            }
    };
    // Row sums over the warp's columns: lane t of a quad keeps the one of row ri.  (As four partial sums a lane each
    // they cost twelve registers, and a spilled register costs a trip to L2: shared memory leaves hardly any L1.)
    const int ri = rowi(t >> 1, t & 1);
    auto row_sum = [&](const float (&a)[4]) {
        const bool odd = t & 1;
        float x0 = odd ? a[1] : a[0], x1 = odd ? a[3] : a[2];
        x0 += __shfl_xor_sync(0xffffffffu, odd ? a[0] : a[1], 1);
        x1 += __shfl_xor_sync(0xffffffffu, odd ? a[2] : a[3], 1);
        return (t & 2 ? x1 : x0) + __shfl_xor_sync(0xffffffffu, t & 2 ? x0 : x1, 2);
    };
    float dG, db, kap = 0.f, d4[4];
    // dW, dKb and dVb are fp16 operands of the next product, but nothing keeps them in fp16's range: a carried state of
    // order 1e3 makes dW leave it, in rows that the decay then takes back.  put() notices, the barrier behind it passes
    // it on, and such a chunk stores the tile again times a power of two, which is put back on the fp32 accumulators.
    // No other chunk changes a bit.  (Bounds that would make the test unnecessary do not exist: T and the state are the
    // caller's.  It costs 0.3 to 0.9 % of a training step of 128 columns, 0.1 % at 64.)
    constexpr float kRoom = 32768.f;
    auto range = [&](const float (&x)[2][NT][4]) {      // (all threads) the power of two that brings the tile below kRoom
        float a = 0.f;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) a = fmaxf(a, fabsf(x[mt][nt][e]));
        a = warp_max(a);
        if (lane == 0) ms.red[warp] = a;
        __syncthreads();
#pragma unroll
        for (int wv = 0; wv < 8; ++wv) a = fmaxf(a, ms.red[wv]);
        __syncthreads();
        const int e = min((int)(__float_as_uint(a) >> 23), 227);                      // (a < 2^(e - 126))
        return a < kRoom ? 1.f : __uint_as_float((unsigned)(126 + 15 + 127 - e) << 23);
    };

    // ---- N = dO U~^T;  Ns = scale_la (N . Gamma), j <= i  -> Y ----
    wait(0);
    {
        float x[2][2][4];
        zero_acc(x);
        mma_block<2, D, false, true>(a_sw(SL::oA), b_pmt(SL::oB, j0), x);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    const int i = rowi(mt, hf), j = j0 + 8 * nt + 2 * t;
                    const float2 Gj = *reinterpret_cast<const float2 *>(&ms.G[j]);
                    const float f0 = p.scale_la * exp_ftz(j <= i ? ms.G[i] - Gj.x : -INFINITY);   // branch-free mask
                    const float f1 = p.scale_la * exp_ftz(j + 1 <= i ? ms.G[i] - Gj.y : -INFINITY);
                    *reinterpret_cast<uint32_t *>(smem + SL::oY + i * 128 + (((j >> 3) ^ (i & 7)) << 4) + 4 * t) =
                        pack_half2(f0 * x[mt][nt][2 * hf], f1 * x[mt][nt][2 * hf + 1]);
                }
    }
    __syncthreads();
    // ---- dq = scale_la gamma dO S0^T + Ns K ----
    wait(1);
    {
        float x[2][NT][4];
        zero_acc(x);
        mma_block<NT, D, false, true>(a_sw(SL::oA), b_pmt(SL::oE, n0), x);
        scale_rows(x, m0 + g, [&](int i) { return p.scale_la * exp_ftz(ms.G[i]); });
        mma_block<NT, 64, false, true>(a_sw(SL::oY), b_swt(SL::oK, n0), x);
        regroup(x);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            uint2 qw[2][NT / 2];
            float4 z[2][NT / 2];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int i = rowi(mt, hf);
#pragma unroll
                for (int u = 0; u < NT / 2; ++u) {
                    qw[hf][u] = *reinterpret_cast<const uint2 *>(p.Qh + ((size_t)bh * p.L + c * kC + i) * D + cb + 16 * u);
                    if (!kNorm) z[hf][u] = add4(p.dq_sm ? p.dq_sm + tok0 + (size_t)i * ts + cb + 16 * u : nullptr);
                }
            }
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const size_t at = tok0 + (size_t)rowi(mt, hf) * ts + cb;
                float a = 0.f;
#pragma unroll
                for (int u = 0; u < NT; u += 2) {
                    const uint2 w = qw[hf][u / 2];
                    const float2 y0 = __half22float2(*reinterpret_cast<const __half2 *>(&w.x));
                    const float2 y1 = __half22float2(*reinterpret_cast<const __half2 *>(&w.y));
                    a = dot4(make_float4(y0.x, y0.y, y1.x, y1.y), x[mt], u, hf, a);
                    if (!kNorm) {
                        const float4 y = z[hf][u / 2];
                        store(dq + at + 8 * u, fmaf(gsc.y, x[mt][u][2 * hf], y.x), fmaf(gsc.y, x[mt][u][2 * hf + 1], y.y),
                              fmaf(gsc.y, x[mt][u + 1][2 * hf], y.z), fmaf(gsc.y, x[mt][u + 1][2 * hf + 1], y.w));
                    }
                }
                d4[2 * mt + hf] = a;
            }
        }
        dG = row_sum(d4);
        __syncthreads();                // dO has been read
        if constexpr (kNorm) norm_store(dq, p.q, p.dq_sm, x, gsc.y, SL::oA);
    }
    // ---- dW = -dU~ S0^T  -> A ----
    wait(2);
    {
        float x[2][NT][4];
        zero_acc(x);
        mma_block<NT, D, true, true>(a_pmt(SL::oC, D), b_pmt(SL::oE, n0), x);
        if (kNorm) named_barrier_sync(2 + (warp & 1), 128);    // norm_store's sums (in this half's rows) have been read
        if (__builtin_expect(__syncthreads_or(put(SL::oA, x, -1.f)), 0)) {      // dW in place; S0 has been read
            const float f = range(x);
            (void)put(SL::oA, x, -f);
            if (tid == 0) ms.fk = ms.fkv = 1.f / f;
            __syncthreads();
        }
    }
    if (tid == 0) {
        mbar_arrive_expect_tx(&ms.bar[3], 2 * SL::kU);
        tma_load_2d(smem + SL::oW, &map_wt, &ms.bar[3], 0, (int)(chunk * D));
        tma_load_2d(smem + SL::oUt, &map_ut, &ms.bar[3], 0, (int)(chunk * D));
    }
    // ---- dKb = T^T dW,  dVb = T^T dU~;  dv ----
    float pp[2][NT][4];
    zero_acc(pp);
    mma_block<NT, 64, true, true>(a_pmt(SL::oT, 64), b_swt(SL::oA, n0), pp);
    {
        float x[2][NT][4];
        zero_acc(x);
        mma_block<NT, 64, true, false>(a_pmt(SL::oT, 64), b_pm(SL::oC, n0), x);
        uint2 vw[2][NT / 2];                                // (every load of 16 rows ahead of their stores)
        float4 z[2][NT / 2];
        auto load_rows = [&](int mt) {
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                for (int u = 0; u < NT / 2; ++u) {
                    const size_t at = tok0 + (size_t)rowi(mt, hf) * ts + cb + 16 * u;
                    vw[hf][u] = *reinterpret_cast<const uint2 *>(p.v + at);
                    z[hf][u] = add4(kBlock && p.dv_x ? p.dv_x + at : nullptr);
                }
        };
        load_rows(0);
        __syncthreads();                // dW and dU~ have been read
        bool over = put(SL::oA, pp, 1.f);
        over |= put(SL::oC, x, 1.f);
        regroup(x);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            if (mt) load_rows(mt);
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int i = rowi(mt, hf);
                const size_t at = tok0 + (size_t)i * ts + cb;
                const bool lin = kBlock || p.route[((size_t)b * p.L + (size_t)c * kC + i) * p.H + h] == 0;
                const float f = gsc.y * ms.bt[i];
                float a = 0.f;
#pragma unroll
                for (int u = 0; u < NT; u += 2) {
                    const float4 y = z[hf][u / 2];
                    a = dot4(bf4(vw[hf][u / 2]), x[mt], u, hf, a);
                    if (lin)
                        store(dv + at + 8 * u, fmaf(f, x[mt][u][2 * hf], y.x), fmaf(f, x[mt][u][2 * hf + 1], y.y),
                              fmaf(f, x[mt][u + 1][2 * hf], y.z), fmaf(f, x[mt][u + 1][2 * hf + 1], y.w));
                }
                d4[2 * mt + hf] = a;
            }
        }
        db = row_sum(d4);
        if (__builtin_expect(__syncthreads_or(over), 0)) {
            regroup(x);                 // (its own inverse)
            const float fk = range(pp), fv = range(x);
            (void)put(SL::oA, pp, fk);
            (void)put(SL::oC, x, fv);
            if (tid == 0) { ms.fv = 1.f / fv; ms.fkv = ms.fk / fk * fv; }
            __syncthreads();
        }
    }
    // ---- M = -(dKb W^T + dVb U^T);  Mg = M . Gamma, j < i -> T;  Ms = diag(beta~) Mg -> A ----
    wait(3);
    {
        float x[2][2][4];
        zero_acc(x);
        mma_block<2, D, false, true>(a_sw(SL::oA), b_swt(SL::oW, j0), x);     // (W^T, U^T: one 64-column tile of D rows)
        scale_rows(x, 0, [&](int) { return ms.fkv; });
        mma_block<2, D, false, true>(a_sw(SL::oC), b_swt(SL::oUt, j0), x);
        fence_proxy_async_smem();       // (threads' stores to A and C before the copies below)
        __syncthreads();
        if (tid == 0) {
            const int row = bh * p.L + c * kC;
            mbar_arrive_expect_tx(&ms.bar[4], D * D * 2 + SL::kU);
            bulk_load_1d(smem + SL::oC, p.dS16 + chunk * D * D, SL::kU < D * D * 2 ? SL::kU : D * D * 2, &ms.bar[4]);
            if (D == 128)
                bulk_load_1d(smem + SL::oW, p.dS16 + chunk * D * D + D * 64, SL::kU, &ms.bar[4]);
            for (int kb = 0; kb < KB; ++kb) tma_load_2d(smem + SL::oUt + kb * 8192, &map_qh, &ms.bar[4], kb * 64, row);
        }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    const int i = rowi(mt, hf), j = j0 + 8 * nt + 2 * t;
                    const float2 Gj = *reinterpret_cast<const float2 *>(&ms.G[j]);
                    const float y0 = -exp_ftz(j < i ? ms.G[i] - Gj.x : -INFINITY) * (ms.fv * x[mt][nt][2 * hf]);
                    const float y1 = -exp_ftz(j + 1 < i ? ms.G[i] - Gj.y : -INFINITY) * (ms.fv * x[mt][nt][2 * hf + 1]);
                    const uint32_t off = i * 128 + (((j >> 3) ^ (i & 7)) << 4) + 4 * t;
                    *reinterpret_cast<uint32_t *>(smem + SL::oT + off) = pack_half2(y0, y1);
                    *reinterpret_cast<uint32_t *>(smem + SL::oA + off) = pack_half2(ms.bt[i] * y0, ms.bt[i] * y1);
                }
    }
    __syncthreads();
    // ---- P = gamma dKb + Mg K ----
    scale_rows(pp, m0 + g, [&](int i) { return ms.fk * exp_ftz(ms.G[i]); });
    mma_block<NT, 64, false, true>(a_sw(SL::oT), b_swt(SL::oK, n0), pp);
    dot_sw(SL::oK, pp, d4);
    {
        const float a = row_sum(d4);
        db += a;
        dG = fmaf(ms.bt[ri], a, dG);
    }
    // ---- R = (gamma_C / gamma) dK~ + Ms^T K + Ns^T Q;  dk = beta~ P + R ----
    if (kNorm) __syncthreads();         // Mg has been read: norm_store's sums go there
    wait(4);
    {
        float x[2][NT][4];
        zero_acc(x);
        if (committed) {                // (an uncommitted block's exit-state gradient reaches nothing but the decay)
            // D = 128: keys 64 .. of dS1 are where W was
            const uint32_t oS = D == 128 && n0 >= 64 ? SL::oW - 8 * D * 16 : SL::oC;
            mma_block<NT, D, true, true>(a_pmt(SL::oB, D), b_pmt(oS, n0), x);
            const float GC = ms.G[63];
            scale_rows(x, m0 + g, [&](int i) { return exp_ftz(GC - ms.G[i]); });
            dot_sw(SL::oK, x, d4);
            kap = row_sum(d4);
        }
        mma_block<NT, 64, true, true>(a_swt(SL::oA), b_swt(SL::oK, n0), x);
        mma_block<NT, 64, true, true>(a_swt(SL::oY), b_swt(SL::oUt, n0), x);
        dot_sw(SL::oK, x, d4);
        dG -= row_sum(d4);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const float bt = ms.bt[rowi(mt, hf)];
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    x[mt][nt][2 * hf] = fmaf(bt, pp[mt][nt][2 * hf], x[mt][nt][2 * hf]);
                    x[mt][nt][2 * hf + 1] = fmaf(bt, pp[mt][nt][2 * hf + 1], x[mt][nt][2 * hf + 1]);
                }
            }
        regroup(x);
        if (!kNorm) {
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int i = rowi(mt, hf);
                    const size_t at = tok0 + (size_t)i * ts + cb;
                    if (!kBlock && p.route[((size_t)b * p.L + (size_t)c * kC + i) * p.H + h] != 0) continue;
#pragma unroll
                    for (int u = 0; u < NT; u += 2) {
                        const float4 z = add4(kBlock && p.dk_x ? p.dk_x + at + 8 * u : nullptr);
                        store(dk + at + 8 * u, fmaf(gsc.y, x[mt][u][2 * hf], z.x), fmaf(gsc.y, x[mt][u][2 * hf + 1], z.y),
                              fmaf(gsc.y, x[mt][u + 1][2 * hf], z.z), fmaf(gsc.y, x[mt][u + 1][2 * hf + 1], z.w));
                    }
                }
        }
        if constexpr (kNorm) norm_store(dk, p.k, p.dk_x, x, gsc.y, SL::oT);
    }
    // ---- <dS1, S0>, element for element (the same layout twice) ----
    {
        const uint4 *s0 = reinterpret_cast<const uint4 *>(p.S16 + chunk * D * D);
        constexpr int kN = D * D / 8 / kCbThreads;
        uint4 y[kN];
#pragma unroll
        for (int e = 0; e < kN; ++e) y[e] = __ldg(s0 + tid + e * kCbThreads);
        float a = 0.f;
#pragma unroll
        for (int e = 0; e < kN; ++e) {
            const int idx = tid + e * kCbThreads;
            const uint32_t o = idx * 16 < SL::kU ? SL::oC + idx * 16 : SL::oW + idx * 16 - SL::kU;
            const uint4 x = *reinterpret_cast<const uint4 *>(smem + o);
            const uint32_t xw[4] = {x.x, x.y, x.z, x.w}, yw[4] = {y[e].x, y[e].y, y[e].z, y[e].w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 xf = __half22float2(*reinterpret_cast<const __half2 *>(&xw[u]));
                const float2 yf = __half22float2(*reinterpret_cast<const __half2 *>(&yw[u]));
                a = fmaf(xf.x, yf.x, fmaf(xf.y, yf.y, a));
            }
        }
        a = warp_sum(a);
        if (lane == 0) ms.red[warp] = a;
    }
    __syncthreads();                    // every operand has been read
    // ---- per-token sums: the 4 column blocks in a fixed order ----
    float *rs = reinterpret_cast<float *>(smem);                            // dG, kappa, dbeta: [3][4][64]
    rs[wc * 64 + ri] = dG;
    rs[256 + wc * 64 + ri] = kap;
    rs[512 + wc * 64 + ri] = db;
    __syncthreads();
    if (tid < 64) {
        // dg_j = sum_{i >= j} dG_i + sum_i kappa_i + gamma_C <dS1, S0>  (i, j: tokens of the chunk)
        auto sum4 = [&](int w) {
            const float *x = rs + 256 * w + tid;
            return (x[0] + x[64]) + (x[128] + x[192]);
        };
        float suf = sum4(0);
        const float kp = warp_sum(sum4(1)), bsum = sum4(2);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_down_sync(0xffffffffu, suf, o);
            if (lane + o < 32) suf += y;
        }
        if (lane == 0) { ms.red[8 + warp] = suf; ms.red[10 + warp] = kp; }
        named_barrier_sync(1, 64);
        float gs = 0.f;
#pragma unroll
        for (int wv = 0; wv < 8; ++wv) gs += ms.red[wv];
        const float kall = ms.red[10] + ms.red[11];
        const float extra = kall + exp_ftz(ms.G[63]) * gs + (warp == 0 ? ms.red[9] : 0.f);
        if (kBlock && p.kap_c && tid == 0) p.kap_c[chunk] = gsc.y * kall;
        const size_t tk = ((size_t)b * p.L + (size_t)c * kC + tid) * p.H + h;
        p.dg[tk] = gsc.y * (suf + extra);
        p.dbeta[tk] = !kBlock && p.route[tk] ? 0.f : gsc.y * bsum;
    }
    if (tid == 0) {
        for (int i = 0; i < 5; ++i) mbar_wait_drain(&ms.bar[i], 0);       // no copy in flight at retirement
        if (ms.abort_flag) atomicMin(p.status, (int)NATSL_ERR_TIMEOUT);
    }
}

template <int D, bool kBlock, bool kNorm, typename TO>
cudaError_t chunk_bwd_impl(const CbArgs &a, const void *dO16, const void *Kh, const void *Wt, const void *U16,
                           void *dq, void *dk, void *dv, Shape s, cudaStream_t st) {
    const int NC = s.L / kC;
    const uint64_t BH = (uint64_t)s.B * s.H;
    CUtensorMap mdo, mkh, mqh, mwt, mut;
    if (!tch::make_map_2d(&mdo, dO16, BH * s.L, D, 64) || !tch::make_map_2d(&mkh, Kh, BH * s.L, D, 64) ||
        !tch::make_map_2d(&mqh, a.Qh, BH * s.L, D, 64) || !tch::make_map_2d(&mwt, Wt, BH * NC * D, 64, D) ||
        !tch::make_map_2d(&mut, U16, BH * NC * D, 64, D))
        return cudaErrorInvalidValue;
    auto kernel = gdn_chunk_bwd_kernel<D, kBlock, kNorm, TO>;
    cudaError_t e = allow_smem(kernel, CbLayout<D>::kTotal);
    if (e != cudaSuccess) return e;
    dim3 grid(NC, s.B * s.H);
    kernel<<<grid, kCbThreads, CbLayout<D>::kTotal, st>>>(mdo, mkh, mqh, mwt, mut, (TO *)dq, (TO *)dk, (TO *)dv, a);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gdn_chunk_bwd(const GdnTcWs &ws, const GdnTcExport &ex, const GdnTcGrads &gr, const void *q,
                                 const void *k, const void *v, const float *beta, const uint8_t *route,
                                 const float *dq_sm, float scale_la, void *dq, void *dk, void *dv, float *dg,
                                 float *dbeta, bool block, const float *dk_x, const float *dv_x, float *kap_c,
                                 int32_t *status, Shape s, cudaStream_t st, HeadGroups hg) {
    const bool normed = hg.norm_eps >= 0.f;
    const CbArgs a{(const __half *)ex.Ut16, (const __half *)gr.dU16, (const __half *)ex.S16, (const __half *)gr.dS16,
                   (const __half *)ex.T16, (const __half *)ws.Qh, (const __nv_bfloat16 *)v, ex.Gcum, beta, dq_sm, route,
                   dk_x, dv_x, scale_la, dg, dbeta, (const __nv_bfloat16 *)q, (const __nv_bfloat16 *)k, hg.norm_eps,
                   hg.G, kap_c, status, s.L, s.H, debug_wait_kcycles()};
#define RUN(BL, NO, T)                                                                                               \
    do {                                                                                                             \
        if (s.d == 128) return chunk_bwd_impl<128, BL, NO, T>(a, gr.dO16, ws.Kh, ws.Wt, ex.U16, dq, dk, dv, s, st); \
        return chunk_bwd_impl<64, BL, NO, T>(a, gr.dO16, ws.Kh, ws.Wt, ex.U16, dq, dk, dv, s, st);                  \
    } while (0)
    if (block) {
        if (normed) RUN(true, true, __nv_bfloat16);
        RUN(true, false, __nv_bfloat16);
    }
    if (normed) RUN(false, false, float);
    RUN(false, false, __nv_bfloat16);
#undef RUN
}

}  // namespace natsl
