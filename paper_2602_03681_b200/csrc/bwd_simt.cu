// fp32 CUDA-core backward of the hybrid layer.
//
// The paper states the properties the backward must have (Section 4.2: the softmax logit
// gradient is P (dP - <do, o>); k, v gradients of an operation vanish for tokens inactive for
// it) but gives no backward of the gated delta rule.  This file differentiates the chunkwise
// forward of fwd_simt.cu.  Per chunk, with entry state S0, exit-state gradient dS1, output
// gradient dO and the forward quantities W, U, P, U~ (same notation as fwd_simt.cu):
//
//   dU~ = P^T dO + K~ dS1                       K~ = diag(gamma_C / gamma) K
//   dS0 = Qg^T dO + gamma_C dS1 - W^T dU~       Qg = scale_la diag(gamma) Q      (reverse scan)
//   dQg = dO S0^T     dW = -dU~ S0^T     dK~ = U~ dS1^T     N = lower(dO U~^T)
//   [dKb | dVb] = (I + A)^-T [dW | dU~]         Kb = diag(beta~ gamma) K, Vb = diag(beta~) V
//   M  = -strict_lower(dKb W^T + dVb U^T)       (gradient w.r.t. A)
//   dq = scale_la gamma dQg + (N . scale_la Gamma) K
//   dk = beta~ gamma dKb + (gamma_C/gamma) dK~ + (M . beta~ Gamma) K + (M . beta~ Gamma)^T K
//        + (N . scale_la Gamma)^T Q
//   dv = beta~ dVb
//   every gamma / Gamma factor contributes to dG_i (G = in-chunk cumulative log decay), and
//   dg_j = sum_{i >= j} dG_i;  dbeta = (1 - route) dbeta~.
//
// The dense products run through one generic batched tile-GEMM kernel over (batch, head,
// chunk); the sequential part is the reverse scan.  Softmax-branch gradients are formed over
// the compacted K/V list only and scattered back to the retained tokens.
#include <cuda_fp16.h>

#include "common.cuh"
#include "natsl_internal.h"

namespace natsl {

namespace {

constexpr int kThreads = 256;

// ------------------------------------------------------------------------------------------
// generic batched GEMM: C = alpha * op(A) op(B) (+ C), 64x64 output tiles, fp32 FMAs (fp32 storage; with bf16 storage
// only when fp32 arithmetic is asked for).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ const float *mat_base(const BMat &m, int b, int h, int ch) {
    return m.p + (size_t)b * m.sb + (size_t)h * m.sh + (size_t)ch * m.sc;
}

template <bool TA, bool TB, int MASK>
__global__ void __launch_bounds__(kThreads)
bgemm_kernel(BMat A, BMat B, BMat Cm, int K, float alpha, int accumulate, int H, int NC) {
    constexpr int kLd = 68;
    __shared__ __align__(16) float As[16][kLd];
    __shared__ __align__(16) float Bs[16][kLd];
    const int z = blockIdx.z, ch = z % NC, bh = z / NC, b = bh / H, h = bh % H;
    const float *Ap = mat_base(A, b, h, ch), *Bp = mat_base(B, b, h, ch);
    float *Cp = const_cast<float *>(mat_base(Cm, b, h, ch));
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
    float acc[4][4];          // rows ty*4 + i, columns tx*4 + j
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    for (int k0 = 0; k0 < K; k0 += 16) {
        if (!TA) {   // A[m][k], k contiguous
            const int r = t >> 2, kk = (t & 3) * 4;
            const float4 x = *reinterpret_cast<const float4 *>(Ap + (size_t)(m0 + r) * A.ld + k0 + kk);
            As[kk][r] = x.x; As[kk + 1][r] = x.y; As[kk + 2][r] = x.z; As[kk + 3][r] = x.w;
        } else {     // A[k][m], m contiguous
            const int kk = t >> 4, r4 = (t & 15) * 4;
            *reinterpret_cast<float4 *>(&As[kk][r4]) =
                *reinterpret_cast<const float4 *>(Ap + (size_t)(k0 + kk) * A.ld + m0 + r4);
        }
        if (!TB) {   // B[k][n], n contiguous
            const int kk = t >> 4, c4 = (t & 15) * 4;
            *reinterpret_cast<float4 *>(&Bs[kk][c4]) =
                *reinterpret_cast<const float4 *>(Bp + (size_t)(k0 + kk) * B.ld + n0 + c4);
        } else {     // B[n][k], k contiguous
            const int c = t >> 2, kk = (t & 3) * 4;
            const float4 x = *reinterpret_cast<const float4 *>(Bp + (size_t)(n0 + c) * B.ld + k0 + kk);
            Bs[kk][c] = x.x; Bs[kk + 1][c] = x.y; Bs[kk + 2][c] = x.z; Bs[kk + 3][c] = x.w;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const float4 a = *reinterpret_cast<const float4 *>(&As[kk][ty * 4]);
            const float4 bb = *reinterpret_cast<const float4 *>(&Bs[kk][tx * 4]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = m0 + ty * 4 + i;
        float *cr = Cp + (size_t)row * Cm.ld + n0 + tx * 4;
        float o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int col = n0 + tx * 4 + j;
            float val = alpha * acc[i][j];
            if (MASK == 1 && col > row) val = 0.f;
            if (MASK == 2 && col >= row) val = 0.f;
            o[j] = val;
        }
        if (accumulate) {
            const float4 old = *reinterpret_cast<const float4 *>(cr);
            o[0] += old.x; o[1] += old.y; o[2] += old.z; o[3] += old.w;
        }
        *reinterpret_cast<float4 *>(cr) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

// ------------------------------------------------------------------------------------------
// storage type -> fp32 copies of q, k, v
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void to_f32_kernel(const T *__restrict__ a, const T *__restrict__ b, const T *__restrict__ c,
                              float *__restrict__ a32, float *__restrict__ b32,
                              float *__restrict__ c32, size_t n4) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (size_t)gridDim.x * blockDim.x) {
        if (a) store4(a32 + 4 * i, load4(a + 4 * i));      // (a, b: optional)
        if (b) store4(b32 + 4 * i, load4(b + 4 * i));
        store4(c32 + 4 * i, load4(c + 4 * i));
    }
}

// ------------------------------------------------------------------------------------------
// combination backward (row-local): do_la, do_nla, dw, Dsm = <do_nla, o_nla>
// ------------------------------------------------------------------------------------------
// max |dout| over the whole tensor, as the bit pattern of a non-negative float (ordered like an
// integer), into the status page; the word is zeroed by the caller beforehand.
// (Magnitudes of bf16 values order like their bits: packed 16-bit maxima, 64 bytes in flight per thread; one atomic
// per CTA -- one per warp was a queue of 9000 on one address.)
template <typename T>
__global__ void __launch_bounds__(256)
dout_amax_kernel(const T *__restrict__ dout, size_t n16, int32_t *status) {
    __shared__ int part[8];
    const uint4 *src = reinterpret_cast<const uint4 *>(dout);          // 16-byte pieces
    auto fold = [](uint32_t m, uint32_t u) {
        return sizeof(T) == 2 ? __vmaxu2(m, u & 0x7fff7fffu) : max(m, u & 0x7fffffffu);
    };
    uint32_t m = 0u;
    const size_t stride = (size_t)gridDim.x * 256;
    size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    for (; i + 3 * stride < n16; i += 4 * stride) {
        uint4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = src[i + u * stride];
#pragma unroll
        for (int u = 0; u < 4; ++u) m = fold(fold(fold(fold(m, x[u].x), x[u].y), x[u].z), x[u].w);
    }
    for (; i < n16; i += stride) {
        const uint4 x = src[i];
        m = fold(fold(fold(fold(m, x.x), x.y), x.z), x.w);
    }
    int bits = (int)(sizeof(T) == 2 ? max(m >> 16, m & 0xffffu) << 16 : m);
    bits = __reduce_max_sync(0xffffffffu, bits);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = bits;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int x = 1; x < 8; ++x) bits = max(bits, part[x]);
        if (bits > 0) atomicMax(status + kGradAmaxWord, bits);
    }
}

// Four neighbouring columns per lane (one vector per array and lane), D / 4 lanes per row, so a warp takes
// two rows at D = 64: the kernel sits at the head of the backward's dependency chain and is bound by how
// many bytes a warp has in flight.
// G > 1 (grouped softmax heads, Section 4.3): the softmax branch's output is normalised per slice of
// D / G columns, so its part of the backward (do_nla, dw_nla, D_i = <do_i, o_i>) is formed per slice;
// Dsm is then [B,H,G,L].  A slice is an aligned group of D / (4 G) lanes: one xor butterfly gives the
// slice's sum on its way to the row's.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
combine_bwd_kernel(const float *__restrict__ o_la, const float *__restrict__ o_nla,
                   const T *__restrict__ dout, const float *__restrict__ w, float eps,
                   float *__restrict__ do_la, float *__restrict__ do_nla, float *__restrict__ dw,
                   float *__restrict__ Dsm, __half *__restrict__ do16,
                   __half *__restrict__ dola16, __half *__restrict__ dolag16,
                   const float *__restrict__ Gd, float scale_la, const int32_t *gsc, int G, int B, int L, int H) {
    constexpr int kE = 8, kLpr = D / kE, kRpw = 32 / kLpr;  // columns per lane, lanes per row, rows per warp
    const float gs = grad_scale(gsc).x;      // scale of the fp16 operand copies (and of Dsm with them)
    const int lane = threadIdx.x & 31, sub = lane / kLpr, li = lane % kLpr;
    const int lps = kLpr / G;                               // lanes per slice
    const float inv_ds = (float)G / D;
    const size_t row = ((size_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * kRpw + sub;
    const bool live = row < (size_t)B * L * H;              // (all lanes stay for the shuffles)
    const size_t rr = live ? row : 0;
    const int h = rr % H;
    const size_t bl = rr / H;
    const int l = bl % L, b = bl / L;
    const size_t at = rr * D + li * kE;
    float ol[kE], on[kE], dy[kE];
    auto load8 = [](const float *p, float (&x)[kE]) {
        const float4 u = *reinterpret_cast<const float4 *>(p), v = *reinterpret_cast<const float4 *>(p + 4);
        x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
    };
    load8(o_la + at, ol);
    load8(o_nla + at, on);
    if constexpr (sizeof(T) == 2) {
        const uint4 u = *reinterpret_cast<const uint4 *>(dout + at);
        const uint32_t uw[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            dy[2 * x] = __uint_as_float(uw[x] << 16);
            dy[2 * x + 1] = __uint_as_float(uw[x] & 0xffff0000u);
        }
    } else {
        load8(reinterpret_cast<const float *>(dout) + at, dy);
    }
    const float wn = w ? w[rr * 2] : 0.5f, wl = w ? w[rr * 2 + 1] : 0.5f;
    // scale_la gamma_l of the token (decay from its chunk's entry), for the reverse scan's operand
    const float sg = dolag16 ? scale_la * Gd[((size_t)(b * H + h) * (L / kC) + l / kC) * 128 + l % kC] : 0.f;
    // All sums follow from four: |o_la|^2 and <dy, o_la> over the row, |o_nla|^2 and <dy, o_nla> over the slice.
    float sl = 0.f, cl = 0.f, sn = 0.f, cn = 0.f;
#pragma unroll
    for (int x = 0; x < kE; ++x) {
        sl = fmaf(ol[x], ol[x], sl); cl = fmaf(dy[x], ol[x], cl);
        sn = fmaf(on[x], on[x], sn); cn = fmaf(dy[x], on[x], cn);
    }
#pragma unroll
    for (int o = 1; o < kLpr; o <<= 1) {
        sl += __shfl_xor_sync(0xffffffffu, sl, o);
        cl += __shfl_xor_sync(0xffffffffu, cl, o);
        if (o < lps) {                                      // (uniform)
            sn += __shfl_xor_sync(0xffffffffu, sn, o);
            cn += __shfl_xor_sync(0xffffffffu, cn, o);
        }
    }
    const float fl = rsqrtf(sl / D + eps), fn = rsqrtf(sn * inv_ds + eps);
    const float dwl = fl * cl, dwn_s = fn * cn;             // <dy, y_la> of the row, <dy, y_nla> of the slice
    float dwn = dwn_s;
    for (int o = lps; o < kLpr; o <<= 1) dwn += __shfl_xor_sync(0xffffffffu, dwn, o);
    const float ml = wl * dwl / D, mn = wn * dwn_s * inv_ds;
    if (!live) return;
    float dl[kE], dn[kE];
#pragma unroll
    for (int x = 0; x < kE; ++x) {
        dl[x] = fl * (wl * dy[x] - ol[x] * fl * ml);
        dn[x] = fn * (wn * dy[x] - on[x] * fn * mn);
    }
    // (the tensor-core kernels read the fp16 copies only)
    auto put8 = [](float *p, const float (&x)[kE]) {
        *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
        *reinterpret_cast<float4 *>(p + 4) = make_float4(x[4], x[5], x[6], x[7]);
    };
    if (do_la) put8(do_la + at, dl);
    if (do_nla) put8(do_nla + at, dn);
    const size_t at16 = (((size_t)b * H + h) * L + l) * D + li * kE;
    auto put16 = [](__half *p, float f, const float (&x)[kE]) {
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const __half2 y = __floats2half2_rn(f * x[2 * e], f * x[2 * e + 1]);
            o[e] = *reinterpret_cast<const uint32_t *>(&y);
        }
        *reinterpret_cast<uint4 *>(p) = make_uint4(o[0], o[1], o[2], o[3]);
    };
    if (do16) put16(do16 + at16, gs, dn);
    if (dolag16) {
        put16(dola16 + at16, gs, dl);
        put16(dolag16 + at16, gs * sg, dl);
    }
    if (li % lps == 0)                                      // <do_nla, o_nla> of the slice
        Dsm[(((size_t)b * H + h) * G + li / lps) * L + l] = gs * fn * (wn * cn - fn * mn * sn);
    if (li == 0 && dw) { dw[rr * 2] = dwn; dw[rr * 2 + 1] = dwl; }
}

// ------------------------------------------------------------------------------------------
// softmax backward, query side: dq_sm.  grid = (L/64, B*H), same tiling as the forward.
// ------------------------------------------------------------------------------------------
// G softmax heads per linear head (Section 4.3): the kernel's head is a slice of D columns of rows of
// DL = G D columns; lse and Dsm are [B,H,G,L].
template <int D, int G>
__global__ void __launch_bounds__(kThreads)
softmax_bwd_dq_kernel(const float *__restrict__ q32, const float *__restrict__ k_sm32,
                      const float *__restrict__ v_sm32, int cap, const int32_t *__restrict__ sm_idx,
                      const int32_t *__restrict__ sm_chunk_prefix,
                      const float *__restrict__ do_nla, const float *__restrict__ lse,
                      const float *__restrict__ Dsm, float scale_sm, float *__restrict__ dq_sm,
                      int L, int H) {
    extern __shared__ float smem[];
    float *Qs = smem;                      // [64][D]
    float *dOs = Qs + kC * D;              // [64][D]
    float *Kt = dOs + kC * D;              // [32][D+1]
    float *Vt = Kt + 32 * (D + 1);         // [32][D+1]
    int *pos = reinterpret_cast<int *>(Vt + 32 * (D + 1));

    constexpr int DL = D * G;
    const int c = blockIdx.x, bhg = blockIdx.y, bh = bhg / G, col0 = (bhg % G) * D, b = bh / H, h = bh % H;
    const int NC = L / kC;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t ts = (size_t)H * DL;
    const size_t tok0 = ((size_t)b * L + (size_t)c * kC) * H + h;
    const int n_end = min(sm_chunk_prefix[(size_t)bh * (NC + 1) + c + 1], cap);

    for (int idx = threadIdx.x; idx < kC * D / 4; idx += kThreads) {
        const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
        store4(Qs + r * D + c4, load4(q32 + tok0 * DL + (size_t)r * ts + col0 + c4));
        store4(dOs + r * D + c4, load4(do_nla + tok0 * DL + (size_t)r * ts + col0 + c4));
    }
    constexpr int kQ = 8, kCols = D / 32;
    float acc[kQ][kCols], lse_r[kQ], dsm_r[kQ];
#pragma unroll
    for (int r = 0; r < kQ; ++r) {
        const int i = c * kC + warp * kQ + r;
        lse_r[r] = lse[(size_t)bhg * L + i];
        dsm_r[r] = Dsm[(size_t)bhg * L + i];
#pragma unroll
        for (int x = 0; x < kCols; ++x) acc[r][x] = 0.f;
    }
    const float *kb = k_sm32 + (size_t)bh * cap * DL + col0, *vb = v_sm32 + (size_t)bh * cap * DL + col0;
    for (int j0 = 0; j0 < n_end; j0 += 32) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < 32 * D / 4; idx += kThreads) {
            const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
            float4 kx = make_float4(0.f, 0.f, 0.f, 0.f), vx = kx;
            if (j0 + r < n_end) {
                kx = load4(kb + (size_t)(j0 + r) * DL + c4);
                vx = load4(vb + (size_t)(j0 + r) * DL + c4);
            }
            float *kp = Kt + r * (D + 1) + c4, *vp = Vt + r * (D + 1) + c4;
            kp[0] = kx.x; kp[1] = kx.y; kp[2] = kx.z; kp[3] = kx.w;
            vp[0] = vx.x; vp[1] = vx.y; vp[2] = vx.z; vp[3] = vx.w;
        }
        if (threadIdx.x < 32)
            pos[threadIdx.x] = (j0 + threadIdx.x < n_end) ? sm_idx[(size_t)bh * L + j0 + threadIdx.x]
                                                          : 0x7fffffff;
        __syncthreads();
        const int my_pos = pos[lane];
        const float *kr = Kt + lane * (D + 1), *vr = Vt + lane * (D + 1);
#pragma unroll
        for (int r = 0; r < kQ; ++r) {
            const int i = c * kC + warp * kQ + r;
            const float *qr = Qs + (warp * kQ + r) * D, *dor = dOs + (warp * kQ + r) * D;
            float s = 0.f, dp = 0.f;
#pragma unroll 8
            for (int x = 0; x < D; ++x) {
                s = fmaf(qr[x], kr[x], s);
                dp = fmaf(dor[x], vr[x], dp);
            }
            const float pj = (my_pos <= i) ? __expf(s * scale_sm - lse_r[r]) : 0.f;
            const float ds = pj * (dp - dsm_r[r]);
            for (int j = 0; j < 32; ++j) {
                const float db = __shfl_sync(0xffffffffu, ds, j);
#pragma unroll
                for (int x = 0; x < kCols; ++x)
                    acc[r][x] = fmaf(db, Kt[j * (D + 1) + lane + 32 * x], acc[r][x]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < kQ; ++r) {
        const size_t t = tok0 + (size_t)(warp * kQ + r) * H;
#pragma unroll
        for (int x = 0; x < kCols; ++x) dq_sm[t * DL + col0 + lane + 32 * x] = scale_sm * acc[r][x];
    }
}

// ------------------------------------------------------------------------------------------
// softmax backward, key side: dk_sm, dv_sm per compacted key.  grid = (ceil(cap/32), B*H).
// ------------------------------------------------------------------------------------------
template <int D, int G>
__global__ void __launch_bounds__(kThreads)
softmax_bwd_dkv_kernel(const float *__restrict__ q32, const float *__restrict__ k_sm32,
                       const float *__restrict__ v_sm32, int cap, const int32_t *__restrict__ sm_idx,
                       const int32_t *__restrict__ sm_chunk_prefix,
                       const float *__restrict__ do_nla, const float *__restrict__ lse,
                       const float *__restrict__ Dsm, float scale_sm, float *__restrict__ dk_sm,
                       float *__restrict__ dv_sm, float *__restrict__ dmask, int L, int H) {
    // dmask [B,H,cap] (or nullptr): per retained key j the sum over its queries of
    // dM_ij = p_ij (dp_ij - <do_i, o_i>), the mask gradient of Section 4.2
    extern __shared__ float smem[];
    float *Kt = smem;                       // [32][D+1]
    float *Vt = Kt + 32 * (D + 1);          // [32][D+1]
    float *Qs = Vt + 32 * (D + 1);          // [64][D]
    float *dOs = Qs + kC * D;               // [64][D]
    float *Ps = dOs + kC * D;               // [64][33]
    float *Dss = Ps + kC * 33;              // [64][33]
    float *lse_s = Dss + kC * 33;           // [64]
    float *dsm_s = lse_s + kC;              // [64]
    int *pos = reinterpret_cast<int *>(dsm_s + kC);

    constexpr int DL = D * G;
    const int bhg = blockIdx.y, bh = bhg / G, col0 = (bhg % G) * D, b = bh / H, h = bh % H;
    const int NC = L / kC;
    const int n_sm = min(sm_chunk_prefix[(size_t)bh * (NC + 1) + NC], cap);
    const int j0 = blockIdx.x * 32;
    if (j0 >= n_sm) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t ts = (size_t)H * DL;
    const float *kb = k_sm32 + (size_t)bh * cap * DL + col0, *vb = v_sm32 + (size_t)bh * cap * DL + col0;

    for (int idx = threadIdx.x; idx < 32 * D / 4; idx += kThreads) {
        const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
        float4 kx = make_float4(0.f, 0.f, 0.f, 0.f), vx = kx;
        if (j0 + r < n_sm) {
            kx = load4(kb + (size_t)(j0 + r) * DL + c4);
            vx = load4(vb + (size_t)(j0 + r) * DL + c4);
        }
        float *kp = Kt + r * (D + 1) + c4, *vp = Vt + r * (D + 1) + c4;
        kp[0] = kx.x; kp[1] = kx.y; kp[2] = kx.z; kp[3] = kx.w;
        vp[0] = vx.x; vp[1] = vx.y; vp[2] = vx.z; vp[3] = vx.w;
    }
    if (threadIdx.x < 32)
        pos[threadIdx.x] = (j0 + threadIdx.x < n_sm) ? sm_idx[(size_t)bh * L + j0 + threadIdx.x]
                                                     : 0x7fffffff;
    __syncthreads();
    const int my_pos = pos[lane];
    const int c_first = pos[0] / kC;
    constexpr int kPer = D / 8;
    const int kj = threadIdx.x >> 3, cs = threadIdx.x & 7;
    float adk[kPer], adv[kPer], adm = 0.f;
#pragma unroll
    for (int x = 0; x < kPer; ++x) { adk[x] = 0.f; adv[x] = 0.f; }

    for (int c = c_first; c < NC; ++c) {
        const size_t tok0 = ((size_t)b * L + (size_t)c * kC) * H + h;
        __syncthreads();
        for (int idx = threadIdx.x; idx < kC * D / 4; idx += kThreads) {
            const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
            store4(Qs + r * D + c4, load4(q32 + tok0 * DL + (size_t)r * ts + col0 + c4));
            store4(dOs + r * D + c4, load4(do_nla + tok0 * DL + (size_t)r * ts + col0 + c4));
        }
        if (threadIdx.x < kC) {
            lse_s[threadIdx.x] = lse[(size_t)bhg * L + c * kC + threadIdx.x];
            dsm_s[threadIdx.x] = Dsm[(size_t)bhg * L + c * kC + threadIdx.x];
        }
        __syncthreads();
        const float *kr = Kt + lane * (D + 1), *vr = Vt + lane * (D + 1);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int il = warp * 8 + r, i = c * kC + il;
            const float *qr = Qs + il * D, *dor = dOs + il * D;
            float s = 0.f, dp = 0.f;
#pragma unroll 8
            for (int x = 0; x < D; ++x) {
                s = fmaf(qr[x], kr[x], s);
                dp = fmaf(dor[x], vr[x], dp);
            }
            const float pj = (my_pos <= i) ? __expf(s * scale_sm - lse_s[il]) : 0.f;
            Ps[il * 33 + lane] = pj;
            Dss[il * 33 + lane] = pj * (dp - dsm_s[il]);
        }
        __syncthreads();
        for (int il = 0; il < kC; ++il) {
            const float pj = Ps[il * 33 + kj], ds = Dss[il * 33 + kj];
            adm += ds;
            const float *dor = dOs + il * D + cs, *qr = Qs + il * D + cs;
#pragma unroll
            for (int x = 0; x < kPer; ++x) {
                adv[x] = fmaf(pj, dor[8 * x], adv[x]);
                adk[x] = fmaf(ds, qr[8 * x], adk[x]);
            }
        }
    }
    if (j0 + kj < n_sm) {
        float *dkr = dk_sm + ((size_t)bh * cap + j0 + kj) * DL + col0 + cs;
        float *dvr = dv_sm + ((size_t)bh * cap + j0 + kj) * DL + col0 + cs;
#pragma unroll
        for (int x = 0; x < kPer; ++x) { dkr[8 * x] = scale_sm * adk[x]; dvr[8 * x] = adv[x]; }
        if (dmask && cs == 0) dmask[(size_t)bhg * cap + j0 + kj] = adm;
    }
}

// ------------------------------------------------------------------------------------------
// Block-level routing (Section 4.1, inner-chunk correlations): a query in a linear block also reads
// the causal part of its own block, whose tokens are not among the retained ones.  One CTA per
// linear block adds that part of the softmax branch's backward in fp32:
//   p_ij = exp(scale s_ij - lse_i), ds_ij = p_ij (dp_ij - D_i), j <= i, with lse_i and
//   D_i = <do_i, o_i> of the whole softmax row;
//   dq_sm += scale dS K;  dk_x = scale dS^T Q,  dv_x = P^T dO  (written: the tokens of a linear
//   block have no other softmax-branch gradient).  grid = (L/64, B*H); softmax blocks return.
// Dsm arrives times the gradient scale of the tensor-core kernels (gsc; 1 without them).
// ------------------------------------------------------------------------------------------
// G softmax heads per linear head: a CTA's head is a slice of D columns of rows of DL = G D columns;
// lse and Dsm are [B,H,G,L]; q32, k32 are the softmax operation's copies of q and k.
template <int D, int G>
__global__ void __launch_bounds__(kThreads)
softmax_bwd_own_block_simt_kernel(const float *__restrict__ q32, const float *__restrict__ k32,
                                  const float *__restrict__ v32, const float *__restrict__ do_nla,
                                  const float *__restrict__ lse, const float *__restrict__ Dsm,
                                  const uint8_t *__restrict__ route, float scale_sm,
                                  float *__restrict__ dq_sm, float *__restrict__ dk_x,
                                  float *__restrict__ dv_x, const int32_t *gsc, int L, int H) {
    extern __shared__ float smem[];
    float *Qs = smem;                        // [64][D+1]
    float *Ks = Qs + kC * (D + 1);
    float *Vs = Ks + kC * (D + 1);
    float *dOs = Vs + kC * (D + 1);
    float *Ps = dOs + kC * (D + 1);          // [64][65]
    float *dSs = Ps + kC * (kC + 1);         // [64][65]
    constexpr int DL = D * G;
    const int c = blockIdx.x, bhg = blockIdx.y, bh = bhg / G, col0 = (bhg % G) * D, b = bh / H, h = bh % H;
    const size_t ts = (size_t)H * DL;
    const size_t tok0 = ((size_t)b * L + (size_t)c * kC) * H + h;
    if (route[tok0]) return;                 // a softmax block: its tokens are retained ones
    const float ginv = grad_scale(gsc).y;
    for (int idx = threadIdx.x; idx < kC * D / 4; idx += kThreads) {
        const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
        const size_t src = tok0 * DL + (size_t)r * ts + col0 + c4;
        const float4 a = load4(q32 + src), bb = load4(k32 + src), cc = load4(v32 + src), dd = load4(do_nla + src);
        float *p0 = Qs + r * (D + 1) + c4, *p1 = Ks + r * (D + 1) + c4, *p2 = Vs + r * (D + 1) + c4,
              *p3 = dOs + r * (D + 1) + c4;
        p0[0] = a.x; p0[1] = a.y; p0[2] = a.z; p0[3] = a.w;
        p1[0] = bb.x; p1[1] = bb.y; p1[2] = bb.z; p1[3] = bb.w;
        p2[0] = cc.x; p2[1] = cc.y; p2[2] = cc.z; p2[3] = cc.w;
        p3[0] = dd.x; p3[1] = dd.y; p3[2] = dd.z; p3[3] = dd.w;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < kC * kC; idx += kThreads) {
        const int i = idx >> 6, j = idx & 63;
        float pj = 0.f, ds = 0.f;
        if (j <= i) {
            const float *qr = Qs + i * (D + 1), *kr = Ks + j * (D + 1), *dor = dOs + i * (D + 1), *vr = Vs + j * (D + 1);
            float s = 0.f, dp = 0.f;
#pragma unroll 8
            for (int x = 0; x < D; ++x) {
                s = fmaf(qr[x], kr[x], s);
                dp = fmaf(dor[x], vr[x], dp);
            }
            const size_t row = (size_t)bhg * L + (size_t)c * kC + i;
            pj = __expf(s * scale_sm - lse[row]);
            ds = pj * (dp - ginv * Dsm[row]);
        }
        Ps[i * (kC + 1) + j] = pj;
        dSs[i * (kC + 1) + j] = ds;
    }
    __syncthreads();
    // thread (row r, column group cg): D / 4 columns cg, cg + 4, ... of dq_r, dk_r, dv_r
    const int r = threadIdx.x >> 2, cg = threadIdx.x & 3;
    for (int x = cg; x < D; x += 4) {
        float aq = 0.f, ak = 0.f, av = 0.f;
        for (int j = 0; j <= r; ++j) aq = fmaf(dSs[r * (kC + 1) + j], Ks[j * (D + 1) + x], aq);
        for (int i = r; i < kC; ++i) {
            ak = fmaf(dSs[i * (kC + 1) + r], Qs[i * (D + 1) + x], ak);
            av = fmaf(Ps[i * (kC + 1) + r], dOs[i * (D + 1) + x], av);
        }
        const size_t dst = tok0 * DL + (size_t)r * ts + col0 + x;
        dq_sm[dst] += scale_sm * aq;
        dk_x[dst] = scale_sm * ak;
        dv_x[dst] = av;
    }
}

// ------------------------------------------------------------------------------------------
// reverse scan over chunks: dU~ (stored), chunk-exit dS (stored), <dS1, S0> partials.
// grid = (D/32, B*H), mirrors gdn_scan_simt_kernel.
// ------------------------------------------------------------------------------------------
constexpr int kDvs = 32;

template <int D>
__global__ void __launch_bounds__(kThreads)
gdn_rscan_kernel(const float *__restrict__ q32, const float *__restrict__ k32,
                 const float *__restrict__ Gcum, const float *__restrict__ W,
                 const float *__restrict__ P, const float *__restrict__ do_la,
                 const float *__restrict__ chunk_states, float scale_la, float *__restrict__ dUt,
                 float *__restrict__ dS_c, float *__restrict__ gS, const float *__restrict__ dstate_out,
                 float *__restrict__ dstate_in, const uint8_t *__restrict__ block_route, int L, int H) {
    // block_route (block-level routing): a softmax block's update was not committed to the state, so
    // its exit-state gradient reaches the entry state through the decay only: no K~ dS term in dU~, and
    // the stored chunk-exit gradient (which the dK~ product reads) is zero; <dS1, S0> is not.
    extern __shared__ float smem[];
    float *dSs = smem;                       // [D][32]
    float *Ws = dSs + D * kDvs;              // [64][D+1]
    float *Qs = Ws + kC * (D + 1);           // [64][D+1]
    float *Ks = Qs + kC * (D + 1);           // [64][D+1]
    float *Ps = Ks + kC * (D + 1);           // [64][65]
    float *dOs = Ps + kC * (kC + 1);         // [64][33]
    float *dUs = dOs + kC * (kDvs + 1);      // [64][33]
    float *Gs = dUs + kC * (kDvs + 1);       // [64]
    float *red = Gs + kC;                    // [8]

    const int slice = blockIdx.x, bh = blockIdx.y, b = bh / H, h = bh % H;
    const int NC = L / kC;
    const size_t ts = (size_t)H * D;
    const int c0 = slice * kDvs;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    for (int idx = threadIdx.x; idx < D * kDvs; idx += kThreads)     // gradient arriving at the final state
        dSs[idx] = dstate_out ? dstate_out[((size_t)bh * D + idx / kDvs) * D + c0 + idx % kDvs] : 0.f;

    for (int c = NC - 1; c >= 0; --c) {
        const size_t tok0 = ((size_t)b * L + (size_t)c * kC) * H + h;
        const float commit = block_route && block_route[tok0] ? 0.f : 1.f;
        __syncthreads();
        // store the chunk-exit gradient and the partial <dS1, S0>
        {
            float part = 0.f;
            for (int idx = threadIdx.x; idx < D * kDvs; idx += kThreads) {
                const int a = idx / kDvs, cc = idx % kDvs;
                const size_t gi = (((size_t)bh * NC + c) * D + a) * D + c0 + cc;
                dS_c[gi] = commit * dSs[idx];
                part = fmaf(dSs[idx], chunk_states[gi], part);
            }
            part = warp_sum(part);
            if (lane == 0) red[warp] = part;
        }
        for (int idx = threadIdx.x; idx < kC * D / 4; idx += kThreads) {
            const int r = idx / (D / 4), c4 = (idx % (D / 4)) * 4;
            const float4 wv = load4(W + tok0 * D + (size_t)r * ts + c4);
            const float4 qv = load4(q32 + tok0 * D + (size_t)r * ts + c4);
            const float4 kv = load4(k32 + tok0 * D + (size_t)r * ts + c4);
            float *wp = Ws + r * (D + 1) + c4, *qp = Qs + r * (D + 1) + c4, *kp = Ks + r * (D + 1) + c4;
            wp[0] = wv.x; wp[1] = wv.y; wp[2] = wv.z; wp[3] = wv.w;
            qp[0] = qv.x; qp[1] = qv.y; qp[2] = qv.z; qp[3] = qv.w;
            kp[0] = kv.x; kp[1] = kv.y; kp[2] = kv.z; kp[3] = kv.w;
        }
        {
            const float *Pc = P + ((size_t)bh * NC + c) * kC * kC;
            for (int idx = threadIdx.x; idx < kC * kC; idx += kThreads)
                Ps[(idx >> 6) * (kC + 1) + (idx & 63)] = Pc[idx];
            for (int idx = threadIdx.x; idx < kC * kDvs; idx += kThreads) {
                const int r = idx / kDvs, cc = idx % kDvs;
                dOs[r * (kDvs + 1) + cc] = do_la[(tok0 + (size_t)r * H) * D + c0 + cc];
            }
            if (threadIdx.x < kC) Gs[threadIdx.x] = Gcum[(size_t)bh * L + c * kC + threadIdx.x];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            float tot = 0.f;
            for (int wv = 0; wv < kThreads / 32; ++wv) tot += red[wv];
            gS[((size_t)bh * NC + c) * (D / kDvs) + slice] = tot;
        }
        const float gl = Gs[kC - 1];
        const int r = threadIdx.x >> 2, cb = (threadIdx.x & 3) * 8;
        // dU~_r = sum_{i>=r} P[i][r] dO_i + (gamma_C/gamma_r) k_r dS
        {
            float acc[8], acc2[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) { acc[x] = 0.f; acc2[x] = 0.f; }
            for (int i = r; i < kC; ++i) {
                const float pv = Ps[i * (kC + 1) + r];
                const float *dr = dOs + i * (kDvs + 1) + cb;
#pragma unroll
                for (int x = 0; x < 8; ++x) acc[x] = fmaf(pv, dr[x], acc[x]);
            }
            const float *kr = Ks + r * (D + 1);
            for (int a = 0; a < D; ++a) {
                const float kv = kr[a];
                const float *sr = dSs + a * kDvs + cb;
#pragma unroll
                for (int x = 0; x < 8; ++x) acc2[x] = fmaf(kv, sr[x], acc2[x]);
            }
            const float kt = commit * __expf(gl - Gs[r]);
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                acc[x] = fmaf(kt, acc2[x], acc[x]);
                dUs[r * (kDvs + 1) + cb + x] = acc[x];
            }
            float *dst = dUt + (tok0 + (size_t)r * H) * D + c0 + cb;
            store4(dst, make_float4(acc[0], acc[1], acc[2], acc[3]));
            store4(dst + 4, make_float4(acc[4], acc[5], acc[6], acc[7]));
        }
        __syncthreads();
        // dS0 = Qg^T dO + gamma_C dS1 - W^T dU~
        {
            constexpr int kPer = D / 8, kTpr = kDvs / kPer;
            const int a = threadIdx.x / kTpr, cs = (threadIdx.x % kTpr) * kPer;
            const float gC = __expf(gl);
            float acc[kPer];
#pragma unroll
            for (int x = 0; x < kPer; ++x) acc[x] = gC * dSs[a * kDvs + cs + x];
            for (int i = 0; i < kC; ++i) {
                const float qg = scale_la * __expf(Gs[i]) * Qs[i * (D + 1) + a];
                const float wv = Ws[i * (D + 1) + a];
                const float *dor = dOs + i * (kDvs + 1) + cs, *dur = dUs + i * (kDvs + 1) + cs;
#pragma unroll
                for (int x = 0; x < kPer; ++x) acc[x] = fmaf(qg, dor[x], fmaf(-wv, dur[x], acc[x]));
            }
            __syncthreads();
#pragma unroll
            for (int x = 0; x < kPer; ++x) dSs[a * kDvs + cs + x] = acc[x];
            if (c == 0 && dstate_in) {      // what is left after the first chunk: the initial state's gradient
#pragma unroll
                for (int x = 0; x < kPer; ++x) dstate_in[((size_t)bh * D + a) * D + c0 + cs + x] = acc[x];
            }
        }
    }
}

// ------------------------------------------------------------------------------------------
// transposed triangular solve: [dKb | dVb] = (I + A)^-T [dW | dU~], A = diag(beta~) Abar.
// grid = (L/C, B*H); one right-hand-side column per thread.
// ------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(kThreads)
gdn_tsolve_kernel(const float *__restrict__ Abar, const float *__restrict__ beta,
                  const uint8_t *__restrict__ route, const float *__restrict__ dW,
                  const float *__restrict__ dUt, float *__restrict__ dKb, float *__restrict__ dVb,
                  int L, int H) {
    __shared__ float As[kC * kC];
    __shared__ float bts[kC];
    const int c = blockIdx.x, bh = blockIdx.y, b = bh / H, h = bh % H;
    const size_t ts = (size_t)H * D;
    const size_t tok0 = ((size_t)b * L + (size_t)c * kC) * H + h;
    if (threadIdx.x < kC) {
        const size_t t = tok0 + (size_t)threadIdx.x * H;
        bts[threadIdx.x] = route && route[t] ? 0.f : beta[t];   // route == nullptr: beta~ = beta
    }
    __syncthreads();
    const float *Ab = Abar + ((size_t)bh * (L / kC) + c) * kC * kC;
    for (int idx = threadIdx.x; idx < kC * kC; idx += kThreads) As[idx] = bts[idx >> 6] * Ab[idx];
    __syncthreads();
    if (threadIdx.x < 2 * D) {
        const bool first = threadIdx.x < D;
        const int col = first ? threadIdx.x : threadIdx.x - D;
        const float *src = (first ? dW : dUt) + tok0 * D + col;
        float x[kC];
#pragma unroll
        for (int i = kC - 1; i >= 0; --i) {
            float acc = src[(size_t)i * ts];
#pragma unroll
            for (int j = i + 1; j < kC; ++j) acc = fmaf(-As[j * kC + i], x[j], acc);
            x[i] = acc;
        }
        float *dst = (first ? dKb : dVb) + tok0 * D + col;
#pragma unroll
        for (int i = 0; i < kC; ++i) dst[(size_t)i * ts] = x[i];
    }
}

// ------------------------------------------------------------------------------------------
// Mg = M . Gamma, Ms = diag(beta~) Mg, Ns = scale_la N . Gamma    (all 64x64 per chunk)
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads)
mask_scale_kernel(const float *__restrict__ M, const float *__restrict__ N,
                  const float *__restrict__ Gcum, const float *__restrict__ beta,
                  const uint8_t *__restrict__ route, float scale_la, float *__restrict__ Mg,
                  float *__restrict__ Ms, float *__restrict__ Ns, int L, int H) {
    __shared__ float Gs[kC], bts[kC];
    const int NC = L / kC;
    const int c = blockIdx.x, bh = blockIdx.y, b = bh / H, h = bh % H;
    if (threadIdx.x < kC) {
        const size_t t = ((size_t)b * L + (size_t)c * kC + threadIdx.x) * H + h;
        bts[threadIdx.x] = route && route[t] ? 0.f : beta[t];
        Gs[threadIdx.x] = Gcum[(size_t)bh * L + c * kC + threadIdx.x];
    }
    __syncthreads();
    const size_t base = ((size_t)bh * NC + c) * kC * kC;
    for (int idx = threadIdx.x; idx < kC * kC; idx += kThreads) {
        const int i = idx >> 6, j = idx & 63;
        const float gam = j <= i ? __expf(Gs[i] - Gs[j]) : 0.f;
        const float mg = M[base + idx] * gam;
        Mg[base + idx] = mg;
        Ms[base + idx] = bts[i] * mg;
        Ns[base + idx] = scale_la * N[base + idx] * gam;
    }
}

// ------------------------------------------------------------------------------------------
// assembly: dq (all tokens), dk/dv (linear tokens), per-row dG, kappa, dbeta.
// one warp per (token, head) row.
// ------------------------------------------------------------------------------------------
template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
gdn_assemble_kernel(const float *__restrict__ q32, const float *__restrict__ k32,
                    const float *__restrict__ v32, const float *__restrict__ Gcum,
                    const float *__restrict__ beta, const uint8_t *__restrict__ route,
                    const float *__restrict__ dQg, const float *__restrict__ dKb,
                    const float *__restrict__ dVb, const float *__restrict__ dKt,
                    const float *__restrict__ X1p, const float *__restrict__ X2,
                    const float *__restrict__ X3, const float *__restrict__ X4,
                    const float *__restrict__ dq_sm, const float *__restrict__ dk_x,
                    const float *__restrict__ dv_x, float scale_la, T *__restrict__ dq,
                    T *__restrict__ dk, T *__restrict__ dv, float *__restrict__ dGrow,
                    float *__restrict__ kappa, float *__restrict__ dbeta, int B, int L, int H) {
    constexpr int kCols = D / 32;
    const int lane = threadIdx.x & 31;
    const size_t row = (size_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    if (row >= (size_t)B * L * H) return;
    const int h = row % H;
    const size_t bl = row / H;
    const int l = bl % L, b = bl / L;
    const size_t bhl = ((size_t)b * H + h) * L;
    const float Gi = Gcum[bhl + l], GC = Gcum[bhl + (l | (kC - 1))];
    // route == nullptr (block-level routing): every token takes part in the delta rule, and every
    // token's dk, dv also has a softmax-branch part, given in dk_x, dv_x (fp32, token-major)
    const bool lin = !route || route[row] == 0;
    const float bt = lin ? beta[row] : 0.f;
    const float gam = __expf(Gi), kt = __expf(GC - Gi);
    float kdKb = 0.f, qdQg = 0.f, kdKt = 0.f, kX1 = 0.f, kX2 = 0.f, qX3 = 0.f, kX4 = 0.f, vdVb = 0.f;
#pragma unroll
    for (int x = 0; x < kCols; ++x) {
        const size_t i = row * D + lane + 32 * x;
        const float qv = q32[i], kv = k32[i], vv = v32[i];
        const float a_dQg = dQg[i], a_dKb = dKb[i], a_dVb = dVb[i], a_dKt = dKt[i];
        const float x1 = X1p[i], x2 = X2[i], x3 = X3[i], x4 = X4[i];
        kdKb = fmaf(kv, a_dKb, kdKb); qdQg = fmaf(qv, a_dQg, qdQg); kdKt = fmaf(kv, a_dKt, kdKt);
        kX1 = fmaf(kv, x1, kX1); kX2 = fmaf(kv, x2, kX2); qX3 = fmaf(qv, x3, qX3);
        kX4 = fmaf(kv, x4, kX4); vdVb = fmaf(vv, a_dVb, vdVb);
        dq[i] = from_f32<T>(scale_la * gam * a_dQg + x3 + (dq_sm ? dq_sm[i] : 0.f));
        if (lin) {
            dk[i] = from_f32<T>(bt * gam * a_dKb + kt * a_dKt + bt * x1 + x2 + x4 + (dk_x ? dk_x[i] : 0.f));
            dv[i] = from_f32<T>(bt * a_dVb + (dv_x ? dv_x[i] : 0.f));
        }
    }
    kdKb = warp_sum(kdKb); qdQg = warp_sum(qdQg); kdKt = warp_sum(kdKt); kX1 = warp_sum(kX1);
    kX2 = warp_sum(kX2); qX3 = warp_sum(qX3); kX4 = warp_sum(kX4); vdVb = warp_sum(vdVb);
    if (lane == 0) {
        const float kap = kt * kdKt;
        dGrow[bhl + l] = bt * gam * kdKb + scale_la * gam * qdQg - kap + bt * kX1 - kX2 + qX3 - kX4;
        kappa[bhl + l] = kap;
        dbeta[row] = lin ? gam * kdKb + vdVb + kX1 : 0.f;
    }
}

// dg_j = sum_{i>=j in chunk} dG_i, with the chunk-end extras added to the last row.
__global__ void dg_kernel(const float *__restrict__ dGrow, const float *__restrict__ kappa,
                          const float *__restrict__ gS, const float *__restrict__ Gcum, int n_slices,
                          float *__restrict__ dg, int B, int L, int H) {
    const int NC = L / kC;
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)B * H * NC) return;
    const int c = idx % NC;
    const size_t bh = idx / NC;
    const int h = bh % H, b = bh / H;
    const size_t base = bh * L + (size_t)c * kC;
    float extra = 0.f;
    for (int i = 0; i < kC; ++i) extra += kappa[base + i];
    float gs = 0.f;
    for (int s = 0; s < n_slices; ++s) gs += gS[idx * n_slices + s];
    extra += __expf(Gcum[base + kC - 1]) * gs;
    float run = extra;
    for (int i = kC - 1; i >= 0; --i) {
        run += dGrow[base + i];
        dg[((size_t)b * L + (size_t)c * kC + i) * H + h] = run;
    }
}

// dk, dv of the retained tokens: scatter the compacted softmax-branch gradients.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
scatter_sm_kernel(const float *__restrict__ dk_sm, const float *__restrict__ dv_sm, int cap,
                  const int32_t *__restrict__ sm_idx, const int32_t *__restrict__ sm_chunk_prefix,
                  T *__restrict__ dk, T *__restrict__ dv, int L, int H) {
    constexpr int kVec = D / 4, kRows = kThreads / kVec;
    const int bh = blockIdx.y, b = bh / H, h = bh % H;
    const int NC = L / kC;
    const int n = min(sm_chunk_prefix[(size_t)bh * (NC + 1) + NC], cap);
    const int row = blockIdx.x * kRows + threadIdx.x / kVec, c4 = (threadIdx.x % kVec) * 4;
    if (row >= n) return;
    const int tok = sm_idx[(size_t)bh * L + row];
    const size_t dst = (((size_t)b * L + tok) * H + h) * D + c4;
    const size_t src = ((size_t)bh * cap + row) * D + c4;
    store4(dk + dst, load4(dk_sm + src));
    store4(dv + dst, load4(dv_sm + src));
}

template <typename Kn>
cudaError_t set_smem(Kn kernel, size_t bytes) {
    return allow_smem(kernel, (int)bytes);
}

}  // namespace

// ------------------------------------------------------------------------------------------
// host launchers
// ------------------------------------------------------------------------------------------
cudaError_t launch_bgemm(bool ta, bool tb, int mask, BMat A, BMat B, BMat C, int m, int n, int k,
                         float alpha, bool accumulate, Shape s, cudaStream_t st) {
    const int NC = s.L / kC;
    if (m % 64 || n % 64 || k % 16) return cudaErrorInvalidValue;
    dim3 grid(n / 64, m / 64, s.B * s.H * NC);
#define NATSL_BG(TA, TB, MK) \
    bgemm_kernel<TA, TB, MK><<<grid, kThreads, 0, st>>>(A, B, C, k, alpha, accumulate ? 1 : 0, s.H, NC)
    if (!ta && !tb && mask == 0) NATSL_BG(false, false, 0);
    else if (!ta && tb && mask == 0) NATSL_BG(false, true, 0);
    else if (ta && !tb && mask == 0) NATSL_BG(true, false, 0);
    else if (!ta && tb && mask == 1) NATSL_BG(false, true, 1);
    else if (!ta && tb && mask == 2) NATSL_BG(false, true, 2);
    else return cudaErrorInvalidValue;
#undef NATSL_BG
    count_launch();
    return cudaGetLastError();
}

template <typename T>
static cudaError_t to_f32_impl(const void *a, const void *b, const void *c, float *a32, float *b32,
                               float *c32, size_t n, cudaStream_t st) {
    to_f32_kernel<T><<<1184, 256, 0, st>>>((const T *)a, (const T *)b, (const T *)c, a32, b32, c32,
                                           n / 4);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_to_f32(const void *a, const void *b, const void *c, float *a32, float *b32,
                          float *c32, size_t n, bool bf16, cudaStream_t st) {
    return bf16 ? to_f32_impl<__nv_bfloat16>(a, b, c, a32, b32, c32, n, st)
                : to_f32_impl<float>(a, b, c, a32, b32, c32, n, st);
}

template <typename T, int D>
static cudaError_t combine_bwd_impl(const float *o_la, const float *o_nla, const void *dout,
                                    const float *w, float eps, float *do_la, float *do_nla,
                                    float *dw, float *Dsm, void *do16, void *dola16, void *dolag16,
                                    const float *Gd, float scale_la, const int32_t *gsc, Shape s,
                                    cudaStream_t st, int G) {
    const size_t rows = (size_t)s.B * s.L * s.H;
    constexpr int kRowsPerBlock = (kThreads / 32) * (32 / (D / 8));
    combine_bwd_kernel<T, D><<<(unsigned)((rows + kRowsPerBlock - 1) / kRowsPerBlock), kThreads, 0, st>>>(
        o_la, o_nla, (const T *)dout, w, eps, do_la, do_nla, dw, Dsm, (__half *)do16, (__half *)dola16,
        (__half *)dolag16, Gd, scale_la, gsc, G, s.B, s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_dout_amax(const void *dout, size_t n, bool bf16, int32_t *status, cudaStream_t st) {
    const size_t n16 = n / (bf16 ? 8 : 4);
    const unsigned blocks = (unsigned)((n16 + 255) / 256 < 1184 ? (n16 + 255) / 256 : 1184);
    if (bf16) dout_amax_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>((const __nv_bfloat16 *)dout, n16, status);
    else dout_amax_kernel<float><<<blocks, 256, 0, st>>>((const float *)dout, n16, status);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_combine_bwd(const float *o_la, const float *o_nla, const void *dout,
                               const float *w, float eps, float *do_la, float *do_nla, float *dw,
                               float *Dsm, void *do16, void *dola16, void *dolag16, const float *Gd,
                               float scale_la, const int32_t *gsc, Shape s, cudaStream_t st, int G) {
    if (G < 1 || s.d % (32 * G) != 0) return cudaErrorInvalidValue;
    if (s.bf16) {
        if (s.d == 128) return combine_bwd_impl<__nv_bfloat16, 128>(o_la, o_nla, dout, w, eps, do_la, do_nla, dw, Dsm, do16, dola16, dolag16, Gd, scale_la, gsc, s, st, G);
        return combine_bwd_impl<__nv_bfloat16, 64>(o_la, o_nla, dout, w, eps, do_la, do_nla, dw, Dsm, do16, dola16, dolag16, Gd, scale_la, gsc, s, st, G);
    }
    if (s.d == 128) return combine_bwd_impl<float, 128>(o_la, o_nla, dout, w, eps, do_la, do_nla, dw, Dsm, do16, dola16, dolag16, Gd, scale_la, gsc, s, st, G);
    return combine_bwd_impl<float, 64>(o_la, o_nla, dout, w, eps, do_la, do_nla, dw, Dsm, do16, dola16, dolag16, Gd, scale_la, gsc, s, st, G);
}

template <int D, int G = 1>
static cudaError_t softmax_bwd_impl(const float *q32, const float *k_sm32, const float *v_sm32,
                                    int cap, const int32_t *sm_idx, const int32_t *pre,
                                    const float *do_nla, const float *lse, const float *Dsm,
                                    float scale_sm, float *dq_sm, float *dk_sm, float *dv_sm,
                                    float *dmask, Shape s, cudaStream_t st) {
    const size_t smem_q = sizeof(float) * (2 * kC * D + 2 * 32 * (D + 1) + 32);
    const size_t smem_k = sizeof(float) * (2 * 32 * (D + 1) + 2 * kC * D + 2 * kC * 33 + 2 * kC + 32);
    cudaError_t e = set_smem(softmax_bwd_dq_kernel<D, G>, smem_q);
    if (e != cudaSuccess) return e;
    e = set_smem(softmax_bwd_dkv_kernel<D, G>, smem_k);
    if (e != cudaSuccess) return e;
    dim3 gq(s.L / kC, s.B * s.H * G);
    softmax_bwd_dq_kernel<D, G><<<gq, kThreads, smem_q, st>>>(q32, k_sm32, v_sm32, cap, sm_idx, pre,
                                                           do_nla, lse, Dsm, scale_sm, dq_sm, s.L, s.H);
    count_launch();
    dim3 gk((cap + 31) / 32, s.B * s.H * G);
    softmax_bwd_dkv_kernel<D, G><<<gk, kThreads, smem_k, st>>>(q32, k_sm32, v_sm32, cap, sm_idx, pre,
                                                            do_nla, lse, Dsm, scale_sm, dk_sm, dv_sm,
                                                            dmask, s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_softmax_bwd(const float *q32, const float *k_sm32, const float *v_sm32, int cap,
                               const int32_t *sm_idx, const int32_t *sm_chunk_prefix,
                               const float *do_nla, const float *lse, const float *Dsm,
                               float scale_sm, float *dq_sm, float *dk_sm, float *dv_sm, Shape s,
                               cudaStream_t st, float *dmask, int G) {
    if (G > 1) {      // grouped softmax heads: slices of 32 or 64 columns
#define NATSL_GROUPED(DS, GG)                                                                                 \
        if (s.d == DS * GG && G == GG)                                                                        \
            return softmax_bwd_impl<DS, GG>(q32, k_sm32, v_sm32, cap, sm_idx, sm_chunk_prefix, do_nla, lse, Dsm, \
                                            scale_sm, dq_sm, dk_sm, dv_sm, dmask, s, st)
        NATSL_GROUPED(32, 2);
        NATSL_GROUPED(64, 2);
        NATSL_GROUPED(32, 4);
#undef NATSL_GROUPED
        return cudaErrorInvalidValue;
    }
    if (s.d == 128) return softmax_bwd_impl<128>(q32, k_sm32, v_sm32, cap, sm_idx, sm_chunk_prefix, do_nla, lse, Dsm, scale_sm, dq_sm, dk_sm, dv_sm, dmask, s, st);
    return softmax_bwd_impl<64>(q32, k_sm32, v_sm32, cap, sm_idx, sm_chunk_prefix, do_nla, lse, Dsm, scale_sm, dq_sm, dk_sm, dv_sm, dmask, s, st);
}

template <int D, int G = 1>
static cudaError_t own_block_impl(const float *q32, const float *k32, const float *v32, const float *do_nla,
                                  const float *lse, const float *Dsm, const uint8_t *route, float scale_sm,
                                  float *dq_sm, float *dk_x, float *dv_x, const int32_t *gsc, Shape s,
                                  cudaStream_t st) {
    const size_t smem = sizeof(float) * (4 * kC * (D + 1) + 2 * kC * (kC + 1));
    cudaError_t e = set_smem(softmax_bwd_own_block_simt_kernel<D, G>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(s.L / kC, s.B * s.H * G);
    softmax_bwd_own_block_simt_kernel<D, G><<<grid, kThreads, smem, st>>>(q32, k32, v32, do_nla, lse, Dsm, route,
                                                                      scale_sm, dq_sm, dk_x, dv_x, gsc, s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_softmax_bwd_own_block_simt(const float *q32, const float *k32, const float *v32,
                                              const float *do_nla, const float *lse, const float *Dsm,
                                              const uint8_t *route, float scale_sm, float *dq_sm,
                                              float *dk_x, float *dv_x, const int32_t *gsc, Shape s,
                                              cudaStream_t st, int G) {
    if (G > 1) {
#define NATSL_GROUPED(DS, GG)                                                                               \
        if (s.d == DS * GG && G == GG)                                                                      \
            return own_block_impl<DS, GG>(q32, k32, v32, do_nla, lse, Dsm, route, scale_sm, dq_sm, dk_x, dv_x, \
                                          gsc, s, st)
        NATSL_GROUPED(32, 2);
        NATSL_GROUPED(64, 2);
        NATSL_GROUPED(32, 4);
#undef NATSL_GROUPED
        return cudaErrorInvalidValue;
    }
    if (s.d == 128) return own_block_impl<128>(q32, k32, v32, do_nla, lse, Dsm, route, scale_sm, dq_sm, dk_x, dv_x, gsc, s, st);
    return own_block_impl<64>(q32, k32, v32, do_nla, lse, Dsm, route, scale_sm, dq_sm, dk_x, dv_x, gsc, s, st);
}

template <int D>
static cudaError_t rscan_impl(const float *q32, const float *k32, const float *Gcum, const float *W,
                              const float *P, const float *do_la, const float *chunk_states,
                              float scale_la, float *dUt, float *dS_c, float *gS,
                              const float *dstate_out, float *dstate_in, const uint8_t *block_route, Shape s,
                              cudaStream_t st) {
    const size_t smem = sizeof(float) * (D * kDvs + 3 * kC * (D + 1) + kC * (kC + 1) +
                                         2 * kC * (kDvs + 1) + kC + 8);
    cudaError_t e = set_smem(gdn_rscan_kernel<D>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(D / kDvs, s.B * s.H);
    gdn_rscan_kernel<D><<<grid, kThreads, smem, st>>>(q32, k32, Gcum, W, P, do_la, chunk_states,
                                                      scale_la, dUt, dS_c, gS, dstate_out, dstate_in, block_route,
                                                      s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_gdn_rscan(const float *q32, const float *k32, const float *Gcum, const float *W,
                             const float *P, const float *do_la, const float *chunk_states,
                             float scale_la, float *dUt, float *dS_c, float *gS,
                             const float *dstate_out, float *dstate_in, Shape s, cudaStream_t st,
                             const uint8_t *block_route) {
    if (s.d == 128)
        return rscan_impl<128>(q32, k32, Gcum, W, P, do_la, chunk_states, scale_la, dUt, dS_c, gS, dstate_out, dstate_in, block_route, s, st);
    return rscan_impl<64>(q32, k32, Gcum, W, P, do_la, chunk_states, scale_la, dUt, dS_c, gS, dstate_out, dstate_in, block_route, s, st);
}

cudaError_t launch_gdn_tsolve(const float *Abar, const float *beta, const uint8_t *route,
                              const float *dW, const float *dUt, float *dKb, float *dVb, Shape s,
                              cudaStream_t st) {
    dim3 grid(s.L / kC, s.B * s.H);
    if (s.d == 128)
        gdn_tsolve_kernel<128><<<grid, kThreads, 0, st>>>(Abar, beta, route, dW, dUt, dKb, dVb, s.L, s.H);
    else
        gdn_tsolve_kernel<64><<<grid, kThreads, 0, st>>>(Abar, beta, route, dW, dUt, dKb, dVb, s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_mask_scale(const float *M, const float *N, const float *Gcum, const float *beta,
                              const uint8_t *route, float scale_la, float *Mg, float *Ms, float *Ns,
                              Shape s, cudaStream_t st) {
    dim3 grid(s.L / kC, s.B * s.H);
    mask_scale_kernel<<<grid, kThreads, 0, st>>>(M, N, Gcum, beta, route, scale_la, Mg, Ms, Ns, s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

template <typename T, int D>
static cudaError_t scatter_impl(const AssembleArgs &a, void *dk, void *dv, Shape s, cudaStream_t st) {
    constexpr int kRows = kThreads / (D / 4);
    dim3 grid((a.cap + kRows - 1) / kRows, s.B * s.H);
    scatter_sm_kernel<T, D><<<grid, kThreads, 0, st>>>(a.dk_sm, a.dv_sm, a.cap, a.sm_idx, a.sm_prefix,
                                                       (T *)dk, (T *)dv, s.L, s.H);
    count_launch();
    return cudaGetLastError();
}

template <typename T, int D>
static cudaError_t assemble_impl(const AssembleArgs &a, void *dq, void *dk, void *dv, Shape s,
                                 cudaStream_t st) {
    const size_t rows = (size_t)s.B * s.L * s.H;
    gdn_assemble_kernel<T, D><<<(unsigned)((rows + 7) / 8), kThreads, 0, st>>>(
        a.q32, a.k32, a.v32, a.Gcum, a.beta, a.route, a.dQg, a.dKb, a.dVb, a.dKt, a.X1p, a.X2, a.X3,
        a.X4, a.dq_sm, a.dk_x, a.dv_x, a.scale_la, (T *)dq, (T *)dk, (T *)dv, a.dGrow, a.kappa, a.dbeta, s.B,
        s.L, s.H);
    count_launch();
    const int NC = s.L / kC;
    const size_t nch = (size_t)s.B * s.H * NC;
    dg_kernel<<<(unsigned)((nch + 127) / 128), 128, 0, st>>>(a.dGrow, a.kappa, a.gS, a.Gcum,
                                                            s.d / kDvs, a.dg, s.B, s.L, s.H);
    count_launch();
    if (a.no_scatter) return cudaGetLastError();   // (the retained tokens' gradients came in through dk_x, dv_x)
    return scatter_impl<T, D>(a, dk, dv, s, st);
}

cudaError_t launch_scatter_sm(const AssembleArgs &a, void *dk, void *dv, Shape s, cudaStream_t st) {
    if (s.bf16) {
        if (s.d == 128) return scatter_impl<__nv_bfloat16, 128>(a, dk, dv, s, st);
        return scatter_impl<__nv_bfloat16, 64>(a, dk, dv, s, st);
    }
    if (s.d == 128) return scatter_impl<float, 128>(a, dk, dv, s, st);
    return scatter_impl<float, 64>(a, dk, dv, s, st);
}

cudaError_t launch_gdn_assemble(const AssembleArgs &a, void *dq, void *dk, void *dv, Shape s,
                                cudaStream_t st) {
    if (s.bf16) {
        if (s.d == 128) return assemble_impl<__nv_bfloat16, 128>(a, dq, dk, dv, s, st);
        return assemble_impl<__nv_bfloat16, 64>(a, dq, dk, dv, s, st);
    }
    if (s.d == 128) return assemble_impl<float, 128>(a, dq, dk, dv, s, st);
    return assemble_impl<float, 64>(a, dq, dk, dv, s, st);
}

}  // namespace natsl
