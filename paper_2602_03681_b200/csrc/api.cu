// C ABI of the library: argument validation, workspace carving and kernel sequencing.
// Nothing here allocates, synchronises (except natsl_device_status) or touches the CPU oracle.
#include <cstring>

#include "natsl_internal.h"

#include <algorithm>
#include <atomic>
#include <mutex>

using namespace natsl;

namespace natsl {
// Test hooks (natsl_debug_set_wait_limit): a bound for the device-side waits of the following
// launches, and whether the scan withholds the per-chunk flags the softmax kernel waits for.
static std::atomic<uint32_t> g_debug_wait_kcycles{0};
static std::atomic<int> g_debug_withhold_flags{0};
int debug_wait_kcycles() { return (int)g_debug_wait_kcycles.load(std::memory_order_relaxed); }
static std::atomic<uint64_t> g_launches{0};
void count_launch(int n) { g_launches.fetch_add((uint64_t)n, std::memory_order_relaxed); }
}  // namespace natsl

namespace {

constexpr size_t kAlign = 256;
constexpr size_t kStatusBytes = 256;

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }
bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

struct Carver {
    char *base;
    size_t off = 0;
    explicit Carver(void *b) : base(static_cast<char *>(b)) {}
    template <typename T> T *take(size_t n) {
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += align_up(n * sizeof(T));
        return p;
    }
};

int check_params(const natsl_params *p, bool needs_L) {
    if (!p) return NATSL_ERR_NULL;
    if (p->dtype != NATSL_F32 && p->dtype != NATSL_BF16) return NATSL_ERR_DTYPE;
    if (p->B <= 0 || p->H <= 0) return NATSL_ERR_SHAPE;
    if (p->d != 64 && p->d != 128) return NATSL_ERR_SHAPE;
    if (p->C != kC) return NATSL_ERR_SHAPE;
    if (needs_L && (p->L <= 0 || p->L % p->C != 0)) return NATSL_ERR_SHAPE;
    if (!(p->eps > 0.f)) return NATSL_ERR_SHAPE;
    if (p->G < 0 || (p->G > 1 && p->d % p->G != 0)) return NATSL_ERR_SHAPE;
    if ((p->flags & NATSL_QK_NORM) && !(p->norm_eps >= 0.f)) return NATSL_ERR_SHAPE;
    return NATSL_OK;
}

// Grouped softmax heads / per-operation q, k normalisation (Section 4.3): what the forward supports.
bool grouped_or_normed(const natsl_params *p) { return p->G > 1 || (p->flags & NATSL_QK_NORM); }
HeadGroups head_groups(const natsl_params *p) {
    HeadGroups hg;
    hg.G = p->G > 1 ? p->G : 1;
    hg.norm_eps = (p->flags & NATSL_QK_NORM) ? p->norm_eps : -1.f;
    return hg;
}

Shape shape_of(const natsl_params *p) { return Shape{p->B, p->H, p->L, p->d, p->dtype == NATSL_BF16}; }

struct FwdWs {
    int32_t *status, *emit_flags, *sm_idx, *prefix;
    void *k_sm, *v_sm, *v16;
    void *kn16;                 // prefill in pieces with NATSL_QK_NORM: normalised fp16 keys of the whole cache
    void *o_la16;               // tensor-core path: the linear read-out as fp16 [B,L,H,d]
    float *W, *U, *P, *o_la;    // fp32 CUDA-core path only
    float *q_la, *k_la, *q_sm, *k_nsm;   // fp32 storage with NATSL_QK_NORM: normalised copies of q and k
    GdnTcWs tc;                 // tensor-core path only
    float *seg_incr, *seg_trans, *seg_start;   // segmented scan: [B*H, nseg, d, d] each
    size_t bytes;
};

bool use_tensor_cores(const natsl_params *p) {
    return p->dtype == NATSL_BF16 && !(p->flags & NATSL_FORCE_SIMT);
}

// Whether the scan is a programmatic dependent of the kernels before it too, which saves the gap of a launch.  Its CTAs, one
// to a multiprocessor, are then placed in the order in which the prepare kernel's drain, i.e. crowded into a few GPCs,
// whose share of the L2 bandwidth the scans fight for (60 of them behind several waves: 310-370 us instead of 128).  So:
// one CTA per pair only while most multiprocessors have no second prepare CTA; several segments, which take every
// multiprocessor anyway, behind up to about one wave.  Without -> with, us a call: one CTA per pair, 128 chunks 34.5 -> 33.0,
// 160 38.5 -> 36.3, 224 34.8 -> 34.4, 240 47.2 -> 48.2, 450 47.7 -> 55.1, 512 51.2 -> 63.0; segments, 256 chunks 53.1 -> 49.8,
// 512 67.7 -> 69.1, 576 88.9 -> 85.9, 640 123.6 -> 117.6, 1024 108.9 -> 113.3 and 129.9 -> 137.1.
bool scan_follows_closely(const natsl_params *p, bool segmented) {
    return (long long)p->B * p->H * (p->L / kC) <= (segmented ? 4 * 148 : 160);
}

// Segments of the forward scan (tensor-core path).  A (batch, head) costs one CTA per SM for as long as its chain of
// chunks, so with few of them most of the GPU waits.  Up to a number of pairs a first pass over the segments (1.6 us per chunk
// against 1.8 with outputs) gains more than it costs: there are as many segments as keep its 2 nseg - 3 runs per pair
// in one wave, at least 4 chunks long (shorter ones gain less than their step of the chain), and at least three --
// with two the two passes are as long as one over everything.  22 pairs: 4 segments, 16: 6, 4: 20.
// Where the line lies: three segments would fit one wave up to 49 pairs, but the softmax kernel, which runs beside the pass
// with outputs, then starts a pass later, and the more it has to do the fewer pairs pay for that: own-block tiles, two softmax
// heads, many softmax tokens (whose share is not known here), and short sequences, whose passes do not hide the launches.  Time with
// segments against one pass over everything, 2048 to 16384 tokens, 5 to 40 % softmax tokens: 128 columns 16 pairs 0.82 to 0.92, 18
// pairs 0.72 to 0.99, 22 pairs 0.84 to 1.17, 24 pairs 0.85 to 1.14, 32 pairs 1.12 to 1.15; 64 columns 24 pairs 0.86, 28 pairs 0.91 to
// 1.06, 32 pairs 0.96 to 1.18, 36 pairs 1.08.  From 4096 tokens on, at 5, 10, 20, 40 %, in the order 4096 | 8192 | 16384 tokens:
//   128 columns          23 pairs 0.86 0.88 0.93 1.02 | 0.81 0.83 0.90 1.06 | 0.79 0.84 0.95 1.07
//                        26 pairs 0.91 0.95 1.02 1.12 | 0.89 0.93 1.05 1.12 | 0.88 0.97 1.02 1.11
//   own-block tiles      18 pairs 0.85 0.88 0.95 1.06 | 0.80 0.84 0.92 1.06 | 0.80 0.88 0.98 1.10
//                        20 pairs 0.93 0.95 1.01 1.13 | 0.87 0.92 1.02 1.10 | 0.86 0.94 1.06 1.12
//   two softmax heads    16 pairs 0.79 0.85 0.96 1.15 | 0.73 0.83 1.00 1.09 | 0.75 0.92 1.06 1.09
//                        20 pairs 0.94 1.00 1.12 1.22 | 0.86 0.96 1.09 1.13 | 0.89 1.03 1.10 1.07
//   both, normalised     15 pairs 0.86 0.91 0.99 1.14 | 0.79 0.86 1.01 1.08 | 0.80 0.92 1.04 1.07
//                        18 pairs 0.92 0.97 1.08 1.13 | 0.92 0.98 1.06 1.11 | 0.95 1.03 1.07 1.06
//   64 col., own-block   20 pairs 0.83 0.86 0.96 1.15 | 0.77 0.83 0.97 1.08 | 0.78 0.91 1.02 1.06
//                        24 pairs 0.91 0.97 1.08 1.13 | 0.85 0.94 1.04 1.08 | 0.89 1.01 1.08 1.07
// (One pass -> segments, us, 8192 tokens, 5 %: own-block tiles 15 pairs 265 -> 186, two softmax heads 15 pairs 255 -> 181, 64 columns
// with own-block tiles 20 pairs 228 -> 175, 23 pairs 296 -> 237; own-block tiles 15 pairs of 16384 tokens 502 -> 344.)
// At 2048 tokens: own-block tiles 15 pairs 0.92 to 1.00, 18 pairs 0.98 to 1.06; two softmax heads 14 pairs 0.91 to 1.07, 16 pairs 0.94 to
// 1.14; both 14 pairs 0.93 to 1.10, 16 pairs 0.98 to 1.18; 64 columns with own-block tiles 18 pairs 0.90 to 1.16, 20 pairs 0.91 to 1.14.
// Shorter sequences keep the lower lines for another reason too: segments need scratch, and calls of 15 to 18 pairs of 1024
// tokens that fit natsl_hybrid_fwd_static's array (23 to 27 of 32 MiB) would not any more; of 4096 tokens none fits it anyway.
int segment_pairs(const natsl_params *p) {
    const bool own = p->flags & NATSL_BLOCK_ROUTING, lng = p->L >= 4096;
    if (p->d == 64) return !own && p->G <= 1 ? 30 : own && lng ? 20 : 18;
    if (p->G > 1) return !lng ? 14 : own ? 15 : 16;
    if (own) return lng ? 18 : 14;
    return lng ? 23 : 22;
}
// The two passes must save 8 chunks of the chain, which is what two more launches and the chaining take.
// The last segment takes what remains, up to twice as much: the first pass does not run it, and in the second the
// softmax kernel fills the other multiprocessors.  *chunks: of the others, even, so that they are whole query tiles.
int scan_segments(const natsl_params *p, int *chunks = nullptr) {
    if (!use_tensor_cores(p) || (p->flags & NATSL_SINGLE_PASS_SCAN)) return 1;
    const int NC = p->L / kC, BH = p->B * p->H;
    if (BH > segment_pairs(p) || NC < 16) return 1;
    const int most = std::min((148 / BH + 3) / 2, 32);
    const int n = std::max(4, ((NC + most) / (most + 1) + 1) & ~1);
    if (chunks) *chunks = n;
    const int nseg = std::min(most, NC / n);
    const int last = NC - (nseg - 1) * n;      // (three quarters: the first pass's chunks against the second's)
    return nseg >= 3 && 4 * (NC - last) - 3 * n >= 32 ? nseg : 1;
}

FwdWs carve_fwd(const natsl_params *p, void *ws) {
    Carver c(ws);
    FwdWs f;
    const size_t B = p->B, H = p->H, L = p->L, d = p->d, NC = L / kC;
    const size_t esz = p->dtype == NATSL_BF16 ? 2 : 4;
    f.status = c.take<int32_t>(kStatusBytes / 4);
    // one counter per chunk, raised by the scan as the chunk's read-out is complete (tensor-core path)
    f.emit_flags = c.take<int32_t>(use_tensor_cores(p) ? B * H * NC : 0);
    f.sm_idx = c.take<int32_t>(B * H * L);
    f.prefix = c.take<int32_t>(B * H * (NC + 1));
    f.k_sm = c.take<char>(B * H * L * d * esz);
    f.v_sm = c.take<char>(B * H * L * d * esz);
    if (use_tensor_cores(p)) {
        // fp16 V of the retained tokens; when the call appends to a cache, of the whole cache
        const size_t capv = (p->flags & NATSL_APPEND_CACHE) && p->sm_cap > 0 ? (size_t)p->sm_cap : L;
        f.v16 = c.take<char>(B * H * capv * d * 2);
        f.kn16 = c.take<char>((p->flags & NATSL_APPEND_CACHE) && (p->flags & NATSL_QK_NORM) ? B * H * capv * d * 2 : 0);
        f.tc.Qh = f.tc.Kh = nullptr;
        f.tc.Wt = c.take<char>(B * H * L * d * 2);
        f.tc.Tb = c.take<char>(B * H * NC * kC * kC * 2);
        f.tc.Ph = c.take<char>(B * H * NC * kC * kC * 2);
        f.tc.Gd = c.take<float>(B * H * L * 2);
        f.tc.Rn = c.take<float>((p->flags & NATSL_QK_NORM) ? B * H * L * 2 : 0);
        f.W = f.U = f.P = nullptr;
        const size_t nseg = scan_segments(p), segf = nseg > 1 ? B * H * nseg * d * d : 0;
        f.seg_incr = c.take<float>(segf);
        f.seg_trans = c.take<float>(segf);
        f.seg_start = c.take<float>(segf);
        f.o_la16 = c.take<char>(B * L * H * d * 2);
        f.o_la = nullptr;
    } else {
        f.v16 = nullptr;
        f.kn16 = nullptr;
        f.o_la16 = nullptr;
        f.tc = GdnTcWs{};
        f.seg_incr = f.seg_trans = f.seg_start = nullptr;
        f.W = c.take<float>(B * L * H * d);
        f.U = c.take<float>(B * L * H * d);
        f.P = c.take<float>(B * H * NC * kC * kC);
        f.o_la = c.take<float>(B * L * H * d);
    }
    const size_t nrm = !use_tensor_cores(p) && (p->flags & NATSL_QK_NORM) ? B * L * H * d : 0;
    f.q_la = c.take<float>(nrm);
    f.k_la = c.take<float>(nrm);
    f.q_sm = c.take<float>(nrm);
    f.k_nsm = c.take<float>(nrm);
    f.bytes = c.off;
    return f;
}

struct BwdWs {
    int32_t *status, *emit_flags, *sm_idx, *prefix, *lin_idx, *n_lin, *sm_len;
    size_t head_bytes;                                       // status page + emit_flags: cleared per forward
    float *o_la, *o_nla, *lse, *Dsm, *Gcum;                  // branch outputs, row sums, cumulative decays
    float *dq_sm, *dk_sm, *dv_sm;                            // softmax branch: dq token-major, dk, dv compacted
    float *dk_x, *dv_x, *dmask;                              // block-level routing: the softmax branch's dk, dv of every
                                                             // token (token-major), mask gradients per retained key
    // fp32 CUDA-core path
    float *k_sm32, *v_sm32;                                  // [B,H,L,d] compacted, fp32
    float *q32, *k32, *v32;                                  // token-major fp32 copies
    float *qs32, *ks32;                                      // NATSL_QK_NORM: RMS-normalised q, k (q32, k32 then hold the
                                                             // L2-normalised ones)
    float *W, *U, *Ut, *do_la, *do_nla;                      // token-major
    float *dUt, *dQg, *dW, *dKt, *dKb, *dVb, *X1p, *X2, *X3, *X4;
    float *P, *Abar, *M, *N, *Mg, *Ms, *Ns;                  // [B,H,NC,64,64]
    float *S_c, *dS_c;                                       // [B,H,NC,d,d]
    float *dGrow, *kappa, *gS;                               // [B,H,L] (gS: [B,H,NC,d/32])
    // tensor-core path
    void *k_smb, *k16, *v16, *Qh, *dO16;                     // softmax branch: 16-bit [B,H,L,d]
    void *o_la16;                                            // linear read-out as fp16 [B,L,H,d]
    GdnTcWs tc;                                              // the forward's chunkwise intermediates
    GdnTcExport ex;                                          // ... and what it keeps for the backward
    GdnTcGrads gr;                                           // fp16 gradient operands of the linear branch
    float *kap_c;                                            // [B,H,NC]
    float *dq32, *dk32, *dv32;                               // NATSL_QK_NORM: gradients before the normalisations' backward
    size_t bytes;
};

// Only what the selected path uses is carved (a buffer the path does not touch gets no bytes and a
// pointer nobody dereferences).  Buffers with disjoint lifetimes share their bytes on the tensor-core path:
// o_nla (dead once the combination's backward has run) / dq_sm, o_la / dq32, and the fp16 o_la / the
// fp16 gradient copy dO16.
BwdWs carve_bwd(const natsl_params *p, void *ws) {
    Carver c(ws);
    BwdWs f;
    const size_t B = p->B, H = p->H, L = p->L, d = p->d, NC = L / kC;
    const size_t TM = B * L * H * d, CC = B * H * NC * kC * kC, ST = B * H * NC * d * d, BHL = B * H * L;
    const bool tcs = use_tensor_cores(p), simt = !tcs;
    const bool block = (p->flags & NATSL_BLOCK_ROUTING) != 0, normed = (p->flags & NATSL_QK_NORM) != 0;
    const size_t Gg = p->G > 1 ? (size_t)p->G : 1;           // softmax heads per linear head: lse, Dsm per softmax head
    auto tm = [&](bool need) { return c.take<float>(need ? TM : 0); };
    auto cc = [&](bool need) { return c.take<float>(need ? CC : 0); };
    auto half = [&](bool need, size_t n) { return static_cast<void *>(c.take<char>(need ? n * 2 : 0)); };
    f.status = c.take<int32_t>(kStatusBytes / 4);
    f.emit_flags = c.take<int32_t>(tcs ? B * H * NC : 0);    // per-chunk counters of the scan (forward part)
    f.head_bytes = c.off;
    f.sm_idx = c.take<int32_t>(BHL);
    f.prefix = c.take<int32_t>(B * H * (NC + 1));
    f.lin_idx = c.take<int32_t>(simt ? BHL : 0);
    f.n_lin = c.take<int32_t>(simt ? B * H * NC : 0);
    f.sm_len = c.take<int32_t>(simt ? B * H : 0);
    f.o_la = tm(true);
    f.o_nla = tm(true);
    f.lse = c.take<float>(BHL * Gg);
    f.Dsm = c.take<float>(BHL * Gg);
    f.Gcum = c.take<float>(BHL);
    f.dq_sm = tcs ? f.o_nla : tm(true);
    f.dk_sm = tm(true); f.dv_sm = tm(true);
    f.dk_x = tm(block); f.dv_x = tm(block);
    f.dmask = c.take<float>(block ? BHL * Gg : 0);
    // fp32 CUDA-core path
    f.k_sm32 = tm(simt); f.v_sm32 = tm(simt);
    f.q32 = tm(simt); f.k32 = tm(simt); f.v32 = tm(simt);
    f.qs32 = tm(simt && normed); f.ks32 = tm(simt && normed);
    f.W = tm(simt); f.U = tm(simt); f.Ut = tm(simt); f.do_la = tm(simt); f.do_nla = tm(simt);
    f.dUt = tm(simt); f.dQg = tm(simt); f.dW = tm(simt); f.dKt = tm(simt); f.dKb = tm(simt); f.dVb = tm(simt);
    f.X1p = tm(simt); f.X2 = tm(simt); f.X3 = tm(simt); f.X4 = tm(simt);
    f.P = cc(simt); f.Abar = cc(simt); f.M = cc(simt); f.N = cc(simt); f.Mg = cc(simt); f.Ms = cc(simt); f.Ns = cc(simt);
    f.S_c = c.take<float>(simt ? ST : 0);
    f.dS_c = c.take<float>(simt ? ST : 0);
    f.dGrow = c.take<float>(simt ? BHL : 0);
    f.kappa = c.take<float>(simt ? BHL : 0);
    f.gS = c.take<float>(simt ? B * H * NC * (d / 32) : 0);
    // tensor-core path
    f.k_smb = half(tcs, TM); f.k16 = half(tcs, TM); f.v16 = half(tcs, TM); f.Qh = half(tcs, TM);
    f.dO16 = half(tcs, TM);
    f.o_la16 = f.dO16;
    f.gr.dO16 = half(tcs, TM); f.gr.dOg16 = half(tcs, TM); f.gr.dU16 = half(tcs, TM); f.gr.dS16 = half(tcs, ST);
    f.tc = GdnTcWs{};
    f.tc.Qh = f.Qh;                           // without the normalisation the same fp16 copy of q serves both branches
    f.tc.Kh = half(tcs, TM);
    f.tc.Wt = half(tcs, TM);
    f.tc.Tb = half(tcs, CC);
    f.tc.Ph = half(tcs, CC);
    f.tc.Gd = c.take<float>(tcs ? BHL * 2 : 0);
    f.tc.Rn = c.take<float>(tcs && normed ? BHL * 2 : 0);
    f.ex = GdnTcExport{};
    f.ex.U16 = half(tcs, TM); f.ex.T16 = half(tcs, CC); f.ex.S16 = half(tcs, ST); f.ex.Ut16 = half(tcs, TM);
    f.ex.Gcum = f.Gcum;
    f.kap_c = c.take<float>(tcs && block ? B * H * NC : 0);
    f.dq32 = f.o_la;
    f.dk32 = tm(tcs && normed && !block); f.dv32 = tm(tcs && normed && !block);
    f.bytes = c.off;
    return f;
}

}  // namespace

namespace {

// In the backward the linear branch's reverse scan and the key-side softmax kernel do not depend on the query-side
// one, so they run beside it: on a library-owned stream per device, forked from the caller's stream with one event and joined back
// with another before the results meet.  Stream and events are created on first use and kept;
// a mutex covers the enqueue of a call, since the two event objects are shared by all calls.
struct SideStream {
    cudaStream_t st = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    bool tried = false;
};
SideStream g_side[64];
std::mutex g_side_mu;

// Joins the side stream back into the caller's stream when a call leaves early after the fork,
// so that no library-owned stream is left with work the caller's stream does not wait for.
struct SideJoin {
    SideStream *side = nullptr;
    cudaStream_t st = nullptr;
    bool pending = false;
    void forked(SideStream *s, cudaStream_t caller) { side = s; st = caller; pending = true; }
    cudaError_t join() {
        if (!pending) return cudaSuccess;
        pending = false;
        cudaError_t e = cudaEventRecord(side->join, side->st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, side->join, 0);
        return e;
    }
    ~SideJoin() { (void)join(); }
};


SideStream *side_stream_locked() {   // g_side_mu held; nullptr: run everything on the caller's stream
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    SideStream &s = g_side[dev];
    if (!s.tried) {
        s.tried = true;
        if (cudaStreamCreateWithFlags(&s.st, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&s.fork, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&s.join, cudaEventDisableTiming) != cudaSuccess) {
            s.st = nullptr;
            (void)cudaGetLastError();
        }
    }
    return s.st ? &s : nullptr;
}

}  // namespace

// The forward as the backward needs it: the same kernels as natsl_hybrid_fwd's, which here also leave
// the chunkwise quantities the gradient kernels read (chunk-entry states, U~, (I + A)^-1, cumulative
// decays, log-sum-exp, raw branch outputs) in the backward workspace `f`.  natsl_hybrid_bwd runs it
// itself unless the caller did, through natsl_hybrid_fwd with NATSL_SAVE_FOR_BWD (then `out` and
// `state_out` are produced as well).
static int bwd_forward_part(const void *q, const void *k, const void *v, const float *g,
                            const float *beta, const uint8_t *route, void *out, float *state_out,
                            const natsl_params *p, const BwdWs &f, cudaStream_t st) {
    const Shape s = shape_of(p);
    Shape s32 = s;              // the same shapes with fp32 storage (the fp32 copies)
    s32.bf16 = false;
    const long long B = p->B, H = p->H, L = p->L, d = p->d;
    const bool block = (p->flags & NATSL_BLOCK_ROUTING) != 0;
    const uint8_t *block_route = block ? route : nullptr;
    const bool tensor_cores = use_tensor_cores(p);
    int32_t *flags = tensor_cores && !(p->flags & NATSL_SINGLE_STREAM) ? f.emit_flags : nullptr;
#define NATSL_TRY(call) do { if ((call) != cudaSuccess) return NATSL_ERR_CUDA; } while (0)
    const HeadGroups hg = head_groups(p);
    if (tensor_cores) {
        // (the kernels of natsl_hybrid_fwd, overlapped like there)
        const bool pdl = !(p->flags & NATSL_SINGLE_STREAM);
        NATSL_TRY(launch_gdn_prepare_tc(q, k, v, g, beta, block ? nullptr : route, p->scale_la, f.tc, f.ex,
                                        f.status, s, st, (int)(kStatusBytes / 4), hg.norm_eps, pdl));
        NATSL_TRY(launch_route_gather_tc(k, v, route, f.sm_idx, f.prefix, nullptr, f.k_smb, nullptr, f.v16, f.k16, p->L,
                                         p->L, f.emit_flags, s, st, pdl, hg));
        NATSL_TRY(launch_gdn_scan_tc(q, k, v, f.tc, p->scale_la, p->state_in, state_out, ScanOut{f.o_la16, f.o_la, flags},
                                     f.ex, ScanSegments{0, 1, 0, nullptr, nullptr, nullptr}, block_route,
                                     f.status, s, st, pdl && scan_follows_closely(p, false), hg.norm_eps >= 0.f));
        NATSL_TRY(launch_softmax_combine_tc(q, f.k_smb, f.v16, p->L, p->L, f.sm_idx, f.prefix, f.o_la16,
                                            flags, p->w, p->scale_sm, p->eps, out, f.o_nla, f.lse, nullptr, p->L,
                                            BlockRouting{block_route, k, v}, false, f.status, s, st, hg));
        return NATSL_OK;
    }
    NATSL_TRY(cudaMemsetAsync(f.status, 0, f.head_bytes, st));
    NATSL_TRY(launch_route_compact(route, f.sm_idx, f.prefix, f.lin_idx, f.n_lin, f.sm_len, nullptr,
                                   block ? f.status : nullptr, p->L, p->B, p->L, p->H, st));
    // fp32 copies of the inputs; with NATSL_QK_NORM q32, k32 become the L2-normalised rows (everything of the linear
    // branch reads those), qs32, ks32 the slice-wise RMS-normalised ones (softmax branch)
    const float *qs = f.q32, *ks = f.k32;
    const bool qk = hg.norm_eps < 0.f;
    NATSL_TRY(launch_to_f32(qk ? q : nullptr, qk ? k : nullptr, v, f.q32, f.k32, f.v32,
                            (size_t)(B * L * H * d), s.bf16, st));
    if (!qk) {
        NATSL_TRY(launch_qk_norm_f32((const float *)q, (const float *)k, f.q32, f.k32, f.qs32, f.ks32, (size_t)(B * L * H), p->d, hg.G,
                                     hg.norm_eps, st));
        qs = f.qs32; ks = f.ks32;
    }
    NATSL_TRY(launch_gather_kv(ks, f.v32, f.sm_idx, f.prefix, f.k_sm32, f.v_sm32, p->L, f.status, s32, st));
    NATSL_TRY(launch_gdn_prepare_simt(f.q32, f.k32, f.v32, g, beta, block ? nullptr : route, p->scale_la,
                                      f.W, f.U, f.P, f.Abar, f.Gcum, s32, st));
    NATSL_TRY(launch_gdn_scan_simt(f.q32, f.k32, g, f.W, f.U, f.P, p->scale_la, p->state_in, state_out,
                                   f.S_c, f.Ut, f.o_la, block_route, s32, st));
    NATSL_TRY(launch_softmax_combine_simt(qs, f.k_sm32, f.v_sm32, p->L, f.sm_idx, f.prefix,
                                          f.o_la, p->w, p->scale_sm, p->eps, out, f.o_nla,
                                          f.lse, BlockRouting{block_route, ks, f.v32}, s32, st, hg.G));
#undef NATSL_TRY
    return NATSL_OK;
}

extern "C" {

uint64_t natsl_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char *natsl_stage_name(int op, int i) {
    static const char *fwd[] = {"route_compact+gather_kv", "gdn_prepare", "gdn_scan",
                                "softmax_combine"};
    if (op == NATSL_OP_FWD && i >= 0 && i < 4) return fwd[i];
    if (op == NATSL_OP_DECODE && i == 0) return "decode_step";
    return nullptr;
}

const char *natsl_strerror(int status) {
    switch (status) {
        case NATSL_OK: return "ok";
        case NATSL_ERR_NULL: return "a required pointer is NULL";
        case NATSL_ERR_SHAPE: return "unsupported shape (need B,H,L>0, L%64==0, d in {64,128}, C==64, eps>0)";
        case NATSL_ERR_DTYPE: return "dtype must be NATSL_F32 or NATSL_BF16";
        case NATSL_ERR_ALIGN: return "tensor base pointer not 16-byte aligned";
        case NATSL_ERR_WORKSPACE: return "workspace missing or too small";
        case NATSL_ERR_CUDA: return "CUDA launch or runtime error";
        case NATSL_ERR_CACHE_FULL: return "retained-KV cache full";
        case NATSL_ERR_UNSUPPORTED: return "request not implemented in this build";
        case NATSL_ERR_ROUTE: return "block-level routing: route changes inside a block";
        case NATSL_ERR_TIMEOUT: return "a bounded device-side wait expired";
        case NATSL_ERR_TOO_LARGE: return "problem needs more scratch than the library's built-in array (NATSL_STATIC_WS_BYTES)";
        default: return "unknown natsl status";
    }
}

int natsl_workspace_size(const natsl_params *p, int op, size_t *bytes) {
    if (!bytes) return NATSL_ERR_NULL;
    int rc = check_params(p, op != NATSL_OP_DECODE);
    if (rc != NATSL_OK) return rc;
    switch (op) {
        case NATSL_OP_FWD: *bytes = carve_fwd(p, nullptr).bytes; return NATSL_OK;
        case NATSL_OP_BWD: *bytes = carve_bwd(p, nullptr).bytes; return NATSL_OK;
        case NATSL_OP_DECODE: *bytes = decode_workspace_bytes(p->B, p->H, p->d); return NATSL_OK;
        case NATSL_OP_COMPACT: *bytes = 0; return NATSL_OK;
        default: return NATSL_ERR_UNSUPPORTED;
    }
}

int natsl_route_compact(const uint8_t *route, int32_t *sm_idx, int32_t *sm_chunk_prefix,
                        int32_t *lin_idx, int32_t *n_lin, const natsl_params *p, void *, size_t,
                        void *stream) {
    int rc = check_params(p, true);
    if (rc != NATSL_OK) return rc;
    if (!route || !sm_idx || !sm_chunk_prefix || !lin_idx || !n_lin) return NATSL_ERR_NULL;
    cudaError_t e = launch_route_compact(route, sm_idx, sm_chunk_prefix, lin_idx, n_lin, nullptr,
                                         nullptr, nullptr, 0, p->B, p->L, p->H,
                                         static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? NATSL_OK : NATSL_ERR_CUDA;
}

int natsl_score_layer(const void *x, const float *w_score, float *scores, uint8_t *route,
                      int32_t d_model, const natsl_params *p, void *stream) {
    int rc = check_params(p, true);
    if (rc != NATSL_OK) return rc;
    if (!x || !w_score || !route) return NATSL_ERR_NULL;
    // a row of X is read in 16-byte pieces
    const int per16 = p->dtype == NATSL_BF16 ? 8 : 4;
    // (the pooled rows of a CTA's two chunks and their scores live in shared memory)
    if (d_model <= 0 || d_model % per16 != 0 || ((size_t)d_model + 2 * (size_t)p->H) * 8 > kScoreSmemMax)
        return NATSL_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(w_score)) return NATSL_ERR_ALIGN;
    cudaError_t e = launch_score_layer(x, w_score, scores, route, d_model, shape_of(p),
                                       static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? NATSL_OK : NATSL_ERR_CUDA;
}

int natsl_hybrid_fwd(const void *q, const void *k, const void *v, const float *g,
                     const float *beta, const uint8_t *route, void *out, const natsl_params *p,
                     void *ws, size_t ws_bytes, void *stream) {
    int rc = check_params(p, true);
    if (rc != NATSL_OK) return rc;
    if (!q || !k || !v || !g || !beta || !route || !out) return NATSL_ERR_NULL;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(ws))
        return NATSL_ERR_ALIGN;
    const bool want_cache = p->k_sm || p->v_sm || p->sm_len;
    if (want_cache && !(p->k_sm && p->v_sm && p->sm_len && p->sm_cap > 0)) return NATSL_ERR_NULL;
    if (want_cache && (!aligned16(p->k_sm) || !aligned16(p->v_sm))) return NATSL_ERR_ALIGN;
    if ((p->o_la && !aligned16(p->o_la)) || (p->o_nla && !aligned16(p->o_nla))) return NATSL_ERR_ALIGN;
    const bool tensor_cores = use_tensor_cores(p);
    if (tensor_cores && !(p->scale_sm > 0.f)) return NATSL_ERR_SHAPE;   // (its kernel takes the maximum of raw logits)
    const bool block = (p->flags & NATSL_BLOCK_ROUTING) != 0;
    const bool append = (p->flags & NATSL_APPEND_CACHE) != 0;
    if (append && !tensor_cores) return NATSL_ERR_UNSUPPORTED;
    if (append && !want_cache) return NATSL_ERR_NULL;
    const HeadGroups hg = head_groups(p);
    if (grouped_or_normed(p)) {
        if (tensor_cores) {
            if (hg.G > 1 && !(hg.G == 2 && p->d == 128)) return NATSL_ERR_UNSUPPORTED;
            // (the saved forward is the backward's forward part: built where the backward is)
            if ((p->flags & NATSL_SAVE_FOR_BWD) && hg.G > 1 && p->d != 128) return NATSL_ERR_UNSUPPORTED;
        } else {
            if (p->dtype != NATSL_F32) return NATSL_ERR_UNSUPPORTED;
            if (hg.G > 1 && (hg.G > 4 || p->d / hg.G < 32)) return NATSL_ERR_UNSUPPORTED;
        }
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (p->flags & NATSL_SAVE_FOR_BWD) {
        // The forward of a training step: run in the backward's workspace, where it leaves what
        // natsl_hybrid_bwd (with NATSL_SAVED_FWD) would otherwise compute again.
        if (append || want_cache || p->o_la || p->o_nla || p->lse || p->stage_events) return NATSL_ERR_UNSUPPORTED;
        const BwdWs fb = carve_bwd(p, ws);
        if (!ws || ws_bytes < fb.bytes) return NATSL_ERR_WORKSPACE;
        return bwd_forward_part(q, k, v, g, beta, route, out, p->state_out, p, fb, st);
    }
    FwdWs f = carve_fwd(p, ws);
    if (!ws || ws_bytes < f.bytes) return NATSL_ERR_WORKSPACE;
    const Shape s = shape_of(p);
    const BlockRouting br{block ? route : nullptr, k, v};

#define NATSL_TRY(call) do { if ((call) != cudaSuccess) return NATSL_ERR_CUDA; } while (0)
    int stage = 0;
    auto mark = [&]() -> cudaError_t {
        if (p->stage_events && stage < p->n_stage_events)
            return cudaEventRecord(static_cast<cudaEvent_t>(p->stage_events[stage++]), st);
        return cudaSuccess;
    };
    void *k_sm = want_cache ? p->k_sm : f.k_sm, *v_sm = want_cache ? p->v_sm : f.v_sm;
    const int32_t cap = want_cache ? p->sm_cap : p->L;
    const int32_t capv = append ? p->sm_cap : p->L;          // rows per head of the fp16 V copy
    // A cache the call returns keeps the keys as given (the decode step normalises them as it reads them);
    // with the normalisation the softmax kernel then reads a normalised copy in the workspace instead.
    const bool raw_cache = want_cache && hg.norm_eps >= 0.f;
    void *k_norm = append ? f.kn16 : f.k_sm;     // (appending: normalised copies of the whole cache, capv rows per head)
    const void *k_soft = raw_cache ? k_norm : k_sm, *v_soft = raw_cache ? f.v_sm : v_sm;
    const int32_t cap_soft = raw_cache ? capv : cap;
    if (tensor_cores) {
        // Four kernels (six with a segmented scan):
        //   prepare (linear branch's set-up) | compaction + gather (softmax branch's), which needs nothing of it and,
        //   as its programmatic dependent, runs where its last wave leaves room, | scan, which waits for both, |
        //   softmax branch + combination, a programmatic dependent of the scan: it starts once the scan's CTAs are
        //   all resident, runs its Q K^T / P V loop beside it on the multiprocessors the scan leaves free, and picks
        //   up o_la chunk by chunk behind the counters the scan raises.
        // Per-stage events and NATSL_SINGLE_STREAM switch the overlap off (kernels in sequence).
        const bool beside = !p->stage_events && !(p->flags & NATSL_SINGLE_STREAM);
        int seg_chunks = 0;
        const int nseg = scan_segments(p, &seg_chunks);
        const bool pdl = beside && scan_follows_closely(p, nseg > 1);
        auto prepare = [&]() {   // block-level routing: every token takes part in the delta rule of its own block
            return launch_gdn_prepare_tc(q, k, v, g, beta, block ? nullptr : route, p->scale_la, f.tc, GdnTcExport{},
                                         f.status, s, st, (int)(kStatusBytes / 4), hg.norm_eps, beside);
        };
        auto gather = [&]() {
            return launch_route_gather_tc(k, v, route, f.sm_idx, f.prefix, append ? p->sm_len : nullptr, k_sm,
                                          want_cache ? v_sm : nullptr, f.v16, raw_cache ? k_norm : nullptr, cap, capv,
                                          f.emit_flags, s, st, beside, hg, raw_cache);
        };
        NATSL_TRY(mark());
        NATSL_TRY(beside ? prepare() : gather());    // (in sequence: in the order of the stages' names)
        NATSL_TRY(mark());
        NATSL_TRY(beside ? gather() : prepare());
        NATSL_TRY(mark());
        int32_t *flags_scan = beside && !g_debug_withhold_flags.load(std::memory_order_relaxed) ? f.emit_flags : nullptr;
        const int32_t *flags_softmax = beside ? f.emit_flags : nullptr;
        const ScanOut so{f.o_la16, p->o_la, flags_scan};
        if (nseg > 1) {   // few (batch, head) pairs: segments in parallel, chained by their transitions
            ScanSegments sg{1, nseg, seg_chunks, f.seg_incr, f.seg_trans, f.seg_start};
            NATSL_TRY(launch_gdn_scan_tc(q, k, v, f.tc, p->scale_la, p->state_in, nullptr, so, GdnTcExport{}, sg,
                                         br.route, f.status, s, st, pdl, hg.norm_eps >= 0.f));
            NATSL_TRY(launch_scan_combine(sg, s, st, pdl));
            sg.mode = 2;
            NATSL_TRY(launch_gdn_scan_tc(q, k, v, f.tc, p->scale_la, p->state_in, p->state_out, so, GdnTcExport{}, sg,
                                         br.route, f.status, s, st, pdl, hg.norm_eps >= 0.f));
        } else {
            NATSL_TRY(launch_gdn_scan_tc(q, k, v, f.tc, p->scale_la, p->state_in, p->state_out, so, GdnTcExport{},
                                         ScanSegments{0, 1, 0, nullptr, nullptr, nullptr}, br.route,
                                         f.status, s, st, pdl, hg.norm_eps >= 0.f));
        }
        NATSL_TRY(mark());
        NATSL_TRY(launch_softmax_combine_tc(q, k_soft, f.v16, cap_soft, capv, f.sm_idx, f.prefix, f.o_la16,
                                            flags_softmax, p->w, p->scale_sm, p->eps, out, p->o_nla,
                                            p->lse, want_cache ? p->sm_len : nullptr, cap, br, append, f.status, s, st, hg, nseg,
                                            seg_chunks / 2));
        NATSL_TRY(mark());
        return NATSL_OK;
    }
    // fp32 arithmetic: prepare | compaction + gather, beside it | scan, which waits for both, | softmax branch, beside the
    // scan up to its epilogue.  With per-stage events: in sequence, in the order of the stages' names.
    const bool beside = !p->stage_events;
    NATSL_TRY(mark());
    if (!beside) NATSL_TRY(cudaMemsetAsync(f.status, 0, kStatusBytes, st));
    // NATSL_QK_NORM: normalised copies first
    const void *q_la = q, *k_la = k, *q_sm = q, *k_nsm = k;
    if (hg.norm_eps >= 0.f) {
        NATSL_TRY(launch_qk_norm_f32((const float *)q, (const float *)k, f.q_la, f.k_la, f.q_sm, f.k_nsm,
                                     (size_t)p->B * p->L * p->H, p->d, hg.G, hg.norm_eps, st));
        q_la = f.q_la; k_la = f.k_la; q_sm = f.q_sm; k_nsm = f.k_nsm;
    }
    float *o_la = p->o_la ? p->o_la : f.o_la;
    auto gather = [&]() {
        const RowsJob soft{k_nsm, raw_cache ? f.k_sm : k_sm, raw_cache ? f.v_sm : v_sm, cap_soft};
        return launch_route_gather_rows(route, v, soft, raw_cache ? RowsJob{k, k_sm, v_sm, cap} : RowsJob{}, f.sm_idx, f.prefix,
                                        want_cache ? p->sm_len : nullptr, cap, f.status, block, s, st, beside);
    };
    if (!beside) NATSL_TRY(gather());
    NATSL_TRY(mark());
    NATSL_TRY(launch_gdn_prepare_simt(q_la, k_la, v, g, beta, block ? nullptr : route, p->scale_la, f.W,
                                      f.U, f.P, nullptr, nullptr, s, st, beside ? f.status : nullptr, (int)(kStatusBytes / 4)));
    if (beside) NATSL_TRY(gather());
    NATSL_TRY(mark());
    NATSL_TRY(launch_gdn_scan_simt(q_la, k_la, g, f.W, f.U, f.P, p->scale_la, p->state_in,
                                   p->state_out, nullptr, nullptr, o_la, br.route, s, st, scan_follows_closely(p, true)));
    NATSL_TRY(mark());
    // (an own-block tile of block-level routing reads the layer's keys: the softmax operation's copy)
    NATSL_TRY(launch_softmax_combine_simt(q_sm, k_soft, v_soft, cap_soft, f.sm_idx, f.prefix, o_la, p->w,
                                          p->scale_sm, p->eps, out, p->o_nla, p->lse,
                                          BlockRouting{br.route, k_nsm, v}, s, st, hg.G));
    NATSL_TRY(mark());
#undef NATSL_TRY
    return NATSL_OK;
}

int natsl_hybrid_bwd(const void *q, const void *k, const void *v, const float *g,
                     const float *beta, const uint8_t *route, const void *dout, void *dq, void *dk,
                     void *dv, float *dg, float *dbeta, float *dw, const natsl_params *p, void *ws,
                     size_t ws_bytes, void *stream) {
    int rc = check_params(p, true);
    if (rc != NATSL_OK) return rc;
    if (!q || !k || !v || !g || !beta || !route || !dout || !dq || !dk || !dv || !dg || !dbeta)
        return NATSL_ERR_NULL;
    if (p->flags & NATSL_APPEND_CACHE) return NATSL_ERR_UNSUPPORTED;
    const HeadGroups hg = head_groups(p);
    if (grouped_or_normed(p)) {      // grouped heads, q/k normalisation: the paths with separate chunk-level products
        if (use_tensor_cores(p)) {      // softmax heads of 64 or 128 columns
            if (!((p->d == 128 && hg.G <= 2) || (p->d == 64 && hg.G == 1))) return NATSL_ERR_UNSUPPORTED;
        } else {
            if (p->dtype != NATSL_F32) return NATSL_ERR_UNSUPPORTED;
            if (hg.G > 1 && (hg.G > 4 || p->d / hg.G < 32)) return NATSL_ERR_UNSUPPORTED;
        }
    }
    if (use_tensor_cores(p) && !(p->scale_sm > 0.f)) return NATSL_ERR_SHAPE;
    const bool block = (p->flags & NATSL_BLOCK_ROUTING) != 0;
    if (p->dscore && !block) return NATSL_ERR_UNSUPPORTED;   // score gradients: one decision per block
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(dout) || !aligned16(dq) ||
        !aligned16(dk) || !aligned16(dv) || !aligned16(ws))
        return NATSL_ERR_ALIGN;
    BwdWs f = carve_bwd(p, ws);
    if (!ws || ws_bytes < f.bytes) return NATSL_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const Shape s = shape_of(p);
    Shape s32 = s;              // the same shapes with fp32 storage (the fp32 copies)
    s32.bf16 = false;
    const long long B = p->B, H = p->H, L = p->L, d = p->d, NC = L / kC;
    auto TM = [&](const float *x) { return BMat{x, L * H * d, d, (long long)kC * H * d, (int)(H * d)}; };
    auto CC = [&](const float *x) { return BMat{x, H * NC * kC * kC, NC * kC * kC, (long long)kC * kC, kC}; };
    auto ST = [&](const float *x) { return BMat{x, H * NC * d * d, NC * d * d, d * d, (int)d}; };
    const int di = p->d;
    const uint8_t *block_route = block ? route : nullptr;
    const bool tensor_cores = use_tensor_cores(p), normed = hg.norm_eps >= 0.f;

    // ---- forward, keeping what the backward needs (unless the caller's forward already did) ----
    if (!(p->flags & NATSL_SAVED_FWD)) {
        rc = bwd_forward_part(q, k, v, g, beta, route, nullptr, nullptr, p, f, st);
        if (rc != NATSL_OK) return rc;
    }
#define NATSL_TRY(call) do { if ((call) != cudaSuccess) return NATSL_ERR_CUDA; } while (0)
    // From here on two more pairs of independent stages run side by side on the library's side
    // stream: the reverse scan of the linear branch beside the softmax branch's backward.
    std::unique_lock<std::mutex> side_lock;
    SideStream *side = nullptr;
    SideJoin side_join;
    if (tensor_cores && !(p->flags & NATSL_SINGLE_STREAM)) {
        side_lock = std::unique_lock<std::mutex>(g_side_mu);
        side = side_stream_locked();
        if (!side) side_lock.unlock();
    }
    cudaStream_t st0 = side ? side->st : st;
    // ---- combination and softmax branch ----
    // Tensor cores: the fp16 gradient operands are scaled by a power of two taken from max |dout|,
    // so that a loss-scaled or a tiny dout stays inside fp16's range (grad_scale, common.cuh).
    if (tensor_cores) NATSL_TRY(launch_dout_amax(dout, (size_t)(B * L * H * d), s.bf16, f.status, st));
    const int32_t *gsc = tensor_cores ? f.status : nullptr;
    NATSL_TRY(launch_combine_bwd(f.o_la, f.o_nla, dout, p->w, p->eps, tensor_cores ? nullptr : f.do_la,
                                 tensor_cores ? nullptr : f.do_nla, dw, f.Dsm,
                                 tensor_cores ? f.dO16 : nullptr, tensor_cores ? f.gr.dO16 : nullptr,
                                 tensor_cores ? f.gr.dOg16 : nullptr, f.tc.Gd, p->scale_la, gsc, s, st, hg.G));
    AssembleArgs a{f.q32, f.k32, f.v32, f.Gcum, beta, block ? nullptr : route, f.dQg, f.dKb, f.dVb, f.dKt, f.X1p, f.X2,
                   f.X3, f.X4, normed ? nullptr : f.dq_sm, f.dk_sm, f.dv_sm, f.gS, f.sm_idx, f.prefix, p->L,
                   p->scale_la, f.dGrow, f.kappa, dbeta, dg};
    if (tensor_cores) {
        // Dependencies from here on: the query-side softmax kernel, the key-side one (both with the normalisation:
        // behind the softmax operation's copy of q) and the reverse scan need only what is already there; the chunk kernel needs the reverse scan and, unless q and k are normalised, the
        // query-side kernel's dq; the scatter of the retained tokens' dk, dv needs the key-side kernel.
        // Token-level routing: query-side kernel, key-side kernel, scatter on the caller's stream (the key-side one
        // starts in the query-side one's tail, on the multiprocessors the reverse scan leaves free), reverse scan and
        // chunk kernel on the side stream.
        // Block-level routing: reverse scan, key-side kernel, scatter on the side stream, the others on the caller's:
        // every token has a softmax-branch dk, dv (retained tokens: scattered from the
        // compacted gradients; linear blocks: their own block's kernel, which needs the query-side one only), both
        // in fp32 token-major buffers that the chunk kernel adds (through the normalisation's Jacobian, where there is
        // one) and so waits for.
        if (side) {
            NATSL_TRY(cudaEventRecord(side->fork, st));
            NATSL_TRY(cudaStreamWaitEvent(st0, side->fork, 0));
            side_join.forked(side, st);
        }
        NATSL_TRY(launch_gdn_rscan_tc(f.tc, f.gr, p->dstate_out, p->dstate_in, block_route, f.status, s, st0));
        if (side && block) NATSL_TRY(cudaEventRecord(side->join, st0));
        // The fp16 copy of q that both softmax kernels read: the prepare kernel's, or, normalised, the softmax
        // operation's own, which goes where the forward had its gathered keys (nothing reads them any more; the
        // reverse scan beside it reads the linear operation's copy).  It is written on the caller's stream, so a
        // key-side kernel on the side stream waits for it there.
        const void *q16 = f.Qh;
        if (normed) {
            NATSL_TRY(launch_to_f16_bhld(q, f.k_smb, s, hg, st));
            q16 = f.k_smb;
            if (side && block) {
                NATSL_TRY(cudaEventRecord(side->fork, st));
                NATSL_TRY(cudaStreamWaitEvent(st0, side->fork, 0));
            }
        }
        NATSL_TRY(launch_softmax_bwd_tc(q16, f.dO16, f.k16, f.v16, p->L, f.sm_idx, f.prefix, f.lse, f.Dsm,
                                        p->scale_sm, f.dq_sm, f.dk_sm, f.dv_sm, p->dscore ? f.dmask : nullptr,
                                        f.status, s, st, block ? st0 : st, side && !block ? side->fork : nullptr, hg));
        if (block) {
            if (side) NATSL_TRY(cudaStreamWaitEvent(st, side->join, 0));     // the reverse scan has finished
            NATSL_TRY(launch_scatter_sm(a, f.dk_x, f.dv_x, s32, st0));
            NATSL_TRY(launch_softmax_bwd_own_block(q, k, v, f.dO16, f.lse, f.Dsm, route, p->scale_sm, f.dq_sm, f.dk_x,
                                                   f.dv_x, gsc, s, st, hg));
            NATSL_TRY(side_join.join());      // the side stream's last kernels
            NATSL_TRY(launch_gdn_chunk_bwd(f.tc, f.ex, f.gr, q, k, v, beta, route, f.dq_sm, p->scale_la, dq, dk, dv, dg,
                                           dbeta, true, f.dk_x, f.dv_x, p->dscore ? f.kap_c : nullptr, f.status, s, st,
                                           hg));
            if (p->dscore)
                NATSL_TRY(launch_dscore(route, f.prefix, f.dmask, f.kap_c, nullptr, p->L, p->dscore, s, st, hg.G));
            return NATSL_OK;
        }
        // Token-level routing.  With the normalisation a token's k has one gradient, of one copy or the other: they
        // stay in fp32 until its backward, a last kernel that rounds once.
        void *dq_o = normed ? f.dq32 : dq, *dk_o = normed ? f.dk32 : dk, *dv_o = normed ? f.dv32 : dv;
        if (side && !normed) NATSL_TRY(cudaStreamWaitEvent(st0, side->fork, 0));      // dq_sm
        NATSL_TRY(launch_gdn_chunk_bwd(f.tc, f.ex, f.gr, q, k, v, beta, route, normed ? nullptr : f.dq_sm, p->scale_la,
                                       dq_o, dk_o, dv_o, dg, dbeta, false, nullptr, nullptr, nullptr, f.status, s, st0,
                                       hg));
        // the retained tokens' dk, dv (rows the chunk kernel does not write)
        NATSL_TRY(launch_scatter_sm(a, dk_o, dv_o, normed ? s32 : s, st));
        NATSL_TRY(side_join.join());
        if (normed)
            NATSL_TRY(launch_qk_norm_bwd_f32(q, k, true, route, f.dq32, f.dq_sm, f.dk32, f.dv32, dq, dk, dv,
                                             (size_t)(B * L * H), p->d, hg.G, hg.norm_eps, st, nullptr));
        return NATSL_OK;
    }
    // ---- fp32 CUDA-core path: softmax branch, reverse scan, chunk-level products as tile GEMMs, assembly ----
    NATSL_TRY(launch_softmax_bwd(normed ? f.qs32 : f.q32, f.k_sm32, f.v_sm32, p->L, f.sm_idx, f.prefix, f.do_nla, f.lse,
                                 f.Dsm, p->scale_sm, f.dq_sm, f.dk_sm, f.dv_sm, s, st, p->dscore ? f.dmask : nullptr,
                                 hg.G));
    NATSL_TRY(launch_gdn_rscan(f.q32, f.k32, f.Gcum, f.W, f.P, f.do_la, f.S_c, p->scale_la, f.dUt, f.dS_c, f.gS,
                               p->dstate_out, p->dstate_in, s, st, block_route));
    // (block-level routing: beta~ = beta for every token, so the kernels below get no route)
    const uint8_t *route_bt = block ? nullptr : route;
    if (block) {
        // Every token has a softmax-branch dk, dv: the retained tokens' from the compacted gradients, the
        // tokens of linear blocks' from their own block (each token is written by exactly one of the
        // two); the assembly adds them to the linear branch's -- with the normalisation dk_x, a gradient with
        // respect to the softmax operation's copy, stays apart until its backward.
        NATSL_TRY(launch_scatter_sm(a, f.dk_x, f.dv_x, s32, st));
        NATSL_TRY(launch_softmax_bwd_own_block_simt(normed ? f.qs32 : f.q32, normed ? f.ks32 : f.k32, f.v32, f.do_nla, f.lse,
                                                    f.Dsm, route, p->scale_sm, f.dq_sm, f.dk_x, f.dv_x, gsc, s32, st,
                                                    hg.G));
        a.dk_x = normed ? nullptr : f.dk_x;
        a.dv_x = f.dv_x;
        a.no_scatter = true;
    }
    auto gemm = [&](bool ta, bool tb, int mask, BMat x, BMat y, BMat z, int m, int n, int k_, float alpha, bool acc) {
        return launch_bgemm(ta, tb, mask, x, y, z, m, n, k_, alpha, acc, s32, st);
    };
    NATSL_TRY(gemm(false, true, 0, TM(f.do_la), ST(f.S_c), TM(f.dQg), kC, di, di, 1.f, false));
    NATSL_TRY(gemm(false, true, 0, TM(f.dUt), ST(f.S_c), TM(f.dW), kC, di, di, -1.f, false));
    NATSL_TRY(gemm(false, true, 0, TM(f.Ut), ST(f.dS_c), TM(f.dKt), kC, di, di, 1.f, false));
    NATSL_TRY(gemm(false, true, 1, TM(f.do_la), TM(f.Ut), CC(f.N), kC, kC, di, 1.f, false));
    NATSL_TRY(launch_gdn_tsolve(f.Abar, beta, route_bt, f.dW, f.dUt, f.dKb, f.dVb, s, st));
    NATSL_TRY(gemm(false, true, 2, TM(f.dKb), TM(f.W), CC(f.M), kC, kC, di, -1.f, false));
    NATSL_TRY(gemm(false, true, 2, TM(f.dVb), TM(f.U), CC(f.M), kC, kC, di, -1.f, true));
    NATSL_TRY(launch_mask_scale(f.M, f.N, f.Gcum, beta, route_bt, p->scale_la, f.Mg, f.Ms, f.Ns, s, st));
    NATSL_TRY(gemm(false, false, 0, CC(f.Mg), TM(f.k32), TM(f.X1p), kC, di, kC, 1.f, false));
    NATSL_TRY(gemm(true, false, 0, CC(f.Ms), TM(f.k32), TM(f.X2), kC, di, kC, 1.f, false));
    NATSL_TRY(gemm(false, false, 0, CC(f.Ns), TM(f.k32), TM(f.X3), kC, di, kC, 1.f, false));
    NATSL_TRY(gemm(true, false, 0, CC(f.Ns), TM(f.q32), TM(f.X4), kC, di, kC, 1.f, false));
    NATSL_TRY(launch_gdn_assemble(a, dq, dk, dv, s, st));
    // With the normalisation (fp32 storage) the assembly's dq, dk are gradients with respect to the normalised
    // rows; a last kernel applies the two row-local Jacobians in place.
    if (normed)
        NATSL_TRY(launch_qk_norm_bwd_f32(q, k, false, route, (const float *)dq, f.dq_sm, (const float *)dk, nullptr,
                                         dq, dk, nullptr, (size_t)(B * L * H), p->d, hg.G, hg.norm_eps, st,
                                         block ? f.dk_x : nullptr));
    if (p->dscore)   // softmax blocks: the mask gradients of their keys; linear blocks: the kappa of their tokens
        NATSL_TRY(launch_dscore(route, f.prefix, f.dmask, nullptr, f.kappa, p->L, p->dscore, s, st, hg.G));
#undef NATSL_TRY
    return NATSL_OK;
}

int natsl_decode_step(const void *q, const void *k, const void *v, const float *g,
                      const float *beta, const uint8_t *route, float *state, void *k_cache,
                      void *v_cache, int32_t *cache_len, int32_t cache_cap, void *out,
                      const natsl_params *p, void *ws, size_t ws_bytes, void *stream) {
    int rc = check_params(p, false);
    if (rc != NATSL_OK) return rc;
    if (!q || !k || !v || !g || !beta || !route || !state || !k_cache || !v_cache || !cache_len ||
        !out)
        return NATSL_ERR_NULL;
    if (cache_cap <= 0) return NATSL_ERR_SHAPE;
    const HeadGroups hg = head_groups(p);
    if (hg.G > 1 && (hg.G > 4 || p->d / hg.G < 32)) return NATSL_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(state) ||
        !aligned16(k_cache) || !aligned16(v_cache) || !aligned16(ws))
        return NATSL_ERR_ALIGN;
    if (!ws || ws_bytes < decode_workspace_bytes(p->B, p->H, p->d)) return NATSL_ERR_WORKSPACE;
    cudaError_t e = launch_decode_step(q, k, v, g, beta, route, p->w, state, k_cache, v_cache,
                                       cache_len, cache_cap, out, p->scale_la, p->scale_sm, p->eps,
                                       ws, shape_of(p),
                                       static_cast<cudaStream_t>(stream), hg);
    return e == cudaSuccess ? NATSL_OK : NATSL_ERR_CUDA;
}

int natsl_decode_block_end(const uint8_t *route_block, const float *g_block, float *state,
                           float *state_start, int32_t *cache_len, int32_t block_len,
                           const natsl_params *p, void *ws, size_t ws_bytes, void *stream) {
    int rc = check_params(p, false);
    if (rc != NATSL_OK) return rc;
    if (!route_block || !g_block || !state || !state_start || !cache_len) return NATSL_ERR_NULL;
    if (block_len <= 0) return NATSL_ERR_SHAPE;
    if (!aligned16(state) || !aligned16(state_start) || !aligned16(ws)) return NATSL_ERR_ALIGN;
    if (!ws || ws_bytes < decode_workspace_bytes(p->B, p->H, p->d)) return NATSL_ERR_WORKSPACE;
    cudaError_t e = launch_decode_block_end(route_block, g_block, state, state_start, cache_len,
                                            block_len, ws, shape_of(p),
                                            static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? NATSL_OK : NATSL_ERR_CUDA;
}

void natsl_debug_set_wait_limit(uint32_t kcycles, int withhold_scan_flags) {
    g_debug_wait_kcycles.store(kcycles > 0x7fffffffu ? 0x7fffffffu : kcycles, std::memory_order_relaxed);
    g_debug_withhold_flags.store(withhold_scan_flags ? 1 : 0, std::memory_order_relaxed);
}

int natsl_device_status(void *ws, void *stream) {
    if (!ws) return NATSL_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t word = 0;
    if (cudaMemcpyAsync(&word, ws, sizeof(word), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return NATSL_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return NATSL_ERR_CUDA;
    if (word != 0 && cudaMemsetAsync(ws, 0, sizeof(word), st) != cudaSuccess) return NATSL_ERR_CUDA;
    return word;
}

}  // extern "C"
