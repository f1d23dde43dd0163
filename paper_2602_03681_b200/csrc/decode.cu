// Decode step (Section 4.1, per-token generation): decay the fp32 d x d state, apply the gated
// delta rule (linear token) or retain the token's K/V (softmax token) -- or both, while the
// decision of the token's block is still open -- read both branches and combine their
// RMS-normalised outputs (Section 4.3, Norm equation).  decode_block_end_kernel rolls back the
// operation that was not chosen once a block is complete.
//
// HBM-bound for many (sequence, head) pairs, a chain of latencies for few: per pair the state is read
// and written once (2 d^2 4 bytes) and the retained K/V are read once.  The work of a pair is split into
// items: `parts` cache items, each a slice of the retained K/V, and kStateParts state items, each a group
// of the state's value columns (the columns of the delta rule are independent).  Whichever item of the
// pair finishes last (an atomic ticket, nobody waits) merges the partial results, adds the new token's own
// term, normalises, combines, writes `out`, appends the token to the cache and bumps its length.
// A pair's slices go by its length: see decode_split.
//   * Few pairs: every item has a CTA of its own and the cache is cut as finely as the machine has room
//     for (up to 16 slices), because a slice is walked serially.
//   * Many pairs: persistent CTAs, two per SM.  The copy warp runs ahead into the next item's slice (96 KB in
//     flight per CTA), the work warps leave their part of an item in shared memory and go on, and a finisher
//     warp merges it, takes the ticket and finishes the step behind them, so that neither the ticket's
//     round trip nor the final merge ever stands between two items.
// The kernel is a programmatic dependent of the work before it in the stream: barriers and the ring are
// set up while that finishes, nothing global is touched before it has.
// Work per cached key: eight lanes share a row (four rows per warp and pass), each with whole 16-byte
// pieces 128 bytes apart (conflict-free); products as packed fp32 pairs; the running maximum moves only when
// a logit exceeds it by 2^8, so the accumulator is rescaled once or twice per slice instead of per key.
// (With sixteen lanes per row and a rescale per key the kernel issued 2.5 x the instructions and sat at 83 %
// of the copy rate, 74 % with grouped heads.)
// Grouped softmax heads and per-operation q/k normalisation (Section 4.3; template parameters): the G softmax
// heads of a linear head are the G slices of d / G columns, each with its own logit, running maximum and
// sum; the state items work on the L2-normalised q and k, and the cache keeps the keys as given: a cached
// key is RMS-normalised per slice as it is read (its sum of squares rides along with the logit's
// reduction), because normalised keys rounded to the cache's bf16 would cost 2.8e-2 of the branch output's
// RMS.
#include <algorithm>
#include "common.cuh"
#include "natsl_internal.h"
#include "tc_common.cuh"

namespace natsl {

namespace {

using namespace tc;

constexpr int kWorkThreads = 256;
constexpr int kWarps = kWorkThreads / 32;
constexpr int kThreads = kWorkThreads + 64;      // + one warp that issues the bulk copies, + the finisher
constexpr int kTileKeys = 32;                    // one key per group of eight lanes and pass
constexpr int kRingBytes = 96 * 1024;
constexpr int kStateParts = 2;
constexpr int kMaxParts = 16;
constexpr int kCtasPerSm = 2;
constexpr int kMaxItems = 128;                   // items of a CTA

// ---- How a pair's cache is cut: by its length, known on the device only.  The host works the count out for every class of
// lengths (1 to 300 keys, to 600, to 900, to 1200, more) that the capacity allows and passes the counts along. ----
// Cache items per (sequence, head), when every item is to be resident at once (0: not possible) ...
inline int parts_resident(int BH, int resident) {
    const int p = resident / BH - kStateParts;
    return p > kMaxParts ? kMaxParts : (p > 0 ? p : 0);
}
// ... and when the CTAs go round: the count whose items fill the last round best, an item's start and merge counted as
// 5 % of a round; from one item per 300 keys (a round of nearly empty items takes 4 us: 504 pairs of 100 keys 45 us a step
// with four items each), four at most.
inline int parts_persistent(int BH, int resident, int keys) {
    const int from = std::min(4, std::max(1, (keys + 299) / 300));
    int best = from;
    float least = 1e30f;
    for (int p = from; p <= kMaxParts; ++p) {
        const float n = (float)BH * (p + kStateParts), per = n / resident;
        const float cost = (float)(int)(per + 0.999f) / per + 0.05f * p;
        if (cost < least) { least = cost; best = p; }
    }
    return best;
}
// Resident where it can be, unless that makes only one or two items of a cache of more than 600 keys for each:
// they then take much longer than the state items, and half of the CTAs wait for them.  Per step, resident -> going round:
// 96 pairs of 1638 keys 26.3 -> 18.6 us, 90 pairs of the normalised mode, 800 keys, 19.2 -> 14.9; 64 pairs of 1638 keys
// 16.3 -> 15.1; but 72 pairs of 800 keys 12.9 -> 13.9, 96 of 200 8.6 -> 11.1.
inline int decode_parts(int BH, int resident, int keys) {
    const int p = parts_resident(BH, resident);
    return p > 2 || (p > 0 && keys <= 600 * p) ? p : parts_persistent(BH, resident, keys);
}
// What the kernel gets: `parts` items are laid out for every pair, those beyond the count of its length are empty.  Where
// all classes that the capacity allows agree nothing is empty, and the kernel that does not ask runs.  (With the count
// taken from the capacity, 4096 rows cost short sequences: 64 pairs of 200 keys 10.6 us a step, 7.9 by length, 504 of 100
// 43.4 and 33.8, 1024 of 100 85.9 and 65.1.)
// Order of the items: the first `front` cache items and the state items of every pair, then the rest.  Where the shortest
// class's items fill no more than two rounds these are the front, so that short caches are spread as evenly as if nothing
// were empty (96 pairs of 200 keys in 4096 rows 12.4 -> 8.3 us, 100 of 600 15.8 -> 12.6); elsewhere the front is everything
// (with a front, 1024 pairs of 1638 keys 161 -> 173: first the states, then the caches).
constexpr int kClassKeys = 300, kClasses = 5, kClassBits = 5;
struct DecSplit { int parts, front; uint32_t by_class; bool varied; };
inline DecSplit decode_split(int BH, int resident, int cap) {
    DecSplit sp{0, 0, 0u, false};
    int first = 0;
    for (int c = 0; c < kClasses; ++c) {
        const int keys = c + 1 < kClasses ? std::min(cap, (c + 1) * kClassKeys) : cap;
        const int p = decode_parts(BH, resident, keys);
        if (c == 0) first = p;
        sp.by_class |= (uint32_t)p << (c * kClassBits);
        sp.parts = std::max(sp.parts, p);
        sp.varied |= p != first;
    }
    sp.front = BH * (first + kStateParts) <= 2 * resident ? first : sp.parts;
    return sp;
}
__device__ __forceinline__ int class_parts(uint32_t by_class, int keys) {
    const int c = min(max((keys + kClassKeys - 1) / kClassKeys, 1), kClasses) - 1;
    return (by_class >> (c * kClassBits)) & ((1u << kClassBits) - 1u);
}

template <typename T> struct Vec16;   // 16 bytes of T as fp32 values
template <> struct Vec16<float> {
    static constexpr int kN = 4;
    __device__ static void unpack(const uint4 u, float (&x)[4]) {
        x[0] = __uint_as_float(u.x); x[1] = __uint_as_float(u.y);
        x[2] = __uint_as_float(u.z); x[3] = __uint_as_float(u.w);
    }
};
template <> struct Vec16<__nv_bfloat16> {
    static constexpr int kN = 8;
    __device__ static void unpack(const uint4 u, float (&x)[8]) {
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
};

// Workspace: [0,256) status word; then tickets [BH] i32; o_la [BH][D] f32; partials [BH][parts][D+8] f32 (m[G] in base-2
// units and z[G] in the first 8 with G <= 4, then acc[D]).
constexpr int kPartHead = 8;
__host__ __device__ inline size_t dec_off_tickets() { return 256; }
__host__ __device__ inline size_t dec_off_ola(size_t BH) { return (256 + BH * 4 + 255) / 256 * 256; }
__host__ __device__ inline size_t dec_off_partials(size_t BH, int D) {
    return dec_off_ola(BH) + (BH * D * 4 + 255) / 256 * 256;
}

template <typename T, int D, int G> struct DecLayout {
    static constexpr int kRowBytes = D * (int)sizeof(T);
    static constexpr int kTileBytes = kTileKeys * kRowBytes;
    static constexpr int kStages = kRingBytes / (2 * kTileBytes);      // K and V tile per stage
    static constexpr int kSlotFloats = 8 * 128;                        // [8 warps][D] or [slots][D / 2]
    static constexpr int oScratch = kRingBytes;                        // two slots, then the state items' own
    static constexpr int oMz = oScratch + 3 * kSlotFloats * 4;         // [2][8 warps][G] (m, z)
    static constexpr int kTotal = oMz + 2 * kWarps * G * 8;
};

// kVaried: the count of a pair's cache items depends on its length.
template <typename T, int D, int G, bool kNorm, bool kVaried>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
decode_step_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v,
                   const float *__restrict__ g, const float *__restrict__ beta,
                   const uint8_t *__restrict__ route, const float *__restrict__ w,
                   float *__restrict__ state, T *__restrict__ k_cache, T *__restrict__ v_cache,
                   int32_t *__restrict__ cache_len, int cap, T *__restrict__ out, float scale_la,
                   float scale_sm, float eps, uint8_t *__restrict__ ws, int BH, DecSplit split, float norm_eps) {
    using SL = DecLayout<T, D, G>;
    constexpr int kStages = SL::kStages, kRowBytes = SL::kRowBytes, kTileBytes = SL::kTileBytes;
    constexpr int ds = D / G;                      // columns per softmax head
    constexpr int kE = Vec16<T>::kN;               // elements per 16-byte piece
    constexpr int kJ = kRowBytes / 128;            // pieces per lane of a row's eight lanes
    constexpr int kSp = ds * (int)sizeof(T) / 16;  // pieces per softmax head
    static_assert(kSp % 4 == 0 && (kSp == 4 || kSp % 8 == 0), "softmax heads of at least 64 bytes");
    constexpr int kLg = kSp >= 8 ? G : kJ;         // logits a lane takes part in
    constexpr int kJpl = kJ / kLg;                 // pieces per logit and lane
    constexpr int kLanes = kSp >= 8 ? 8 : 4;       // lanes that share a logit
    constexpr float kLog2e = 1.4426950408889634f;
    constexpr int kCols = D / kStateParts;         // state item: value columns
    constexpr int kLpr = kCols / 4;                // lanes per (half) state row
    constexpr int kRpl = 32 / kLpr;                // rows per warp-wide access
    constexpr int kSlots = kWarps * kRpl;          // row slots in the CTA
    constexpr int kR = D / kSlots;                 // rows per thread
    static_assert(kSlots * kCols <= SL::kSlotFloats, "scratch too small");

    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t full[kStages], empty[kStages], done[2], taken[2];
    __shared__ uint64_t looked, first_read;
    __shared__ uint32_t s_empty[kMaxItems / 32], s_closed[kMaxItems / 32];
    __shared__ int s_len[kMaxItems], s_pair[kMaxItems];
    __shared__ int2 s_tiles[kMaxItems];
    __shared__ int s_abort[2];   // s_abort[1]: wait limit (see mbar_wait)
    auto slot_of = [&](int i) { return reinterpret_cast<float *>(smem + SL::oScratch) + i * SL::kSlotFloats; };
    float2 *mz = reinterpret_cast<float2 *>(smem + SL::oMz);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int parts = split.parts, front = split.front, per_head = parts + kStateParts, total = BH * per_head;
    const int n_front = BH * (front + kStateParts);
    int32_t *status = reinterpret_cast<int32_t *>(ws);
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], kWarps); }
        for (int s = 0; s < 2; ++s) { mbar_init(&done[s], kWarps); mbar_init(&taken[s], 1); }
        mbar_init(&looked, 1);
        mbar_init(&first_read, kWarps);
        s_abort[0] = 0;
        s_abort[1] = 0;
        fence_mbar_init();
    }
    if (kVaried && tid < kMaxItems / 32) s_empty[tid] = 0u;
    __syncthreads();
    volatile int *abort_flag = s_abort;
    grid_dependency_wait();
    launch_dependents();

    // This CTA's items: blockIdx.x, blockIdx.x + gridDim.x, ...; part >= parts: a state item.
    // (Counted: with the item's number as the loops' test a step of two items per CTA took 1 us longer, 64 pairs 14.3 for 13.3.)
    auto item_no = [&](int ord) { return (int)blockIdx.x + ord * (int)gridDim.x; };
    const int n_items = (total - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
    auto has = [&](int ord) { return ord < n_items; };
    auto locate = [&](int item, int &part, int &bh) {
        if (!kVaried || item < n_front) {
            bh = item / (front + kStateParts);
            part = item - bh * (front + kStateParts);
            if (kVaried && part >= front) part += parts - front;
        } else {
            bh = (item - n_front) / (parts - front);
            part = front + (item - n_front) - bh * (parts - front);
        }
    };
    // The copy warp looks up the lengths of all of them and lists what it will copy; cache items that the length leaves
    // empty get no turn, the finisher takes their tickets at once.
    // The length changes with the pair's last ticket, so every ticket of a CTA comes behind every read of that length in
    // the CTA: the copy warp's, through `looked`, the work warps', through the item's turn or, where the first item, which
    // they do not wait for the look-up with, has none, through `first_read`.
    auto parts_of = [&](int n_old) { return kVaried ? class_parts(split.by_class, n_old) : parts; };
    auto empty_item = [&](int ord) { return (s_empty[ord >> 5] >> (ord & 31)) & 1u; };
    // Tiles of a cache item.  A stored length outside [0, cap] (a prefill whose cache overflowed, a caller's
    // mistake) is clamped, so that no copy can leave the pair's rows; the finisher reports it.
    auto tiles_of = [&](int part, int n_old, bool cache_full, int &t_begin, int &t_end) {
        const int tiles = cache_full ? 0 : (n_old + kTileKeys - 1) / kTileKeys;
        const int np = parts_of(n_old), tpp = (tiles + np - 1) / np;
        t_begin = min(part * tpp, tiles);
        t_end = min(t_begin + tpp, tiles);
    };

    if (warp == kWarps) {
        // ---------------- copy warp: the cache slices of all items of this CTA, back to back ----------------
        int t = 0, t_end = 0, bh = 0, n_old = 0, it = 0; // (it: tiles issued so far)
        bool ok = true;
        auto issue = [&]() {                             // tile t of pair bh
            const int s = it % kStages;
            ok = mbar_wait(&empty[s], ((it / kStages) & 1) ^ 1, abort_flag);
            if (!ok) return;
            const int rows = min(kTileKeys, n_old - t * kTileKeys);
            const uint32_t bytes = (uint32_t)rows * kRowBytes;
            const size_t at = (size_t)bh * cap * kRowBytes + (size_t)t * kTileBytes;
            mbar_arrive_expect_tx(&full[s], 2 * bytes);
            bulk_load_1d(smem + (2 * s) * kTileBytes, reinterpret_cast<const uint8_t *>(k_cache) + at, bytes, &full[s]);
            bulk_load_1d(smem + (2 * s + 1) * kTileBytes, reinterpret_cast<const uint8_t *>(v_cache) + at, bytes, &full[s]);
            ++t;
            ++it;
        };
        int part = parts, pr = 0, len = 0, rv = 0;       // of this lane's item of the batch: a cache item or none
        auto look_up = [&](int ord) {
            part = parts;
            if (has(ord)) locate(item_no(ord), part, pr);
            if (part < parts) { len = cache_len[pr]; rv = route[pr]; }
        };
        look_up(lane);
        if (lane == 0 && part < parts) {                 // the first item: a ring of tiles ahead of the others' lengths
            bh = pr;
            n_old = min(max(len, 0), cap);
            tiles_of(part, n_old, rv != 0 && n_old >= cap, t, t_end);
            while (t < t_end && it < kStages && ok) issue();
        }
        __syncwarp();
        int n = 0;                                       // listed: cache items with tiles behind the first item
        for (int o0 = 0; has(kVaried ? o0 : o0 + 1); o0 += 32) {
            const int ord = o0 + lane;
            if (o0) look_up(ord);
            bool empty_one = false, copies = false;
            int t0 = 0, t1 = 0;
            if (part < parts) {
                len = min(max(len, 0), cap);
                empty_one = part >= parts_of(len);
                tiles_of(part, len, rv != 0 && len >= cap, t0, t1);
                copies = ord > 0 && t1 > t0;
            }
            const unsigned me = __ballot_sync(0xffffffffu, empty_one), mc = __ballot_sync(0xffffffffu, copies);
            if (copies) {
                const int at = n + __popc(mc & ((1u << lane) - 1u));
                s_pair[at] = pr;
                s_tiles[at] = make_int2(t0, t1);
                s_len[at] = len;
            }
            if (kVaried && lane == 0) s_empty[o0 >> 5] = me;
            n += __popc(mc);
        }
        __syncwarp();
        if (lane != 0) return;
        mbar_arrive(&looked);                            // (a release: no length is read behind it)
        for (int i = 0; ok; ++i) {
            if (t < t_end) issue();
            int bh_next = 0, n_next = 0;                 // (while that tile travels)
            int2 t_next = make_int2(0, 0);
            if (i < n) { bh_next = s_pair[i]; n_next = s_len[i]; t_next = s_tiles[i]; }
            while (t < t_end && ok) issue();
            if (i >= n) break;
            bh = bh_next; n_old = n_next; t = t_next.x; t_end = t_next.y;
        }
        for (int u = max(0, it - kStages); u < it; ++u)  // no copy in flight when the CTA retires, aborted or not
            mbar_wait_drain(&full[u % kStages], (u / kStages) & 1);
        return;
    }

    if (warp == kWarps + 1) {
        // ---------------- finisher warp: merges what the work warps leave per item; the last item of a
        // (sequence, head) anywhere finishes the step.  Lane l owns columns V l .. V l + V - 1. ----------------
        constexpr int V = D / 32, kLs = 32 / G;          // columns per lane, lanes per softmax head
        constexpr int kPs = D + kPartHead;
        auto slice_sum = [&](float x) {
#pragma unroll
            for (int o = kLs / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            return x;
        };
        const int sg = lane / kLs;
        int32_t *tickets = reinterpret_cast<int32_t *>(ws + dec_off_tickets());
        const bool known = mbar_wait(&looked, 0, abort_flag) && (!kVaried || mbar_wait(&first_read, 0, abort_flag));
        // The empty items' tickets, a lane each; who gets a pair's last one finishes it when its place in the order comes.
        // (After a time-out, which is reported, all of the CTA's tickets are still taken, so that they end at zero.)
        for (int o0 = 0; kVaried && known && has(o0); o0 += 32) {
            const int ord = o0 + lane;
            bool closes = false;
            if (has(ord) && empty_item(ord)) {
                int pt, pr;
                locate(item_no(ord), pt, pr);
                closes = atom_add_acq_rel(tickets + pr, 1) == per_head - 1;
            }
            const unsigned m = __ballot_sync(0xffffffffu, closes);
            if (lane == 0) s_closed[o0 >> 5] = m;
        }
        __syncwarp();
#pragma unroll 1
        for (int i = 0, ord = 0; has(ord); ++ord) {
            const bool turn = !kVaried || !known || !__any_sync(0xffffffffu, empty_item(ord));
            if (!turn && !__any_sync(0xffffffffu, (s_closed[ord >> 5] >> (ord & 31)) & 1u)) continue;
            int part, bh;
            locate(item_no(ord), part, bh);
            int32_t *ticket = tickets + bh;
            float *partials = reinterpret_cast<float *>(ws + dec_off_partials(BH, D)) + (size_t)bh * parts * kPs;
            float *ola_ws = reinterpret_cast<float *>(ws + dec_off_ola(BH)) + (size_t)bh * D;
            const float *sc = slot_of(i & 1);
            const bool ok = turn && mbar_wait(&done[i & 1], (i >> 1) & 1, abort_flag);
            if (!ok) {
            } else if (part < parts) {                   // eight warps' (m, z, acc) -> one partial
                float M = -INFINITY, Z = 0.f, o[V];
#pragma unroll
                for (int x = 0; x < V; ++x) o[x] = 0.f;
                const float2 *mzs = mz + (i & 1) * kWarps * G;
#pragma unroll
                for (int wv = 0; wv < kWarps; ++wv) M = fmaxf(M, mzs[wv * G + sg].x);
                const float Mu = M == -INFINITY ? 0.f : M;
#pragma unroll
                for (int wv = 0; wv < kWarps; ++wv) {
                    const float2 e = mzs[wv * G + sg];
                    const float f = ex2_ftz(e.x - Mu);
                    Z = fmaf(e.y, f, Z);
#pragma unroll
                    for (int x = 0; x < V; ++x) o[x] = fmaf(sc[wv * D + lane * V + x], f, o[x]);
                }
                float *pp = partials + (size_t)part * kPs;
#pragma unroll
                for (int x = 0; x < V; ++x) pp[kPartHead + lane * V + x] = o[x];
                if (lane % kLs == 0) { pp[sg] = M; pp[4 + sg] = Z; }
            } else {                                     // the row slots' shares of this half of the read-out
                constexpr int kVc = (kCols + 31) / 32;
                float a[kVc];
#pragma unroll
                for (int x = 0; x < kVc; ++x) a[x] = 0.f;
#pragma unroll 8
                for (int sl = 0; sl < kSlots; ++sl)
#pragma unroll
                    for (int x = 0; x < kVc; ++x) a[x] += sc[sl * kCols + lane * kVc + x];
#pragma unroll
                for (int x = 0; x < kVc; ++x) ola_ws[(part - parts) * kCols + lane * kVc + x] = scale_la * a[x];
            }
            // ticket (release by lane 0 behind the warp's barrier, acquire by it before the warp's barrier)
            __syncwarp();
            int last = !turn;
            if (lane == 0) {
                if (turn) {
                    mbar_arrive(&taken[i & 1]);
                    last = atom_add_acq_rel(ticket, 1) == per_head - 1;
                }
                if (last) *ticket = 0;                   // ready for the next step
            }
            i += turn;
            last = __shfl_sync(0xffffffffu, last, 0);
            if (!last) continue;
            // All of the pair's partial results and the token's rows in one round trip.
            float pa[kMaxParts][V], ol[V], qv[V], kv[V], vv[V], pm[G], pz[G];
#pragma unroll
            for (int pt = 0; pt < kMaxParts; ++pt)
#pragma unroll
                for (int x = 0; x < V; ++x)
                    pa[pt][x] = pt < parts ? __ldcg(partials + pt * kPs + kPartHead + lane * V + x) : 0.f;
#pragma unroll
            for (int a = 0; a < G; ++a) {
                pm[a] = lane < parts ? __ldcg(partials + lane * kPs + a) : -INFINITY;
                pz[a] = lane < parts ? __ldcg(partials + lane * kPs + 4 + a) : 0.f;
            }
            const int rv = route[bh], n_raw = cache_len[bh];
#pragma unroll
            for (int x = 0; x < V; ++x) {
                ol[x] = __ldcg(ola_ws + lane * V + x);
                qv[x] = to_f32(q[(size_t)bh * D + lane * V + x]);
                kv[x] = to_f32(k[(size_t)bh * D + lane * V + x]);
                vv[x] = to_f32(v[(size_t)bh * D + lane * V + x]);
            }
            const float wn = w ? w[(size_t)bh * 2] : 0.5f, wl = w ? w[(size_t)bh * 2 + 1] : 0.5f;
            const bool r = rv != 0;                      // append, and attend to itself
            const int n_old = min(max(n_raw, 0), cap), np = parts_of(n_old);
#pragma unroll
            for (int a = 0; kVaried && a < G; ++a) {     // (partials of empty items are another step's)
                if (lane >= np) { pm[a] = -INFINITY; pz[a] = 0.f; }
            }
            if (n_raw != n_old && lane == 0) atomicMin(status, (int)NATSL_ERR_CACHE_FULL);
            if (r && n_old >= cap) {                     // no room: the sequence is left untouched
#pragma unroll
                for (int x = 0; x < V; ++x) out[(size_t)bh * D + lane * V + x] = from_f32<T>(0.f);
                if (lane == 0) atomicMin(status, (int)NATSL_ERR_CACHE_FULL);
                continue;
            }
            float qq = 0.f, kk = 0.f, self = 0.f;
#pragma unroll
            for (int x = 0; x < V; ++x) {
                qq = fmaf(qv[x], qv[x], qq);
                kk = fmaf(kv[x], kv[x], kk);
                self = fmaf(qv[x], kv[x], self);
            }
            self = slice_sum(self) * scale_sm * kLog2e;
            if (kNorm) self *= rsqrtf(slice_sum(qq) / ds + norm_eps) * rsqrtf(slice_sum(kk) / ds + norm_eps);
            if (!r) self = -INFINITY;                    // (the token attends to itself when it is retained)
            float M = self, Z = 0.f, pf[G], on[V];
#pragma unroll
            for (int a = 0; a < G; ++a) {
                const float Ma = warp_max(pm[a]);
                if (a == sg) M = fmaxf(M, Ma);
            }
            const float Mu = M == -INFINITY ? 0.f : M;
#pragma unroll
            for (int a = 0; a < G; ++a) {
                pf[a] = ex2_ftz(pm[a] - __shfl_sync(0xffffffffu, Mu, a * kLs));
                const float Za = warp_sum(pz[a] * pf[a]);
                if (a == sg) Z = Za;
            }
            const float fs = ex2_ftz(self - Mu);
            Z += fs;
#pragma unroll
            for (int x = 0; x < V; ++x) on[x] = vv[x] * fs;
#pragma unroll
            for (int pt = 0; pt < kMaxParts; ++pt) {
                if (pt >= parts) break;
                float f = __shfl_sync(0xffffffffu, pf[0], pt);
#pragma unroll
                for (int a = 1; a < G; ++a) {
                    const float fa = __shfl_sync(0xffffffffu, pf[a], pt);
                    if (a == sg) f = fa;
                }
#pragma unroll
                for (int x = 0; x < V; ++x) on[x] = fmaf(!kVaried || pt < np ? pa[pt][x] : 0.f, f, on[x]);
            }
            const float iz = Z > 0.f ? 1.f / Z : 0.f;    // (no visible key: o_nla = 0)
            float tn = 0.f, tl = 0.f;
#pragma unroll
            for (int x = 0; x < V; ++x) {
                on[x] *= iz;
                tn = fmaf(on[x], on[x], tn);
                tl = fmaf(ol[x], ol[x], tl);
            }
            const float fn = wn * rsqrtf(slice_sum(tn) / ds + eps), fl = wl * rsqrtf(warp_sum(tl) / D + eps);
#pragma unroll
            for (int x = 0; x < V; ++x) {
                out[(size_t)bh * D + lane * V + x] = from_f32<T>(fn * on[x] + fl * ol[x]);
                if (r) {   // retain the token: every reader of the old length has finished
                    k_cache[((size_t)bh * cap + n_old) * D + lane * V + x] = from_f32<T>(kv[x]);
                    v_cache[((size_t)bh * cap + n_old) * D + lane * V + x] = from_f32<T>(vv[x]);
                }
            }
            if (r && lane == 0) cache_len[bh] = n_old + 1;
        }
        if (lane == 0 && s_abort[0]) atomicMin(status, (int)NATSL_ERR_TIMEOUT);
        return;
    }

    int it = 0;                                          // tiles consumed so far
#pragma unroll 1
    for (int i = 0, ord = 0; has(ord); ++i, ++ord) {
        if (kVaried && ord) {
            // (after a time-out: go on, for the warps meet at the state items' barriers; what is not looked up gets a turn)
            if (ord == 1) (void)mbar_wait(&looked, 0, abort_flag);
            if (__any_sync(0xffffffffu, empty_item(ord))) { --i; continue; }
        }
        int part, bh;
        locate(item_no(ord), part, bh);
        // route 0: linear token (delta rule); 1: softmax token (appended to the cache); 2: token of a
        // block whose decision is still open -- both (Section 4.1, pseudo-update of both hidden states)
        const int rv = route[bh], n_raw = cache_len[bh];
        if (kVaried && ord == 0) {
            const bool none = __any_sync(0xffffffffu, part < parts && part >= parts_of(min(max(n_raw, 0), cap)));
            if (lane == 0) mbar_arrive(&first_read);
            if (none) { --i; continue; }
        }
        float *slot_out = slot_of(i & 1);
        if (part < parts) {
            // ---------------- cache item: one slice of the retained K/V ----------------
            const int row = warp * 4 + (lane >> 3), l8 = lane & 7;
            uint64_t qf[kJ][kE / 2], acc[kJ][kE / 2];
            float m[kLg], z[kLg];
            {
                float qx[kJ][kE];
#pragma unroll
                for (int j = 0; j < kJ; ++j)
                    Vec16<T>::unpack(__ldg(reinterpret_cast<const uint4 *>(q + (size_t)bh * D) + j * 8 + l8), qx[j]);
#pragma unroll
                for (int a = 0; a < kLg; ++a) {
                    float f = scale_sm * kLog2e;
                    if (kNorm) {                         // RMS over the softmax head's columns
                        float ss = 0.f;
#pragma unroll
                        for (int jj = 0; jj < kJpl; ++jj)
#pragma unroll
                            for (int x = 0; x < kE; ++x) ss = fmaf(qx[a * kJpl + jj][x], qx[a * kJpl + jj][x], ss);
#pragma unroll
                        for (int o = kLanes / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                        f *= rsqrtf(ss / ds + norm_eps);
                    }
#pragma unroll
                    for (int jj = 0; jj < kJpl; ++jj)
#pragma unroll
                        for (int x = 0; x < kE / 2; ++x) {
                            const int j = a * kJpl + jj;
                            qf[j][x] = pack2(qx[j][2 * x] * f, qx[j][2 * x + 1] * f);
                            acc[j][x] = 0ull;
                        }
                    m[a] = -INFINITY;
                    z[a] = 0.f;
                }
            }
            const int n_old = min(max(n_raw, 0), cap);
            int t, t_end;
            tiles_of(part, n_old, rv != 0 && n_old >= cap, t, t_end);
            bool ok = true;
            for (; t < t_end; ++t, ++it) {
                const int st = it % kStages;
                ok = mbar_wait(&full[st], (it / kStages) & 1, abort_flag);
                if (!ok) break;
                const uint8_t *kt = smem + (2 * st) * kTileBytes + row * kRowBytes + l8 * 16, *vt = kt + kTileBytes;
                const bool valid = t * kTileKeys + row < n_old;     // (rows past the slice hold stale bytes)
                float sc[kLg], kk[kLg];
#pragma unroll
                for (int a = 0; a < kLg; ++a) {
                    uint64_t s2 = 0ull, k2 = 0ull;
#pragma unroll
                    for (int jj = 0; jj < kJpl; ++jj) {
                        const int j = a * kJpl + jj;
                        float kx[kE];
                        Vec16<T>::unpack(*reinterpret_cast<const uint4 *>(kt + j * 128), kx);
#pragma unroll
                        for (int x = 0; x < kE / 2; ++x) {
                            const uint64_t kp = pack2(kx[2 * x], kx[2 * x + 1]);
                            s2 = fma2(qf[j][x], kp, s2);
                            if (kNorm) k2 = fma2(kp, kp, k2);      // the key's sum of squares rides along
                        }
                    }
                    const float2 sf = unpack2(s2), kf = unpack2(k2);
                    sc[a] = sf.x + sf.y;
                    kk[a] = kf.x + kf.y;
                }
                uint4 vraw[kJ];
#pragma unroll
                for (int j = 0; j < kJ; ++j) vraw[j] = *reinterpret_cast<const uint4 *>(vt + j * 128);
#pragma unroll
                for (int o = kLanes / 2; o > 0; o >>= 1)
#pragma unroll
                    for (int a = 0; a < kLg; ++a) {
                        sc[a] += __shfl_xor_sync(0xffffffffu, sc[a], o);
                        if (kNorm) kk[a] += __shfl_xor_sync(0xffffffffu, kk[a], o);
                    }
                if (lane == 0) mbar_arrive(&empty[st]);  // (behind the shuffles: every lane's reads are done)
                bool raise = false;
#pragma unroll
                for (int a = 0; a < kLg; ++a) {
                    if (kNorm) sc[a] *= rsqrtf(fmaf(kk[a], 1.f / ds, norm_eps));
                    raise |= valid && sc[a] > m[a] + 8.f;
                }
                if (__any_sync(0xffffffffu, raise)) {
#pragma unroll
                    for (int a = 0; a < kLg; ++a) {
                        const float m_new = valid ? fmaxf(m[a], sc[a]) : m[a];
                        const float corr = m[a] == m_new ? 1.f : ex2_ftz(m[a] - m_new);
                        z[a] *= corr;
                        m[a] = m_new;
                        const uint64_t c2 = pack2(corr, corr);
#pragma unroll
                        for (int jj = 0; jj < kJpl; ++jj)
#pragma unroll
                            for (int x = 0; x < kE / 2; ++x) acc[a * kJpl + jj][x] = mul2(acc[a * kJpl + jj][x], c2);
                    }
                }
                if (valid) {
#pragma unroll
                    for (int a = 0; a < kLg; ++a) {
                        const float pj = ex2_ftz(sc[a] - m[a]);
                        z[a] += pj;
                        const uint64_t p2 = pack2(pj, pj);
#pragma unroll
                        for (int jj = 0; jj < kJpl; ++jj) {
                            const int j = a * kJpl + jj;
                            float vx[kE];
                            Vec16<T>::unpack(vraw[j], vx);
#pragma unroll
                            for (int x = 0; x < kE / 2; ++x) acc[j][x] = fma2(p2, pack2(vx[2 * x], vx[2 * x + 1]), acc[j][x]);
                        }
                    }
                }
            }
            // the four rows of the warp by shuffles, then the warp's (m, z, acc) to the item's slot
            // (after a time-out: go on without it, the other warps count on this one at the state items' barriers)
            if (!ok || !mbar_wait(&taken[i & 1], ((i >> 1) & 1) ^ 1, abort_flag)) continue;
#pragma unroll
            for (int a = 0; a < kLg; ++a) {
                float M = fmaxf(m[a], __shfl_xor_sync(0xffffffffu, m[a], 8));
                M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 16));
                const float f = m[a] == -INFINITY ? 0.f : ex2_ftz(m[a] - M);
                z[a] *= f;
                z[a] += __shfl_xor_sync(0xffffffffu, z[a], 8);
                z[a] += __shfl_xor_sync(0xffffffffu, z[a], 16);
                if (lane < 8 && l8 % kLanes == 0)
                    mz[((i & 1) * kWarps + warp) * G + (kSp >= 8 ? a : 2 * a + (l8 >> 2))] = make_float2(M, z[a]);
#pragma unroll
                for (int jj = 0; jj < kJpl; ++jj) {
                    const int j = a * kJpl + jj;
#pragma unroll
                    for (int x = 0; x < kE / 2; ++x) {
                        float2 y = unpack2(acc[j][x]);
                        y.x *= f;
                        y.y *= f;
                        y.x += __shfl_xor_sync(0xffffffffu, y.x, 8);
                        y.y += __shfl_xor_sync(0xffffffffu, y.y, 8);
                        y.x += __shfl_xor_sync(0xffffffffu, y.x, 16);
                        y.y += __shfl_xor_sync(0xffffffffu, y.y, 16);
                        if (lane < 8) *reinterpret_cast<float2 *>(&slot_out[warp * D + (j * 8 + l8) * kE + 2 * x]) = y;
                    }
                }
            }
        } else {
            // ---------------- state item: half of the value columns, all rows ----------------
            // (warp-local operands: row slot `slot` holds rows slot kR ..; its k and q values, the token's
            // norms and the v values come straight from global memory, in flight together with the state)
            const int c0 = (part - parts) * kCols;
            const int slot = warp * kRpl + lane / kLpr, col = (lane % kLpr) * 4;
            float *sp = state + (size_t)bh * D * D + c0 + (size_t)(slot * kR) * D + col;
            float4 s[kR];
#pragma unroll
            for (int rr = 0; rr < kR; ++rr) s[rr] = *reinterpret_cast<const float4 *>(sp + (size_t)rr * D);
            float kx[kR], qx[kR], vx[4];
#pragma unroll
            for (int rr = 0; rr < kR; ++rr) {
                kx[rr] = to_f32(k[(size_t)bh * D + slot * kR + rr]);
                qx[rr] = to_f32(q[(size_t)bh * D + slot * kR + rr]);
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) vx[x] = to_f32(v[(size_t)bh * D + c0 + col + x]);
            const float alpha = __expf(g[bh]), bt = beta[bh];
            if (kNorm) {                                 // L2 over the row (the linear operation's q, k)
                float sq = 0.f, sk = 0.f;
#pragma unroll
                for (int x = 0; x < D / 32; ++x) {
                    const float a = to_f32(q[(size_t)bh * D + lane + 32 * x]), b = to_f32(k[(size_t)bh * D + lane + 32 * x]);
                    sq = fmaf(a, a, sq);
                    sk = fmaf(b, b, sk);
                }
                const float rq = rsqrtf(warp_sum(sq) + norm_eps), rk = rsqrtf(warp_sum(sk) + norm_eps);
#pragma unroll
                for (int rr = 0; rr < kR; ++rr) { qx[rr] *= rq; kx[rr] *= rk; }
            }
            const bool skip = rv != 0 && min(max(n_raw, 0), cap) >= cap;   // no room: left untouched
            const bool fold = rv != 1;                                     // delta rule
            float (*redv)[kCols] = reinterpret_cast<float (*)[kCols]>(slot_of(2));   // [kSlots][kCols]
#pragma unroll
            for (int rr = 0; rr < kR; ++rr) {
                s[rr].x *= alpha; s[rr].y *= alpha; s[rr].z *= alpha; s[rr].w *= alpha;
            }
            if (fold) {   // uniform over the CTA
                float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int rr = 0; rr < kR; ++rr) {
                    p.x = fmaf(kx[rr], s[rr].x, p.x); p.y = fmaf(kx[rr], s[rr].y, p.y);
                    p.z = fmaf(kx[rr], s[rr].z, p.z); p.w = fmaf(kx[rr], s[rr].w, p.w);
                }
                *reinterpret_cast<float4 *>(&redv[slot][col]) = p;
                named_barrier_sync(1, kWorkThreads);
                float4 e = make_float4(vx[0], vx[1], vx[2], vx[3]);
#pragma unroll
                for (int sl = 0; sl < kSlots; ++sl) {
                    const float4 t = *reinterpret_cast<const float4 *>(&redv[sl][col]);
                    e.x -= t.x; e.y -= t.y; e.z -= t.z; e.w -= t.w;
                }
#pragma unroll
                for (int rr = 0; rr < kR; ++rr) {
                    const float bk = bt * kx[rr];
                    s[rr].x = fmaf(bk, e.x, s[rr].x); s[rr].y = fmaf(bk, e.y, s[rr].y);
                    s[rr].z = fmaf(bk, e.z, s[rr].z); s[rr].w = fmaf(bk, e.w, s[rr].w);
                }
                named_barrier_sync(1, kWorkThreads);     // (redv is written again by the next state item)
            }
            float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int rr = 0; rr < kR; ++rr) {
                p.x = fmaf(qx[rr], s[rr].x, p.x); p.y = fmaf(qx[rr], s[rr].y, p.y);
                p.z = fmaf(qx[rr], s[rr].z, p.z); p.w = fmaf(qx[rr], s[rr].w, p.w);
                if (!skip) *reinterpret_cast<float4 *>(sp + (size_t)rr * D) = s[rr];
            }
            if (!mbar_wait(&taken[i & 1], ((i >> 1) & 1) ^ 1, abort_flag)) continue;
            *reinterpret_cast<float4 *>(&slot_out[slot * kCols + col]) = p;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&done[i & 1]);
    }
}

// End of a block of R tokens decoded with the decision open: a softmax block resets the state to
// its value at the block's start times the block's decay (the block's K/V stay in the cache); a
// linear block keeps the state and drops its R cache entries.  state_start then holds the new
// state: the start of the next block.  One CTA per (sequence, head).
__global__ void __launch_bounds__(256)
decode_block_end_kernel(const uint8_t *__restrict__ route_block, const float *__restrict__ g_block,
                        float *__restrict__ state, float *__restrict__ state_start,
                        int32_t *__restrict__ cache_len, int R, int n4, int32_t *status) {
    const int bh = blockIdx.x;
    float4 *S = reinterpret_cast<float4 *>(state) + (size_t)bh * n4;
    float4 *S0 = reinterpret_cast<float4 *>(state_start) + (size_t)bh * n4;
    if (route_block[bh]) {
        const float decay = expf(g_block[bh]);
        for (int i = threadIdx.x; i < n4; i += blockDim.x) {
            float4 a = S0[i];
            a.x *= decay; a.y *= decay; a.z *= decay; a.w *= decay;
            S[i] = a;
            S0[i] = a;
        }
    } else {
        for (int i = threadIdx.x; i < n4; i += blockDim.x) S0[i] = S[i];
        if (threadIdx.x == 0) {
            const int n = cache_len[bh];
            if (n < R) atomicMin(status, (int)NATSL_ERR_ROUTE);   // the block's entries are not there
            else cache_len[bh] = n - R;
        }
    }
}

}  // namespace

cudaError_t launch_decode_block_end(const uint8_t *route_block, const float *g_block, float *state,
                                    float *state_start, int32_t *cache_len, int32_t block_len,
                                    void *ws, Shape s, cudaStream_t st) {
    decode_block_end_kernel<<<s.B * s.H, 256, 0, st>>>(route_block, g_block, state, state_start,
                                                       cache_len, block_len, s.d * s.d / 4,
                                                       reinterpret_cast<int32_t *>(ws));
    count_launch();
    return cudaGetLastError();
}

size_t decode_workspace_bytes(int B, int H, int d) {
    const size_t BH = (size_t)B * H;
    return dec_off_partials(BH, d) + (BH * kMaxParts * (d + kPartHead) * 4 + 255) / 256 * 256;
}

template <typename T, int D, int G, bool kNorm>
static cudaError_t decode_impl(const void *q, const void *k, const void *v, const float *g,
                               const float *beta, const uint8_t *route, const float *w,
                               float *state, void *k_cache, void *v_cache, int32_t *cache_len,
                               int32_t cap, void *out, float scale_la, float scale_sm, float eps,
                               void *ws, Shape s, cudaStream_t st, float norm_eps) {
    if constexpr (D / G * (int)sizeof(T) < 64) {
        return cudaErrorInvalidValue;
    } else {
        const int BH = s.B * s.H, resident = kCtasPerSm * sm_count();
        const DecSplit split = decode_split(BH, resident, cap);
        const int per_head = split.parts + kStateParts;
        auto kernel = split.varied ? decode_step_kernel<T, D, G, kNorm, true> : decode_step_kernel<T, D, G, kNorm, false>;
        cudaError_t e = allow_smem(kernel, DecLayout<T, D, G>::kTotal);
        if (e != cudaSuccess) return e;
        // Persistent beyond one resident set, up to the items a CTA can list; the stride then has no factor in common with
        // the items per pair (of the front), so that every CTA gets the same mix of cache and state items.
        auto gcd = [](int a, int b) { while (b) { const int c = a % b; a = b; b = c; } return a; };
        int grid = BH * per_head;
        if (grid > resident) {
            const int least = (grid + kMaxItems - 1) / kMaxItems;
            grid = resident;
            while (grid > 1 && gcd(grid, split.front + kStateParts) != 1) --grid;
            if (grid < least)
                for (grid = least; gcd(grid, split.front + kStateParts) != 1;) ++grid;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = DecLayout<T, D, G>::kTotal;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, kernel, (const T *)q, (const T *)k, (const T *)v, g, beta, route, w, state,
                               (T *)k_cache, (T *)v_cache, cache_len, (int)cap, (T *)out, scale_la, scale_sm, eps,
                               (uint8_t *)ws, BH, split, norm_eps);
        count_launch();
        return e;
    }
}

cudaError_t launch_decode_step(const void *q, const void *k, const void *v, const float *g,
                               const float *beta, const uint8_t *route, const float *w,
                               float *state, void *k_cache, void *v_cache, int32_t *cache_len,
                               int32_t cache_cap, void *out, float scale_la, float scale_sm,
                               float eps, void *ws, Shape s, cudaStream_t st, HeadGroups hg) {
#define ARGS q, k, v, g, beta, route, w, state, k_cache, v_cache, cache_len, cache_cap, out, \
             scale_la, scale_sm, eps, ws, s, st, hg.norm_eps
#define BY_GROUPS(T, D)                                                                                     \
    if (hg.norm_eps >= 0.f) {                                                                               \
        if (hg.G == 4) return decode_impl<T, D, 4, true>(ARGS);                                             \
        if (hg.G == 2) return decode_impl<T, D, 2, true>(ARGS);                                             \
        if (hg.G == 1) return decode_impl<T, D, 1, true>(ARGS);                                             \
    } else {                                                                                                \
        if (hg.G == 4) return decode_impl<T, D, 4, false>(ARGS);                                            \
        if (hg.G == 2) return decode_impl<T, D, 2, false>(ARGS);                                            \
        if (hg.G == 1) return decode_impl<T, D, 1, false>(ARGS);                                            \
    }                                                                                                       \
    return cudaErrorInvalidValue
    if (s.bf16) {
        if (s.d == 128) { BY_GROUPS(__nv_bfloat16, 128); }
        BY_GROUPS(__nv_bfloat16, 64);
    }
    if (s.d == 128) { BY_GROUPS(float, 128); }
    BY_GROUPS(float, 64);
#undef BY_GROUPS
#undef ARGS
}

}  // namespace natsl
