// The part that the two gather kernels of the forward share: a CTA of grid = (slices of the chunks, B*H) lists its own
// chunks' retained tokens, finds out how many lie before them and walks over their rows.
#pragma once
#include "common.cuh"

namespace natsl {

constexpr int kRouteThreads = 256;
constexpr int kMaxSlice = 32;                        // chunks per CTA

struct RouteLists {                                  // in shared memory
    int list[kMaxSlice * kC];                        // a chunk's retained tokens, compacted within its 64 places
    int counts[kMaxSlice], wsum[kRouteThreads / 32];
};
struct RouteSlice {
    int c_lo, nc;                                    // first chunk, chunks
    int base, mine;                                  // entries before the slice, retained tokens in it
    bool mixed;                                      // a chunk seen by this thread's warp holds tokens of both kinds
};

// One 64-bit ballot word per chunk of the slice; what lies before it is counted by the CTA itself, route bytes out of L2:
// a few microseconds however long the sequence (one CTA per (batch, head) walking all chunks took 28 us at 512).
// rt: route + (first token of the batch) H + h.  prefix [L/C + 1] of the pair: entries before each chunk, base0 of them from
// earlier calls.
__device__ __forceinline__ RouteSlice list_slice(RouteLists &rl, const uint8_t *rt, int32_t *prefix, int base0,
                                                 int slice_chunks, int NC, int H) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    RouteSlice sl;
    sl.c_lo = blockIdx.x * slice_chunks;
    sl.nc = min(slice_chunks, NC - sl.c_lo);
    sl.mixed = false;
    for (int c = warp; c < sl.nc; c += kRouteThreads / 32) {
        const size_t l0 = (size_t)(sl.c_lo + c) * kC;
        const uint8_t a0 = rt[(l0 + lane) * H], a1 = rt[(l0 + 32 + lane) * H];
        const unsigned lo = __ballot_sync(0xffffffffu, a0 != 0), hi = __ballot_sync(0xffffffffu, a1 != 0);
        const unsigned lt = (1u << lane) - 1u;
        const int nlo = __popc(lo), n = nlo + __popc(hi);
        if (a0) rl.list[c * kC + __popc(lo & lt)] = (int)l0 + lane;
        if (a1) rl.list[c * kC + nlo + __popc(hi & lt)] = (int)l0 + 32 + lane;
        sl.mixed |= n != 0 && n != kC;
        if (lane == 0) rl.counts[c] = n;
    }
    int before = 0;
    const int n_before = sl.c_lo * kC;
    for (int l = tid; l < n_before; l += 8 * kRouteThreads) {                 // eight loads in flight
        uint8_t x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int ll = l + u * kRouteThreads;
            x[u] = ll < n_before ? rt[(size_t)ll * H] : (uint8_t)0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) before += x[u] != 0;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) rl.wsum[warp] = before;
    __syncthreads();
    sl.base = base0;
#pragma unroll
    for (int wv = 0; wv < kRouteThreads / 32; ++wv) sl.base += rl.wsum[wv];
    sl.mine = 0;
    for (int c = 0; c < sl.nc; ++c) sl.mine += rl.counts[c];
    if (tid < sl.nc) {
        int pre = sl.base;
        for (int c = 0; c < tid; ++c) pre += rl.counts[c];
        prefix[sl.c_lo + tid] = pre;
    }
    if (sl.c_lo + sl.nc == NC && tid == 0) prefix[NC] = sl.base + sl.mine;
    return sl;
}

// copy(entry, token) for the slice's retained tokens: each group of kLanes threads takes every (256 / kLanes)-th one
template <int kLanes, typename F> __device__ __forceinline__ void for_each_row(const RouteLists &rl, const RouteSlice &sl, F copy) {
    int row0 = sl.base, c = 0, in_c = threadIdx.x / kLanes;                   // in_c: index within chunk c's list
    while (true) {
        while (c < sl.nc && in_c >= rl.counts[c]) { in_c -= rl.counts[c]; row0 += rl.counts[c]; ++c; }
        if (c >= sl.nc) break;
        copy(row0 + in_c, rl.list[c * kC + in_c]);
        in_c += kRouteThreads / kLanes;
    }
}

// Chunks per slice for about ctas_per_sm CTAs on each of 148 multiprocessors over all (batch, head) pairs, at most 32 slices
// per pair (each counts what lies before it).
inline int slice_chunks_of(int NC, int BH, int ctas_per_sm) {
    int slices = (ctas_per_sm * 148 + BH - 1) / BH;
    slices = slices > 32 ? 32 : slices;
    const int cps = (NC + slices - 1) / slices;
    return cps > kMaxSlice ? kMaxSlice : cps;
}

}  // namespace natsl
