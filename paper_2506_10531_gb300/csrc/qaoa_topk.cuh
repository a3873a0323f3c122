// qaoa_topk.cuh -- block-wide top-k selection for the reductions over states and lists in global
// memory (blocks of TK_NT = 256 threads): a lower bound from the threads' maxima, the few entries
// that reach it collected in shared memory, and their ranks. A list of k entries is unique under
// (probability descending, index ascending), so the result does not depend on the order of the
// collection.
#pragma once
#include "qaoa_common.cuh"

namespace qaoa {

constexpr int TK_NT = 256;
constexpr int TK_CAP = 256;   // collected entries; more (massive ties): kth_collected

struct __align__(16) TopScratch {
    float wb[16 * (TK_NT / 32)];
    TopEnt cand[TK_CAP];
    TopEnt wl[(TK_NT / 32) * 32];
    TopEnt run[16];             // the result: k entries, empty ones hold probability -1
    TopEnt kth;
    float bound;
    int cnt, over;
};
constexpr int TK_RETRY = 4;   // collections after an overflow, each above a better bound, before sorted insertion

// The k-th largest (1 <= k <= 16) of one value per thread of the block: every warp offers its k
// largest and the k-th largest of those is found by rank. Also clears the collection counters.
__device__ __forceinline__ float block_kth_largest(float v, int k, TopScratch& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float srt = warp_sort_desc(v);
    if (lane < k) s.wb[warp * k + lane] = srt;
    if (threadIdx.x == 0) { s.cnt = 0; s.over = 0; }
    __syncthreads();
    const int nl = (TK_NT / 32) * k;   // a multiple of 8
    if ((int)threadIdx.x < nl) {
        const float me = s.wb[threadIdx.x];
        const int t = (int)threadIdx.x;
        const float4* w4 = reinterpret_cast<const float4*>(s.wb);
        int rank = 0;
#pragma unroll 4
        for (int q4 = 0; q4 < nl / 4; ++q4) {
            const float4 o = w4[q4];
            const int q = 4 * q4;
            rank += (o.x > me || (o.x == me && q < t)) ? 1 : 0;
            rank += (o.y > me || (o.y == me && q + 1 < t)) ? 1 : 0;
            rank += (o.z > me || (o.z == me && q + 2 < t)) ? 1 : 0;
            rank += (o.w > me || (o.w == me && q + 3 < t)) ? 1 : 0;
        }
        if (rank == k - 1) s.bound = me;
    }
    __syncthreads();
    return s.bound;
}

__device__ __forceinline__ void collect_entry(double p, uint32_t z, TopScratch& s) {
    const int pos = atomicAdd(&s.cnt, 1);
    if (pos < TK_CAP) s.cand[pos] = TopEnt{p, z};
    else s.over = 1;
}

// After an overflow (s.over, behind a barrier): the k-th best of the TK_CAP entries that were kept, which
// at least k of all entries are or beat, for another collection; clears the counters. Ties of one
// probability are told apart by their index here, where the FP32 bound cannot, and a warp's sorted insertion
// takes about 1 us per 32 of them (a flat state of n = 21, top-8: 260 us by insertion, 77 so). Called by
// all threads; ends with a barrier.
__device__ __forceinline__ TopEnt kth_collected(int k, TopScratch& s) {
    static_assert(TK_CAP == TK_NT, "an entry per thread");
    const TopEnt me = s.cand[threadIdx.x];
    int rank = 0;
    for (int j = 0; j < TK_CAP; ++j) rank += better(s.cand[j].p, s.cand[j].z, me.p, me.z) ? 1 : 0;
    if (rank == k - 1) s.kth = me;
    __syncthreads();
    if (threadIdx.x == 0) { s.cnt = 0; s.over = 0; }
    const TopEnt t = s.kth;
    __syncthreads();
    return t;
}

// s.run = the k best of the collected entries and, with have_run, the entries of s.run. Called by
// all threads after a barrier that follows the collection; ends with a barrier.
__device__ __forceinline__ void rank_collected(int k, bool have_run, TopScratch& s) {
    const int na = s.cnt, nr = have_run ? k : 0;
    for (int c = threadIdx.x; c < na + nr; c += TK_NT) {
        const TopEnt me = c < na ? s.cand[c] : s.run[c - na];
        int rank = 0;
        for (int j = 0; j < na; ++j) rank += better(s.cand[j].p, s.cand[j].z, me.p, me.z) ? 1 : 0;
        for (int j = 0; j < nr; ++j) rank += better(s.run[j].p, s.run[j].z, me.p, me.z) ? 1 : 0;
        if (rank < k) s.wl[rank] = me;
    }
    // equal empty entries share a rank: the slots past the real entries are filled here
    __syncthreads();
    int real = na;
    for (int j = 0; j < nr; ++j) real += is_entry(s.run[j].p) ? 1 : 0;
    __syncthreads();
    if ((int)threadIdx.x < k) s.run[threadIdx.x] = (int)threadIdx.x < real ? s.wl[threadIdx.x] : TopEnt{-1.0, 0xffffffffu};
    __syncthreads();
}

// s.run = the k best over the block's warps of their sorted lists (one entry per lane < k) and,
// with have_run, the entries of s.run. Called by all threads; ends with a barrier.
__device__ __forceinline__ void merge_warp_lists(const WarpTopK& top, int k, bool have_run, TopScratch& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane < k) s.wl[warp * 32 + lane] = TopEnt{top.p, top.z};
    __syncthreads();
    if (warp == 0) {
        WarpTopK f;
        f.init(k);
        const TopEnt r = (have_run && lane < k) ? s.run[lane] : TopEnt{-1.0, 0xffffffffu};
        f.offer_exact(r.p, r.z, have_run && lane < k);
        for (int w = 0; w < TK_NT / 32; ++w) {
            const bool ok = lane < k;
            const TopEnt e = ok ? s.wl[w * 32 + lane] : TopEnt{-1.0, 0xffffffffu};
            f.offer_exact(e.p, e.z, ok);
        }
        __syncwarp();
        if (lane < k) s.run[lane] = TopEnt{f.p, f.z};
    }
    __syncthreads();
}

// s.run = the k best of nent listed entries, entry e read as at(e) (probability -1: empty). The
// bound is the k-th largest of the threads' maxima rounded down to FP32: k entries reach it, and
// usually little more than k do. Called by all threads; ends with a barrier.
template <typename At>
__device__ __forceinline__ void merge_entries(uint64_t nent, int k, TopScratch& s, At&& at) {
    double best = -1.0;
#pragma unroll 4
    for (uint64_t e = threadIdx.x; e < nent; e += TK_NT) {
        const double p = at(e).p;
        if (pbits(p) > pbits(best)) best = p;
    }
    const float b = block_kth_largest(is_entry(best) ? __double2float_rd(best) : -1.0f, k, s);
    const long long lo = b >= 0.0f ? pbits((double)b) : 0;   // 0: every entry
    if (pbits(best) >= lo) {
        for (uint64_t e = threadIdx.x; e < nent; e += TK_NT) {
            const TopEnt x = at(e);
            if (pbits(x.p) >= lo) collect_entry(x.p, x.z, s);
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int t = 0; s.over && t < TK_RETRY; ++t) {
        const TopEnt b2 = kth_collected(k, s);
        for (uint64_t e = threadIdx.x; e < nent; e += TK_NT) {
            const TopEnt x = at(e);
            if (is_entry(x.p) && !better(b2.p, b2.z, x.p, x.z)) collect_entry(x.p, x.z, s);
        }
        __syncthreads();
    }
    if (!s.over) {
        rank_collected(k, false, s);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpTopK top;
    top.init(k);
    for (uint64_t e0 = (uint64_t)warp * 32; e0 < nent; e0 += TK_NT) {
        const uint64_t e = e0 + lane;
        const TopEnt x = e < nent ? at(e) : TopEnt{-1.0, 0xffffffffu};
        top.offer_exact(x.p, x.z, e < nent);
    }
    merge_warp_lists(top, k, false, s);
}

}  // namespace qaoa
