// k_reduce.cu -- the standalone reductions over a state in HBM: <C> = sum |psi|^2 E (Section IV)
// and the k most probable bitstrings. Blocks of 256 threads take 2048 amplitudes at a time (eight
// per thread, all loads in flight before the first use; FP32 products of those eight, FP64
// above), keep one top-k list each, and a second small kernel merges the blocks' partials; up to
// n = 12 one block does it all and writes the results itself.
// What bounds it: at n = 19 (6 MB, L2) latency -- the loads of one round and the barriers of the
// selection; from about n = 23 HBM. Against one block per 8192
// amplitudes with a serial insertion per candidate and a serial merge: the calls on a single
// n = 19 instance (energies, p = 3, <C>, top-8) 149 -> 100 us together.
#include "qaoa_engine.cuh"
#include "qaoa_stream.h"
#include "qaoa_topk.cuh"

namespace qaoa {

namespace {

constexpr int RPT = 8;                     // amplitudes per thread and round
constexpr uint64_t RCH = TK_NT * RPT;      // amplitudes per block and round

// The round below after its collection overflowed (thousands of amplitudes tie with the bound): collections
// above better bounds, then sorted insertion. A function of its own that reads the amplitudes again, so
// that the round does not hold them for it (inlined, top-8 of a complex128 state of n = 26 took 422 us, 314 so).
template <typename C>
__device__ __noinline__ void topk_round_over(const C* __restrict__ psi, uint64_t z0, uint64_t D, int k, bool have_run,
                                             float lo, TopScratch& s) {
#pragma unroll 1
    for (int t = 0; s.over && t < TK_RETRY; ++t) {
        const TopEnt b = kth_collected(k, s);
#pragma unroll 1
        for (int i = 0; i < RPT; ++i) {
            const uint64_t z = z0 + (uint64_t)i * TK_NT + threadIdx.x;
            if (z >= D) break;
            const C x = psi[z];
            const float pf = (float)x.x * (float)x.x + (float)x.y * (float)x.y;
            if (!(pf * 1.00000095367431640625f >= lo)) continue;
            const double p = exact_prob(x);
            if (!better(b.p, b.z, p, (uint32_t)z) && (!have_run || better(p, (uint32_t)z, s.run[k - 1].p, s.run[k - 1].z)))
                collect_entry(p, (uint32_t)z, s);
        }
        __syncthreads();
    }
    if (!s.over) {
        rank_collected(k, have_run, s);
        return;
    }
    WarpTopK top;
    top.init(k);
#pragma unroll 1
    for (int i = 0; i < RPT; ++i) {
        const uint64_t z = z0 + (uint64_t)i * TK_NT + threadIdx.x;
        C x;
        x.x = x.y = 0;
        if (z < D) x = psi[z];
        top.offer(x, (uint32_t)z, z < D);
    }
    merge_warp_lists(top, k, have_run, s);
}

// One round of the selection over the block's RCH amplitudes: s.run (valid with have_run) becomes
// the k best of itself and the amplitudes v[i] at z0 + i * TK_NT + tid (those < D). An FP32
// test with the margins of WarpTopK::offer comes first; FP64 runs for the few that pass.
template <typename C>
__device__ __forceinline__ void topk_round(const C (&v)[RPT], const C* __restrict__ psi, uint64_t z0, uint64_t D, int k,
                                           bool have_run, TopScratch& s) {
    float pf[RPT], pmax = -1.0f;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const bool in = z0 + (uint64_t)i * TK_NT + threadIdx.x < D;
        pf[i] = in ? (float)v[i].x * (float)v[i].x + (float)v[i].y * (float)v[i].y : -2.0f;
        pmax = fmaxf(pmax, pf[i]);
    }
    float lo;
    if (have_run) {
        lo = is_entry(s.run[k - 1].p) ? __double2float_rd(s.run[k - 1].p) * 0.99999904632568359375f : -1.0f;   // (1 - 2^-20)
        if (threadIdx.x == 0) { s.cnt = 0; s.over = 0; }
        if (!__syncthreads_or(pmax * 1.00000095367431640625f >= lo)) return;
    } else {
        const float b = block_kth_largest(pmax, k, s);
        lo = b > 0.0f ? b * 0.99999904632568359375f : -1.0f;
    }
    if (pmax * 1.00000095367431640625f >= lo) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            if (!(pf[i] * 1.00000095367431640625f >= lo)) continue;
            const uint32_t z = (uint32_t)(z0 + (uint64_t)i * TK_NT + threadIdx.x);
            const double p = exact_prob(v[i]);
            if (!have_run || better(p, z, s.run[k - 1].p, s.run[k - 1].z)) collect_entry(p, z, s);
        }
    }
    __syncthreads();
    if (s.over) topk_round_over(psi, z0, D, k, have_run, lo, s);
    else rank_collected(k, have_run, s);
}

// expect / topk: what is wanted. One block (gridDim.x == 1) writes expect_out, idx_out, prob_out;
// else the partials.
template <typename T, bool EXPECT, bool TOPK>
__global__ void __launch_bounds__(TK_NT) k_reduce_state(int n, const typename Num<T>::C* __restrict__ psi,
                                                        const T* __restrict__ E, int k, double* part_expect,
                                                        double* part_topp, uint32_t* part_topz, double* expect_out,
                                                        uint64_t* idx_out, double* prob_out) {
    using C = typename Num<T>::C;
    __shared__ TopScratch ts;
    __shared__ double red[TK_NT / 32];
    const uint64_t D = 1ull << n;
    double ex = 0.0;
    bool have_run = false;
    for (uint64_t z0 = (uint64_t)blockIdx.x * RCH; z0 < D; z0 += (uint64_t)gridDim.x * RCH) {
        C v[RPT];
        T e[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const uint64_t z = z0 + (uint64_t)i * TK_NT + threadIdx.x;
            v[i].x = v[i].y = T(0);
            e[i] = T(0);
            if (z < D) {
                v[i] = psi[z];
                if (EXPECT) e[i] = E[z];
            }
        }
        if (EXPECT) {
            T acc = T(0);
#pragma unroll
            for (int i = 0; i < RPT; ++i) acc += (v[i].x * v[i].x + v[i].y * v[i].y) * e[i];
            ex += (double)acc;
        }
        if (TOPK) {
            topk_round(v, psi, z0, D, k, have_run, ts);
            have_run = true;
        }
    }
    const bool one = gridDim.x == 1;
    if (EXPECT) {
        const double tot = block_sum(ex, red);
        if (threadIdx.x == 0) {
            if (!one) part_expect[blockIdx.x] = tot;
            else if (expect_out) *expect_out = tot;
        }
    }
    if (TOPK && (int)threadIdx.x < k) {
        const TopEnt x = ts.run[threadIdx.x];
        if (!one) {
            part_topp[(uint64_t)blockIdx.x * k + threadIdx.x] = x.p;
            part_topz[(uint64_t)blockIdx.x * k + threadIdx.x] = x.z;
        } else {
            if (idx_out) idx_out[threadIdx.x] = (uint64_t)x.z;
            if (prob_out) prob_out[threadIdx.x] = x.p;
        }
    }
}

template <bool EXPECT, bool TOPK>
__global__ void __launch_bounds__(TK_NT) k_reduce_finalize(int nparts, const double* part_expect,
                                                           const double* part_topp, const uint32_t* part_topz, int k,
                                                           double* expect, uint64_t* topk_idx, double* topk_prob) {
    __shared__ TopScratch ts;
    __shared__ double red[TK_NT / 32];
    if (EXPECT) {
        double acc = 0.0;
        const int per = (nparts + TK_NT - 1) / TK_NT;
        for (int t = threadIdx.x * per; t < (int)(threadIdx.x + 1) * per && t < nparts; ++t) acc += part_expect[t];
        const double tot = block_sum(acc, red);
        if (threadIdx.x == 0 && expect) *expect = tot;
    }
    if (TOPK) {
        merge_entries((uint64_t)nparts * k, k, ts, [=](uint64_t e) { return TopEnt{part_topp[e], part_topz[e]}; });
        if ((int)threadIdx.x < k) {
            const TopEnt x = ts.run[threadIdx.x];
            if (topk_idx) topk_idx[threadIdx.x] = (uint64_t)x.z;
            if (topk_prob) topk_prob[threadIdx.x] = x.p;
        }
    }
}

template <typename T, bool EXPECT, bool TOPK>
cudaError_t reduce_t(int n, const void* psi, const void* E, int k, double* pe, double* pp, uint32_t* pz,
                     double* expect, uint64_t* idx, double* prob, cudaStream_t st) {
    const int parts = reduce_parts(n);
    k_reduce_state<T, EXPECT, TOPK><<<parts, TK_NT, 0, st>>>(n, static_cast<const typename Num<T>::C*>(psi),
                                                            static_cast<const T*>(E), k, pe, pp, pz, expect, idx, prob);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || parts == 1) return e;
    k_reduce_finalize<EXPECT, TOPK><<<1, TK_NT, 0, st>>>(parts, pe, pp, pz, k, expect, idx, prob);
    return cudaGetLastError();
}

template <typename T>
cudaError_t reduce_any(int n, const void* psi, const void* E, int k, double* pe, double* pp, uint32_t* pz,
                       double* expect, uint64_t* idx, double* prob, cudaStream_t st) {
    if (E && k > 0) return reduce_t<T, true, true>(n, psi, E, k, pe, pp, pz, expect, idx, prob, st);
    if (E) return reduce_t<T, true, false>(n, psi, E, k, pe, pp, pz, expect, idx, prob, st);
    return reduce_t<T, false, true>(n, psi, E, k, pe, pp, pz, expect, idx, prob, st);
}

}  // namespace

cudaError_t launch_reduce_state(bool dbl, int n, const void* psi, const void* E, int k, double* part_expect,
                                double* part_topp, uint32_t* part_topz, double* expect, uint64_t* topk_idx,
                                double* topk_prob, cudaStream_t st) {
    return dbl ? reduce_any<double>(n, psi, E, k, part_expect, part_topp, part_topz, expect, topk_idx, topk_prob, st)
               : reduce_any<float>(n, psi, E, k, part_expect, part_topp, part_topz, expect, topk_idx, topk_prob, st);
}

}  // namespace qaoa
