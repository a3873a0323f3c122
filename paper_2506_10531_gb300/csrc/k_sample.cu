// k_sample.cu -- measurement shots of a complex64 state: inverse-CDF sampling over |psi|^2 with
// uniforms supplied by the caller (Section IV reads the sub-solution from measured shots; the
// default path of this library takes the top-k bitstrings instead).
//
// The 2^n probabilities are cut into F = 2^(n - fb) fine parts of 2^fb contiguous amplitudes
// (fb = 4 up to n = 20, then n - 16, so F <= 65536) and runs of up to 256 fine parts form a
// coarse part (C <= 256 of them):
//   1. k_sample_sums: one block per coarse part: the FP64 sum of each fine part, their exclusive
//      prefix inside the coarse part, and the coarse part's total;
//   2. k_sample_draw: every block first scans the C coarse totals (at most 256 values, cheaper
//      than a launch of its own); a shot's target t = u * total is then located by two binary
//      searches (coarse offsets in shared memory, fine prefixes in L2) and a walk through one
//      fine part.
// What bounds it: FP64 issue (GB300 has two FP64 lanes per SM and clock), so the design counts
// FP64 operations: three per amplitude for the sums; the searches compare the non-negative
// doubles as integers; a shot's walk is one thread over its 16 amplitudes (1.5 FP64 warp
// instructions per shot; a warp per shot with shuffle scans needs 8 per 32 amplitudes walked).
// Only for fb >= 7 half a warp walks a part together.
// Up to 8 qubits the draw forms the sums itself (small_sums) and k_sample_sums does not run.
// Every loop is bounded by the part length; nothing waits on another block. A batch of states of
// equal n (a DQAOA cycle's sub-QUBO states, 2^n amplitudes apart) runs as one launch of each
// kernel, the state index in blockIdx.y; each state has its own scratch (F + C doubles),
// uniforms and shots. Complex64 loads are 8 bytes wide: a state needs no more alignment.
// Measured on GB300 against parts of 2^(n-12) amplitudes, a one-thread scan over 4096 of them and a
// warp per shot: one n = 20 state, 65536 shots, 748 -> 41 us (sums 17, draw 23); 128 states of
// n = 12, 1024 shots each, 2380 -> 49 us (sums 10, draw 38).
#include <cuda_runtime.h>

#include "qaoa_common.cuh"
#include "qaoa_host.h"

namespace qaoa {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int NTS = 256;   // threads per block; also the most fine parts of a coarse part

// Fine-part bits, fine parts per coarse part (log2) and coarse parts (log2) of an n-qubit state.
struct SampleGeo {
    int fb, jb, cb;
};
__host__ __device__ inline SampleGeo sample_geo(int n) {
    SampleGeo g;
    g.fb = n > 20 ? n - 16 : (n < 4 ? n : 4);
    const int f = n - g.fb;
    g.jb = f < 8 ? f : 8;
    g.cb = f - g.jb;
    return g;
}

// |v|^2 in FP64: the products of two floats are exact, the fused add rounds once (the value of
// exact_prob in one operation fewer)
__device__ __forceinline__ double prob64(float2 v) {
    return __fma_rn((double)v.x, (double)v.x, __dmul_rn((double)v.y, (double)v.y));
}

// Inclusive prefix over W lanes: at each level the upper half of a group adds the lower half's
// total. The sums never decrease from lane to lane and a zero leaves its neighbour's sum as it
// is, bit for bit, so a part or an amplitude without probability spans no target.
template <int W>
__device__ __forceinline__ double lane_scan(double v) {
    const int lane = threadIdx.x & (W - 1);
#pragma unroll
    for (int d = 1; d < W; d <<= 1) {
        const double o = __shfl_sync(FULL, v, (lane & ~(2 * d - 1)) | (d - 1), W);
        if (lane & d) v = o + v;
    }
    return v;
}

// Exclusive prefix of one value per thread over the block (fixed order, properties as lane_scan);
// the total in *tot.
__device__ __forceinline__ double block_excl_scan(double v, double* wsum, double* tot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double incl = lane_scan<32>(v);
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    double off = 0.0, all = 0.0;
#pragma unroll
    for (int i = 0; i < NTS / 32; ++i) {
        if (i < w) off += wsum[i];
        all += wsum[i];
    }
    *tot = all;
    const double left = __shfl_up_sync(FULL, incl, 1);
    return lane == 0 ? off : off + left;
}

// One block per coarse part of 2^(fb + jb) amplitudes. Fine parts of up to 128 amplitudes: 4096
// amplitudes at a time are read coalesced, their probabilities pass through shared memory (rows of
// 16 padded to 17) and thread t adds the 16 of row t; neighbouring threads combine their rows
// when a fine part has more than one. Longer fine parts: one warp per part, lanes strided.
__global__ void __launch_bounds__(NTS) k_sample_sums(const float2* __restrict__ psi, int n,
                                                     double* __restrict__ scratch) {
    __shared__ double row[NTS * 17];
    __shared__ double fine[NTS];
    __shared__ double wsum[NTS / 32];
    const SampleGeo g = sample_geo(n);
    const uint32_t J = 1u << g.jb;
    psi += ((uint64_t)blockIdx.y << n) + ((uint64_t)blockIdx.x << (g.fb + g.jb));
    double* pre = scratch + (size_t)blockIdx.y * (((size_t)1 << (n - g.fb)) + ((size_t)1 << g.cb));
    double* coarse = pre + ((size_t)1 << (n - g.fb));
    pre += (size_t)blockIdx.x << g.jb;
    if (g.fb <= 7) {
        const uint32_t D = 1u << (g.fb + g.jb);   // amplitudes of the block
        const int rb = g.fb < 4 ? 0 : g.fb - 4;   // rows per fine part (log2)
        for (uint32_t c0 = 0; c0 < D; c0 += NTS * 16) {
            float2 v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const uint32_t u = c0 + (uint32_t)i * NTS + threadIdx.x;
                v[i] = u < D ? psi[u] : make_float2(0.0f, 0.0f);
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const uint32_t u = (uint32_t)i * NTS + threadIdx.x;
                row[u + (u >> 4)] = prob64(v[i]);
            }
            __syncthreads();
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < 16; ++i) s += row[threadIdx.x * 17 + i];
            for (int d = 0; d < rb; ++d) s += __shfl_xor_sync(FULL, s, 1 << d);
            const uint32_t f = (c0 >> g.fb) + (threadIdx.x >> rb);
            if ((threadIdx.x & ((1u << rb) - 1u)) == 0 && f < J) fine[f] = s;
            __syncthreads();
        }
    } else {
        const uint32_t L = 1u << g.fb;
        for (uint32_t f = threadIdx.x >> 5; f < J; f += NTS / 32) {
            const float2* p = psi + ((uint64_t)f << g.fb) + (threadIdx.x & 31);
            double a = 0.0, b = 0.0;
#pragma unroll 4
            for (uint32_t u = 0; u < L; u += 64) {
                const float2 v0 = p[u], v1 = p[u + 32];
                a = __fma_rn((double)v0.x, (double)v0.x, a);
                b = __fma_rn((double)v1.x, (double)v1.x, b);
                a = __fma_rn((double)v0.y, (double)v0.y, a);
                b = __fma_rn((double)v1.y, (double)v1.y, b);
            }
            const double s = warp_sum(a + b);
            if ((threadIdx.x & 31) == 0) fine[f] = s;
        }
        __syncthreads();
    }
    double tot;
    const double ex = block_excl_scan(threadIdx.x < J ? fine[threadIdx.x] : 0.0, wsum, &tot);
    if (threadIdx.x < J) pre[threadIdx.x] = ex;
    if (threadIdx.x == 0) coarse[blockIdx.x] = tot;
}

// The last of `count` non-decreasing offsets (off[0] = 0) that is <= t, as integers: every offset
// is a non-negative double, and a negative t lies below all of them in either reading.
__device__ __forceinline__ uint32_t last_le(const double* off, uint32_t count, double t) {
    const long long tb = pbits(t);
    uint32_t lo = 0;
    for (uint32_t step = count >> 1; step; step >>= 1)   // count is a power of two
        if (pbits(off[lo + step]) <= tb) lo += step;
    return lo;
}

// The largest double below the positive double v (v itself when v <= 0): targets stay below the
// total of the part they are searched in, so a tail of empty parts is never chosen.
__device__ __forceinline__ double below(double v) {
    return pbits(v) > 0 ? __longlong_as_double(pbits(v) - 1) : v;
}

// Up to 8 qubits every block of shots forms the at most 16 fine sums and their prefix for itself, in the
// order of k_sample_sums (same bits): one launch instead of two (n = 3, 16 shots: 18.5 us in two, 8.3 in
// one; 12.4 us in three of a block per amplitude). pre, total: shared. Called by all threads.
constexpr int SMALL_N = 8;
__device__ __forceinline__ void small_sums(const float2* __restrict__ psi, int n, double* pre, double* total) {
    const SampleGeo g = sample_geo(n);
    const int J = 1 << g.jb, L = 1 << g.fb, f = (int)threadIdx.x;
    if (f < 32) {
        double s = 0.0;
        if (f < J)
            for (int i = 0; i < L; ++i) s += prob64(psi[f * L + i]);
        for (int d = 1; d < J; d <<= 1) {   // lane_scan over the first J lanes
            const double o = __shfl_sync(FULL, s, (f & ~(2 * d - 1)) | (d - 1));
            if (f & d) s = o + s;
        }
        const double left = __shfl_up_sync(FULL, s, 1);
        if (f < J) pre[f] = f == 0 ? 0.0 : left;
        if (f == J - 1) *total = s;
    }
    __syncthreads();
}

// One thread per shot (fine parts of up to 64 amplitudes), or HALF: 16 lanes per shot; SMALL: no sums in
// scratch (n <= SMALL_N, blocks of 64 threads).
template <bool HALF, bool SMALL = false>
__global__ void __launch_bounds__(NTS) k_sample_draw(const float2* __restrict__ psi, int n,
                                                     const double* __restrict__ scratch, int64_t shots,
                                                     const double* __restrict__ u, uint64_t* __restrict__ out) {
    __shared__ double off[NTS];
    __shared__ double wsum[NTS / 32];
    const SampleGeo g = sample_geo(n);
    const uint32_t C = 1u << g.cb, J = 1u << g.jb;
    const double* pre = scratch + (size_t)blockIdx.y * (((size_t)1 << (n - g.fb)) + C);
    const double* coarse = pre + ((size_t)1 << (n - g.fb));
    psi += (uint64_t)blockIdx.y << n;
    u += (size_t)blockIdx.y * shots;
    out += (size_t)blockIdx.y * shots;
    double total;
    if constexpr (SMALL) {
        small_sums(psi, n, off, wsum);
        total = wsum[0];
        pre = off;
    } else {
        off[threadIdx.x] = block_excl_scan(threadIdx.x < C ? coarse[threadIdx.x] : 0.0, wsum, &total);
        __syncthreads();
    }
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t s = HALF ? id >> 4 : id;
    const bool live = s < shots;
    if (!HALF && !live) return;
    // (+ 0: a target of -0 is 0, and lies behind leading amplitudes without probability like it)
    const double t = fmin(__fma_rn(u[live ? s : shots - 1], total, 0.0), below(total));
    const uint32_t c = SMALL ? 0u : last_le(off, C, t);
    const double r = SMALL ? t : fmin(t - off[c], below(coarse[c]));
    const uint32_t f = last_le(pre + ((size_t)c << g.jb), J, r);
    double acc = pre[((size_t)c << g.jb) + f];
    const uint64_t base = (((uint64_t)c << g.jb) + f) << g.fb;
    const uint32_t L = 1u << g.fb;
    const float2* p = psi + base;
    uint32_t hit = 0xffffffffu, lastnz = 0xffffffffu;
    if (!HALF) {
        for (uint32_t c0 = 0; c0 < L && hit == 0xffffffffu; c0 += 16) {
            float2 v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = c0 + i < L ? p[c0 + i] : make_float2(0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const double q = prob64(v[i]);
                acc += q;
                if (hit == 0xffffffffu && c0 + i < L && acc > r) hit = c0 + i;
                if (pbits(q) > 0) lastnz = c0 + i;
            }
        }
        // no running sum exceeded the target (rounding at the part's end): its last nonzero amplitude
        if (hit == 0xffffffffu) hit = lastnz != 0xffffffffu ? lastnz : 0u;
        out[s] = base + hit;
    } else {
        // each of the 16 lanes sums its own L / 16 contiguous amplitudes, a scan finds the lane
        // that holds the target, and its run is walked 16 amplitudes at a time by all lanes
        const int hl = threadIdx.x & 15;
        const uint32_t S = L >> 4;
        const float2* pl = p + (uint32_t)hl * S;
        double a = 0.0, b = 0.0;
#pragma unroll 4
        for (uint32_t i = 0; i < S; i += 2) {
            const float2 v0 = pl[i], v1 = pl[i + 1];
            a = __fma_rn((double)v0.x, (double)v0.x, a);
            b = __fma_rn((double)v1.x, (double)v1.x, b);
            a = __fma_rn((double)v0.y, (double)v0.y, a);
            b = __fma_rn((double)v1.y, (double)v1.y, b);
        }
        const double mine = a + b;
        const double incl = lane_scan<16>(mine);
        const int sh = threadIdx.x & 16;
        const uint32_t over = (__ballot_sync(FULL, acc + incl > r) >> sh) & 0xffffu;
        const uint32_t some = (__ballot_sync(FULL, pbits(mine) > 0) >> sh) & 0xffffu;
        // the first lane past the target, else the last one that holds any probability
        const int w = over ? __ffs((int)over) - 1 : (some ? 31 - __clz((int)some) : 0);
        const double wl = __shfl_sync(FULL, incl, w > 0 ? w - 1 : 0, 16);
        if (w > 0) acc += wl;
        const float2* pw = p + (uint32_t)w * S;
        for (uint32_t c0 = 0; c0 < S; c0 += 16) {      // the same trip count in every lane
            const uint32_t i = c0 + hl;
            const double q = i < S ? prob64(pw[i]) : 0.0;
            const double in2 = lane_scan<16>(q);
            const uint32_t h2 = (__ballot_sync(FULL, i < S && acc + in2 > r) >> sh) & 0xffffu;
            const uint32_t nz = (__ballot_sync(FULL, pbits(q) > 0) >> sh) & 0xffffu;
            if (hit == 0xffffffffu && h2) hit = c0 + (uint32_t)__ffs((int)h2) - 1u;
            if (nz) lastnz = c0 + 31u - (uint32_t)__clz((int)nz);
            acc += __shfl_sync(FULL, in2, 15, 16);
        }
        if (hit == 0xffffffffu) hit = lastnz != 0xffffffffu ? lastnz : 0u;
        if (live && hl == 0) out[s] = base + (uint64_t)w * S + hit;
    }
}

}  // namespace

size_t sample_scratch_bytes(int n) {
    const SampleGeo g = sample_geo(n);
    return (((size_t)1 << (n - g.fb)) + ((size_t)1 << g.cb)) * sizeof(double);
}

cudaError_t launch_sample(int n, const void* psi, int count, int64_t shots, const double* u, uint64_t* out,
                          double* scratch, cudaStream_t st) {
    if (count < 1 || count > 65535) return cudaErrorInvalidValue;
    const SampleGeo g = sample_geo(n);
    const float2* ps = static_cast<const float2*>(psi);
    if (n <= SMALL_N) {
        constexpr int nt = 64;
        if (shots > 0)
            k_sample_draw<false, true><<<dim3((unsigned)((shots + nt - 1) / nt), (unsigned)count), nt, 0, st>>>(ps, n, scratch, shots, u, out);
        return cudaGetLastError();
    }
    k_sample_sums<<<dim3(1u << g.cb, (unsigned)count), NTS, 0, st>>>(ps, n, scratch);
    if (shots > 0) {
        const bool half = g.fb >= 7;
        const int64_t lanes = shots * (half ? 16 : 1);
        const dim3 grid((unsigned)((lanes + NTS - 1) / NTS), (unsigned)count);
        if (half) k_sample_draw<true><<<grid, NTS, 0, st>>>(ps, n, scratch, shots, u, out);
        else k_sample_draw<false><<<grid, NTS, 0, st>>>(ps, n, scratch, shots, u, out);
    }
    return cudaGetLastError();
}

}  // namespace qaoa
