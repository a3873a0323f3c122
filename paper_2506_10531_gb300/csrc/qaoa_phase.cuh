// qaoa_phase.cuh -- cost phases and energies of a 2^13-amplitude tile from Q itself, so that the
// forward TMA tiers neither build nor read an energy vector: 4 of the 20 bytes per amplitude of a
// pass with a cost phase, and all of the energy build.
//
// E(z) is a sum over the set bits and pairs of set bits of z, and so is the phase gamma E / 2 pi in
// turns. Phases are kept as 32-bit fractions of a turn: every term gamma W_ij / 2 pi is rounded once
// to 2^-32 turns in FP64 (W_ij = Q_ij + Q_ji, W_ii = Q_ii) and the sums wrap modulo one turn by
// themselves, so a sum is off by about 1e-8 rad (rms; at most 2^-33 turns a term, 3e-7 rad over the 465 terms
// of n = 30) whatever the energy. Its conversion to FP32 and the scaling to radians put up to 3e-7 rad more
// on it (rms 8e-8) and the hardware sine and cosine their 2^-21 -- FP32 energies put up to 1e-6 gamma on a
// phase. The energies of the final reduction are the same sums in FP32.
//
// With tile bit a standing for qubit q_a (a < c: a, else a - c + s; all tiles of a pass alike) and F
// the set bits the tile fixes, z = F + the tile bits u:
//   value(z) = V_F + sum_{a in u} d_a + sum_{a<b in u} W_{q_a q_b},  d_a = W_{q_a q_a} + sum_{f in F} W_{q_a f}.
// Thread t of 256 owns the elements whose low eight tile bits are t; e = tile bits 8..12:
//   value = base(t) + sum_{k in e} w_k(t) + pairs(e),
//   base(t) = V_F + pairs(t) + sum_{a in t} d_a,   w_k(t) = cross_k(t) + d_{8+k},
// pairs(t), cross_k(t) (per thread) and pairs(e) (32 values) are formed once per instance and pass,
// d and V_F (14 sums over F, a lane per qubit) once per tile, and the sum over k takes one
// addition per element in Gray-code order: a handful of instructions per amplitude.
#pragma once
#include "qaoa_engine.cuh"

namespace qaoa {
namespace tma {

struct PhaseTab {
    uint32_t W[32 * 32];      // symmetric; fractions of a turn, or FP32 bits
    uint32_t pairs[32];
    uint32_t d[16];           // d_0..d_12, V_F
    uint32_t own[6][256];     // per thread: pairs(t), cross_0..cross_4
    float scale;              // 2 pi 2^-32; NaN when a term is not finite
};

// F: FP32 energies, else fractions of a turn.
template <bool F>
__device__ __forceinline__ uint32_t tab_add(uint32_t a, uint32_t b) {
    return F ? __float_as_uint(__uint_as_float(a) + __uint_as_float(b)) : a + b;
}
// The entry of the pair (a, b) = (Q_ij, Q_ji), or of the diagonal (Q_ii, 0).
template <bool F>
__device__ __forceinline__ uint32_t tab_term(float a, float b, double g, bool& bad) {
    if (F) return __float_as_uint(__fadd_rn(a, b));
    double x = g * ((double)a + (double)b);
    if (!(fabs(x) < 500000.0)) {
        bad = bad || !(fabs(x) <= 1.0e300);
        x -= rint(x);
    }
    return (uint32_t)__double2loint(x + 1572864.0);   // 1.5 2^20: the low word counts 2^-32 turns
}
__device__ __forceinline__ int tile_qubit(int a, int c, int s) { return a < c ? a : a - c + s; }

// The table of an n-qubit instance (Q: n x n floats) for tiles with c low bits and s (kind A: c = 13);
// g = gamma / 2 pi (unused with F). All 256 threads call it; contains one barrier; the table may be
// read after the next one.
template <bool F>
__device__ __forceinline__ void tab_build(PhaseTab& t, const float* Q, int n, double g, int c, int s) {
    bool bad = false;
    // The pairs i <= j without gaps (FP64 issues at 1/64 of the FP32 rate, a warp at a time; with half of the
    // threads on i > j one instance of n = 18, p = 3, took 62.8 us, 59.5 so): rows k and
    // n - k (odd n; n - 1 - k for even) of the triangle together fill a row of n | 1.
    const int wd = n | 1, total = n * (n + 1) / 2;
    for (int x = threadIdx.x; x < total; x += 256) {
        const int k = x / wd, b = x - k * wd, over = b - (n - k);
        const int i = over < 0 ? k : n - k - 1 + (n & 1), j = i + (over < 0 ? b : over);
        t.W[i * 32 + j] = t.W[j * 32 + i] = tab_term<F>(Q[i * n + j], i == j ? 0.0f : Q[j * n + i], g, bad);
    }
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) t.scale = bad ? __int_as_float(0x7fffffff) : 1.4629180792671596e-9f;   // 2 pi 2^-32
    int q[13];
#pragma unroll
    for (int a = 0; a < 13; ++a) q[a] = tile_qubit(a, c, s);
    const uint32_t u = threadIdx.x;
    if (u < 32u) {
        uint32_t v = 0u;
#pragma unroll
        for (int a = 0; a < 5; ++a)
#pragma unroll
            for (int b = a + 1; b < 5; ++b)
                if ((u >> a) & (u >> b) & 1u) v = tab_add<F>(v, t.W[q[8 + a] * 32 + q[8 + b]]);
        t.pairs[u] = v;
    }
    uint32_t p = 0u, w[5] = {0u, 0u, 0u, 0u, 0u};
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const uint32_t ma = 0u - ((u >> a) & 1u);
#pragma unroll
        for (int b = a + 1; b < 8; ++b) p = tab_add<F>(p, t.W[q[a] * 32 + q[b]] & ma & (0u - ((u >> b) & 1u)));
#pragma unroll
        for (int k = 0; k < 5; ++k) w[k] = tab_add<F>(w[k], t.W[q[a] * 32 + q[8 + k]] & ma);
    }
    t.own[0][u] = p;
#pragma unroll
    for (int k = 0; k < 5; ++k) t.own[1 + k][u] = w[k];
}

// d and V_F of a tile that fixes the set bits F of z. All 256 threads call it (the table readable);
// the result may be read after the next barrier.
template <bool F>
__device__ __forceinline__ void tab_tile(PhaseTab& t, uint32_t fixed, int c, int s) {
    const int lane = threadIdx.x & 31;
    const bool on = (fixed >> lane) & 1u;
#pragma unroll 1
    for (int i = threadIdx.x >> 5; i < 14; i += 8) {
        uint32_t v = 0u;
        const int q = i < 13 ? tile_qubit(i, c, s) : 0;
        if (on) {
            if (i < 13) {
                v = t.W[q * 32 + lane];
            } else {
                v = t.W[lane * 33];
                for (uint32_t b = fixed & ((1u << lane) - 1u); b; b &= b - 1u)
                    v = tab_add<F>(v, t.W[lane * 32 + __ffs((int)b) - 1]);
            }
        }
        if (F) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = tab_add<F>(v, __shfl_xor_sync(0xffffffffu, v, o));
        } else {
            v = __reduce_add_sync(0xffffffffu, v);
        }
        if (lane == 0) t.d[i] = i < 13 ? tab_add<F>(v, t.W[q * 33]) : v;
    }
}

// A thread's values of the tile (after the barrier that follows tab_tile).
struct TileVals {
    const PhaseTab* t;
    uint32_t base, w[5];
    template <bool F>
    __device__ __forceinline__ void init(const PhaseTab& tab) {
        t = &tab;
        const uint32_t u = threadIdx.x;
        base = tab_add<F>(tab.d[13], tab.own[0][u]);
#pragma unroll
        for (int a = 0; a < 8; ++a) base = tab_add<F>(base, tab.d[a] & (0u - ((u >> a) & 1u)));
#pragma unroll
        for (int k = 0; k < 5; ++k) w[k] = tab_add<F>(tab.own[1 + k][u], tab.d[8 + k]);
    }
    // the value at the thread's elements whose bits 8..A-1 are r and whose window bits are clear
    template <bool F, int A>
    __device__ __forceinline__ uint32_t start(int r) const {
        uint32_t v = base;
#pragma unroll
        for (int k = 0; k < A - 8; ++k) v = tab_add<F>(v, w[k] & (0u - ((uint32_t)(r >> k) & 1u)));
        return v;
    }
};

// fn(i, sin, cos) of the phase at every element i of group r of window [A, 13), A >= 8.
template <int A, int R, typename Fn>
__device__ __forceinline__ void tab_phases(const TileVals& x, int r, Fn&& fn) {
    static_assert(A >= 8 && A + R == 13, "windows that reach the top of the tile");
    const uint32_t* pr = x.t->pairs + r;
    const float scale = x.t->scale;
    uint32_t cur = x.start<false, A>(r);
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
        const int i = gray_elem(k);
        if (k) {
            int b = 0;
            while (!((k >> b) & 1) && b < R - 1) ++b;
            cur = ((i >> b) & 1) ? cur + x.w[A - 8 + b] : cur - x.w[A - 8 + b];
        }
        float s, c;
        __sincosf((float)(int)(cur + pr[i << (A - 8)]) * scale, &s, &c);
        fn(i, s, c);
    }
}
// fn(i, E) at the same elements.
template <int A, int R, typename Fn>
__device__ __forceinline__ void tab_energies(const TileVals& x, int r, Fn&& fn) {
    static_assert(A >= 8 && A + R == 13, "windows that reach the top of the tile");
    constexpr int RL = R < 2 ? R : 2, RH = R - RL;
    const uint32_t* pr = x.t->pairs + r;
    float lo[1 << RL], hi[1 << RH];
    lo[0] = 0.0f;
#pragma unroll
    for (int b = 0; b < RL; ++b)
#pragma unroll
        for (int m = 0; m < (1 << b); ++m) lo[m | (1 << b)] = lo[m] + __uint_as_float(x.w[A - 8 + b]);
    hi[0] = __uint_as_float(x.start<true, A>(r));
#pragma unroll
    for (int b = 0; b < RH; ++b)
#pragma unroll
        for (int m = 0; m < (1 << b); ++m) hi[m | (1 << b)] = hi[m] + __uint_as_float(x.w[A - 8 + RL + b]);
#pragma unroll
    for (int i = 0; i < (1 << R); ++i)
        fn(i, (hi[i >> RL] + lo[i & ((1 << RL) - 1)]) + __uint_as_float(pr[i << (A - 8)]));
}

}  // namespace tma
}  // namespace qaoa
