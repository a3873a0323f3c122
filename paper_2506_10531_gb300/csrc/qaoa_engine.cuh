// qaoa_engine.cuh -- the shared-memory tile engine of libqaoa.
//
// A tile is 2^tb amplitudes of one QAOA state held in shared memory (swizzled, see swz()).
// The whole state is a tile in the resident tier; the streaming tier moves tiles between HBM
// and shared memory. Inside a tile the mixer (Section IV, Eq. 2: exp(-i beta X_q) on every
// qubit) is applied in *sub-passes*: a sub-pass loads groups of 2^R amplitudes that differ
// only in a window of R consecutive tile bits [a, a+R) into registers, applies the
// butterflies of the window's qubits (a bit mask chooses which), and writes them back. Each
// thread owns whole groups; the 32 lanes of a warp own groups that differ in the lowest tile
// bits outside the window, so with the swizzle every access of a warp hits distinct banks.
//
// Layers are scheduled in a "snake": within a layer the windows are visited in one order,
// in the next layer in the reverse order, so the last window of layer l and the first window
// of layer l+1 are the same and share one sub-pass: mixer_l(window), cost_{l+1} (elementwise),
// mixer_{l+1}(window). With G windows per layer this takes 1 + p (G - 1) sub-passes instead of
// p G. The adjoint runs the same sub-passes in reverse order with each operation inverted.
#pragma once
#include "qaoa_common.cuh"

namespace qaoa {

// Per-layer constants staged in shared memory. Every layer mixes with unscaled shears (see
// butterfly); the factor its n qubits leave is post (-1)^(cot |z|), |z| the set bits of the global
// index, applied by the next layer's cost phase (pre, pcot) or, for the last layer, by the last
// sub-pass. The adjoint undoes the mixers with three in-place shears instead (lift_inverse), which
// leave no factor: t is then tan(beta / 2) and sn sin(beta), beta taken modulo pi into
// [-pi/2, pi/2] (a sign that both of its states share).
template <typename T>
struct LayerConst {
    PhaseK<T> ph;   // gamma_l
    T t;            // tan(beta_l), or cot(beta_l) with cot; adjoint: tan(beta_l / 2)
    T sn;           // adjoint: sin(beta_l)
    T pre;          // factor of layer l - 1, applied with this layer's cost phase
    T post;         // factor this layer leaves
    int cot, pcot;  // this layer's and layer l - 1's form
};

// A pending factor on the elements of a group: f0 on those with an even number of set window
// bits, f1 on the others (parity: of the set bits of the group's base index).
template <typename T>
struct Pending {
    T f[2];
    __device__ __forceinline__ Pending(T post, int cot, int parity) {
        f[0] = (cot && (parity & 1)) ? -post : post;
        f[1] = cot ? -f[0] : f[0];
    }
};

// x^n by repeated squaring in the working precision (no FP64 on the complex64 path).
template <typename T>
__device__ __forceinline__ T ipow(T x, int n) {
    T r = T(1);
    while (n) {
        if (n & 1) r *= x;
        x *= x;
        n >>= 1;
    }
    return r;
}

// (1 + t^2)^(-n/2): the factor n shears with the rounded t leave, so that a layer keeps the norm.
// In complex64 as a product of two-float numbers: the n-th power of a factor rounded to float
// put up to n 2^-24 on every amplitude.
struct Two {
    float h, l;
    __device__ __forceinline__ Two mul(const Two& o) const {
        const float p = h * o.h;
        const float e = fmaf(h, o.l, fmaf(l, o.h, fmaf(h, o.h, -p)));
        const float s = p + e;
        return Two{s, e - (s - p)};
    }
};
__device__ __forceinline__ float shear_norm(float t, int n) {
    const float qh = fmaf(t, t, 1.0f), ql = fmaf(t, t, 1.0f - qh);      // 1 + t^2 = qh + ql
    const float r0 = rsqrtf(qh), s = r0 * r0, se = fmaf(r0, r0, -s);
    float d = fmaf(-qh, s, 1.0f);                                       // 1 - (1 + t^2) r0^2
    d = fmaf(-qh, se, fmaf(-ql, s, d));
    Two x{r0, 0.5f * r0 * d}, r{1.0f, 0.0f};
    for (; n; n >>= 1) {
        if (n & 1) r = r.mul(x);
        x = x.mul(x);
    }
    return r.h + r.l;
}
// complex128: the same with unnormalised pairs (h + l, l a few roundings of h), whose dependent
// chain is a third of the products' above: FP64 latency is what a layer's constants cost (256 grid points
// of n = 10: 60.2 us with the plain power of the rounded factor, 60.6 us so). That power put 22 2^-53
// on the squared norm of 64 states of n = 10, p = 1; the pairs leave less than 5.
__device__ __forceinline__ double shear_norm(double t, int n) {
    const double qh = fma(t, t, 1.0), ql = fma(t, t, 1.0 - qh);         // 1 + t^2 = qh + ql
    const double r0 = rsqrt(qh), s = r0 * r0, se = fma(r0, r0, -s);
    const double d = fma(-qh, se, fma(-ql, s, fma(-qh, s, 1.0)));       // 1 - (1 + t^2) r0^2
    double xh = r0, xl = 0.5 * r0 * d;
    const auto square = [&] {
        const double q = xh * xh;
        xl = fma(2.0 * xh, xl, fma(xh, xh, -q));
        xh = q;
    };
    for (; !(n & 1); n >>= 1) square();                                 // n >= 1
    double rh = xh, rl = xl;
    while (n >>= 1) {
        square();
        if (n & 1) {
            const double p = rh * xh;
            rl = fma(rh, xl, fma(rl, xh, fma(rh, xh, -p)));
            rh = p;
        }
    }
    return rh + rl;
}

// Fill the constants of p layers of an n-qubit instance (one thread per layer; contains a
// __syncthreads, so every thread of the block calls it). The factor of a cot layer is
// (sign(s) / sqrt(1 + t^2))^n (-1)^(n - |z|): everything but (-1)^|z| is folded into post.
template <typename T>
__device__ __forceinline__ void set_layer_consts(LayerConst<T>* lc, const T* gamma, const T* beta,
                                                 int p, int n, bool adjoint) {
    for (int l = threadIdx.x; l < p; l += blockDim.x) {
        T sb, cb;
        sincos_full(beta[l], sb, cb);
        LayerConst<T> k;
        make_phase(gamma[l], k.ph);
        k.pre = k.post = T(1);
        k.sn = T(0);
        k.cot = k.pcot = 0;
        if (adjoint) {
            if (cb < T(0)) { sb = -sb; cb = -cb; }
            k.t = sb / (T(1) + cb);
            k.sn = sb;
        } else {
            k.cot = fabs(cb) < fabs(sb) ? 1 : 0;
            const T f = k.cot ? sb : cb;
            k.t = (k.cot ? cb : sb) / f;
            const bool neg = k.cot ? f > T(0) : f < T(0);     // the sign of -s or c
            k.post = shear_norm(k.t, n);
            if (neg && (n & 1)) k.post = -k.post;
        }
        lc[l] = k;
    }
    __syncthreads();
    for (int l = 1 + (int)threadIdx.x; l < p; l += blockDim.x) {
        lc[l].pre = lc[l - 1].post;
        lc[l].pcot = lc[l - 1].cot;
    }
    __syncthreads();
}

// Constants of the engine's forward runs. complex128 uses LayerConst. Measured shots are drawn from
// complex64 states of the resident tier and of the single-instance calls (and, in sampled sessions of 15 and
// more variables, from batched plans of the TMA tiers, which take LayerConst and phases from Q), and
// a shot is a whole number that moves when a probability moves by one rounding: the engine's runs
// keep one arithmetic (gamma / pi in one float, shears where |cos| >= |sin| and scaled
// rotations elsewhere, factors as powers of the rounded cosine) and one order of the qubits in a
// layer (blocks of `block` qubits ascending in even layers, descending in odd ones, ascending
// inside a block) whatever windows, tiles or block sizes a launch takes. The forward half of a
// gradient takes LayerConst in complex64 too: the powers of a rounded cosine put a norm error of n 2^-25
// a layer on psi and lam alike, and the adjoint undoes the phases of the two-float gamma (n = 20,
// p = 4, medians of 24 gradients against 64 bits: dgamma 1.9e-6, dbeta 1.1e-6, <C> 6e-7; with
// FwdConst32 on both sides 3.0e-6, 2.7e-6, 1.8e-6).
struct FwdConst32 {
    float gpi;     // gamma_l / pi
    float c, s;    // cos(beta_l), sin(beta_l)
    float t;       // tan(beta_l) when shear != 0
    float pre;     // scale applied with this layer's cost phase (pending factor of layer l-1)
    float post;    // scale still pending after this layer (used for the last layer)
    int shear;
};
template <typename T> struct FwdOf;
template <> struct FwdOf<float> { using K = FwdConst32; };
template <> struct FwdOf<double> { using K = LayerConst<double>; };
template <typename T> using FwdConst = typename FwdOf<T>::K;

__device__ __forceinline__ void set_fwd_consts(FwdConst32* lc, const float* gamma, const float* beta, int p, int n) {
    for (int l = threadIdx.x; l < p; l += blockDim.x) {
        float sb, cb;
        sincosf(beta[l], &sb, &cb);
        FwdConst32 k;
        k.gpi = gamma[l] * 0.31830988618379067154f;   // 1 / pi
        k.c = cb;
        k.s = sb;
        k.shear = fabsf(cb) >= fabsf(sb) ? 1 : 0;
        k.t = k.shear ? sb / cb : 0.0f;
        k.post = k.shear ? ipow(cb, n) : 1.0f;
        k.pre = 1.0f;
        lc[l] = k;
    }
    __syncthreads();
    for (int l = 1 + (int)threadIdx.x; l < p; l += blockDim.x) lc[l].pre = lc[l - 1].post;
    __syncthreads();
}
__device__ __forceinline__ void set_fwd_consts(LayerConst<double>* lc, const double* gamma, const double* beta, int p,
                                               int n) {
    set_layer_consts<double>(lc, gamma, beta, p, n, false);
}
__device__ __forceinline__ void set_fwd_consts(LayerConst<float>* lc, const float* gamma, const float* beta, int p, int n) {
    set_layer_consts<float>(lc, gamma, beta, p, n, false);
}
// The constants of a forward run, GRAD: that of a gradient.
template <typename T, bool GRAD> struct FwdFor { using K = FwdConst<T>; };
template <typename T> struct FwdFor<T, true> { using K = LayerConst<T>; };

// One sub-pass: window start a, butterfly mask over the window bits, layers [la, lb]
// (lb <= la + 1), whether the cost of layer la opens the sub-pass; post != 0 applies the
// pending shear factor of layer lb after its mixer (set by the caller on the very last
// sub-pass of a state).
struct SubPass {
    int a, mask, la, lb, ph_first, post;
};

// Windows of a layer over the mixed tile bits [m0, m1): window w covers bits
// [m0 + w R, min(m0 + (w+1) R, m1)); its register window is shifted down when it would run
// past the tile top so that it always spans R valid bits.
__device__ __forceinline__ void window_of(int w, int m0, int m1, int tb, int R, int& a, int& mask) {
    const int lo = m0 + w * R;
    const int hi = min(lo + R, m1);
    a = min(lo, tb - R);
    if (a < 0) a = 0;
    mask = ((1 << (hi - lo)) - 1) << (lo - a);
}

__device__ __forceinline__ int num_windows(int m0, int m1, int R) { return (m1 - m0 + R - 1) / R; }

// Walk of the snake over layers L0..L0+nl-1, forward from begin() or backward from end(): sub-pass
// 0 is window order[0] of layer 0, afterwards layer l has G - 1 sub-passes, so the position is
// advanced without a division (a thread's sub-pass is a few hundred instructions; forming the
// position from its number took a fifth of that). ph_first of the very first sub-pass is given
// by first_ph. top_phase: a single layer that opens with its cost phase runs its windows top
// down, so the phase shares the top window (the mixer windows of one layer commute); the TMA
// adjoint keeps every energy read in a window whose lanes cover the low tile bits that way.
struct Snake {
    int G, nl, L0, first_ph, m0, m1, tb, R;
    bool top;
    int l, pos;
    __device__ __forceinline__ Snake(int nl_, int L0_, int first_ph_, int m0_, int m1_, int tb_, int R_,
                                     bool top_phase = false)
        : G(num_windows(m0_, m1_, R_)), nl(nl_), L0(L0_), first_ph(first_ph_), m0(m0_), m1(m1_), tb(tb_), R(R_),
          top(top_phase && nl_ == 1 && first_ph_), l(0), pos(0) {}
    __device__ __forceinline__ void to_last() {
        l = nl - 1;
        pos = G > 1 ? G - 1 : 0;
    }
    __device__ __forceinline__ bool first() const { return l == 0 && pos == 0; }
    __device__ __forceinline__ bool last() const { return l == nl - 1 && pos == (G > 1 ? G - 1 : 0); }
    __device__ __forceinline__ void next() {
        if (G <= 1 || pos == G - 1) { ++l; pos = G > 1 ? 1 : 0; }
        else ++pos;
    }
    __device__ __forceinline__ void prev() {
        if (G <= 1) --l;
        else if (pos == 1 && l > 0) { --l; pos = G - 1; }
        else --pos;
    }
    __device__ __forceinline__ SubPass get() const {
        SubPass sp;
        const bool fwd = (l & 1) == 0 && !top;
        const int w = fwd ? pos : G - 1 - pos;
        sp.la = L0 + l;
        sp.lb = (G > 1 && pos == G - 1 && l + 1 < nl) ? sp.la + 1 : sp.la;
        sp.ph_first = first() ? first_ph : (G <= 1 ? 1 : 0);
        window_of(w, m0, m1, tb, R, sp.a, sp.mask);
        sp.post = 0;
        return sp;
    }
};

// Register windows of a layer over bits [0, n) that keep the qubit order of blocks of `block` qubits
// (FwdConst): each block is cut into windows of at most R qubits; odd layers take the blocks top
// down, and the windows of a block always upwards (odd: their order). Made on the host.
struct WinSched {
    int nw;
    signed char a[10], mask[10], odd[10];
};
inline WinSched win_sched(int n, int block, int R) {
    WinSched w{};
    for (int b = 0; b < n; b += block)
        for (int q = b; q < n && q < b + block; q += R) {
            const int size = (b + block < n ? b + block : n) - q < R ? (b + block < n ? b + block : n) - q : R;
            const int a = q + R <= n ? q : (n > R ? n - R : 0);
            w.a[w.nw] = (signed char)a;
            w.mask[w.nw++] = (signed char)(((1 << size) - 1) << (q - a));
        }
    const int per = (block + R - 1) / R;
    int k = 0;
    for (int b = (w.nw + per - 1) / per - 1; b >= 0; --b)
        for (int i = b * per; i < (b + 1) * per && i < w.nw; ++i) w.odd[k++] = (signed char)i;
    return w;
}

// Local index of element i of group g for window start a (R window bits).
template <int R>
__device__ __forceinline__ uint32_t group_base(uint32_t g, int a) {
    const uint32_t low = g & ((1u << a) - 1u);
    const uint32_t high = g >> a;
    return low | (high << (a + R));
}

// Mixer of layer constants k on the masked window bits of a register group (rotated frame,
// unscaled).
template <int R, bool COT, bool FULL, typename C, typename T>
__device__ __forceinline__ void mix_group(C (&v)[1 << R], int mask, T t) {
#pragma unroll
    for (int j = 0; j < R; ++j) {
        if (FULL || (mask & (1 << j))) {
#pragma unroll
            for (int i = 0; i < (1 << R); ++i)
                if (!(i & (1 << j))) butterfly<COT>(v[i], v[i | (1 << j)], t);
        }
    }
}
// Whole windows have a path of their own without the qubit tests: a butterfly's result lands in
// new registers, and every point where branches meet moves them back.
template <int R, typename C, typename T>
__device__ __forceinline__ void mix_layer(C (&v)[1 << R], int mask, const LayerConst<T>& k) {
    constexpr int ALL = (1 << R) - 1;
    if (k.cot) {
        if (mask == ALL) mix_group<R, true, true>(v, mask, k.t);
        else mix_group<R, true, false>(v, mask, k.t);
    } else {
        if (mask == ALL) mix_group<R, false, true>(v, mask, k.t);
        else mix_group<R, false, false>(v, mask, k.t);
    }
}

template <int R, typename Fn>
__device__ __forceinline__ void each_pair(float2 (&v)[1 << R], int mask, Fn&& fn) {
#pragma unroll
    for (int j = 0; j < R; ++j) {
        if (mask & (1 << j)) {
#pragma unroll
            for (int i = 0; i < (1 << R); ++i)
                if (!(i & (1 << j))) fn(v[i], v[i | (1 << j)]);
        }
    }
}
template <int R>
__device__ __forceinline__ void mix_layer(float2 (&v)[1 << R], int mask, const FwdConst32& k) {
    if (k.shear) {
        const float t = k.t;
        if (mask == (1 << R) - 1) each_pair<R>(v, (1 << R) - 1, [t](float2& a, float2& b) { butterfly<false>(a, b, t); });
        else each_pair<R>(v, mask, [t](float2& a, float2& b) { butterfly<false>(a, b, t); });
    } else {
        const float c = k.c, s = k.s;
        each_pair<R>(v, mask, [c, s](float2& a, float2& b) { butterfly_scaled(a, b, c, s); });
    }
}
// The cost phase of a forward layer with the factor the layer before left, on one amplitude: i,
// parity as in Pending.
struct FwdPhase32 {
    float g, pre;
    __device__ __forceinline__ FwdPhase32(const FwdConst32& k, int) : g(k.gpi), pre(k.pre) {}
    __device__ __forceinline__ void apply(float2& v, int, float e) const {
        float s, c;
        sincos_gpi(g, e, s, c);
        rot_neg(v, s * pre, c * pre);
    }
};
template <typename T>
struct FwdPhase {
    PhaseK<T> ph;
    Pending<T> pre;
    __device__ __forceinline__ FwdPhase(const LayerConst<T>& k, int parity) : ph(k.ph), pre(k.pre, k.pcot, parity) {}
    __device__ __forceinline__ void apply(typename Num<T>::C& v, int i, T e) const {
        T s, c;
        sincos_phase(ph, e, s, c);
        rot_neg(v, s * pre.f[__popc(i) & 1], c * pre.f[__popc(i) & 1]);
    }
};
__device__ __forceinline__ FwdPhase32 fwd_phase(const FwdConst32& k, int parity) { return FwdPhase32(k, parity); }
template <typename T>
__device__ __forceinline__ FwdPhase<T> fwd_phase(const LayerConst<T>& k, int parity) { return FwdPhase<T>(k, parity); }

// Apply a pending factor to every amplitude of a group.
template <int R, typename C, typename T>
__device__ __forceinline__ void scale_group(C (&v)[1 << R], const Pending<T>& f) {
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) {
        v[i].x *= f.f[__popc(i) & 1];
        v[i].y *= f.f[__popc(i) & 1];
    }
}

// The factor the last layer leaves.
template <int R>
__device__ __forceinline__ void finish_group(float2 (&v)[1 << R], const FwdConst32& k, int) {
    if (!k.shear) return;
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) {
        v[i].x *= k.post;
        v[i].y *= k.post;
    }
}
template <int R, typename C, typename T>
__device__ __forceinline__ void finish_group(C (&v)[1 << R], const LayerConst<T>& k, int parity) {
    scale_group<R>(v, Pending<T>(k.post, k.cot, parity));
}

// Mixer inverse on two states with the accumulation of Im <lam| X_q |psi> over the masked
// qubits. Any point of the layer's mixer gives the same value (X_q commutes with every
// exp(-i beta X_q')). In the rotated frame X_q becomes Y_q, so over the pairs (a, b)
//   Im <lam|X_q|psi> = sum Re(conj(lam~_b) psi~_a) - Re(conj(lam~_a) psi~_b),
// two packed FMAs per pair.
template <int R, typename C, typename T>
__device__ __forceinline__ T mix_group_adj(C (&v)[1 << R], C (&u)[1 << R], int mask, T tu, T s) {
    C p, m;
    p.x = p.y = m.x = m.y = T(0);
#pragma unroll
    for (int j = 0; j < R; ++j) {
        if (mask & (1 << j)) {
#pragma unroll
            for (int i = 0; i < (1 << R); ++i)
                if (!(i & (1 << j))) {
                    const int b = i | (1 << j);
                    p = fma_v(u[b], v[i], p);
                    m = fma_v(u[i], v[b], m);
                    lift_inverse(v[i], v[b], tu, s);
                    lift_inverse(u[i], u[b], tu, s);
                }
        }
    }
    return (p.x + p.y) - (m.x + m.y);
}

// Shared-memory layout of a tile: position of amplitude u (p) and of energy u (e). The engine's
// own swizzle for both; the TMA tiers use the hardware's 128-byte swizzle for amplitudes and
// unswizzled energies. Both maps are linear over GF(2).
template <typename T>
struct SwzLayout {
    __device__ __forceinline__ static uint32_t p(uint32_t u) { return swz<T>(u); }
    __device__ __forceinline__ static uint32_t e(uint32_t u) { return swz<T>(u); }
};

// Element addresses of a group. Both maps are linear over GF(2) and a group's base index and its
// window offsets (i << A) have disjoint bits, so
//   p(base | (i << A)) = p(base) ^ p(i << A),   p(i << A) = xor of p(1 << (A + j)) over the set
// bits j of i: walking i in Gray-code order, each element's byte offset is the last one XOR one
// of R per-window values. The window start A is a run-time value, so that one copy of a sub-pass
// serves every window: with a copy per window start the sub-passes waited for instructions (GB300,
// stall "no instruction": 17.8 of 22 cycles per issue in a single n = 8 run, 4.5 of 14 in a batch
// of 500 instances of n = 12). One copy: that batch 76.6 -> 72.1 us, an uneven training step
// (48 instances, n = 8..24) 10.30 -> 10.02 ms, serving ticks 4% shorter.
template <int R>
struct WinSteps {
    uint32_t s[R];   // byte steps
};
template <int R, typename Map>
__device__ __forceinline__ WinSteps<R> win_steps(int a, uint32_t bytes, Map&& map) {
    WinSteps<R> w;
#pragma unroll
    for (int j = 0; j < R; ++j) w.s[j] = map(1u << (a + j)) * bytes;
    return w;
}
// Element of step k of the Gray walk, and the byte step from step k - 1 to step k (of the window
// bits from `from` on; steps are compile-time indices of unrolled loops).
__host__ __device__ constexpr int gray_elem(int k) { return k ^ (k >> 1); }
template <int R>
__device__ __forceinline__ uint32_t gray_step(const WinSteps<R>& w, int k, int from = 0) {
    int j = from;
    while (j < R - 1 && !((k >> (j - from)) & 1)) ++j;
    return w.s[j];
}

// 32-bit shared-memory accesses (the tile pointers reach the sub-passes through structs, where the
// compiler would fall back to generic 64-bit addressing).
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void lds(uint32_t a, float& v) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory"); }
__device__ __forceinline__ void lds(uint32_t a, double& v) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory"); }
__device__ __forceinline__ void lds(uint32_t a, float2& v) {
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds(uint32_t a, double2& v) {
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds2(uint32_t a, float2& v, float2& w) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(w.x), "=f"(w.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void sts(uint32_t a, const float2& v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void sts(uint32_t a, const double2& v) {
    asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void sts2(uint32_t a, const float2& v, const float2& w) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(w.x), "f"(w.y) : "memory");
}

// Load / store the 2^R elements of a group whose element 0 lies b0 bytes into the tile at shared
// address p. complex64 windows starting at bit 0 (pairs) move aligned pairs with one 16-byte shared
// access (the swizzle keeps pairs adjacent; conflict-free that way).
template <int R>
__device__ __forceinline__ void load_group(uint32_t p, uint32_t b0, bool pairs, const WinSteps<R>& w,
                                           float2 (&v)[1 << R]) {
    if (pairs) {
#pragma unroll
        for (int k = 0; k < (1 << (R - 1)); ++k) {
            if (k) b0 ^= gray_step(w, k, 1);
            const int i = 2 * gray_elem(k);
            lds2(p + b0, v[i], v[i + 1]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < (1 << R); ++k) {
            if (k) b0 ^= gray_step(w, k);
            lds(p + b0, v[gray_elem(k)]);
        }
    }
}
template <int R>
__device__ __forceinline__ void store_group(uint32_t p, uint32_t b0, bool pairs, const WinSteps<R>& w,
                                            const float2 (&v)[1 << R]) {
    if (pairs) {
#pragma unroll
        for (int k = 0; k < (1 << (R - 1)); ++k) {
            if (k) b0 ^= gray_step(w, k, 1);
            const int i = 2 * gray_elem(k);
            sts2(p + b0, v[i], v[i + 1]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < (1 << R); ++k) {
            if (k) b0 ^= gray_step(w, k);
            sts(p + b0, v[gray_elem(k)]);
        }
    }
}
template <int R>
__device__ __forceinline__ void load_group(uint32_t p, uint32_t b0, bool, const WinSteps<R>& w,
                                           double2 (&v)[1 << R]) {
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
        if (k) b0 ^= gray_step(w, k);
        lds(p + b0, v[gray_elem(k)]);
    }
}
template <int R>
__device__ __forceinline__ void store_group(uint32_t p, uint32_t b0, bool, const WinSteps<R>& w,
                                            const double2 (&v)[1 << R]) {
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
        if (k) b0 ^= gray_step(w, k);
        sts(p + b0, v[gray_elem(k)]);
    }
}
// fn(i, e) for every element i of a group with its energy e (element 0 lies b0 bytes into the
// energies at shared address p)
template <int R, typename T, typename Fn>
__device__ __forceinline__ void for_energies(uint32_t p, uint32_t b0, const WinSteps<R>& w, Fn&& fn) {
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
        if (k) b0 ^= gray_step(w, k);
        T e;
        lds(p + b0, e);
        fn(gray_elem(k), e);
    }
}

// Shared state of one tile.
template <typename T>
struct TileRef {
    typename Num<T>::C* psi;   // 2^tb amplitudes, swizzled
    typename Num<T>::C* lam;   // adjoint state (or nullptr)
    const T* E;                // 2^tb energies, swizzled
    int tb;                    // tile bits
};

// A copy of x that the compiler cannot trace to it: what is formed from it is formed there.
__device__ __forceinline__ int opaque(int x) {
    asm volatile("" : "+r"(x));
    return x;
}

// Forward sub-pass over all groups of the tile. Groups of 64 registers (5 complex64 qubits, 4 complex128)
// form the steps of the energies' walk anew at each cost phase: held across the mixers they cost 112 bytes
// of spills in the resident kernel (304 instances of n = 13, p = 6: 74.3 us so, 68.8 now; qaoa_run_layers at
// n = 22, p = 5: 210 us, 187 now). Smaller groups have the registers (n = 11, 1000 instances: 54.7 us, 56.7 anew).
//   init:  amplitudes start as |+> (amp0 i^{|z|} in the rotated frame; pc0 = number of set
//          global bits that the tile index itself fixes) instead of being read
template <typename T, int R, typename K>
__device__ __forceinline__ void subpass_fwd(const TileRef<T>& t, const SubPass& sp,
                                            const K* lc, bool init, T amp0, int pc0) {
    using C = typename Num<T>::C;
    const auto map = [](uint32_t u) { return swz<T>(u); };
    const uint32_t apsi = smem_addr(t.psi), aE = smem_addr(t.E);
    constexpr bool tight = (sizeof(C) << R) >= 256;
    const WinSteps<R> ws = win_steps<R>(sp.a, sizeof(C), map), we0 = win_steps<R>(sp.a, sizeof(T), map);
    const uint32_t ngroups = 1u << (t.tb - R);
    for (uint32_t g = threadIdx.x; g < ngroups; g += blockDim.x) {
        const uint32_t base = group_base<R>(g, sp.a);
        const uint32_t sb = swz<T>(base);
        C v[1 << R];
        if (init) {
            // |+> in the rotated frame: amp0 i^{|z|}, |z| = pc0 + |base| + |i|; the four
            // values i^m amp0 are formed once and picked by the compile-time |i|
            const int pb = pc0 + __popc(base);
            C a;
            a.x = amp0;
            a.y = T(0);
            const C q0 = times_i_pow(a, pb), q1 = times_i_pow(a, pb + 1);
            const C q2 = times_i_pow(a, pb + 2), q3 = times_i_pow(a, pb + 3);
#pragma unroll
            for (int i = 0; i < (1 << R); ++i) {
                const int m = __popc(i) & 3;
                v[i] = m == 0 ? q0 : (m == 1 ? q1 : (m == 2 ? q2 : q3));
            }
        } else {
            load_group<R>(apsi, sb * (uint32_t)sizeof(C), sp.a == 0, ws, v);
        }
#pragma unroll 1
        for (int l = sp.la; l <= sp.lb; ++l) {
            if (l > sp.la || sp.ph_first) {
                const WinSteps<R> we = tight ? win_steps<R>(opaque(sp.a), sizeof(T), map) : we0;
                const auto ph = fwd_phase(lc[l], pc0 + __popc(base));
                for_energies<R, T>(aE, sb * (uint32_t)sizeof(T), we, [&](int i, T e) { ph.apply(v[i], i, e); });
            }
            mix_layer<R>(v, sp.mask, lc[l]);
        }
        if (sp.post) finish_group<R>(v, lc[sp.lb], pc0 + __popc(base));
        store_group<R>(apsi, sb * (uint32_t)sizeof(C), sp.a == 0, ws, v);
    }
}

// Adjoint sub-pass: the forward sub-pass `sp` undone on psi and lam, accumulating for layer l,
// slot = top - l (0 or 1),
//   acc[slot] += Im <lam| sum_q X_q |psi> (window qubits),  acc[2 + slot] += Im <lam| E |psi> (its
// cost phase). lam_from_E: lam = E psi is formed on load (first adjoint sub-pass).
template <typename T, int R, typename Lay = SwzLayout<T>>
__device__ __forceinline__ void subpass_adj(const TileRef<T>& t, const SubPass& sp,
                                            const LayerConst<T>* lc, bool lam_from_E, int top, T (&acc)[4]) {
    using C = typename Num<T>::C;
    const uint32_t apsi = smem_addr(t.psi), alam = smem_addr(t.lam), aE = smem_addr(t.E);
    const WinSteps<R> ws = win_steps<R>(sp.a, sizeof(C), [](uint32_t u) { return Lay::p(u); });
    const WinSteps<R> we = win_steps<R>(sp.a, sizeof(T), [](uint32_t u) { return Lay::e(u); });
    const uint32_t ngroups = 1u << (t.tb - R);
    for (uint32_t g = threadIdx.x; g < ngroups; g += blockDim.x) {
        const uint32_t base = group_base<R>(g, sp.a);
        const uint32_t sb = Lay::p(base) * (uint32_t)sizeof(C), eb = Lay::e(base) * (uint32_t)sizeof(T);
        C v[1 << R], u[1 << R];
        load_group<R>(apsi, sb, sp.a == 0, ws, v);
        if (lam_from_E) {
            for_energies<R, T>(aE, eb, we, [&](int i, T e) {
                u[i].x = e * v[i].x;
                u[i].y = e * v[i].y;
            });
        } else {
            load_group<R>(alam, sb, sp.a == 0, ws, u);
        }
#pragma unroll 1
        for (int l = sp.lb; l >= sp.la; --l) {
            const T ab = mix_group_adj<R>(v, u, sp.mask, lc[l].t, lc[l].sn);
            if (l == top) acc[0] += ab; else acc[1] += ab;
            if (l > sp.la || sp.ph_first) {
                const PhaseK<T> ph = lc[l].ph;
                T ag[4] = {T(0), T(0), T(0), T(0)};
                for_energies<R, T>(aE, eb, we, [&](int i, T e) {
                    ag[i & 3] = fma(e, im_conj_mul(u[i], v[i]), ag[i & 3]);
                    T s, c;
                    sincos_phase(ph, e, s, c);
                    rot_neg(v[i], -s, c);
                    rot_neg(u[i], -s, c);
                });
                const T agt = (ag[0] + ag[1]) + (ag[2] + ag[3]);
                if (l == top) acc[2] += agt; else acc[3] += agt;
            }
        }
        store_group<R>(apsi, sb, sp.a == 0, ws, v);
        store_group<R>(alam, sb, sp.a == 0, ws, u);
    }
}

// ---- energies of a tile -----------------------------------------------------------------
// E(z) = z^T Q z for the 2^L tile indices u of one n-qubit instance, z = zfix | u (zfix holds
// global bits >= L that the tile fixes, e.g. the CTA rank of a cluster). With u split into
// three bit fields lo = [0, B), ha = [B, B+A), hb = [B+A, L) and S = the set bits of zfix:
//   E(z) = E_S + El[lo] + Ea[ha] + Eb[hb] + Xa[lo][ha] + Xb[lo][hb] + Xab[ha][hb],
//   El[lo]  = sum_{i,j in lo} Q_ij + sum_{i in lo, j in S} (Q_ij + Q_ji)   (Ea, Eb likewise),
//   Xa[lo][ha] = sum_{i in lo, j in ha} (Q_ij + Q_ji)                        (Xb, Xab likewise).
// Every pair of set bits of z falls in exactly one term. The tables are small (a few KB)
// and built in parallel; then every element is six table reads and six adds, independent of
// all other elements (no serial walk). scratch: tile_energy_scratch(L) values of T.
__host__ __device__ inline void energy_fields(int L, int& B, int& A) {
    B = (L + 1) / 2;
    A = (L - B) / 2;
}
__host__ __device__ inline size_t tile_energy_scratch(int L) {
    int B, A;
    energy_fields(L, B, A);
    const int Hb = L - B - A;
    return 1 + ((size_t)1 << B) + ((size_t)1 << A) + ((size_t)1 << Hb) +
           ((size_t)1 << (B + A)) + ((size_t)1 << (B + Hb)) + ((size_t)1 << (A + Hb));
}

template <typename T>
__device__ __forceinline__ T pair_sum(const T* Qs, int n, uint32_t x, int xs, uint32_t y, int ys) {
    // sum over set bits i of x (shifted by xs) and j of y (shifted by ys) of Q_ij + Q_ji
    T acc = T(0);
    for (uint32_t bi = x; bi; bi &= bi - 1u) {
        const int i = xs + __ffs((int)bi) - 1;
        for (uint32_t bj = y; bj; bj &= bj - 1u) {
            const int j = ys + __ffs((int)bj) - 1;
            acc += Qs[i * n + j] + Qs[j * n + i];
        }
    }
    return acc;
}
template <typename T>
__device__ __forceinline__ T self_sum(const T* Qs, int n, uint32_t x, int xs, uint32_t zfix) {
    // sum_{i,j in x} Q_ij + sum_{i in x, j in zfix} (Q_ij + Q_ji)
    T acc = T(0);
    for (uint32_t bi = x; bi; bi &= bi - 1u) {
        const int i = xs + __ffs((int)bi) - 1;
        for (uint32_t bj = x; bj; bj &= bj - 1u) acc += Qs[i * n + xs + __ffs((int)bj) - 1];
        for (uint32_t bj = zfix; bj; bj &= bj - 1u) {
            const int j = __ffs((int)bj) - 1;
            acc += Qs[i * n + j] + Qs[j * n + i];
        }
    }
    return acc;
}

template <typename T>
__device__ __forceinline__ void build_tile_energy(int n, int L, uint32_t zfix, const T* Qs, T* E,
                                                  T* scratch) {
    int B, A;
    energy_fields(L, B, A);
    const int Hb = L - B - A;
    const uint32_t NL = 1u << B, NA = 1u << A, NB = 1u << Hb;
    T* Es = scratch;
    T* El = Es + 1;
    T* Ea = El + NL;
    T* Eb = Ea + NA;
    T* Xa = Eb + NB;            // [ha][lo]: consecutive lanes read consecutive lo (no conflicts)
    T* Xb = Xa + NL * NA;       // [hb][lo]
    T* Xab = Xb + NL * NB;      // [ha][hb] (one address per warp: broadcast)
    const uint32_t total = 1u + NL + NA + NB + NL * NA + NL * NB + NA * NB;
    for (uint32_t x = threadIdx.x; x < total; x += blockDim.x) {
        uint32_t y = x;
        if (y == 0) {                                   // E_S
            T acc = T(0);
            for (uint32_t bi = zfix; bi; bi &= bi - 1u) {
                const int i = __ffs((int)bi) - 1;
                for (uint32_t bj = zfix; bj; bj &= bj - 1u) acc += Qs[i * n + __ffs((int)bj) - 1];
            }
            Es[0] = acc;
            continue;
        }
        y -= 1;
        if (y < NL) { El[y] = self_sum(Qs, n, y, 0, zfix); continue; }
        y -= NL;
        if (y < NA) { Ea[y] = self_sum(Qs, n, y, B, zfix); continue; }
        y -= NA;
        if (y < NB) { Eb[y] = self_sum(Qs, n, y, B + A, zfix); continue; }
        y -= NB;
        if (y < NL * NA) { Xa[y] = pair_sum(Qs, n, y & (NL - 1u), 0, y >> B, B); continue; }
        y -= NL * NA;
        if (y < NL * NB) { Xb[y] = pair_sum(Qs, n, y & (NL - 1u), 0, y >> B, B + A); continue; }
        y -= NL * NB;
        Xab[y] = pair_sum(Qs, n, y >> Hb, B, y & (NB - 1u), B + A);
    }
    __syncthreads();
    const T es = Es[0];
    for (uint32_t u = threadIdx.x; u < (1u << L); u += blockDim.x) {
        const uint32_t lo = u & (NL - 1u), ha = (u >> B) & (NA - 1u), hb = u >> (B + A);
        E[swz<T>(u)] = ((es + El[lo]) + (Ea[ha] + Eb[hb])) +
                       ((Xa[(ha << B) | lo] + Xb[(hb << B) | lo]) + Xab[(ha << Hb) | hb]);
    }
}

// Fast path of the tile energies when blockDim = 2^(L - HB): thread t owns the low field
// lo = t (B = L - HB bits) and the 2^HB elements u = t | (j << B). With S the set bits of zfix
//   E(z) = [E_S + El(t)] + Eh[j] + X_t(j),   X_t(j) = sum_{b in j} W_b(t),
//   W_b(t) = sum_{i in t} (Q_{i,B+b} + Q_{B+b,i}),
// El(t) and W_b(t) are evaluated by the thread (sums over the set bits of t), Eh (2^HB
// entries, shared) by 2^HB threads, and X_t(j) for all j by subset doubling in registers
// (2^HB - 1 additions). Each element is then one broadcast read, two adds and one store.
// Optional fused start of the state: with psi != nullptr every element is also set to the
// |+> amplitude after the first cost layer, amp0 i^{|z|} e^{-i gamma_0 E(z)} (rotated frame,
// |z| = pc0 + |u|), so the first sub-pass starts with the first mixer.
template <typename T>
struct FusedInit {
    typename Num<T>::C* psi;   // nullptr: energies only
    T amp0, gpi0;              // 2^{-n/2}, gamma_0 / pi
    int pc0;                   // set bits of zfix
    bool two = false;          // the phase from the two-float ph instead of gpi0 (gradients, complex64)
    PhaseK<T> ph{};
};

template <typename T>
__device__ __forceinline__ void fused_init_store(const FusedInit<T>& fi, uint32_t u, uint32_t ix, T e) {
    typename Num<T>::C a;
    T s, c;
    if constexpr (sizeof(T) == 4) {
        if (fi.two) sincos_phase(fi.ph, e, s, c);
        else sincos_gpi(fi.gpi0, e, s, c);
    } else sincospi(fi.gpi0 * e, &s, &c);
    a.x = fi.amp0 * c;          // amp0 e^{-i theta}
    a.y = -fi.amp0 * s;
    fi.psi[ix] = times_i_pow(a, fi.pc0 + __popc(u));
}

template <typename T, int HB>
__device__ __forceinline__ void build_tile_energy_fast(int n, int L, uint32_t zfix, const T* Qs,
                                                       T* E, T* scratch, const FusedInit<T>& fi) {
    const int B = L - HB;
    const uint32_t t = threadIdx.x;
    T* Eh = scratch;                 // 2^HB entries: hi self terms + hi x S
    if (t < (1u << HB)) {
        T acc = T(0);
        const uint32_t hbits = t << B;
        for (uint32_t bi = hbits; bi; bi &= bi - 1u) {
            const int i = __ffs((int)bi) - 1;
            for (uint32_t bj = hbits; bj; bj &= bj - 1u) acc += Qs[i * n + __ffs((int)bj) - 1];
            for (uint32_t bj = zfix; bj; bj &= bj - 1u) {
                const int j = __ffs((int)bj) - 1;
                acc += Qs[i * n + j] + Qs[j * n + i];
            }
        }
        Eh[t] = acc;
    }
    // E_S + El(t), and W_b(t): loops over bit positions (the same for every lane, so each Q
    // read is a shared-memory broadcast) with predicated adds instead of loops over the set
    // bits of t (which diverge across the warp)
    T base = T(0);
    for (uint32_t bi = zfix; bi; bi &= bi - 1u) {
        const int i = __ffs((int)bi) - 1;
        for (uint32_t bj = zfix; bj; bj &= bj - 1u) base += Qs[i * n + __ffs((int)bj) - 1];
    }
    for (int i = 0; i < B; ++i) {
        const bool ti = (t >> i) & 1u;
        T si = Qs[i * n + i];
        for (uint32_t bj = zfix; bj; bj &= bj - 1u) {
            const int j = __ffs((int)bj) - 1;
            si += Qs[i * n + j] + Qs[j * n + i];
        }
        T cross = T(0);
        for (int j = 0; j < i; ++j)
            if ((t >> j) & 1u) cross += Qs[i * n + j] + Qs[j * n + i];
        if (ti) base += si + cross;
    }
    T X[1 << HB];
    X[0] = T(0);
#pragma unroll
    for (int b = 0; b < HB; ++b) {
        T w = T(0);
        const int q = B + b;
        for (int i = 0; i < B; ++i)
            if ((t >> i) & 1u) w += Qs[i * n + q] + Qs[q * n + i];
#pragma unroll
        for (int m = 0; m < (1 << b); ++m) X[m | (1 << b)] = X[m] + w;
    }
    __syncthreads();
    const uint32_t st = swz<T>(t);
#pragma unroll
    for (int j = 0; j < (1 << HB); ++j) {
        const uint32_t ix = st ^ swz<T>((uint32_t)j << B);
        const T ev = base + (Eh[j] + X[j]);
        E[ix] = ev;
        if (fi.psi) fused_init_store(fi, t | ((uint32_t)j << B), ix, ev);
    }
}

// Energies of the tile (fast path when blockDim = 2^(L - HB), HB <= 5), and optionally the
// fused start of the state (see FusedInit). Returns true if the state was started. Not
// inlined: its 2^HB register subset sums would otherwise add to the register pressure of the
// whole calling kernel (spills there cost more than the call).
template <typename T>
__device__ __noinline__ bool build_tile_energy_any(int n, int L, uint32_t zfix, const T* Qs,
                                                      T* E, T* scratch, const FusedInit<T>& fi) {
    const int lg = 31 - __clz((int)blockDim.x);
    switch (L - lg) {
        case 0: build_tile_energy_fast<T, 0>(n, L, zfix, Qs, E, scratch, fi); return fi.psi != nullptr;
        case 1: build_tile_energy_fast<T, 1>(n, L, zfix, Qs, E, scratch, fi); return fi.psi != nullptr;
        case 2: build_tile_energy_fast<T, 2>(n, L, zfix, Qs, E, scratch, fi); return fi.psi != nullptr;
        case 3: build_tile_energy_fast<T, 3>(n, L, zfix, Qs, E, scratch, fi); return fi.psi != nullptr;
        case 4: build_tile_energy_fast<T, 4>(n, L, zfix, Qs, E, scratch, fi); return fi.psi != nullptr;
        case 5: build_tile_energy_fast<T, 5>(n, L, zfix, Qs, E, scratch, fi); return fi.psi != nullptr;
        default: build_tile_energy<T>(n, L, zfix, Qs, E, scratch); return false;
    }
}

// ---- final reductions of a tile -----------------------------------------------------------
// Shared-memory placement of tile index u for the state (p) and the energies (e): the engine's
// swizzle for both (default), or another layout supplied by a tier (a TMA-staged tile).

// Shared scratch of tile_reduce (sizes: wb 16 * nwarps floats, cand TOPK_CAP entries, out 16,
// wlists 32 * nwarps entries, cnt 4 ints).
constexpr int TOPK_CAP = 256;
struct TileTopk {
    float* wb;        // per-warp sorted lane maxima (k per warp)
    TopEnt* cand;     // candidate buffer
    TopEnt* out;      // the tile's top-k (valid after tile_reduce)
    TopEnt* wlists;   // (blockDim/32) * 32 entries, used only by the fallback
    int* cnt;         // [0] candidate count, [1] overflow flag, [2..3] bound (float / double bits)
};

// Collect the elements whose probability can reach `bound_lo` (FP32 filter with the margins of
// WarpTopK::offer; with exact_bound != 0 the exact probability must also be >= *exact_bound)
// into ts.cand. Sets ts.cnt[1] on overflow. Each thread scans only its own elements
// u = tid + j * blockDim, and only if its FP32 maximum over them (pmax, from the pass that
// computed the tile's <C> partial) can reach the bound: a list of k entries has few owners, so
// most threads skip the scan. pmax and the per-element value are two FP32 roundings of the same
// probability, each within 2^-21 of it, hence the wider 2^-18 margin of the thread test.
template <typename T, typename Lay = SwzLayout<T>, typename ZMap>
__device__ __forceinline__ void collect_candidates(const TileRef<T>& t, float pmax, float bound_lo,
                                                   const double* exact_bound, ZMap&& zmap,
                                                   const TileTopk& ts) {
    using C = typename Num<T>::C;
    const uint32_t D = 1u << t.tb;
    if (!(pmax * 1.000003814697265625f >= bound_lo)) return;
    const long long eb = exact_bound ? pbits(*exact_bound) : -1ll;
    for (uint32_t c0 = 0; c0 < D; c0 += 32u * blockDim.x) {
        // FP32 test of up to 32 elements first (independent loads), then the hits one by one
        uint32_t hits = 0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const uint32_t u = c0 + (uint32_t)j * blockDim.x + threadIdx.x;
            if (u < D) {
                const C v = t.psi[Lay::p(u)];
                const float pf = (float)v.x * (float)v.x + (float)v.y * (float)v.y;
                if (pf * 1.00000095367431640625f >= bound_lo) hits |= 1u << j;
            }
        }
        while (hits) {
            const int j = __ffs(hits) - 1;
            hits &= hits - 1;
            const uint32_t u = c0 + (uint32_t)j * blockDim.x + threadIdx.x;
            const double pe = exact_prob(t.psi[Lay::p(u)]);
            if (pbits(pe) >= eb) {
                const int pos = atomicAdd(&ts.cnt[0], 1);
                if (pos < TOPK_CAP) ts.cand[pos] = TopEnt{pe, zmap(u)};
                else ts.cnt[1] = 1;
            }
        }
    }
}

// <C> partial of the tile (FP32 |psi|^2 E over at most 32 elements per thread, FP64 above, added
// to `ex`) and the thread's largest FP32 probability over its elements u = tid + j * blockDim
// (its lane maximum, returned). Called by all threads; no barrier.
template <typename T, typename Lay = SwzLayout<T>>
__device__ __forceinline__ float tile_expect(const TileRef<T>& t, double& ex) {
    using C = typename Num<T>::C;
    const uint32_t D = 1u << t.tb;
    float pmax = -1.0f;
    for (uint32_t c0 = 0; c0 < D; c0 += 32u * blockDim.x) {
        T accp = T(0);
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const uint32_t u = c0 + (uint32_t)j * blockDim.x + threadIdx.x;
            if (u < D) {
                const C v = t.psi[Lay::p(u)];
                const T pr = v.x * v.x + v.y * v.y;
                accp += pr * t.E[Lay::e(u)];
                pmax = fmaxf(pmax, (float)pr);
            }
        }
        ex += (double)accp;
    }
    return pmax;
}

// Top-k list of the whole tile into ts.out, given each thread's lane maximum pmax:
//  1. a lower bound on the tile's k-th largest probability: the k-th largest of all lane
//     maxima (k distinct elements are at least that probable). Each warp sorts its lane
//     maxima and offers its k largest; their k-th largest is found by rank;
//  2. every element whose probability can reach the bound goes to a shared candidate buffer
//     with its exact FP64 probability; on overflow (flat distributions) the bound is raised
//     to the k-th largest exact probability among the buffered elements and the collection
//     repeated with an exact test;
//  3. each candidate's rank = number of candidates better than it (probability descending,
//     index ascending: a strict total order, so ranks are distinct); ranks < k are the list.
// The result does not depend on the order of the buffer, so the reduction is deterministic.
// If the buffer still overflows (massive ties) the warps fall back to sorted insertion lists
// merged by warp 0. zmap(u): global index of tile index u. Called by all threads, k >= 1.
template <typename T, typename Lay = SwzLayout<T>, typename ZMap>
__device__ __forceinline__ void tile_topk(const TileRef<T>& t, int k, float pmax, ZMap&& zmap,
                                          const TileTopk& ts) {
    using C = typename Num<T>::C;
    const uint32_t D = 1u << t.tb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    // (1) the k-th largest lane maximum of the block
    const float srt = warp_sort_desc(pmax);
    if (lane < k) ts.wb[warp * k + lane] = srt;
    if (threadIdx.x == 0) { ts.cnt[0] = 0; ts.cnt[1] = 0; }
    __syncthreads();
    float* bound = reinterpret_cast<float*>(&ts.cnt[2]);
    const int nl = nw * k;
    for (int i = threadIdx.x; i < nl; i += blockDim.x) {
        const float me = ts.wb[i];
        int rank = 0;
        for (int j = 0; j < nl; ++j) {
            const float o = ts.wb[j];
            rank += (o > me || (o == me && j < i)) ? 1 : 0;
        }
        if (rank == k - 1) *bound = me;
    }
    __syncthreads();
    const float thr = *bound;
    const float thr_lo = thr > 0.0f ? thr * 0.99999904632568359375f : -1.0f;   // (1 - 2^-20)
    // (2) candidates
    collect_candidates<T, Lay>(t, pmax, thr_lo, nullptr, zmap, ts);
    __syncthreads();
    if (ts.cnt[1]) {
        // raise the bound to the k-th best buffered exact probability and collect again
        double* b2 = reinterpret_cast<double*>(ts.wlists);
        for (int c = threadIdx.x; c < TOPK_CAP; c += blockDim.x) {
            const TopEnt me = ts.cand[c];
            int rank = 0;
            for (int j = 0; j < TOPK_CAP; ++j) {
                const TopEnt o = ts.cand[j];
                rank += better(o.p, o.z, me.p, me.z) ? 1 : 0;
            }
            if (rank == k - 1) *b2 = me.p;
        }
        __syncthreads();
        const float b2lo = __double2float_rd(*b2) * 0.99999904632568359375f;
        if (threadIdx.x == 0) { ts.cnt[0] = 0; ts.cnt[1] = 0; }
        __syncthreads();
        collect_candidates<T, Lay>(t, pmax, b2lo, b2, zmap, ts);
        __syncthreads();
    }
    const int cnt = min(ts.cnt[0], TOPK_CAP);
    if (!ts.cnt[1]) {
        // (3) rank selection
        for (int c = threadIdx.x; c < cnt; c += blockDim.x) {
            const TopEnt me = ts.cand[c];
            int rank = 0;
            for (int j = 0; j < cnt; ++j) {
                const TopEnt o = ts.cand[j];
                rank += better(o.p, o.z, me.p, me.z) ? 1 : 0;
            }
            if (rank < k) ts.out[rank] = me;
        }
        if (threadIdx.x < (unsigned)k && threadIdx.x >= (unsigned)cnt) ts.out[threadIdx.x] = TopEnt{-1.0, 0xffffffffu};
    } else {
        __syncthreads();
        WarpTopK top;
        top.init(k);
        for (uint32_t u0 = 0; u0 < D; u0 += blockDim.x) {
            const uint32_t u = u0 + threadIdx.x;
            C v;
            v.x = T(0);
            v.y = T(0);
            if (u < D) v = t.psi[Lay::p(u)];
            top.offer(v, zmap(u < D ? u : 0u), u < D);
        }
        if (lane < k) ts.wlists[warp * 32 + lane] = TopEnt{top.p, top.z};
        __syncthreads();
        if (warp == 0) {
            WarpTopK f;
            f.init(k);
            for (int w = 0; w < nw; ++w) {
                const bool ok = lane < k;
                const TopEnt e = ok ? ts.wlists[w * 32 + lane] : TopEnt{-1.0, 0xffffffffu};
                f.offer_exact(e.p, e.z, ok);
            }
            if (lane < k) ts.out[lane] = TopEnt{f.p, f.z};
        }
    }
    __syncthreads();
}

// <C> partial (added to `ex`) and, for k >= 1, the top-k list (ts.out) of the whole tile after
// its last sub-pass. Called by all threads.
template <typename T, typename Lay = SwzLayout<T>, typename ZMap>
__device__ __forceinline__ void tile_reduce(const TileRef<T>& t, int k, ZMap&& zmap,
                                            const TileTopk& ts, double& ex) {
    const float pmax = tile_expect<T, Lay>(t, ex);
    if (k <= 0) return;
    tile_topk<T, Lay>(t, k, pmax, zmap, ts);
}

// Fold the tile into `run`, the top-k list (k entries, all present) of the tiles of the same
// state that this block reduced before: only elements that can beat run's k-th entry are
// collected (usually none once a few tiles are in), and the merged list is the k best of the
// candidates and run by rank. On candidate overflow the tile's own list (tile_topk) is merged
// instead. pmax as from tile_expect. Called by all threads.
template <typename T, typename ZMap>
__device__ __forceinline__ void running_topk(const TileRef<T>& t, int k, float pmax, ZMap&& zmap,
                                             const TileTopk& ts, TopEnt* run) {
    const double* pk = &run[k - 1].p;
    const float lo = __double2float_rd(*pk) * 0.99999904632568359375f;
    if (threadIdx.x == 0) { ts.cnt[0] = 0; ts.cnt[1] = 0; }
    if (!__syncthreads_or(pmax * 1.000003814697265625f >= lo)) return;
    collect_candidates<T>(t, pmax, lo, pk, zmap, ts);
    __syncthreads();
    const TopEnt* a = ts.cand;
    int na = ts.cnt[0];
    if (ts.cnt[1]) {
        __syncthreads();                        // every thread has read the counters that tile_topk resets
        tile_topk<T>(t, k, pmax, zmap, ts);
        a = ts.out;
        na = k;
    }
    if (na == 0) return;                        // uniform: every thread read the same count
    TopEnt* merged = ts.wlists;                 // free here (tile_topk ended with a barrier)
    for (int c = threadIdx.x; c < na + k; c += blockDim.x) {
        const TopEnt me = c < na ? a[c] : run[c - na];
        if (!is_entry(me.p)) continue;
        int rank = 0;
        for (int j = 0; j < na; ++j) rank += better(a[j].p, a[j].z, me.p, me.z) ? 1 : 0;
        for (int j = 0; j < k; ++j) rank += better(run[j].p, run[j].z, me.p, me.z) ? 1 : 0;
        if (rank < k) merged[rank] = me;
    }
    __syncthreads();
    if (threadIdx.x < (unsigned)k) run[threadIdx.x] = merged[threadIdx.x];
    __syncthreads();
}

// Top-k of a small set of candidate lists already in shared memory (count entries, entries
// with p < 0 are empty): rank selection as in tile_reduce; result in out[0..k).
__device__ __forceinline__ void rank_select(const TopEnt* cand, int count, int k, TopEnt* out) {
    for (int c = threadIdx.x; c < count; c += blockDim.x) {
        const TopEnt me = cand[c];
        if (!is_entry(me.p)) continue;
        int rank = 0;
        for (int j = 0; j < count; ++j) {
            const TopEnt o = cand[j];
            rank += (is_entry(o.p) && better(o.p, o.z, me.p, me.z)) ? 1 : 0;
        }
        if (rank < k) out[rank] = me;
    }
}

// Block-wide FP64 sums of four values per thread, fixed order. In a warp the four reductions share
// their first two steps (each lane hands over half of what it holds), six FP64 adds a lane
// instead of twenty: FP64 issues at 1/64 of the FP32 rate. red: 4 * (blockDim / 32) doubles, at
// most 16 warps. Lane j < 4 of warp 0 returns the sum of value j. Called by all threads.
__device__ __forceinline__ double block_sum4(double v0, double v1, double v2, double v3, double* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    const bool o1 = lane & 1, o2 = lane & 2;
    const double a = (o1 ? v2 : v0) + __shfl_xor_sync(0xffffffffu, o1 ? v0 : v2, 1);
    const double b = (o1 ? v3 : v1) + __shfl_xor_sync(0xffffffffu, o1 ? v1 : v3, 1);
    double c = (o2 ? b : a) + __shfl_xor_sync(0xffffffffu, o2 ? a : b, 2);   // lane & 3 holds v0, v2, v1, v3
#pragma unroll
    for (int o = 4; o <= 16; o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    __syncthreads();
    if (lane < 4) red[4 * w + (lane == 1 ? 2 : (lane == 2 ? 1 : lane))] = c;
    __syncthreads();
    double tot = 0.0;
    if (w == 0) {   // lane 4 i + j: value j of warps i and i + 8
        const int i = lane >> 2;
        if (i < nw) tot = red[lane];
        if (i + 8 < nw) tot += red[lane + 32];
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    return tot;
}

// Block-wide sum of one value per thread into slot[0] (thread 0 only); red has blockDim/32
// doubles. Fixed order: deterministic. Must be called by all threads.
__device__ __forceinline__ double block_sum(double v, double* red) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double tot = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < nw; ++i) tot += red[i];
    return tot;
}

}  // namespace qaoa
