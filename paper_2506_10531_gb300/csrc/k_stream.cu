// k_stream.cu -- HBM-streaming tier for states larger than one SM's shared memory, plus the
// standalone energy build.
//
// A layer of Eq. 2 (Section IV) on a 2^n state is split into HBM passes. Each pass moves
// tiles of 2^tb amplitudes between HBM and shared memory and runs the tile engine on them:
//   kind A: the tile is 2^tb contiguous amplitudes; its tile bits are qubits 0..tb-1;
//   kind B: the tile is 2^c contiguous amplitudes (qubits 0..c-1, c >= 4, so every run is at
//           least 128 bytes) times 2^h values of the high qubits [s, s+h), c + h = tb; only the
//           high qubits are mixed.
// The HBM passes follow the same snake order as the windows of a tile (A, B1, B2, ... then
// back), so consecutive layers share a pass; the cost phase of a layer is fused into the pass
// that opens it, |+> is generated in the first pass, and <C> plus the top-k candidates are
// reduced in the last one (per-tile partials, then one fixed-order finalize per instance).
#include "qaoa_engine.cuh"
#include "qaoa_kernels.h"
#include "qaoa_stream.h"
#include "qaoa_topk.cuh"

namespace qaoa {

namespace {

// Tiles of a single state (see the host side): windows, sizes with tiles of their own, first upper qubit.
constexpr int SMALL_R = 3, SMALL_NMIN = 15, SMALL_NMAX = 20, SMALL_LOW = 13, SMALL_RA = 4, SMALL_GRAD_NMAX = 21;

// Windows of a layer for tiles of tb bits whose kind-B chunks keep 2^cmin contiguous amplitudes.
__host__ __device__ inline int stream_windows(int n, int tb, int cmin) {
    return 1 + (n - tb + tb - cmin - 1) / (tb - cmin);
}

// Global index of tile-local index u for tile tau of pass P.
__device__ __forceinline__ uint64_t global_index(const StreamPass& P, uint64_t tau, uint32_t u) {
    if (P.kind == 0) return (tau << P.tb) | u;
    const uint64_t lo = u & ((1u << P.c) - 1u);
    const uint64_t hi = u >> P.c;
    const int midbits = P.s - P.c;
    const uint64_t mid = tau & ((1ull << midbits) - 1ull);
    const uint64_t top = tau >> midbits;
    return lo | (mid << P.c) | (hi << P.s) | (top << (P.s + P.h));
}

// Per-thread strided walk over a tile: element u = u0 + j * step (step a multiple of 2^c for kind
// B, any for kind A) has global index global_index(P, tau, u0) + j * gstep. Returns false when
// kind B's contiguous run is longer than the step (then the index is formed per element).
__device__ __forceinline__ bool linear_walk(const StreamPass& P, uint32_t step, uint64_t& gstep) {
    if (step < 512u) return false;   // the swizzle permutes bits 1..8: a shorter stride would not advance linearly
    if (P.kind == 0) { gstep = step; return true; }
    if (step & ((1u << P.c) - 1u)) return false;
    gstep = (uint64_t)(step >> P.c) << P.s;
    return true;
}

// Stage the tile's amplitudes (16-byte copies) and optionally energies (8-byte copies) of
// tile tau into shared memory, asynchronously. The swizzle only permutes bits below the copy
// stride, so the shared-memory offset advances linearly as well.
template <typename T>
__device__ __forceinline__ void stage_tile(const StreamPass& P, uint64_t tau,
                                           const typename Num<T>::C* gsrc,
                                           typename Num<T>::C* sdst, const T* gE, T* sE) {
    using C = typename Num<T>::C;
    const uint32_t TD = 1u << P.tb;
    constexpr uint32_t PAIR = sizeof(C) == 8 ? 2u : 1u;   // amplitudes per 16-byte copy
    const uint32_t step = PAIR * blockDim.x, u0 = PAIR * threadIdx.x;
    uint64_t gstep;
    if (!gsrc) {
    } else if (linear_walk(P, step, gstep)) {
        const C* g = gsrc + global_index(P, tau, u0);
        C* sp = sdst + swz<T>(u0);
#pragma unroll 4
        for (uint32_t u = u0; u < TD; u += step, g += gstep, sp += step) cp_async16(sp, g);
    } else {
        for (uint32_t u = u0; u < TD; u += step) cp_async16(&sdst[swz<T>(u)], gsrc + global_index(P, tau, u));
    }
    if (gE) {
        constexpr uint32_t EP = 8u / sizeof(T);           // energies per 8-byte copy
        const uint32_t estep = EP * blockDim.x, e0 = EP * threadIdx.x;
        uint64_t egstep;
        if (linear_walk(P, estep, egstep)) {
            const T* g = gE + global_index(P, tau, e0);
            T* sp = sE + swz<T>(e0);
#pragma unroll 4
            for (uint32_t u = e0; u < TD; u += estep, g += egstep, sp += estep) cp_async8(sp, g);
        } else {
            for (uint32_t u = e0; u < TD; u += estep) cp_async8(&sE[swz<T>(u)], gE + global_index(P, tau, u));
        }
    }
}

// Write the tile back (16-byte accesses on both sides), same walk as stage_tile.
template <typename T>
__device__ __forceinline__ void store_tile(const StreamPass& P, uint64_t tau, const typename Num<T>::C* ssrc,
                                          typename Num<T>::C* gdst) {
    using C = typename Num<T>::C;
    const uint32_t TD = 1u << P.tb;
    constexpr uint32_t PAIR = sizeof(C) == 8 ? 2u : 1u;
    const uint32_t step = PAIR * blockDim.x, u0 = PAIR * threadIdx.x;
    uint64_t gstep;
    if (linear_walk(P, step, gstep)) {
        C* g = gdst + global_index(P, tau, u0);
        const C* sp = ssrc + swz<T>(u0);
        for (uint32_t u = u0; u < TD; u += step, g += gstep, sp += step)
            *reinterpret_cast<uint4*>(g) = *reinterpret_cast<const uint4*>(sp);
    } else {
        for (uint32_t u = u0; u < TD; u += step)
            *reinterpret_cast<uint4*>(gdst + global_index(P, tau, u)) =
                *reinterpret_cast<const uint4*>(&ssrc[swz<T>(u)]);
    }
}

template <typename T>
struct StreamSmem {
    typename Num<T>::C* psi;
    T* E;
    void* lc;        // forward constants: K[64]
    double* red;
    TileTopk tk;
    TopEnt* run;     // running top-k of the state's tiles this block reduced (last pass)
};

// The tile's copies HBM -> shared: asynchronous, all in flight before the wait in stream_tile
// (tile bit 0 is global bit 0 and c >= 1, so aligned pairs stay adjacent in both layouts).
template <typename T>
__device__ __forceinline__ void stream_stage(const StreamPass& P, const StreamInst<T>& I, uint64_t tau,
                                             const StreamSmem<T>& s) {
    using C = typename Num<T>::C;
    if (!P.init) stage_tile<T>(P, tau, reinterpret_cast<C*>(I.psi), s.psi, P.need_e ? I.E : nullptr, s.E);
    else if (P.need_e) stage_tile<T>(P, tau, nullptr, nullptr, I.E, s.E);
}

// One staged tile. have_run: this block reduced tile prev_tau of the same state just before (last
// pass, k >= 1); s.run then holds the top-k of all the state's tiles it reduced so far. TOPK:
// the instantiation serves passes with a top-k.
template <typename T, int R, bool TOPK, typename K>
__device__ void stream_tile(const StreamPass& P, const StreamInst<T>& I, uint64_t tau,
                            const StreamSmem<T>& s, bool have_run, uint64_t prev_tau, const StreamSubs& subs) {
    using C = typename Num<T>::C;
    const uint32_t TD = 1u << P.tb;
    C* gpsi = reinterpret_cast<C*>(I.psi);
    cp_async_wait_all();
    __syncthreads();
    // ---- tile engine: snake over the local windows of the mixed bits, layers [la, lb] ----
    const TileRef<T> tile{s.psi, nullptr, s.E, P.tb};
    const int m0 = (P.kind == 0) ? 0 : P.c;
    const T amp0 = (T)I.amp0;
    if (subs.n > 0) {              // listed sub-passes (a single state's small tiles)
        for (int i = 0; i < subs.n; ++i) {
            const StreamSub& b = subs.sub[i];
            SubPass sp{b.a, b.mask, P.la + b.l0, P.la + b.l1, b.phase, P.fin && i == subs.n - 1};
            subpass_fwd<T, R>(tile, sp, static_cast<const K*>(s.lc), P.init && i == 0, amp0, __popcll(tau));
            __syncthreads();
        }
    } else {
        Snake sn(P.lb - P.la + 1, P.la, P.ph_first, m0, P.tb, P.tb, R);
        for (;; sn.next()) {
            SubPass sp = sn.get();
            sp.post = P.fin && sn.last();
            subpass_fwd<T, R>(tile, sp, static_cast<const K*>(s.lc), P.init && sn.first(), amp0, __popcll(tau));
            __syncthreads();
            if (sn.last()) break;
        }
    }
    // ---- shared -> HBM (16-byte accesses on both sides). Between passes the state stays in
    // the rotated frame; the last pass converts back with (-i)^{|z|} (|z| = |tau| + |u|: the
    // tile map only permutes bits). ----
    if (!P.fin || P.keep_frame) {
        store_tile<T>(P, tau, s.psi, gpsi);
    } else if (!P.no_store) {
        const int pt = __popcll(tau);
        constexpr uint32_t PAIR = sizeof(C) == 8 ? 2u : 1u;
        const uint32_t step = PAIR * blockDim.x, u0 = PAIR * threadIdx.x;
        uint64_t gstep;
        if (linear_walk(P, step, gstep)) {
            C* g = gpsi + global_index(P, tau, u0);
            for (uint32_t u = u0; u < TD; u += step, g += gstep) {
                const uint32_t su = swz<T>(u);
                if constexpr (PAIR == 2) {
                    const C a = times_i_pow(s.psi[su], -(pt + __popc(u)));
                    const C b = times_i_pow(s.psi[su + 1], -(pt + __popc(u + 1)));
                    *reinterpret_cast<float4*>(g) = make_float4(a.x, a.y, b.x, b.y);
                } else {
                    *g = times_i_pow(s.psi[su], -(pt + __popc(u)));
                }
            }
        } else {
            for (uint32_t u = threadIdx.x; u < TD; u += blockDim.x)
                gpsi[global_index(P, tau, u)] = times_i_pow(s.psi[swz<T>(u)], -(pt + __popc(u)));
        }
    }
    if (P.fin && !TOPK) {
        if (I.expect) {                        // <C> alone, and only where somebody reads it
            double ex = 0.0;
            tile_expect<T>(tile, ex);
            const double tot = block_sum(ex, s.red);
            if (threadIdx.x == 0) I.part_expect[tau] = tot;
        }
    } else if (P.fin) {
        double ex = 0.0;
        const StreamPass Pm = P;   // by value: the lambda then holds no address of a kernel parameter
        const auto zmap = [Pm, tau](uint32_t u) { return (uint32_t)global_index(Pm, tau, u); };
        const float pmax = tile_expect<T>(tile, ex);
        if (P.k > 0) {
            if (have_run) {
                running_topk<T>(tile, P.k, pmax, zmap, s.tk, s.run);
            } else {
                tile_topk<T>(tile, P.k, pmax, zmap, s.tk);
                if (threadIdx.x < (unsigned)P.k) s.run[threadIdx.x] = s.tk.out[threadIdx.x];
            }
        }
        const double tot = block_sum(ex, s.red);
        if (threadIdx.x == 0) I.part_expect[tau] = tot;
        // the running list goes to this tile's slot and the previous tile's slot is emptied (the
        // same thread wrote it), so each state's slots hold every candidate exactly once
        if (threadIdx.x < (unsigned)P.k) {
            const TopEnt e = s.run[threadIdx.x];
            I.part_topp[tau * P.k + threadIdx.x] = e.p;
            I.part_topz[tau * P.k + threadIdx.x] = e.z;
            if (have_run) {
                I.part_topp[prev_tau * P.k + threadIdx.x] = -1.0;
                I.part_topz[prev_tau * P.k + threadIdx.x] = 0xffffffffu;
            }
        }
    }
    __syncthreads();
}

template <typename T, int R, int NTH, bool TOPK, bool GRAD>   // GRAD: the forward half of gradients
__global__ void __launch_bounds__(NTH, 2) k_stream_pass(const StreamPass P,
                                                     const StreamInst<T>* __restrict__ insts,
                                                     int count, const StreamInst<T> one, const StreamSubs subs) {
    extern __shared__ __align__(16) unsigned char sm[];
    using C = typename Num<T>::C;
    using K = typename FwdFor<T, GRAD>::K;
    const uint32_t TD = 1u << P.tb;
    StreamSmem<T> s;
    size_t o = 0;
    s.psi = reinterpret_cast<C*>(sm + o); o += (size_t)TD * sizeof(C);
    s.E = reinterpret_cast<T*>(sm + o); o += (size_t)TD * sizeof(T);
    s.lc = sm + o; o += 64 * sizeof(LayerConst<T>);
    o = (o + 15) & ~(size_t)15;
    s.red = reinterpret_cast<double*>(sm + o); o += 32 * sizeof(double);
    s.tk.wlists = reinterpret_cast<TopEnt*>(sm + o); o += 8 * 32 * sizeof(TopEnt);
    s.tk.cand = reinterpret_cast<TopEnt*>(sm + o); o += TOPK_CAP * sizeof(TopEnt);
    s.tk.out = reinterpret_cast<TopEnt*>(sm + o); o += 16 * sizeof(TopEnt);
    s.run = reinterpret_cast<TopEnt*>(sm + o); o += 16 * sizeof(TopEnt);
    s.tk.wb = reinterpret_cast<float*>(sm + o); o += 16 * 32 * sizeof(float);
    s.tk.cnt = reinterpret_cast<int*>(sm + o);
    const uint64_t ntiles = 1ull << (P.n - P.tb);
    const uint64_t total = ntiles * (uint64_t)count;
    // layer constants are rebuilt only when the parameters change (instances of a batch often
    // share one parameter vector)
    const T *cur_g = nullptr, *cur_b = nullptr;
    int cur_p = 0;
    // The last pass with a top-k gives each block a run of consecutive tiles instead of a
    // grid-strided share, so that the tiles of one state follow each other and the block carries
    // one top-k list across them. The run lengths are those of the strided share: total / grid,
    // one more for the first total % grid blocks.
    uint64_t b = blockIdx.x, bstep = gridDim.x, bend = total;
    if (P.fin && P.k > 0) {
        const uint64_t q = total / gridDim.x, rem = total % gridDim.x, c = blockIdx.x;
        b = c * q + (c < rem ? c : rem);
        bend = b + q + (c < rem ? 1 : 0);
        bstep = 1;
    }
    int run_ii = -1;
    uint64_t run_tau = 0;
    for (; b < bend; b += bstep) {
        const int ii = (int)(b >> (P.n - P.tb));
        const uint64_t tau = b & (ntiles - 1);
        const StreamInst<T>& I = insts ? insts[ii] : one;
        stream_stage<T>(P, I, tau, s);   // the copies run while the constants are formed
        if (I.gamma != cur_g || I.beta != cur_b || I.p != cur_p) {
            set_fwd_consts(static_cast<K*>(s.lc), I.gamma, I.beta, I.p, P.n);
            cur_g = I.gamma;
            cur_b = I.beta;
            cur_p = I.p;
        }
        stream_tile<T, R, TOPK, K>(P, I, tau, s, run_ii == ii, run_tau, subs);
        run_ii = ii;
        run_tau = tau;
    }
}

// First merge level for instances with many tiles: block (c, i) merges the lists of tiles
// [c * FIN_CHUNK, (c + 1) * FIN_CHUNK) of instance i and writes the result over the list of the
// chunk's first tile (only this block reads the chunk, and it reads everything first).
constexpr uint64_t FIN_CHUNK = 256;

template <typename T>
__global__ void __launch_bounds__(256) k_stream_topk_chunks(const StreamInst<T>* __restrict__ insts,
                                                           int count, uint64_t ntiles, int k,
                                                           const StreamInst<T> one) {
    __shared__ TopScratch ts;
    const int ii = blockIdx.y;
    if (ii >= count) return;
    const StreamInst<T>& I = insts ? insts[ii] : one;
    const uint64_t t0 = (uint64_t)blockIdx.x * FIN_CHUNK;
    const uint64_t nl = (ntiles - t0) < FIN_CHUNK ? (ntiles - t0) : FIN_CHUNK;
    // merge_entries ends with a barrier: every read of the chunk is done before its first list is
    // overwritten
    double* topp = I.part_topp + t0 * k;
    uint32_t* topz = I.part_topz + t0 * k;
    merge_entries(nl * k, k, ts, [=](uint64_t e) { return TopEnt{topp[e], topz[e]}; });
    if (threadIdx.x < (unsigned)k) {
        topp[threadIdx.x] = ts.run[threadIdx.x].p;
        topz[threadIdx.x] = ts.run[threadIdx.x].z;
    }
}

// Per-instance finalize: <C> = fixed-order sum of the tile partials; top-k = merge of the lists
// at tile slots 0, stride, 2 stride, ... (stride 1: every tile's list; FIN_CHUNK after the first
// merge level).
template <typename T>
__global__ void __launch_bounds__(256) k_stream_finalize(const StreamInst<T>* __restrict__ insts,
                                                         int count, uint64_t ntiles, int k,
                                                         uint64_t stride, const StreamInst<T> one) {
    __shared__ double red[32];
    __shared__ TopScratch ts;
    const int ii = blockIdx.x;
    if (ii >= count) return;
    const StreamInst<T>& I = insts ? insts[ii] : one;
    if (ntiles == 0) {             // instances of several sizes
        ntiles = 1ull << (I.n - (sizeof(T) == 8 ? 12 : 13));
        k = I.k;
        stride = k > 0 && ntiles > FIN_CHUNK ? FIN_CHUNK : 1;
    }
    // sum: each thread a contiguous slice (fixed), then the block tree
    double acc = 0.0;
    const uint64_t per = (ntiles + blockDim.x - 1) / blockDim.x;
    const uint64_t b0 = threadIdx.x * per;
    for (uint64_t t = b0; t < b0 + per && t < ntiles; ++t) acc += I.part_expect[t];
    const double tot = block_sum(acc, red);
    if (threadIdx.x == 0 && I.expect) *I.expect = tot;
    if (k > 0) {
        const uint64_t nl = (ntiles + stride - 1) / stride;
        const double* topp = I.part_topp;
        const uint32_t* topz = I.part_topz;
        merge_entries(nl * k, k, ts, [=](uint64_t e) {
            const uint64_t a = (e / k) * stride * k + e % k;
            return TopEnt{topp[a], topz[a]};
        });
        if (threadIdx.x < (unsigned)k) {
            if (I.topk_idx) I.topk_idx[threadIdx.x] = (uint64_t)ts.run[threadIdx.x].z;
            if (I.topk_prob) I.topk_prob[threadIdx.x] = ts.run[threadIdx.x].p;
        }
    }
}

// ---- adjoint passes -----------------------------------------------------------------------
// Two CTAs per SM: psi, lam and E tiles of 2^12 (float) or 2^11 (double) amplitudes each.
constexpr int ADJ_THREADS = 256;
// The forward pass P undone on a tile of psi and lam (both in the rotated frame), with the
// gradient accumulations of the tile engine's adjoint sub-passes: the local snake of P with
// RB_ADJ-bit windows, run in reverse. Per tile, four partial sums are written (as FP64):
//   [0] Im <lam|B|psi> of layer lb, [1] of layer la (lb > la), [2] Im <lam|E|psi> of layer lb,
//   [3] of layer la -- zero where the pass holds no such operation.
template <typename T, int RA>
__device__ void stream_adj_tile(const StreamPass& P, int si, bool lam_first, bool store,
                                const StreamInst<T>& I, uint64_t tau, const StreamSmem<T>& s,
                                typename Num<T>::C* slam, const LayerConst<T>* lc) {
    using C = typename Num<T>::C;
    C* gpsi = reinterpret_cast<C*>(I.psi);
    C* glam = reinterpret_cast<C*>(I.lam);
    cp_async_wait_all();
    __syncthreads();
    const TileRef<T> tile{s.psi, slam, s.E, P.tb};
    const int m0 = (P.kind == 0) ? 0 : P.c;
    Snake sn(P.lb - P.la + 1, P.la, P.ph_first, m0, P.tb, P.tb, RA);
    sn.to_last();
    bool first = lam_first;
    // tile accumulators by the pass's layer slot (0: layer lb, 1: layer la)
    T acc[4] = {T(0), T(0), T(0), T(0)};
    for (;; sn.prev()) {
        const SubPass sp = sn.get();
        subpass_adj<T, RA>(tile, sp, lc, first, P.lb, acc);
        first = false;
        __syncthreads();
        if (sn.first()) break;
    }
    double* out = I.part_grad + ((uint64_t)si << (P.n - P.tb)) * 4 + tau * 4;
    const double v = block_sum4((double)acc[0], (double)acc[1], (double)acc[2], (double)acc[3], s.red);
    if (threadIdx.x < 4) out[threadIdx.x] = v;
    if (store) {
        store_tile<T>(P, tau, s.psi, gpsi);
        store_tile<T>(P, tau, slam, glam);
    }
    __syncthreads();
}

template <typename T, int RA, int NTH>
__global__ void __launch_bounds__(NTH, 2) k_stream_adj_pass(const StreamPass P, int si, int lam_first,
                                                         int store,
                                                         const StreamInst<T>* __restrict__ insts,
                                                         int count, const StreamInst<T> one) {
    extern __shared__ __align__(16) unsigned char sm[];
    using C = typename Num<T>::C;
    const uint32_t TD = 1u << P.tb;
    StreamSmem<T> s;
    size_t o = 0;
    s.psi = reinterpret_cast<C*>(sm + o); o += (size_t)TD * sizeof(C);
    C* slam = reinterpret_cast<C*>(sm + o); o += (size_t)TD * sizeof(C);
    s.E = reinterpret_cast<T*>(sm + o); o += (size_t)TD * sizeof(T);
    LayerConst<T>* lc = reinterpret_cast<LayerConst<T>*>(sm + o); o += 64 * sizeof(LayerConst<T>);
    o = (o + 15) & ~(size_t)15;
    s.red = reinterpret_cast<double*>(sm + o);   // 64 doubles
    const uint64_t ntiles = 1ull << (P.n - P.tb);
    const uint64_t total = ntiles * (uint64_t)count;
    const T *cur_g = nullptr, *cur_b = nullptr;
    int cur_p = 0;
    for (uint64_t b = blockIdx.x; b < total; b += gridDim.x) {
        const int ii = (int)(b >> (P.n - P.tb));
        const uint64_t tau = b & (ntiles - 1);
        const StreamInst<T>& I = insts ? insts[ii] : one;
        stage_tile<T>(P, tau, reinterpret_cast<C*>(I.psi), s.psi, I.E, s.E);
        if (!lam_first) stage_tile<T>(P, tau, reinterpret_cast<C*>(I.lam), slam, nullptr, nullptr);
        if (I.gamma != cur_g || I.beta != cur_b || I.p != cur_p) {
            set_layer_consts<T>(lc, I.gamma, I.beta, I.p, P.n, true);
            cur_g = I.gamma;
            cur_b = I.beta;
            cur_p = I.p;
        }
        stream_adj_tile<T, RA>(P, si, lam_first != 0, store != 0, I, tau, s, slam, lc);
    }
}

// Block (i, l): dgamma_l = 2 sum of the gamma slots of layer l of instance i, dbeta_l = 2 sum of the
// beta slots, over passes in order and tiles in fixed contiguous chunks per thread. (One block per
// instance, its layers one after the other: 15 us at n = 20, p = 4; a layer per block: 6 us.)
template <typename T>
__global__ void __launch_bounds__(256) k_stream_grad_reduce(int tb, int cmin, const StreamInst<T>* __restrict__ insts, int count,
                                                            const StreamInst<T> one) {
    __shared__ double red[32];
    const int ii = blockIdx.x, l = blockIdx.y;
    if (ii >= count) return;
    const StreamInst<T>& I = insts ? insts[ii] : one;
    if (l >= I.p || !I.part_grad) return;   // (a mixed launch also meets instances without a gradient)
    // the passes that hold layer l (stream_plan): the first shared with layer l - 1, the last with
    // layer l + 1, W windows per layer
    const int W = stream_windows(I.n, tb, cmin);
    const uint64_t ntiles = 1ull << (I.n - tb);
    const uint64_t per = (ntiles + blockDim.x - 1) / blockDim.x;
    double gb = 0.0, gg = 0.0;
    for (int s = l * (W - 1); s <= (l + 1) * (W - 1); ++s) {
        const bool ha = s == (l + 1) * (W - 1) && l + 1 < I.p;   // layer l is the pass's la, else its lb
        const double* base = I.part_grad + ((uint64_t)s * ntiles) * 4 + (ha ? 1 : 0);
        for (uint64_t t = threadIdx.x * per; t < (threadIdx.x + 1) * per && t < ntiles; ++t) {
            const double* q = base + t * 4;
            gb += q[0];
            gg += q[2];
        }
    }
    const double v = block_sum4(gb, gg, 0.0, 0.0, red);
    if (threadIdx.x == 0 && I.dbeta) I.dbeta[l] = 2.0 * v;
    if (threadIdx.x == 1 && I.dgamma) I.dgamma[l] = 2.0 * v;
}

// ---- energy build into HBM, row form (n >= 2) ------------------------------------------
// E(z) = sum_i Q_ii z_i + sum_{i<j} W_ij z_i z_j with W_ij = Q_ij + Q_ji (Q need not be
// symmetric). Split z = (hi, lo) with hi the top nh bits and m = n - nh. A thread fixes lo up to
// its two lowest bits and holds the four energies E(hi, lo | v), v = 0..3, and the cross fields
//   P_h(lo | v) = sum_{j in lo|v} W_{m+h, j}              (h < nh),
// then walks hi in Gray-code order: flipping bit b of hi changes every energy by
//   s * (P_b(lo|v) + Q_{b'b'} + sum_{j in hi, j != b} W_{b'j'})   (s = +1 setting, -1 clearing;
// primes: positions m + b, m + j). The hi-only part depends on the step alone, so a table D[k]
// of it (sign included) is built once per block; each step costs one select, eight adds and one
// 16-byte (float) or two (double) stores of four consecutive energies. The walk is at most 2^8
// steps, which bounds the FP32 rounding drift of the running sums.
constexpr int ROWS_NH_MAX = 8;

template <typename T>
__global__ void __launch_bounds__(256) k_energy_rows(int n, int nh, const T* __restrict__ Q,
                                                     T* __restrict__ E, const StreamInst<T>* insts) {
    __shared__ T W[32 * 32];
    __shared__ T D[1 << ROWS_NH_MAX];
    if (insts) {
        Q = insts[blockIdx.y].Q;
        E = const_cast<T*>(insts[blockIdx.y].E);
    }
    for (int x = threadIdx.x; x < n * n; x += blockDim.x) {
        const int i = x / n, j = x - i * n;
        W[x] = (i == j) ? Q[x] : Q[x] + Q[j * n + i];
    }
    __syncthreads();
    const int m = n - nh;
    const int steps = 1 << nh;
    for (int k = 1 + threadIdx.x; k < steps; k += blockDim.x) {
        const int b = __ffs(k) - 1;
        const uint32_t g = (uint32_t)(k - 1) ^ ((uint32_t)(k - 1) >> 1);   // hi before the flip
        const T* row = W + (m + b) * n + m;
        T d = row[b];
        for (int j = 0; j < nh; ++j)
            if (j != b && ((g >> j) & 1u)) d += row[j];
        D[k] = ((g >> b) & 1u) ? -d : d;
    }
    __syncthreads();
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (1ull << (m - 2))) return;
    const uint32_t base = (uint32_t)gid << 2;
    // exact energies of lo = base | v at hi = 0
    T eb = T(0), f0 = W[0], f1 = W[n + 1];
    for (int i = 2; i < m; ++i) {
        if (!((base >> i) & 1u)) continue;
        const T* row = W + i * n;
        T r = row[i];
        for (int j = 2; j < i; ++j)
            if ((base >> j) & 1u) r += row[j];
        eb += r;
        f0 += row[0];
        f1 += row[1];
    }
    T e[4] = {eb, eb + f0, eb + f1, eb + f0 + f1 + W[1]};
    T P[ROWS_NH_MAX][4];
#pragma unroll
    for (int h = 0; h < ROWS_NH_MAX; ++h) {
        if (h < nh) {
            const T* row = W + (m + h) * n;
            T pb = T(0);
            for (int j = 2; j < m; ++j)
                if ((base >> j) & 1u) pb += row[j];
            P[h][0] = pb;
            P[h][1] = pb + row[0];
            P[h][2] = pb + row[1];
            P[h][3] = pb + row[0] + row[1];
        } else {
            P[h][0] = P[h][1] = P[h][2] = P[h][3] = T(0);
        }
    }
    // E is 8-byte aligned (checked when the plan is made); 16-byte stores where it is 16-aligned
    const bool v16 = (reinterpret_cast<uintptr_t>(E) & 15u) == 0;
    auto put = [&](uint32_t hi) {
        T* dst = E + (((uint64_t)hi << m) | base);
        if constexpr (sizeof(T) == 4) {
            if (v16) {
                *reinterpret_cast<float4*>(dst) = make_float4(e[0], e[1], e[2], e[3]);
            } else {
                reinterpret_cast<float2*>(dst)[0] = make_float2(e[0], e[1]);
                reinterpret_cast<float2*>(dst)[1] = make_float2(e[2], e[3]);
            }
        } else {
            if (v16) {
                reinterpret_cast<double2*>(dst)[0] = make_double2(e[0], e[1]);
                reinterpret_cast<double2*>(dst)[1] = make_double2(e[2], e[3]);
            } else {
                dst[0] = e[0]; dst[1] = e[1]; dst[2] = e[2]; dst[3] = e[3];
            }
        }
    };
    put(0u);
    uint32_t hi = 0;
    for (int k = 1; k < steps; ++k) {
        const int b = __ffs(k) - 1;
        hi ^= 1u << b;
        T p0 = T(0), p1 = T(0), p2 = T(0), p3 = T(0);
#pragma unroll
        for (int h = 0; h < ROWS_NH_MAX; ++h)
            if (h == b) { p0 = P[h][0]; p1 = P[h][1]; p2 = P[h][2]; p3 = P[h][3]; }
        if (!((hi >> b) & 1u)) { p0 = -p0; p1 = -p1; p2 = -p2; p3 = -p3; }
        const T d = D[k];
        e[0] += p0 + d;
        e[1] += p1 + d;
        e[2] += p2 + d;
        e[3] += p3 + d;
        put(hi);
    }
}

// ---- energy build into HBM, direct form ---------------------------------------------------
// The row form without a walk (nh = 0: a single complex64 instance of up to 20 qubits), the same
// additions in the same order: E is what qaoa_build_energies has always returned, and what states and
// shots follow from. Bits 2..9 belong to the thread, the bits above to the block, so the loops over the
// block's set bits are uniform and the thread's bits act as masks on unrolled additions, where
// the row form tests every pair of bits (n = 19: 9.4 -> 6.8 us). FP64 keeps the row form: its issue
// rate pays for every masked addition (n = 12: 8.8 us by rows, 10.3 so). Blocks have 256 threads at any n:
// with 2^(n-2) of them a few threads fill W alone (n = 2: 30 us so, 3.7 now).
__device__ __forceinline__ float keep(float x, uint32_t m) { return __uint_as_float(__float_as_uint(x) & m); }
__device__ __forceinline__ double keep(double x, uint32_t m) { return m ? x : 0.0; }

__global__ void __launch_bounds__(256) k_energy_direct(int n, const float* __restrict__ Q, float* __restrict__ E) {
    __shared__ float W[32 * 32];      // zero beyond n
    for (int x = threadIdx.x; x < 32 * 32; x += 256) {
        const int i = x >> 5, j = x & 31;
        float w = 0.0f;
        if (i < n && j < n) w = (i == j) ? Q[i * n + i] : Q[i * n + j] + Q[j * n + i];
        W[x] = w;
    }
    __syncthreads();
    if (n < 10 && threadIdx.x >= 1u << (n - 2)) return;
    uint32_t m[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] = 0u - ((threadIdx.x >> i) & 1u);
    float eb = 0.0f, f0 = W[0], f1 = W[33];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float* row = W + (2 + i) * 32;
        float r = row[2 + i];
#pragma unroll
        for (int j = 0; j < i; ++j) r += keep(row[2 + j], m[j]);
        eb += keep(r, m[i]);
        f0 += keep(row[0], m[i]);
        f1 += keep(row[1], m[i]);
    }
    const uint32_t hi = blockIdx.x;
    for (uint32_t b = hi; b; b &= b - 1u) {
        const int i = 10 + __ffs((int)b) - 1;
        const float* row = W + i * 32;
        float r = row[i];
#pragma unroll
        for (int j = 0; j < 8; ++j) r += keep(row[2 + j], m[j]);
        for (uint32_t d = hi & ((b & (0u - b)) - 1u); d; d &= d - 1u) r += row[10 + __ffs((int)d) - 1];
        eb += r;
        f0 += row[0];
        f1 += row[1];
    }
    float2* dst = reinterpret_cast<float2*>(E + (((uint64_t)hi << 10) | ((uint64_t)threadIdx.x << 2)));   // E is 8-byte aligned
    dst[0] = make_float2(eb, eb + f0);
    dst[1] = make_float2(eb + f1, eb + f0 + f1 + W[1]);
}

// ---- energy build into HBM, tile form ----------------------------------------------------
// A block builds the 2^11 energies of one value hi of the bits above 11 (all 2^n for n < 11). With
// W_ij = Q_ij + Q_ji and S the set bits of hi,
//   E(z) = E_S + sum_{i in lo} d_i + sum_{i<k in lo} W_ik,   d_i = Q_ii + sum_{s in S} W_is,
// the block's d_i and E_S are summed by warps (a lane per bit of hi), a thread adds the terms
// of its low eight bits once and forms its eight energies by subset doubling over bits 8..10,
// against a sum over all bit pairs per energy quadruple in the row form, whose walk over hi is
// too short to pay for its start below about 2^23 energies (n = 20 on GB300: 14.6 us in the row form, 8.4 us
// here). The energies of batched instances; single instances keep the row form's sums (k_energy_direct).
// Sums are
// compensated (Acc: TwoSum, the rounding errors added separately), so that an energy is off by
// little more than its own last rounding (relative 2-norm at n = 19: 9e-8 in the row form,
// 2.5e-8 here): phases gamma E inherit that error. Stores are 4 (8) bytes per lane, coalesced: any
// alignment.
constexpr int ETB = 11;

template <typename T>
struct Acc {
    T s, c;   // value s + c
    __device__ __forceinline__ void add(T x) {
        const T t = s + x, z = t - s;
        c += (s - (t - z)) + (x - z);
        s = t;
    }
    __device__ __forceinline__ void add(const Acc& o) {
        add(o.s);
        c += o.c;
    }
    // (the error of a sum that has become infinite is NaN: its value is the sum's)
    __device__ __forceinline__ T value() const { return c == c ? s + c : s; }
};

// Runs of instances of equal n in one launch: run i owns blocks [b0[i], b0[i + 1]).
struct EnergyRuns {
    int runs;
    uint32_t b0[ENERGY_RUNS + 1];
    int n[ENERGY_RUNS], first[ENERGY_RUNS];
};

template <typename T>
__global__ void __launch_bounds__(256) k_energy_tile(int n, const T* __restrict__ Q, T* __restrict__ E,
                                                     const StreamInst<T>* insts, const EnergyRuns er) {
    __shared__ T W[32 * 32];      // zero beyond n
    __shared__ Acc<T> d[16];
    uint32_t hi = blockIdx.x;
    if (er.runs > 0) {
        int r = 0;
        while (hi >= er.b0[r + 1]) ++r;
        n = er.n[r];
        hi -= er.b0[r];
        const int hb = n > ETB ? n - ETB : 0;
        const StreamInst<T>& I = insts[er.first[r] + (hi >> hb)];
        hi &= (1u << hb) - 1u;
        Q = I.Q;
        E = const_cast<T*>(I.E);
    } else if (insts) {
        Q = insts[blockIdx.y].Q;
        E = const_cast<T*>(insts[blockIdx.y].E);
    }
#pragma unroll
    for (int x = threadIdx.x; x < 32 * 32; x += 256) {
        const int i = x >> 5, j = x & 31;
        T w = T(0);
        if (i < n && j < n) w = (i == j) ? Q[i * n + i] : Q[i * n + j] + Q[j * n + i];
        W[x] = w;
    }
    const int nhi = n > ETB ? n - ETB : 0, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    const bool on = lane < nhi && ((hi >> lane) & 1u);
    for (int b = warp; b <= ETB; b += 8) {          // d_0 .. d_10, and E_S as entry 11
        Acc<T> v{T(0), T(0)};
        if (b < ETB) {
            if (on) v.s = W[b * 32 + ETB + lane];
        } else if (on) {
            const T* row = W + (ETB + lane) * 32 + ETB;
            v.s = row[lane];
            for (int s = 0; s < lane; ++s)
                if ((hi >> s) & 1u) v.add(row[s]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const Acc<T> w{__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o)};
            v.add(w);
        }
        if (b < ETB) v.add(W[b * 32 + b]);
        if (lane == 0) d[b] = v;
    }
    __syncthreads();
    // terms of clear bits are masked out, not multiplied by 0: an infinite entry of Q reaches only the
    // energies that hold its qubits
    const uint32_t t = threadIdx.x;
    uint32_t m[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] = 0u - ((t >> i) & 1u);
    Acc<T> base = d[ETB], w8[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) w8[b] = d[8 + b];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const Acc<T> di = d[i];
        base.add(keep(di.s, m[i]));
        base.c += keep(di.c, m[i]);
#pragma unroll
        for (int k = i + 1; k < 8; ++k) base.add(keep(W[i * 32 + k], m[i] & m[k]));
#pragma unroll
        for (int b = 0; b < 3; ++b) w8[b].add(keep(W[i * 32 + 8 + b], m[i]));
    }
    const T w01 = W[8 * 32 + 9], w02 = W[8 * 32 + 10], w12 = W[9 * 32 + 10];
    Acc<T> x[8];
    x[0] = base;
#pragma unroll
    for (int j = 1; j < 8; ++j) {
        const int top = j >= 4 ? 2 : (j >= 2 ? 1 : 0);   // x[j] from x[j without its top bit]
        x[j] = x[j ^ (1 << top)];
        x[j].add(w8[top]);
        if (top == 1 && (j & 1)) x[j].add(w01);
        if (top == 2 && (j & 1)) x[j].add(w02);
        if (top == 2 && (j & 2)) x[j].add(w12);
    }
    const uint64_t z0 = ((uint64_t)hi << ETB) | t;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint64_t z = z0 + ((uint64_t)j << 8);
        if (n >= ETB || z < (1ull << n)) E[z] = x[j].value();
    }
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------

// Passes of a single complex64 state of up to 20 (forward) or 21 qubits (gradient). With the batched
// tiles (2^13 forward, 2^12 adjoint) such a state is a few dozen tiles, one per CTA and pass, and a pass
// lasts as long as one tile does on a CTA of 256 threads that runs a thousand unrolled instructions once.
//   qaoa_run_layers, n = 15..20: qubits 0..12 in the batched tiles, qubits 13..n-1 in tiles of 2^10
//   amplitudes (runs of at least 8; at n = 21 such runs leave 2^11 and the pass loses to the batched
//   tiles' 256 blocks: p = 3, 88 us against 72; 2^11 at n = 19, 20 gave nothing), eight amplitudes per
//   thread, the windows of a pass listed on the host so that the qubit order stays that of 5-qubit
//   windows over 0..12 and 13..n-1 (see FwdConst: shots are drawn from these states, and that order is
//   why the contiguous tiles keep 13 qubits; 1024 threads on one of them took as long as 256).
//   qaoa_grad (whose states stay inside): tb = (n + 4) / 2 bits forward and adjoint, runs of at
//   least 8 amplitudes, 16 amplitudes per thread.
// GB300: qaoa_run_layers at n = 19, p = 3, passes of 22 to 29 us -> 14 to 18 (qubits 0..12) and 8 to
// 10 us; qaoa_grad at n = 20, p = 4, forward passes 23 to 32 -> 10 to 15 us.
static bool small_tiles(bool dbl, int n, int tb) { return !dbl && n >= 14 && n <= SMALL_GRAD_NMAX && tb == (n + 4) / 2; }

int stream_tile_bits(bool dbl) { return dbl ? 12 : 13; }
int stream_adj_tile_bits(bool dbl) { return dbl ? 11 : 12; }
int stream_one_grad_tile_bits(bool dbl, int n, bool adjoint, int* cmin) {
    const bool small = !dbl && n >= 14 && n <= SMALL_GRAD_NMAX;
    *cmin = small ? 3 : 4;
    return small ? (n + 4) / 2 : (adjoint ? stream_adj_tile_bits(dbl) : stream_tile_bits(dbl));
}
uint64_t stream_one_max_tiles(bool dbl, int n) {
    if (!dbl && n >= SMALL_NMIN && n <= SMALL_NMAX) return 1ull << (n - 10);
    return n > stream_tile_bits(dbl) ? 1ull << (n - stream_tile_bits(dbl)) : 0;
}

// The forward passes of a single state (see above); other sizes and types: the batched plan.
int stream_plan_one(bool dbl, int n, int p, int k, StreamPass* out, StreamSubs* subs, int max_out) {
    for (int i = 0; i < max_out; ++i) subs[i].n = 0;
    if (dbl || n < SMALL_NMIN || n > SMALL_NMAX || k > 0) return stream_plan(dbl, n, p, k, out, max_out);
    if (p + 1 > max_out) return -1;
    // blocks of qubits, each cut into windows of at most SMALL_R
    struct Blk { int q, size; };
    Blk up[2];
    int nu = 0;
    for (int q = SMALL_LOW; q < n; q += 5) up[nu++] = Blk{q, n - q < 5 ? n - q : 5};
    const int tbA = SMALL_LOW, h = n - SMALL_LOW, tbB = 10, c = tbB - h;
    for (int si = 0; si <= p; ++si) {
        StreamPass P{};
        P.n = n;
        P.la = si > 0 ? si - 1 : 0;
        P.lb = si < p ? si : p - 1;
        if (si == 0) P.lb = 0;
        P.init = P.ph_first = si == 0 ? 1 : 0;
        P.fin = si == p ? 1 : 0;
        const bool lower = (si & 1) == 0;
        P.kind = lower ? 0 : 1;
        P.tb = lower ? tbA : tbB;
        P.c = lower ? tbA : c;
        P.s = lower ? tbA : SMALL_LOW;
        P.h = lower ? 0 : h;
        P.need_e = (P.ph_first || P.lb > P.la || P.fin) ? 1 : 0;
        const int shift = c - SMALL_LOW;                  // tile bit of qubit q: q + shift
        for (int l = P.la; !lower && l <= P.lb; ++l)
            for (int i = 0; i < nu; ++i) {
                const Blk& b = up[l > P.la ? nu - 1 - i : i];
                for (int q = b.q; q < b.q + b.size; q += SMALL_R) {
                    const int size = b.q + b.size - q < SMALL_R ? b.q + b.size - q : SMALL_R;
                    const int lo = q + shift, a = lo + SMALL_R <= P.tb ? lo : P.tb - SMALL_R;
                    StreamSub sb{a, ((1 << size) - 1) << (lo - a), l - P.la, l - P.la, 0};
                    const bool opens = i == 0 && q == b.q;
                    sb.phase = opens && (l > P.la || P.ph_first) ? 1 : 0;
                    StreamSubs& L = subs[si];
                    if (opens && l > P.la && L.sub[L.n - 1].a == sb.a && L.sub[L.n - 1].mask == sb.mask) {
                        L.sub[L.n - 1].l1 = sb.l1;         // shared around the cost phase
                        continue;
                    }
                    if (L.n == STREAM_MAX_SUB) return -1;
                    L.sub[L.n++] = sb;
                }
            }
        out[si] = P;
    }
    return p + 1;
}

// HBM windows of a layer: window 0 = kind A (qubits 0..tb-1); windows 1.. = kind B chunks of
// the qubits [tb, n), as equal as possible, each at most tb - cmin qubits (4: runs of at least 128
// bytes; 3 for the small tiles of a single gradient).
int stream_plan(bool dbl, int n, int p, int k, StreamPass* out, int max_out, int tb, int cmin) {
    if (tb < 0) tb = stream_tile_bits(dbl);
    if (n <= tb) return -1;
    const int rest = n - tb;
    const int nB = stream_windows(n, tb, cmin) - 1;
    int chunk_s[16], chunk_h[16];
    int s0 = tb;
    for (int i = 0; i < nB; ++i) {
        const int h = rest / nB + (i < rest % nB ? 1 : 0);
        chunk_s[i] = s0;
        chunk_h[i] = h;
        s0 += h;
    }
    const int G = 1 + nB;
    const int S = (G <= 1) ? p : 1 + p * (G - 1);
    if (S > max_out) return -1;
    for (int si = 0; si < S; ++si) {
        int l, pos;
        if (si < G) { l = 0; pos = si; }
        else { l = 1 + (si - G) / (G - 1); pos = 1 + (si - G) % (G - 1); }
        const int w = (l % 2 == 0) ? pos : (G - 1 - pos);
        StreamPass P{};
        P.n = n;
        P.tb = tb;
        P.la = l;
        P.lb = (pos == G - 1 && l + 1 < p) ? l + 1 : l;
        P.ph_first = (l == 0 && pos == 0) ? 1 : 0;
        P.init = (si == 0) ? 1 : 0;
        P.fin = (si == S - 1) ? 1 : 0;
        P.k = P.fin ? k : 0;
        if (w == 0) {
            P.kind = 0;
            P.c = tb; P.s = tb; P.h = 0;
        } else {
            P.kind = 1;
            P.h = chunk_h[w - 1];
            P.s = chunk_s[w - 1];
            P.c = tb - P.h;
        }
        P.need_e = (P.ph_first || P.lb > P.la || P.fin) ? 1 : 0;
        out[si] = P;
    }
    return S;
}

static size_t stream_smem_bytes(bool dbl, int tb) {
    const size_t TD = (size_t)1 << tb;
    const size_t c = dbl ? 16 : 8, r = dbl ? 8 : 4, lcs = dbl ? sizeof(LayerConst<double>) : sizeof(LayerConst<float>);
    size_t o = TD * c + TD * r + 64 * lcs;
    o = (o + 15) & ~(size_t)15;
    return o + 32 * sizeof(double) + (8 * 32 + TOPK_CAP + 16 + 16) * sizeof(TopEnt) +
           16 * 32 * sizeof(float) + 4 * sizeof(int);
}

template <typename T>
static StreamInst<T> one_of(const void* one) {
    StreamInst<T> o{};
    if (one) o = *static_cast<const StreamInst<T>*>(one);
    return o;
}

template <typename T, int R, int NTH, bool TOPK, bool GRAD = false>
static cudaError_t pass_t(const StreamPass& P, const void* insts, int count, int grid, int threads, cudaStream_t st,
                          const void* one, const StreamSubs* subs = nullptr) {
    const size_t sm = stream_smem_bytes(sizeof(T) == 8, P.tb);
    const cudaError_t e = cudaFuncSetAttribute(k_stream_pass<T, R, NTH, TOPK, GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_stream_pass<T, R, NTH, TOPK, GRAD><<<grid, threads, sm, st>>>(P, static_cast<const StreamInst<T>*>(insts), count, one_of<T>(one),
                                                            subs ? *subs : StreamSubs{});
    return cudaGetLastError();
}

cudaError_t launch_stream_pass(bool dbl, const StreamPass& P, const void* insts, int count,
                               int grid, cudaStream_t st, bool grad, const void* one, const StreamSubs* subs) {
    if (dbl) return pass_t<double, Num<double>::RB, 256, true>(P, insts, count, grid, 256, st, one);
    if (grad) {
        if (P.k > 0) return pass_t<float, Num<float>::RB, 256, true, true>(P, insts, count, grid, 256, st, one);
        if (small_tiles(dbl, P.n, P.tb))
            return pass_t<float, SMALL_RA, 256, false, true>(P, insts, count, grid, 1 << (P.tb - SMALL_RA), st, one);
        return pass_t<float, Num<float>::RB, 256, false, true>(P, insts, count, grid, 256, st, one);
    }
    if (subs && subs->n > 0)
        return pass_t<float, SMALL_R, 256, false>(P, insts, count, grid, 1 << (P.tb - SMALL_R), st, one, subs);
    if (P.k == 0) return pass_t<float, Num<float>::RB, 256, false>(P, insts, count, grid, 256, st, one);
    return pass_t<float, Num<float>::RB, 256, true>(P, insts, count, grid, 256, st, one);
}

bool stream_finalize_two_level(uint64_t ntiles, int k) { return k > 0 && ntiles > FIN_CHUNK; }

cudaError_t launch_stream_topk_chunks(const void* insts, int count, uint64_t ntiles, int k, cudaStream_t st) {
    const dim3 grid((unsigned)((ntiles + FIN_CHUNK - 1) / FIN_CHUNK), (unsigned)count);
    k_stream_topk_chunks<float><<<grid, 256, 0, st>>>(static_cast<const StreamInst<float>*>(insts), count, ntiles, k, StreamInst<float>{});
    return cudaGetLastError();
}

cudaError_t launch_stream_finalize_mixed(const void* insts, int count, cudaStream_t st) {
    k_stream_finalize<float><<<count, 256, 0, st>>>(static_cast<const StreamInst<float>*>(insts), count, 0, 0, 1, StreamInst<float>{});
    return cudaGetLastError();
}

cudaError_t launch_stream_finalize(bool dbl, const void* insts, int count, uint64_t ntiles, int k,
                                   cudaStream_t st, const void* one) {
    uint64_t stride = 1;
    if (stream_finalize_two_level(ntiles, k)) {
        const dim3 grid((unsigned)((ntiles + FIN_CHUNK - 1) / FIN_CHUNK), (unsigned)count);
        if (dbl) k_stream_topk_chunks<double><<<grid, 256, 0, st>>>(static_cast<const StreamInst<double>*>(insts), count, ntiles, k, one_of<double>(one));
        else k_stream_topk_chunks<float><<<grid, 256, 0, st>>>(static_cast<const StreamInst<float>*>(insts), count, ntiles, k, one_of<float>(one));
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        stride = FIN_CHUNK;
    }
    if (dbl) k_stream_finalize<double><<<count, 256, 0, st>>>(static_cast<const StreamInst<double>*>(insts), count, ntiles, k, stride, one_of<double>(one));
    else k_stream_finalize<float><<<count, 256, 0, st>>>(static_cast<const StreamInst<float>*>(insts), count, ntiles, k, stride, one_of<float>(one));
    return cudaGetLastError();
}

// Top bits walked per thread by the row form: enough threads in total (instances x 2^(n-2-nh))
// to fill the GPU, a walk of at most 2^8 steps.
static int rows_nh(int n, int count) {
    int lc = 0;
    while ((2ull << lc) <= (unsigned long long)count) ++lc;
    int nh = n - 20 + lc;
    if (nh > ROWS_NH_MAX) nh = ROWS_NH_MAX;
    if (nh > n - 4) nh = n - 4;
    return nh < 0 ? 0 : nh;
}

template <typename T>
static cudaError_t launch_rows(int n, int count, const void* Q, void* E, const void* insts, cudaStream_t st) {
    const int nh = rows_nh(n, count);
    const uint64_t threads = 1ull << (n - nh - 2);
    const int block = threads < 256 ? (int)threads : 256;
    const unsigned gx = (unsigned)((threads + block - 1) / block);
    const StreamInst<T>* in = static_cast<const StreamInst<T>*>(insts);
    for (int c0 = 0; c0 < count; c0 += 65535) {          // grid.y limit
        const int cy = count - c0 < 65535 ? count - c0 : 65535;
        k_energy_rows<T><<<dim3(gx, (unsigned)cy), block, 0, st>>>(n, nh, static_cast<const T*>(Q),
                                                                  static_cast<T*>(E), in ? in + c0 : nullptr);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Batches: tile form up to 2^22 energies per instance (ENERGY_TILE_NMAX), row form above.

template <typename T>
static cudaError_t launch_tiles(int n, int count, const void* Q, void* E, const void* insts, cudaStream_t st) {
    const unsigned gx = n > ETB ? 1u << (n - ETB) : 1u;
    const StreamInst<T>* in = static_cast<const StreamInst<T>*>(insts);
    for (int c0 = 0; c0 < count; c0 += 65535) {          // grid.y limit
        const int cy = count - c0 < 65535 ? count - c0 : 65535;
        k_energy_tile<T><<<dim3(gx, (unsigned)cy), 256, 0, st>>>(n, static_cast<const T*>(Q), static_cast<T*>(E),
                                                                 in ? in + c0 : nullptr, EnergyRuns{});
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_energy_mixed(const void* insts, int runs, const int* n, const int* first, const int* count,
                                cudaStream_t st) {
    EnergyRuns er{};
    for (int i = 0; i < runs; ++i) {
        er.n[i] = n[i];
        er.first[i] = first[i];
        er.b0[i + 1] = er.b0[i] + ((uint32_t)count[i] << (n[i] > ETB ? n[i] - ETB : 0));
    }
    er.runs = runs;
    k_energy_tile<float><<<er.b0[runs], 256, 0, st>>>(0, nullptr, nullptr, static_cast<const StreamInst<float>*>(insts), er);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_one(int n, const void* Q, void* E, cudaStream_t st) {
    // one qubit, or an address the wider stores cannot take
    if (n < 2 || (reinterpret_cast<uintptr_t>(E) & 7u) != 0) return launch_tiles<T>(n, 1, Q, E, nullptr, st);
    if (sizeof(T) == 8 || rows_nh(n, 1) > 0) return launch_rows<T>(n, 1, Q, E, nullptr, st);
    k_energy_direct<<<n > 10 ? 1u << (n - 10) : 1u, 256, 0, st>>>(n, static_cast<const float*>(Q), static_cast<float*>(E));
    return cudaGetLastError();
}

cudaError_t launch_energy(bool dbl, int n, const void* Q, void* E, cudaStream_t st) {
    return dbl ? launch_one<double>(n, Q, E, st) : launch_one<float>(n, Q, E, st);
}

cudaError_t launch_energy_batch(bool dbl, int n, const void* insts, int count, cudaStream_t st) {
    // every instance's E is at least 8-byte aligned (plan validation)
    if (n <= ENERGY_TILE_NMAX)
        return dbl ? launch_tiles<double>(n, count, nullptr, nullptr, insts, st)
                   : launch_tiles<float>(n, count, nullptr, nullptr, insts, st);
    return dbl ? launch_rows<double>(n, count, nullptr, nullptr, insts, st)
               : launch_rows<float>(n, count, nullptr, nullptr, insts, st);
}

static size_t stream_adj_smem_bytes(bool dbl, int tb) {
    const size_t TD = (size_t)1 << tb;
    const size_t c = dbl ? 16 : 8, r = dbl ? 8 : 4;
    const size_t lcs = dbl ? sizeof(LayerConst<double>) : sizeof(LayerConst<float>);
    size_t o = 2 * TD * c + TD * r + 64 * lcs;
    o = (o + 15) & ~(size_t)15;
    return o + 64 * sizeof(double);
}

template <typename T, int RA, int NTH>
static cudaError_t adj_t(const StreamPass& P, int si, bool lam_first, bool store, const void* insts, int count, int grid,
                         int threads, cudaStream_t st, const void* one) {
    const size_t sm = stream_adj_smem_bytes(sizeof(T) == 8, P.tb);
    const cudaError_t e = cudaFuncSetAttribute(k_stream_adj_pass<T, RA, NTH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_stream_adj_pass<T, RA, NTH><<<grid, threads, sm, st>>>(P, si, lam_first, store, static_cast<const StreamInst<T>*>(insts),
                                                            count, one_of<T>(one));
    return cudaGetLastError();
}

cudaError_t launch_stream_adj_pass(bool dbl, const StreamPass& P, int si, bool lam_first, bool store,
                                   const void* insts, int count, int grid, cudaStream_t st,
                                   const void* one) {
    if (dbl) return adj_t<double, Num<double>::RB_ADJ, ADJ_THREADS>(P, si, lam_first, store, insts, count, grid, ADJ_THREADS, st, one);
    if (small_tiles(dbl, P.n, P.tb))
        return adj_t<float, SMALL_RA, 256>(P, si, lam_first, store, insts, count, grid, 1 << (P.tb - SMALL_RA), st, one);
    return adj_t<float, Num<float>::RB_ADJ, ADJ_THREADS>(P, si, lam_first, store, insts, count, grid, ADJ_THREADS, st, one);
}

cudaError_t launch_stream_grad_reduce(bool dbl, int tb, int cmin, int pmax, const void* insts, int count, cudaStream_t st,
                                      const void* one) {
    const dim3 grid((unsigned)count, (unsigned)pmax);
    if (dbl) k_stream_grad_reduce<double><<<grid, 256, 0, st>>>(tb, cmin, static_cast<const StreamInst<double>*>(insts), count, one_of<double>(one));
    else k_stream_grad_reduce<float><<<grid, 256, 0, st>>>(tb, cmin, static_cast<const StreamInst<float>*>(insts), count, one_of<float>(one));
    return cudaGetLastError();
}

}  // namespace qaoa
