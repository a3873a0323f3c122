// k_tstream.cu -- TMA streaming passes of the HBM tier (complex64 states of n >= 14 qubits whose
// passes walk the whole state in HBM; Section IV, Eq. 2: cost phase and mixer per layer, <C> and
// the top-k bitstrings at the end).
//
// A launch is persistent, two CTAs per SM, walking the tiles of one pass of every instance of its
// plan groups: groups of other sizes and depths share the launches (segments, TsSeg), so that an
// uneven batch takes as many launches as its longest group has passes and small states fill the
// SMs that one group alone would leave idle (a launch per group and pass: 48 uneven training
// instances 7.95 ms a step, 16 served jobs 800 us a tick; shared launches: 5.66 ms, 365 us). A tile is
// 2^13 amplitudes, moved between HBM and shared memory by TMA (cp.async.bulk.tensor; the state with
// the 128-byte swizzle). Phases and energies come from Q itself (qaoa_phase.cuh); instances whose
// energies live in HBM anyway (gradient runs, returned energies) read them, unswizzled, in passes with
// a cost phase or the final reductions. n = 30, p = 2: 16.19 ms, with energies built and read 16.74.
// A CTA loads its next tile as soon as the bulk store of the current one has read the buffer, and the
// other CTA of the SM works while it waits: measured on GB300 at n = 30 this beats one CTA per SM
// with a two-stage ring (8 warps per SM leave the sub-passes latency-bound) by 12% over the passes
// of a solve. What bounds the passes (n = 30): single-layer passes HBM (2.9 ms for 17.2 GB); the
// others, at 2.8-3.8 ms, the latency of 16 warps per SM (0.35-0.45 of the issue slots).
//
// Tiles follow the streaming tier's pass plan (stream_plan): kind A holds qubits 0..12 (2^13
// contiguous amplitudes), kind B the 2^c contiguous amplitudes of qubits 0..c-1 times the 2^h
// values of qubits s..s+h-1 (c = 13 - h, 1 <= h <= 9). Inside a tile the qubits are mixed in
// register windows of at most five bits (tile_pass; the cost phase in the one that reaches bit 12). With
// the lanes of a warp on tile bits outside the window, the swizzle makes every shared access free
// of bank conflicts. The final pass reduces each tile to an FP64 <C> partial and a top-k list;
// the streaming tier's finalize kernel merges them per instance.
#include <cuda.h>

#include "qaoa_engine.cuh"
#include "qaoa_kernels.h"
#include "qaoa_phase.cuh"
#include "qaoa_stream.h"
#include "qaoa_tma.cuh"
#include "qaoa_tstream.h"

namespace qaoa {

namespace {

using namespace tma;

constexpr int TB = 13;
constexpr uint32_t TD = 1u << TB;
constexpr int NT = TMA_NT;

struct TsOff {
    size_t psi, E, lc, red, wbound, wb, cnt, cand, out, wlists, run, mbar, total;
};
__host__ __device__ inline size_t ts_al(size_t x) { return (x + 15) & ~(size_t)15; }
// tab: the phase table in the place of the energy tile
__host__ __device__ inline TsOff ts_offsets(bool tab) {
    TsOff o{};
    size_t x = 0;
    o.psi = x; x += (size_t)TD * 8;   // 1024-aligned at run time
    o.E = x; x = ts_al(x + (tab ? sizeof(PhaseTab) : (size_t)TD * 4));
    o.lc = x; x = ts_al(x + 64 * sizeof(LayerConst<float>));
    o.red = x; x = ts_al(x + 32 * sizeof(float));
    o.wbound = x; x = ts_al(x + sizeof(float));
    o.wb = x; x = ts_al(x + 16 * (NT / 32) * sizeof(float));
    o.cnt = x; x = ts_al(x + 4 * sizeof(int));
    o.cand = x; x = ts_al(x + TOPK_CAP * sizeof(TopEnt));
    o.out = x; x = ts_al(x + 16 * sizeof(TopEnt));
    o.wlists = x; x = ts_al(x + (NT / 32) * 32 * sizeof(TopEnt));
    o.run = x; x = ts_al(x + 16 * sizeof(TopEnt));
    o.mbar = x; x = ts_al(x + sizeof(uint64_t));
    o.total = x + 1024;
    return o;
}

// Geometry of one tile of a pass: global index of tile-local index u is
//   kind A: u | zt,  kind B: (u & lomask) | zt | ((u >> c) << s),
// with zt the bits that the tile index fixes.
struct Geo {
    uint32_t lomask;
    int c, s;
    uint64_t zt;
    bool kindA;
    __device__ __forceinline__ uint64_t z(uint32_t u) const {
        return kindA ? ((uint64_t)u | zt) : ((uint64_t)(u & lomask) | zt | ((uint64_t)(u >> c) << s));
    }
};

// Group g of a window [A, A+R): tile index of its element 0 (the window bits clear).
template <int A, int R>
__device__ __forceinline__ uint32_t wbase(uint32_t g) {
    return (g & ((1u << A) - 1u)) | ((g >> A) << (A + R));
}
// Shared index of element i of a group whose base has shared index pb (the swizzle is linear
// over GF(2); for A >= 7 the window bits lie above the swizzled bits and the XOR is an add).
template <int A>
__device__ __forceinline__ uint32_t wix(uint32_t pb, int i) {
    if constexpr (A >= 7) return pb + ((uint32_t)i << A);
    else return pb ^ psw((uint32_t)i << A);
}

template <int A, int R>
__device__ __forceinline__ void wload(const float2* sp, uint32_t pb, float2 (&v)[1 << R]) {
    if constexpr (A == 0 && R >= 1) {
#pragma unroll
        for (int j = 0; j < (1 << R); j += 2) {
            const float4 q = *reinterpret_cast<const float4*>(sp + (pb ^ (uint32_t)j));
            v[j] = make_float2(q.x, q.y);
            v[j + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < (1 << R); ++i) v[i] = sp[wix<A>(pb, i)];
    }
}
template <int A, int R>
__device__ __forceinline__ void wstore(float2* sp, uint32_t pb, const float2 (&v)[1 << R]) {
    if constexpr (A == 0 && R >= 1) {
#pragma unroll
        for (int j = 0; j < (1 << R); j += 2)
            *reinterpret_cast<float4*>(sp + (pb ^ (uint32_t)j)) = make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y);
    } else {
#pragma unroll
        for (int i = 0; i < (1 << R); ++i) sp[wix<A>(pb, i)] = v[i];
    }
}

// Phases and energies of a top window's elements (group r of the thread): from the tile's energies in
// shared memory, or from the phase table.
struct ValsMem {
    const float* sE;
    template <bool F>
    __device__ __forceinline__ void load() {}
    template <int A, int R, typename Fn>
    __device__ __forceinline__ void phases(const PhaseK<float>& ph, uint32_t base, int, Fn&& fn) const {
#pragma unroll
        for (int i = 0; i < (1 << R); ++i) {
            float s, c;
            sincos_phase(ph, sE[base + ((uint32_t)i << A)], s, c);
            fn(i, s, c);
        }
    }
    template <int A, int R, typename Fn>
    __device__ __forceinline__ void energies(uint32_t base, int, Fn&& fn) const {
#pragma unroll
        for (int i = 0; i < (1 << R); ++i) fn(i, sE[base + ((uint32_t)i << A)]);
    }
};
struct ValsTab {
    const PhaseTab* t;
    TileVals x;
    template <bool F>
    __device__ __forceinline__ void load() {
        x.init<F>(*t);
    }
    template <int A, int R, typename Fn>
    __device__ __forceinline__ void phases(const PhaseK<float>&, uint32_t, int r, Fn&& fn) const {
        tab_phases<A, R>(x, r, fn);
    }
    template <int A, int R, typename Fn>
    __device__ __forceinline__ void energies(uint32_t, int r, Fn&& fn) const {
        tab_energies<A, R>(x, r, fn);
    }
};

// A pass takes a tile through the windows below its top one (upwards, mixing layer la), through the
// top window, which reaches tile bit 12 (mixer of la; a pass that ends a layer and opens the next:
// the cost phase of lb and its mixer; the opening pass: |+> in the rotated frame, phase and mixer of
// layer 0; the final pass: the pending shear factor of the last layer and the thread's FP32 <C> terms
// and maximum |psi|^2), and, where layer lb is mixed too, back down through the lower windows.
//
//   kind A:              [0,4) [4,8) | [8,13)
//   kind B, h high bits: [13-h,8)    | [8,13)   (h > 5; h <= 5: [13-h,13) alone)
//
// One copy of each lower window's code serves both ways and both kinds; the top window has one per
// thing it does (one body with run-time switches spilled 244 bytes: n = 30 18.6 ms, split 16.2). A
// five-bit top window leaves a thread one group with one phase start (windows [c,c+5) and [c+5,13)
// gave it up to eight: 13 shared loads per amplitude at h = 7; two-layer pass at n = 30 4.04 -> 3.82 ms).
enum { TOP_ONE, TOP_TWO, TOP_INIT, TOP_FIN };   // what the top window does besides: nothing, phase and mixer of lb, ...

// Window [A, A+R) below the top: the mixer of layer constants k on every group of the thread
// (2^(13-R) / 256 of them).
template <int A, int R>
__device__ __forceinline__ void low_window(float2* sp, const LayerConst<float>& k) {
    constexpr int NGT = (1 << (TB - R)) / NT;
#pragma unroll 1
    for (int r = 0; r < NGT; ++r) {
        const uint32_t pb = psw(wbase<A, R>(threadIdx.x + (uint32_t)(r * NT)));
        float2 v[1 << R];
        wload<A, R>(sp, pb, v);
        mix_layer<R>(v, (1 << R) - 1, k);
        wstore<A, R>(sp, pb, v);
    }
}

// The top window [A, 13), A >= 8: group r of the thread has base threadIdx.x + 256 r.
template <int MODE, int A, typename Vals>
__device__ __forceinline__ void top_window(float2* sp, const Geo& geo, const LayerConst<float>& ka,
                                           const LayerConst<float>& kb, Vals vals, float amp0, float& accp, float& pmax) {
    constexpr int R = TB - A, NGT = 1 << (A - 8);
    const int pz = __popcll(geo.zt);
    if (MODE != TOP_ONE) vals.template load<MODE == TOP_FIN>();
#pragma unroll 1
    for (int r = 0; r < NGT; ++r) {
        const uint32_t base = threadIdx.x + (uint32_t)(r * NT);
        const uint32_t pb = psw(base);
        float2 v[1 << R];
        if (MODE == TOP_INIT) {
            const int pc = __popc(base) + pz;
            vals.template phases<A, R>(ka.ph, base, r, [&](int i, float s, float c) {
                v[i] = times_i_pow(make_float2(amp0 * c, -amp0 * s), pc + __popc(i));
            });
        } else {
            wload<A, R>(sp, pb, v);
        }
        mix_layer<R>(v, (1 << R) - 1, ka);
        if (MODE == TOP_TWO) {
            const Pending<float> pre(kb.pre, kb.pcot, __popc(base) + pz);
            vals.template phases<A, R>(kb.ph, base, r, [&](int i, float s, float c) {
                rot_neg(v[i], s * pre.f[__popc(i) & 1], c * pre.f[__popc(i) & 1]);
            });
            mix_layer<R>(v, (1 << R) - 1, kb);
        }
        if (MODE == TOP_FIN) {
            scale_group<R>(v, Pending<float>(ka.post, ka.cot, __popc(base) + pz));
            vals.template energies<A, R>(base, r, [&](int i, float e) {
                const float pr = v[i].x * v[i].x + v[i].y * v[i].y;
                accp = fmaf(pr, e, accp);
                pmax = fmaxf(pmax, pr);
            });
        }
        wstore<A, R>(sp, pb, v);
    }
}
template <int MODE, typename Vals>
__device__ __forceinline__ void top_windows(int R, float2* sp, const Geo& geo, const LayerConst<float>& ka,
                                            const LayerConst<float>& kb, const Vals& vals, float amp0, float& accp,
                                            float& pmax) {
    switch (R) {
        case 1: top_window<MODE, 12>(sp, geo, ka, kb, vals, amp0, accp, pmax); break;
        case 2: top_window<MODE, 11>(sp, geo, ka, kb, vals, amp0, accp, pmax); break;
        case 3: top_window<MODE, 10>(sp, geo, ka, kb, vals, amp0, accp, pmax); break;
        case 4: top_window<MODE, 9>(sp, geo, ka, kb, vals, amp0, accp, pmax); break;
        default: top_window<MODE, 8>(sp, geo, ka, kb, vals, amp0, accp, pmax); break;
    }
}

template <typename Vals>
__device__ __forceinline__ void tile_pass(float2* sp, const Geo& geo, const StreamPass& P, const LayerConst<float>* lc,
                                          const Vals& vals, float amp0, float& accp, float& pmax) {
    const bool two = P.lb > P.la || P.init;
    const int nlow = geo.kindA ? 2 : (P.h > 5 ? 1 : 0);
    const int steps = two ? 2 * nlow : nlow;
#pragma unroll 1
    for (int i = P.init ? nlow : 0; i <= steps; ++i) {
        if (i == nlow) {
            const LayerConst<float>&ka = lc[P.la], &kb = lc[P.lb];
            const int R = geo.kindA ? 5 : P.h;
            if (P.init) top_window<TOP_INIT, 8>(sp, geo, ka, kb, vals, amp0, accp, pmax);   // a kind-A pass
            else if (two) top_windows<TOP_TWO>(R, sp, geo, ka, kb, vals, amp0, accp, pmax);
            else if (P.fin) top_windows<TOP_FIN>(R, sp, geo, ka, kb, vals, amp0, accp, pmax);
            else top_windows<TOP_ONE>(R, sp, geo, ka, kb, vals, amp0, accp, pmax);
        } else {
            const LayerConst<float>& k = lc[i < nlow ? P.la : P.lb];
            // kind A: [0,4) first and last; 0 and 4: the window's low bit
            switch (geo.kindA ? ((i & 3) ? 4 : 0) : TB - P.h) {
                case 0: low_window<0, 4>(sp, k); break;
                case 4: low_window<4, 4>(sp, k); break;
                case 5: low_window<5, 3>(sp, k); break;
                case 6: low_window<6, 2>(sp, k); break;
                default: low_window<7, 1>(sp, k); break;
            }
        }
        if (i < steps) __syncthreads();
    }
}

// Element i < 32 of the thread in the top window (reductions): shared and global index.
template <int A>
__device__ __forceinline__ void top_elem(const Geo& geo, int zsh, int i, uint32_t& ix, uint64_t& z) {
    constexpr int R = TB - A;
    const uint32_t base = threadIdx.x + (uint32_t)((i >> R) * NT);
    const int e = i & ((1 << R) - 1);
    ix = wix<A>(psw(base), e);
    z = geo.z(base) + ((uint64_t)e << zsh);
}
__device__ __forceinline__ void last_elem(const Geo& geo, const StreamPass& P, int i, uint32_t& ix, uint64_t& z) {
    switch (P.kind == 0 ? 5 : P.h) {
        case 1: top_elem<12>(geo, P.s, i, ix, z); break;
        case 2: top_elem<11>(geo, P.s, i, ix, z); break;
        case 3: top_elem<10>(geo, P.s, i, ix, z); break;
        case 4: top_elem<9>(geo, P.s, i, ix, z); break;
        default: top_elem<8>(geo, P.kind == 0 ? 8 : 8 - P.c + P.s, i, ix, z); break;
    }
}

// Shape of the tensor map of a pass (TMA coordinates of a tile): kind A; kind B with h <= 8 and
// qubits above the chunk (5-D) or without (4-D); kind B with h = 9, whose 512 high values are
// split over two box dimensions (at most 256 each), 5-D or 4-D; kind A of the adjoint's 12-bit tiles (3-D).
enum : int { TS_A, TS_B5, TS_B4, TS_B9_5, TS_B9_4, TS_A3 };
struct TsPass {
    int bmode;          // TS_*
    int midbits;        // kind B: tile-index bits below the chunk (s - c)
    int map;            // index of this pass's state map among an instance's maps
    int emap;           // index of its energy map
    int maps_per_inst;  // maps per instance in the plan's map array
};

// TMA coordinates of tile tau; the energy maps have the same coordinates as the state maps.
__device__ __forceinline__ void tile_load(const TsPass& T, const CUtensorMap* map, void* dst, uint64_t tau,
                                          uint64_t* bar) {
    const int mid = (int)(tau & ((1ull << T.midbits) - 1ull)), top = (int)(tau >> T.midbits);
    switch (T.bmode) {
        case TS_A: tma_load_4d(dst, map, 0, 0, 0, (int)tau, bar); break;
        case TS_A3: tma_load_3d(dst, map, 0, 0, (int)tau, bar); break;
        case TS_B5: tma_load_5d(dst, map, 0, 0, mid, 0, top, bar); break;
        case TS_B4: tma_load_4d(dst, map, 0, 0, mid, 0, bar); break;
        case TS_B9_5: tma_load_5d(dst, map, 0, mid, 0, 0, top, bar); break;
        default: tma_load_4d(dst, map, 0, mid, 0, 0, bar); break;
    }
}
// L2 prefetch of the tile tile_load would copy (a cache hint only)
__device__ __forceinline__ void tile_prefetch(const TsPass& T, const CUtensorMap* map, uint64_t tau) {
    const int mid = (int)(tau & ((1ull << T.midbits) - 1ull)), top = (int)(tau >> T.midbits);
    switch (T.bmode) {
        case TS_A: tma_prefetch_4d(map, 0, 0, 0, (int)tau); break;
        case TS_A3: tma_prefetch_3d(map, 0, 0, (int)tau); break;
        case TS_B5: tma_prefetch_5d(map, 0, 0, mid, 0, top); break;
        case TS_B4: tma_prefetch_4d(map, 0, 0, mid, 0); break;
        case TS_B9_5: tma_prefetch_5d(map, 0, mid, 0, 0, top); break;
        default: tma_prefetch_4d(map, 0, mid, 0, 0); break;
    }
}
__device__ __forceinline__ void tile_store(const TsPass& T, const CUtensorMap* map, const void* src, uint64_t tau) {
    const int mid = (int)(tau & ((1ull << T.midbits) - 1ull)), top = (int)(tau >> T.midbits);
    switch (T.bmode) {
        case TS_A: tma_store_4d(map, src, 0, 0, 0, (int)tau); break;
        case TS_A3: tma_store_3d(map, src, 0, 0, (int)tau); break;
        case TS_B5: tma_store_5d(map, src, 0, 0, mid, 0, top); break;
        case TS_B4: tma_store_4d(map, src, 0, 0, mid, 0); break;
        case TS_B9_5: tma_store_5d(map, src, 0, mid, 0, 0, top); break;
        default: tma_store_4d(map, src, 0, mid, 0, 0); break;
    }
}

// The segment a CTA works on: a group's pass, formed from the group's numbers by one thread.
struct SegPass {
    uint32_t tile0;
    int si, lam_first;
    StreamPass P;
    TsPass T;
    const StreamInst<float>* insts;
    const CUtensorMap* maps;
};
__host__ __device__ __noinline__ void expand_segment(const TsGroup* groups, const TsSeg& seg, SegPass* x) {
    const TsGroup& g = groups[seg.group];
    const int s = seg.pass, W = g.W;
    int l = 0, pos = s;
    if (s >= W) {
        l = 1 + (s - W) / (W - 1);
        pos = 1 + (s - W) % (W - 1);
    }
    const int w = (l & 1) ? W - 1 - pos : pos;
    StreamPass P{};
    P.n = g.n;
    P.tb = g.tb;
    P.la = l;
    P.lb = (pos == W - 1 && l + 1 < g.p) ? l + 1 : l;
    P.ph_first = P.init = s == 0;
    P.fin = s == g.S - 1;
    P.k = P.fin ? g.k : 0;
    P.kind = w > 0;
    P.h = w > 0 ? g.ch[w - 1] : 0;
    P.s = w > 0 ? g.cs[w - 1] : g.tb;
    P.c = g.tb - P.h;
    P.need_e = P.ph_first || P.lb > P.la || P.fin;
    P.keep_frame = P.fin && g.keep_frame;
    P.no_store = P.fin && g.no_store;
    TsPass T{};
    T.maps_per_inst = g.maps_per_inst;
    T.map = g.adjoint ? 3 * w : w;
    T.emap = g.adjoint ? T.map + 2 : W + w;
    if (w == 0) {
        T.bmode = g.adjoint ? TS_A3 : TS_A;
    } else {
        const bool top = P.s + P.h < P.n;
        T.midbits = P.s - P.c;
        T.bmode = P.h <= 8 ? (top ? TS_B5 : TS_B4) : (top ? TS_B9_5 : TS_B9_4);
    }
    x->tile0 = seg.tile0;
    x->si = s;
    x->lam_first = s == g.S - 1;
    x->P = P;
    x->T = T;
    x->insts = g.insts;
    x->maps = static_cast<const CUtensorMap*>(g.maps);
}
// Move on to the segment of tile q. All threads call it, behind a barrier that follows their last
// use of the segment.
__device__ __forceinline__ void advance_segment(const TsGroup* groups, const TsSeg* segs, int nseg, uint32_t total,
                                                uint32_t q, int& sg, uint32_t& send, SegPass* cur) {
    do {
        ++sg;
        send = sg + 1 < nseg ? segs[sg + 1].tile0 : total;
    } while (q >= send);
    if (threadIdx.x == 0) expand_segment(groups, segs[sg], cur);
    __syncthreads();
}

// TAB: phases and energies come from Q (qaoa_phase.cuh), no energy vector exists; else from the energies
// in HBM (gradient runs, whose adjoint reads them, and instances that return them).
// RUNS: a CTA takes its share of the tiles in a row instead of every gridDim.x-th, so that it meets few
// instances: a table is an instance's, and rebuilding it for every tile took back what the tables give
// (64 instances of n = 20, p = 3: 1218 us with energies, 1371 with a table per tile, 1067 in rows; 16 of n = 22:
// 1295, 1313, 1072). Large instances stay with the stride, whose CTAs read neighbouring tiles at a time
// (n = 30: 1% faster).
template <bool TAB, bool RUNS>
__global__ void __launch_bounds__(NT, 2) k_tstream_pass(const TsGroup* __restrict__ groups,
                                                       const TsSeg* __restrict__ segs, int nseg, uint32_t total,
                                                       unsigned* status) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ SegPass cur, nxt;   // nxt: thread 0's, for loads of the next segment's first tile
    const uint32_t raw = saddr(sm_raw);
    unsigned char* sm = sm_raw + (((raw + 1023u) & ~1023u) - raw);
    const TsOff o = ts_offsets(TAB);
    float2* const sp = reinterpret_cast<float2*>(sm + o.psi);
    float* const sE = reinterpret_cast<float*>(sm + o.E);
    PhaseTab& tab = *reinterpret_cast<PhaseTab*>(sm + o.E);
    LayerConst<float>* lc = reinterpret_cast<LayerConst<float>*>(sm + o.lc);
    float* red = reinterpret_cast<float*>(sm + o.red);
    TileTopk ts;
    ts.wb = reinterpret_cast<float*>(sm + o.wb);
    ts.cnt = reinterpret_cast<int*>(sm + o.cnt);
    ts.cand = reinterpret_cast<TopEnt*>(sm + o.cand);
    ts.out = reinterpret_cast<TopEnt*>(sm + o.out);
    ts.wlists = reinterpret_cast<TopEnt*>(sm + o.wlists);
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + o.mbar);
    if (threadIdx.x == 0) mbar_init(mbar, 1);
    __syncthreads();

    const StreamPass& P = cur.P;
    const TsPass& T = cur.T;
    uint32_t parity = 0;
    bool ok = true;
    int sg = -1;
    uint32_t send = 0;        // first tile past the segment
    const uint32_t per = total / gridDim.x, rem = total % gridDim.x;
    const uint32_t q0 = RUNS ? blockIdx.x * per + min(blockIdx.x, rem) : blockIdx.x;
    const uint32_t qend = RUNS ? q0 + per + (blockIdx.x < rem ? 1u : 0u) : total;
    const uint32_t qstep = RUNS ? 1u : gridDim.x;
    if (q0 < qend) advance_segment(groups, segs, nseg, total, q0, sg, send, &cur);
    // Thread 0: the loads of tile q (segment S). The energies first (their buffer is never stored
    // from), then, once the last tile's store has read the state buffer (wait_store), the state.
    auto issue = [&](uint32_t q, bool wait_store) {
        const SegPass* S = &cur;
        if (q >= send) {
            int j = sg + 1;
            while (j + 1 < nseg && q >= segs[j + 1].tile0) ++j;
            expand_segment(groups, segs[j], &nxt);
            S = &nxt;
        }
        const StreamPass& p = S->P;
        const TsPass& t = S->T;
        const bool need_e = !TAB && p.need_e;
        if (p.init && !need_e) return;
        const int tbits = p.n - TB;
        const uint32_t ql = q - S->tile0, tmask = (1u << tbits) - 1u;
        const CUtensorMap* m = S->maps + (size_t)(ql >> tbits) * t.maps_per_inst;
        mbar_expect_tx(mbar, (p.init ? 0u : TD * 8) + (need_e ? TD * 4 : 0u));
        if (need_e) tile_load(t, m + t.emap, sE, ql & tmask, mbar);
        if (!p.init) {
            if (wait_store) bulk_wait_read();
            tile_load(t, m + t.map, sp, ql & tmask, mbar);
        }
        // the tile after it towards L2, a tile's compute ahead of its own load (in the passes
        // that store no state: with the state stores in flight it slowed the others down)
        const uint32_t q1 = ql + qstep;
        const uint32_t end = S == &cur ? (RUNS ? min(send, qend) : send) - S->tile0 : 0u;
        if ((p.init || (p.fin && p.no_store)) && q1 < end) {
            const CUtensorMap* m1 = S->maps + (size_t)(q1 >> tbits) * t.maps_per_inst;
            if (need_e) tile_prefetch(t, m1 + t.emap, q1 & tmask);
            if (!p.init) tile_prefetch(t, m1 + t.map, q1 & tmask);
        }
    };
    if (q0 < qend && threadIdx.x == 0) issue(q0, false);
    // what the constants and the table belong to, in shared memory: the sub-passes need the registers
    __shared__ const float *cur_g, *cur_b, *cur_q;
    __shared__ int cur_p, cur_n, cur_l;
    if (threadIdx.x == 0) cur_n = 0;
    __syncthreads();
    TopEnt* run = reinterpret_cast<TopEnt*>(sm + o.run);
    bool run_valid = false;   // the run list holds this CTA's best k of the current instance so far
    for (uint32_t q = q0; q < qend; q += qstep) {
        if (q >= send) {
            __syncthreads();
            advance_segment(groups, segs, nseg, total, q, sg, send, &cur);
        }
        const int tbits = P.n - TB;                 // tiles of an instance: 2^tbits
        const uint32_t ql = q - cur.tile0;
        const int ii = (int)(ql >> tbits);
        const uint64_t tau = ql & ((1u << tbits) - 1u);
        const bool store = !P.fin || !P.no_store;
        const StreamInst<float>& I = cur.insts[ii];
        const bool same = P.n == cur_n && I.p == cur_p && I.gamma == cur_g && I.beta == cur_b;
        const int layer = TAB && P.need_e ? (P.fin ? I.p : P.lb) + 64 * (P.kind ? P.s : 0) : -1;   // what the table holds
        const bool retab = layer >= 0 && !(same && I.Q == cur_q && layer == cur_l);
        if (!same || retab) {
            __syncthreads();
            if (!same) set_layer_consts<float>(lc, I.gamma, I.beta, I.p, P.n, false);
            if (TAB && retab) {
                if (P.fin) tab_build<true>(tab, I.Q, P.n, 0.0, P.c, P.s);
                else tab_build<false>(tab, I.Q, P.n, (double)I.gamma[P.lb] * 0.15915494309189533577, P.c, P.s);   // gamma / 2 pi
            }
            if (threadIdx.x == 0) {
                cur_g = I.gamma; cur_b = I.beta; cur_p = I.p; cur_n = P.n;
                if (retab) { cur_q = I.Q; cur_l = layer; }
                if (!same && !retab) cur_q = nullptr;
            }
            __syncthreads();
        }
        Geo geo;
        geo.kindA = P.kind == 0;
        geo.c = P.c;
        geo.s = P.s;
        geo.lomask = (1u << P.c) - 1u;
        if (geo.kindA) {
            geo.zt = tau << TB;
        } else {
            const int midbits = P.s - P.c;
            const uint64_t mid = tau & ((1ull << midbits) - 1ull), top = tau >> midbits;
            geo.zt = (mid << P.c) | (top << (P.s + P.h));
        }
        if (TAB && P.need_e) {
            if (P.fin) tab_tile<true>(tab, (uint32_t)geo.zt, P.c, P.s);
            else tab_tile<false>(tab, (uint32_t)geo.zt, P.c, P.s);
        }
        if (!P.init || (!TAB && P.need_e)) {
            if (ok) ok = mbar_wait_bounded(mbar, parity);
            parity ^= 1u;
        }
        // a pass that loads no state may meet a store of the last tile still reading the buffer
        if (P.init && threadIdx.x == 0) bulk_wait_read();
        ok = __syncthreads_and(ok);
        float accp = 0.0f, pmax = -1.0f;
        if constexpr (TAB) tile_pass(sp, geo, P, lc, ValsTab{&tab}, (float)I.amp0, accp, pmax);
        else tile_pass(sp, geo, P, lc, ValsMem{sE}, (float)I.amp0, accp, pmax);
        if (P.fin) warp_sum_df(accp, red);
        __syncthreads();
        if (P.fin) {
            if (threadIdx.x < 32) {
                const double tot = sum_parts_df(red);
                if (threadIdx.x == 0) I.part_expect[tau] = tot;
            }
            if (P.k > 0) {
                // Top-k: the CTA carries one list (run) across its tiles of an instance and writes
                // it into the slot of its last such tile (the other slots it owns stay empty); the
                // list of an instance is unique, so this does not depend on which tiles a CTA gets.
                const auto elem = [&geo, &P](int i, uint32_t& ix, uint32_t& z) {
                    uint64_t zz;
                    last_elem(geo, P, i, ix, zz);
                    z = (uint32_t)zz;
                };
                const int kk = P.k;
                const auto full_tile = [&]() {   // the tile's own list into ts.out
                    if (!topk_own(sp, kk, pmax, elem, ts, reinterpret_cast<float*>(sm + o.wbound))) {
                        float pm2 = -1.0f;
                        for (uint32_t u = threadIdx.x; u < TD; u += NT) {
                            const float2 v = sp[psw(u)];
                            pm2 = fmaxf(pm2, v.x * v.x + v.y * v.y);
                        }
                        const TileRef<float> tile{sp, nullptr, nullptr, TB};
                        const auto zmap = [&geo](uint32_t u) { return (uint32_t)geo.z(u); };
                        tile_topk<float, TmaLayout>(tile, kk, pm2, zmap, ts);
                    }
                };
                // the k best of `na` entries a[] and the run list, into run (rank selection)
                const auto merge_run = [&](const TopEnt* a, int na) {
                    TopEnt* merged = ts.wlists;
                    for (int c = threadIdx.x; c < na + kk; c += NT) {
                        const TopEnt me = c < na ? a[c] : run[c - na];
                        int rank = 0;
                        for (int j2 = 0; j2 < na; ++j2) rank += better(a[j2].p, a[j2].z, me.p, me.z) ? 1 : 0;
                        for (int j2 = 0; j2 < kk; ++j2) rank += better(run[j2].p, run[j2].z, me.p, me.z) ? 1 : 0;
                        if (rank < kk) merged[rank] = me;
                    }
                    __syncthreads();
                    if (threadIdx.x < (unsigned)kk) run[threadIdx.x] = merged[threadIdx.x];
                    __syncthreads();
                };
                if (!run_valid) {
                    full_tile();
                    if (threadIdx.x < (unsigned)kk) run[threadIdx.x] = ts.out[threadIdx.x];
                    __syncthreads();
                    run_valid = true;
                } else {
                    const float lo = __double2float_rd(run[kk - 1].p) * 0.99999904632568359375f;   // (1 - 2^-20)
                    if (threadIdx.x == 0) { ts.cnt[0] = 0; ts.cnt[1] = 0; }
                    if (__syncthreads_or(pmax * 1.000003814697265625f >= lo)) {
                        if (pmax * 1.000003814697265625f >= lo) {
                            for (int i = 0; i < 32; ++i) {
                                uint32_t ix, z;
                                elem(i, ix, z);
                                const float2 v = sp[ix];
                                if ((v.x * v.x + v.y * v.y) * 1.00000095367431640625f >= lo) {
                                    const int pos = atomicAdd(&ts.cnt[0], 1);
                                    if (pos < TOPK_CAP) {
                                        ts.cand[pos].p = __hiloint2double(__float_as_int(v.y), __float_as_int(v.x));
                                        ts.cand[pos].z = z;
                                    } else {
                                        ts.cnt[1] = 1;
                                    }
                                }
                            }
                        }
                        __syncthreads();
                        if (!ts.cnt[1]) {
                            const int cnt = ts.cnt[0];
                            for (int c = threadIdx.x; c < cnt; c += NT) {
                                const double raw = ts.cand[c].p;
                                ts.cand[c].p = exact_prob(make_float2(__int_as_float(__double2loint(raw)),
                                                                      __int_as_float(__double2hiint(raw))));
                            }
                            __syncthreads();
                            merge_run(ts.cand, cnt);
                        } else {
                            __syncthreads();   // every thread has read the overflow flag
                            full_tile();
                            merge_run(ts.out, kk);
                        }
                    }
                }
                // this tile's slot: the list when it is the CTA's last tile of the instance
                const uint32_t qn = q + qstep;
                const bool last_of_inst = (RUNS && qn >= qend) || qn >= send || (int)((qn - cur.tile0) >> tbits) != ii;
                if (threadIdx.x < (unsigned)kk) {
                    const TopEnt e = last_of_inst ? run[threadIdx.x] : TopEnt{-1.0, 0xffffffffu};
                    I.part_topp[tau * kk + threadIdx.x] = e.p;
                    I.part_topz[tau * kk + threadIdx.x] = e.z;
                }
                if (last_of_inst) run_valid = false;
            }
            if (store && !P.keep_frame) {
                // the state leaves in the standard frame: psi = (-i)^{|z|} psi~
                __syncthreads();
                for (uint32_t u = threadIdx.x; u < TD; u += NT)
                    sp[psw(u)] = times_i_pow(sp[psw(u)], -__popcll(geo.z(u)));
            }
        }
        if (store) {
            fence_async_smem();
            __syncthreads();
            if (threadIdx.x == 0) {
                tile_store(T, cur.maps + (size_t)ii * T.maps_per_inst + T.map, sp, tau);
                bulk_commit();
            }
        } else {
            fence_async_smem();   // the sub-passes' shared writes before the next tile's TMA writes
            __syncthreads();
        }
        // the next tile's loads: the energies at once, the state once this tile's store has read
        // the buffer (the init pass loads only the energies)
        if (q + qstep < qend && threadIdx.x == 0 && ok) issue(q + qstep, true);
    }
    if (threadIdx.x == 0) {
        bulk_wait_all();
        if (!ok) atomicOr(status, 1u);
    }
}

// ---- adjoint passes ---------------------------------------------------------------------------
// The forward pass P undone on 2^12-amplitude tiles of psi and lam (both in the rotated frame),
// with the adjoint sub-passes of the tile engine on the TMA layout (amplitudes in the 128-byte
// swizzle, energies unswizzled): the local snake of P run in reverse, a single layer that opens
// with its cost phase ordered so that the phase (an energy read) shares the top window, where
// the lanes of a warp cover the low tile bits. Per tile the four FP64 gradient partials of the
// cp.async adjoint ([0] Im <lam|B|psi> of layer lb, [1] of la, [2] Im <lam|E|psi> of lb, [3] of
// la) are written; psi and lam go back by TMA unless this is the last adjoint pass. Persistent,
// two CTAs per SM (psi, lam and energies of a tile: 80 KiB), a CTA's next tile loaded once the
// bulk stores of the current one have read the buffers.
constexpr uint32_t TDA = 1u << TSA_TB;

struct TaOff {
    size_t psi, lam, E, lc, red, mbar, total;
};
__host__ __device__ inline TaOff ta_offsets() {
    TaOff o{};
    size_t x = 0;
    o.psi = x; x += (size_t)TDA * 8;   // 1024-aligned at run time (swizzled)
    o.lam = x; x += (size_t)TDA * 8;   // 32 KiB further: still 1024-aligned
    o.E = x; x += (size_t)TDA * 4;
    o.lc = x; x = ts_al(x + 64 * sizeof(LayerConst<float>));
    o.red = x; x = ts_al(x + 32 * sizeof(double));
    o.mbar = x; x = ts_al(x + sizeof(uint64_t));
    o.total = x + 1024;
    return o;
}

__global__ void __launch_bounds__(NT, 2) k_tstream_adj_pass(const TsGroup* __restrict__ groups,
                                                           const TsSeg* __restrict__ segs, int nseg, uint32_t total,
                                                           unsigned* status) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ SegPass cur, nxt;   // nxt: thread 0's, for loads of the next segment's first tile
    const uint32_t raw = saddr(sm_raw);
    unsigned char* sm = sm_raw + (((raw + 1023u) & ~1023u) - raw);
    const TaOff o = ta_offsets();
    float2* spsi = reinterpret_cast<float2*>(sm + o.psi);
    float2* slam = reinterpret_cast<float2*>(sm + o.lam);
    float* sE = reinterpret_cast<float*>(sm + o.E);
    LayerConst<float>* lc = reinterpret_cast<LayerConst<float>*>(sm + o.lc);
    double* red = reinterpret_cast<double*>(sm + o.red);
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + o.mbar);
    // the parameters the constants belong to, in shared memory: the sub-passes need the registers
    __shared__ const float *cur_g, *cur_b;
    __shared__ int cur_p;
    if (threadIdx.x == 0) {
        mbar_init(mbar, 1);
        cur_p = 0;
    }
    __syncthreads();

    constexpr int RA = Num<float>::RB_ADJ;
    const StreamPass& P = cur.P;
    const TsPass& T = cur.T;
    uint32_t parity = 0;
    bool ok = true;
    int sg = -1;
    uint32_t send = 0;
    if (blockIdx.x < total) advance_segment(groups, segs, nseg, total, blockIdx.x, sg, send, &cur);
    // the energies first (never stored from), then, once the last tile's stores have read the
    // state buffers (wait_store), psi and lam
    auto issue = [&](uint32_t q, bool wait_store) {
        const SegPass* S = &cur;
        if (q >= send) {
            int j = sg + 1;
            while (j + 1 < nseg && q >= segs[j + 1].tile0) ++j;
            expand_segment(groups, segs[j], &nxt);
            S = &nxt;
        }
        const TsPass& t = S->T;
        const bool lam_first = S->lam_first, need_e = lam_first || S->P.ph_first || S->P.lb > S->P.la;
        const int tbits = S->P.n - TSA_TB;
        const uint32_t ql = q - S->tile0, tmask = (1u << tbits) - 1u, tau = ql & tmask;
        const CUtensorMap* m = S->maps + (size_t)(ql >> tbits) * t.maps_per_inst;
        mbar_expect_tx(mbar, TDA * 8 + (lam_first ? 0u : TDA * 8) + (need_e ? TDA * 4 : 0u));
        if (need_e) tile_load(t, m + t.emap, sE, tau, mbar);
        if (wait_store) bulk_wait_read();
        tile_load(t, m + t.map, spsi, tau, mbar);
        if (!lam_first) tile_load(t, m + t.map + 1, slam, tau, mbar);
        // the tile after it towards L2, a tile's compute ahead of its own loads
        const uint32_t q1 = ql + gridDim.x;
        if (S == &cur && q1 < send - S->tile0) {
            const CUtensorMap* m1 = S->maps + (size_t)(q1 >> tbits) * t.maps_per_inst;
            if (need_e) tile_prefetch(t, m1 + t.emap, q1 & tmask);
            tile_prefetch(t, m1 + t.map, q1 & tmask);
            if (!lam_first) tile_prefetch(t, m1 + t.map + 1, q1 & tmask);
        }
    };
    if (blockIdx.x < total && threadIdx.x == 0) issue(blockIdx.x, false);
    const TileRef<float> tile{spsi, slam, sE, TSA_TB};
    for (uint32_t q = blockIdx.x; q < total; q += gridDim.x) {
        if (q >= send) {
            __syncthreads();
            advance_segment(groups, segs, nseg, total, q, sg, send, &cur);
        }
        const int tbits = P.n - TSA_TB;
        const uint32_t ql = q - cur.tile0, tau = ql & ((1u << tbits) - 1u);
        const StreamInst<float>& I = cur.insts[ql >> tbits];
        if (I.p != cur_p || I.gamma != cur_g || I.beta != cur_b) {   // (the adjoint's constants do not depend on n)
            __syncthreads();
            set_layer_consts<float>(lc, I.gamma, I.beta, I.p, P.n, true);
            if (threadIdx.x == 0) { cur_g = I.gamma; cur_b = I.beta; cur_p = I.p; }
            __syncthreads();
        }
        if (ok) ok = mbar_wait_bounded(mbar, parity);
        parity ^= 1u;
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        bool first_sub = cur.lam_first;
        Snake sn(P.lb - P.la + 1, P.la, P.ph_first, P.kind == 0 ? 0 : P.c, TSA_TB, TSA_TB, RA, true);
        sn.to_last();
        for (;; sn.prev()) {
            const SubPass sp = sn.get();
            subpass_adj<float, RA, TmaLayout>(tile, sp, lc, first_sub, P.lb, acc);
            first_sub = false;
            __syncthreads();
            if (sn.first()) break;
        }
        double* out = I.part_grad + (((uint64_t)cur.si << tbits) + tau) * 4;
        const double v = block_sum4((double)acc[0], (double)acc[1], (double)acc[2], (double)acc[3], red);
        if (threadIdx.x < 4) out[threadIdx.x] = v;
        if (cur.si > 0) {   // the first pass's states are not needed any more
            fence_async_smem();
            __syncthreads();
            if (threadIdx.x == 0) {
                const CUtensorMap* m = cur.maps + (size_t)(ql >> tbits) * T.maps_per_inst;
                tile_store(T, m + T.map, spsi, tau);
                tile_store(T, m + T.map + 1, slam, tau);
                bulk_commit();
            }
        } else {
            fence_async_smem();   // the sub-passes' shared writes before the next tile's TMA writes
            __syncthreads();
        }
        // the next tile's loads: the energies at once, psi and lam once this tile's stores have
        // read the buffers
        if (q + gridDim.x < total && threadIdx.x == 0 && ok) issue(q + gridDim.x, true);
    }
    if (threadIdx.x == 0) {
        bulk_wait_all();
        if (!ok) atomicOr(status, 1u);
    }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn() {
    static EncodeFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeFn) nullptr;
        return reinterpret_cast<EncodeFn>(f);
    }();
    return fn;
}

bool encode(CUtensorMap* m, void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
            const cuuint32_t* box, bool swz128) {
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, base, dims, strides, box, es,
                       CU_TENSOR_MAP_INTERLEAVE_NONE,
                       swz128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The map of one pass shape over an array of 2^n elements of `w` floats each (w = 2: the
// complex64 state, swizzled; w = 1: the energies, unswizzled). The innermost dimension is the 16
// elements of tile bits 0..3 (16 w floats); the others follow TsPass::bmode.
bool encode_shape(const StreamPass& P, void* base, int w, CUtensorMap* m) {
    const int n = P.n;
    const cuuint64_t f = (cuuint64_t)w * 4;            // bytes per element
    const cuuint32_t d0 = 16u * (cuuint32_t)w;
    const bool swz = w == 2;
    if (P.kind == 0 && P.tb == TSA_TB) {   // (16 elements, 256 lines, tile): the adjoint's tiles
        const cuuint64_t d[3] = {d0, 256, 1ull << (n - TSA_TB)};
        const cuuint64_t s[2] = {16 * f, 4096 * f};
        const cuuint32_t b[3] = {d0, 256, 1};
        return encode(m, base, 3, d, s, b, swz);
    }
    if (P.kind == 0) {   // (16 elements, 256 lines, 2 planes, tile)
        const cuuint64_t d[4] = {d0, 256, 2, 1ull << (n - TB)};
        const cuuint64_t s[3] = {16 * f, 4096 * f, 8192 * f};
        const cuuint32_t b[4] = {d0, 256, 2, 1};
        return encode(m, base, 4, d, s, b, swz);
    }
    const int c = P.c, sh = P.s, h = P.h;
    const bool top = sh + h < n;
    const cuuint64_t topd = 1ull << (n - sh - h);
    if (h <= 8) {   // (16 elements, lines of bits 4..c-1, tile bits c..s-1, hi bits s..s+h-1[, top])
        const cuuint64_t d[5] = {d0, 1ull << (c - 4), 1ull << (sh - c), 1ull << h, topd};
        const cuuint64_t s[4] = {16 * f, (1ull << c) * f, (1ull << sh) * f, (1ull << (sh + h)) * f};
        const cuuint32_t b[5] = {d0, 1u << (c - 4), 1, 1u << h, 1};
        return encode(m, base, top ? 5 : 4, d, s, b, swz);
    }
    // h = 9, c = 4: (16 elements, tile bits 4..s-1, hi bits s..s+7, hi bit s+8[, top])
    const cuuint64_t d[5] = {d0, 1ull << (sh - c), 256, 2, topd};
    const cuuint64_t s[4] = {16 * f, (1ull << sh) * f, (1ull << (sh + 8)) * f, (1ull << (sh + 9)) * f};
    const cuuint32_t b[5] = {d0, 1, 256, 2, 1};
    return encode(m, base, top ? 5 : 4, d, s, b, swz);
}

}  // namespace

bool tstream_available() { return encode_fn() != nullptr; }

size_t tstream_smem_bytes(bool tab) { return ts_offsets(tab).total; }

bool tstream_encode_maps(const StreamPass& P, void* psi, void* E, void* psi_map, void* e_map) {
    if (!encode_fn() || P.tb != TB || P.n <= TB || P.n > 34) return false;
    return encode_shape(P, psi, 2, static_cast<CUtensorMap*>(psi_map)) &&
           (!E || encode_shape(P, E, 1, static_cast<CUtensorMap*>(e_map)));
}

void tstream_group_windows(const StreamPass* passes, int S, TsGroup* g) {
    g->S = S;
    g->W = 1;
    for (int i = 0; i < 4; ++i) g->cs[i] = g->ch[i] = 0;
    // the first pass of every window, in layer 0: contiguous, then the chunks by start qubit
    for (int i = 0; i < S && passes[i].la == 0; ++i)
        if (passes[i].kind == 1 && g->W <= 4) {
            g->cs[g->W - 1] = passes[i].s;
            g->ch[g->W - 1] = passes[i].h;
            ++g->W;
        }
}

cudaError_t launch_tstream_pass(bool tab, const TsGroup* groups, const TsSeg* segs, int nseg, uint32_t total, int grid,
                                bool runs, unsigned* status, cudaStream_t st) {
    const size_t sm = tstream_smem_bytes(tab);
    const auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        kern<<<grid, NT, sm, st>>>(groups, segs, nseg, total, status);
        return cudaGetLastError();
    };
    if (!tab) return go(k_tstream_pass<false, false>);
    return runs ? go(k_tstream_pass<true, true>) : go(k_tstream_pass<true, false>);
}

size_t tstream_adj_smem_bytes() { return ta_offsets().total; }

bool tstream_encode_adj_maps(const StreamPass& P, void* psi, void* lam, void* E, void* maps3) {
    if (!encode_fn() || P.tb != TSA_TB || P.n <= TSA_TB || P.n > 34 || (P.kind == 1 && (P.h > 8 || P.c < 4)))
        return false;
    char* b = static_cast<char*>(maps3);
    return encode_shape(P, psi, 2, reinterpret_cast<CUtensorMap*>(b)) &&
           encode_shape(P, lam, 2, reinterpret_cast<CUtensorMap*>(b + TS_MAP_BYTES)) &&
           encode_shape(P, E, 1, reinterpret_cast<CUtensorMap*>(b + 2 * TS_MAP_BYTES));
}

cudaError_t launch_tstream_adj_pass(const TsGroup* groups, const TsSeg* segs, int nseg, uint32_t total, int grid,
                                    unsigned* status, cudaStream_t st) {
    const size_t sm = tstream_adj_smem_bytes();
    cudaError_t e = cudaFuncSetAttribute(k_tstream_adj_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_tstream_adj_pass<<<grid, NT, sm, st>>>(groups, segs, nseg, total, status);
    return cudaGetLastError();
}

}  // namespace qaoa
