// k_resident.cu -- resident tier: one CTA per QAOA instance, the whole 2^n state (complex64
// up to n = 14, complex128 up to n = 13) and its energy vector held in shared memory for all
// p layers. One persistent launch walks a queue of instance descriptors; each CTA
//   1. builds E(z) = z^T Q z for all z from small tables (Section IV, the QUBO mapped to the
//      diagonal problem Hamiltonian),
//   2. applies the p layers of Eq. 2 (cost phase, then exp(-i beta X_q) on every qubit) from
//      |+> with the snake schedule of the tile engine,
//   3. reduces <C> = sum |psi|^2 E (FP32 per-thread partials over at most 2^R terms, FP64
//      above) and the k most probable bitstrings (the sub-solution of Section IV), fused into
//      the last sub-pass,
//   4. optionally runs the adjoint sweep for d<C>/d(gamma, beta) on the same shared tile.
#include <algorithm>

#include "qaoa_engine.cuh"
#include "qaoa_kernels.h"

namespace qaoa {

namespace {

template <typename T>
struct Smem {
    typename Num<T>::C* psi;
    typename Num<T>::C* lam;
    T* E;
    T* Q;
    LayerConst<T>* lc;     // adjoint; the forward run's constants occupy the same place
    double* red;       // 64 doubles
    TileTopk tk;       // top-k scratch
    T* escr;           // energy-build tables
};

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

template <typename T>
__host__ __device__ inline size_t smem_layout(int n, int p, bool grad, int threads, size_t* off) {
    using C = typename Num<T>::C;
    const size_t D = (size_t)1 << n;
    size_t o = 0;
    off[0] = o; o = align_up(o + D * sizeof(C), 16);                       // psi
    off[1] = o; if (grad) o = align_up(o + D * sizeof(C), 16);             // lam
    off[2] = o; o = align_up(o + D * sizeof(T), 16);                       // E
    off[3] = o; o = align_up(o + (size_t)n * n * sizeof(T), 16);           // Q
    off[4] = o; o = align_up(o + (size_t)p * sizeof(LayerConst<T>), 16);   // layer consts
    off[5] = o; o = align_up(o + 64 * sizeof(double), 16);                 // reduction
    // the energy-build tables are used before the first sub-pass and the top-k scratch after
    // the last one: both live in one region
    const size_t nw = (size_t)(threads + 31) / 32;
    const size_t r0 = o;
    off[7] = o; o = align_up(o + nw * 32 * sizeof(TopEnt), 16);          // fallback lists
    off[8] = o; o = align_up(o + TOPK_CAP * sizeof(TopEnt), 16);         // candidates
    off[9] = o; o = align_up(o + 16 * sizeof(TopEnt), 16);               // tile top-k
    off[10] = o; o = align_up(o + 16 * 32 * sizeof(float) + 4 * sizeof(int), 16);  // bounds, counts
    off[11] = r0;                                                         // energy tables
    const size_t eend = align_up(r0 + tile_energy_scratch(n) * sizeof(T), 16);
    if (eend > o) o = eend;
    return o;
}

template <typename T, int R, typename K>
__device__ void forward_run(const InstDesc<T>& d, const Smem<T>& s, const WinSched& ws, bool started) {
    const int n = d.n, p = d.p;
    const TileRef<T> tile{s.psi, s.lam, s.E, n};
    // started: the energy build already wrote |+> after the first cost layer
    const bool init = !(d.flags & F_INIT_PSI) && !started;
    const T amp0 = (T)exp2(-0.5 * (double)n);
    const K* lc = reinterpret_cast<const K*>(s.lc);
    // layer by layer through the windows in the schedule's order; when a layer's last window is the
    // next one's first, both share a sub-pass around the cost phase
    bool opens = !started, first = true;
    int pos = 0;
    for (int l = 0; l < p;) {
        SubPass sp;
        const int w = (l & 1) ? ws.odd[pos] : pos;
        sp.a = ws.a[w];
        sp.mask = ws.mask[w];
        sp.la = sp.lb = l;
        sp.ph_first = opens;
        opens = false;
        if (++pos == ws.nw) {
            pos = 0;
            opens = true;
            ++l;
            if (l < p && w == ((l & 1) ? ws.odd[0] : 0)) {
                sp.lb = l;
                opens = false;
                if (++pos == ws.nw) { pos = 0; opens = true; ++l; }
            }
        }
        sp.post = l == p;
        subpass_fwd<T, R>(tile, sp, lc, init && first, amp0, 0);
        first = false;
        __syncthreads();
    }
    // <C> and the top-k list of the final state (the list is unique under (probability desc,
    // index asc), whatever the order of the reduction)
    if (!d.expect && d.k == 0) return;   // the state alone is wanted
    double ex = 0.0;
    tile_reduce<T>(tile, d.k, [](uint32_t u) { return u; }, s.tk, ex);
    const double tot = block_sum(ex, s.red);
    if (threadIdx.x == 0 && d.expect) *d.expect = tot;
    if (threadIdx.x < (unsigned)d.k) {
        const TopEnt e = s.tk.out[threadIdx.x];
        if (d.topk_idx) d.topk_idx[threadIdx.x] = (uint64_t)e.z;
        if (d.topk_prob) d.topk_prob[threadIdx.x] = e.p;
    }
    __syncthreads();
}

template <typename T, int R>
__device__ void adjoint_run(const InstDesc<T>& d, const Smem<T>& s) {
    const int n = d.n, p = d.p;
    const TileRef<T> tile{s.psi, s.lam, s.E, n};
    // A thread adds its FP32 terms of a layer in FP64 (db, dg: of layer `cur` and of the one below);
    // a layer's block sum is taken once, when the sweep has left the layer.
    double db[2] = {0.0, 0.0}, dg[2] = {0.0, 0.0};
    int cur = p - 1;
    set_layer_consts<T>(s.lc, d.gamma, d.beta, p, n, true);
    Snake sn(p, 0, 1, 0, n, n, R);
    sn.to_last();
    bool first = true;
    for (;; sn.prev()) {
        const SubPass sp = sn.get();
        while (sp.lb < cur) {   // uniform: layer cur is complete
            const double v = block_sum4(db[0], dg[0], 0.0, 0.0, s.red);
            if (threadIdx.x == 0 && d.dbeta) d.dbeta[cur] = 2.0 * v;
            if (threadIdx.x == 1 && d.dgamma) d.dgamma[cur] = 2.0 * v;
            db[0] = db[1]; dg[0] = dg[1];
            db[1] = dg[1] = 0.0;
            --cur;
        }
        T acc[4] = {T(0), T(0), T(0), T(0)};
        subpass_adj<T, R>(tile, sp, s.lc, first, cur, acc);
        first = false;
        db[0] += (double)acc[0];
        db[1] += (double)acc[1];
        dg[0] += (double)acc[2];
        dg[1] += (double)acc[3];
        __syncthreads();
        if (sn.first()) break;
    }
    while (cur >= 0) {
        const double v = block_sum4(db[0], dg[0], 0.0, 0.0, s.red);
        if (threadIdx.x == 0 && d.dbeta) d.dbeta[cur] = 2.0 * v;
        if (threadIdx.x == 1 && d.dgamma) d.dgamma[cur] = 2.0 * v;
        db[0] = db[1]; dg[0] = dg[1];
        db[1] = dg[1] = 0.0;
        --cur;
    }
    __syncthreads();
}

// Forward register window of an n-qubit instance: rb, narrowed to rmax when asked for n - rmax <= 9
// (at n = 14 the 4-qubit window measured 12% slower), at most n.
__host__ __device__ inline int resident_window(int n, int rb, int rmax) {
    const int r = (rmax < rb && n - rmax <= 9) ? rmax : rb;
    return n < r ? n : r;
}

template <typename T, int R, int RA, bool GRAD>
__device__ void run_instance(const InstDesc<T>& d, unsigned char* sm, const WinSched& ws) {
    using C = typename Num<T>::C;
    const int n = d.n, p = d.p;
    const bool grad = GRAD && (d.flags & F_GRAD) != 0;
    size_t off[12];
    smem_layout<T>(n, p, grad, blockDim.x, off);
    Smem<T> s;
    s.psi = reinterpret_cast<C*>(sm + off[0]);
    s.lam = reinterpret_cast<C*>(sm + off[1]);
    s.E = reinterpret_cast<T*>(sm + off[2]);
    s.Q = reinterpret_cast<T*>(sm + off[3]);
    s.lc = reinterpret_cast<LayerConst<T>*>(sm + off[4]);
    s.red = reinterpret_cast<double*>(sm + off[5]);
    s.tk.wlists = reinterpret_cast<TopEnt*>(sm + off[7]);
    s.tk.cand = reinterpret_cast<TopEnt*>(sm + off[8]);
    s.tk.out = reinterpret_cast<TopEnt*>(sm + off[9]);
    s.tk.wb = reinterpret_cast<float*>(sm + off[10]);
    s.tk.cnt = reinterpret_cast<int*>(sm + off[10] + 16 * 32 * sizeof(float));
    s.escr = reinterpret_cast<T*>(sm + off[11]);
    const uint32_t D = 1u << n;

    static_assert(sizeof(FwdConst<T>) <= sizeof(LayerConst<T>), "the forward constants share the adjoint's place");
    using K = typename FwdFor<T, GRAD>::K;
    set_fwd_consts(reinterpret_cast<K*>(s.lc), d.gamma, d.beta, p, n);
    bool started = false;
    if (d.Q) {
        for (int i = threadIdx.x; i < n * n; i += blockDim.x) s.Q[i] = d.Q[i];
        __syncthreads();
        FusedInit<T> fi{nullptr, T(0), T(0), 0};
        if (!(d.flags & F_INIT_PSI)) {
            fi.psi = s.psi;
            fi.amp0 = (T)exp2(-0.5 * (double)n);
            fi.gpi0 = d.gamma[0] / T(3.14159265358979323846);
            if constexpr (GRAD && sizeof(T) == 4) {
                fi.two = true;
                make_phase(d.gamma[0], fi.ph);
            }
        }
        started = build_tile_energy_any<T>(n, n, 0u, s.Q, s.E, s.escr, fi);
    } else {
        for (uint32_t z = threadIdx.x; z < D; z += blockDim.x) s.E[swz<T>(z)] = d.E_in[z];
    }
    if (d.flags & F_INIT_PSI) {   // into the rotated frame: psi~ = i^{|z|} psi
        const C* pin = reinterpret_cast<const C*>(d.psi_in);
        for (uint32_t z = threadIdx.x; z < D; z += blockDim.x)
            s.psi[swz<T>(z)] = times_i_pow(pin[z], __popc(z));
    }
    __syncthreads();
    if (d.E_out)
        for (uint32_t z = threadIdx.x; z < D; z += blockDim.x) d.E_out[z] = s.E[swz<T>(z)];

    forward_run<T, R, K>(d, s, ws, started);

    if (d.psi_out) {              // back from the rotated frame: psi = (-i)^{|z|} psi~
        C* pout = reinterpret_cast<C*>(d.psi_out);
        for (uint32_t z = threadIdx.x; z < D; z += blockDim.x)
            pout[z] = times_i_pow(s.psi[swz<T>(z)], -__popc(z));
    }
    if constexpr (GRAD) {
        if (grad) adjoint_run<T, RA>(d, s);
    }
}

// WIDE: windows of RB (forward) and RB_ADJ (adjoint) qubits; else narrower ones (rmax, or fewer than RB
// qubits): the same number for both.
template <typename T, bool GRAD, bool WIDE>
__device__ __forceinline__ void dispatch_instance(const InstDesc<T>& d, unsigned char* sm, int rmax, const WinSched& ws) {
    constexpr int RBF = Num<T>::RB, RBA = Num<T>::RB_ADJ;
    if constexpr (WIDE) {
        run_instance<T, RBF, RBA, GRAD>(d, sm, ws);
    } else {
        const int rf = resident_window(d.n, RBF, rmax);
        if constexpr (RBA >= 4) {
            if (rf == 4) return run_instance<T, 4, 4, GRAD>(d, sm, ws);
        }
        if (rf == 3) run_instance<T, 3, 3, GRAD>(d, sm, ws);
        else if (rf == 2) run_instance<T, 2, 2, GRAD>(d, sm, ws);
        else run_instance<T, 1, 1, GRAD>(d, sm, ws);
    }
}

// Persistent walk over `count` descriptors (queue: device counter zeroed before the launch);
// with desc == nullptr the single instance `one` (passed by value) is run by block 0.
// GRAD: a kernel of its own with the adjoint sweep, and WIDE: one for windows of 5 (complex128: 4) qubits,
// so that launches do not carry the registers and code of the others: in one kernel with the narrower
// windows either the wide ones spilled (n = 13, 304 instances, p = 6: 74.3 us; 71.0 before the window starts
// became run-time values; 68.8 now) or, with the spills mended, the narrow ones slowed down (n = 11, 1000
// instances: 54.5 -> 56.9 us; 53.0 now). The launch picks by the size all its instances have.
template <typename T, bool GRAD, bool WIDE>
__global__ void __launch_bounds__(512) k_resident(const InstDesc<T>* __restrict__ desc, int count,
                                                  int* queue, const InstDesc<T> one, int rmax, const WinSched ws) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int s_next;
    if (desc == nullptr) {
        if (blockIdx.x == 0) dispatch_instance<T, GRAD, WIDE>(one, sm, rmax, ws);
        return;
    }
    for (;;) {
        if (threadIdx.x == 0) s_next = atomicAdd(queue, 1);
        __syncthreads();
        const int ii = s_next;
        __syncthreads();
        if (ii >= count) break;
        const InstDesc<T> d = desc[ii];
        dispatch_instance<T, GRAD, WIDE>(d, sm, rmax, ws);
        __syncthreads();
    }
}

int resident_r(bool dbl, int n, int rmax) { return resident_window(n, dbl ? Num<double>::RB : Num<float>::RB, rmax); }

// fn(kernel, descriptor of its type) for the kernel that serves n-qubit instances
template <typename T, typename Fn>
auto with_kernel(bool grad, bool wide, Fn&& fn) {
    if (grad) return wide ? fn(k_resident<T, true, true>, InstDesc<T>{}) : fn(k_resident<T, true, false>, InstDesc<T>{});
    return wide ? fn(k_resident<T, false, true>, InstDesc<T>{}) : fn(k_resident<T, false, false>, InstDesc<T>{});
}
template <typename Fn>
auto with_kernel(bool dbl, int n, bool grad, int rmax, Fn&& fn) {
    const int R = resident_r(dbl, n, rmax);
    return dbl ? with_kernel<double>(grad, R == Num<double>::RB, fn) : with_kernel<float>(grad, R == Num<float>::RB, fn);
}

}  // namespace

int resident_threads(bool dbl, int n, int rmax) {
    const int R = resident_r(dbl, n, rmax);
    const int g = (n > R) ? (1 << (n - R)) : 1;
    return g < 32 ? 32 : (g > 512 ? 512 : g);
}

size_t resident_smem_bytes(bool dbl, int n, int p, bool grad, int rmax) {
    size_t off[12];
    const int th = resident_threads(dbl, n, rmax);
    return dbl ? smem_layout<double>(n, p, grad, th, off) : smem_layout<float>(n, p, grad, th, off);
}

int resident_max_blocks_per_sm(bool dbl, int n, int pmax, bool grad, int rmax) {
    int nb = 0;
    const int th = resident_threads(dbl, n, rmax);
    const size_t sm = resident_smem_bytes(dbl, n, pmax, grad, rmax);
    // the occupancy query counts a block that needs more than 48 KB of dynamic shared memory only
    // once the kernel may use that much, so the limit is raised first (the launch sets it again)
    with_kernel(dbl, n, grad, rmax, [&](auto kern, auto) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, th, sm) != cudaSuccess)
            nb = 0;
        return nb;
    });
    return nb;
}

cudaError_t launch_resident(bool dbl, const void* desc, int count, int n, int pmax, bool grad,
                            int* queue, int grid, cudaStream_t st, const void* one, int rmax, bool block5) {
    const int th = resident_threads(dbl, n, rmax);
    const size_t sm = resident_smem_bytes(dbl, n, pmax, grad, rmax);
    const int R = resident_r(dbl, n, rmax);
    // the qubit order of blocks of the window itself, or of 5 qubits for narrower windows of a
    // single complex64 instance
    const WinSched ws = win_sched(n, block5 ? Num<float>::RB : R, R);
    return with_kernel(dbl, n, grad, rmax, [&](auto kern, auto inst) -> cudaError_t {
        using D = decltype(inst);
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        if (one) inst = *static_cast<const D*>(one);
        kern<<<grid, th, sm, st>>>(static_cast<const D*>(desc), count, queue, inst, rmax, ws);
        return cudaGetLastError();
    });
}

}  // namespace qaoa
