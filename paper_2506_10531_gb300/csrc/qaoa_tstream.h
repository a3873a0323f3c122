// qaoa_tstream.h -- internal interface of the TMA streaming passes (k_tstream.cu): the forward
// and adjoint passes of the HBM tier for complex64, with tiles moved by TMA.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "qaoa_stream.h"

namespace qaoa {

// Shape of the tensor map of a pass (TMA coordinates of a tile): kind A; kind B with h <= 8 and
// qubits above the chunk (5-D) or without (4-D); kind B with h = 9, whose 512 high values are
// split over two box dimensions (at most 256 each), 5-D or 4-D.
enum : int { TS_A = 0, TS_B5 = 1, TS_B4 = 2, TS_B9_5 = 3, TS_B9_4 = 4, TS_A3 = 5 };   // TS_A3: kind A of
// the adjoint's 12-bit tiles, 3-D
// Tile bits of the adjoint passes (the adjoint plan of stream_plan with stream_adj_tile_bits).
constexpr int TSA_TB = 12;

struct TsPass {
    int bmode;          // TS_*
    int midbits;        // kind B: tile-index bits below the chunk (s - c)
    int map;            // index of this pass's state map among an instance's maps
    int emap;           // index of its energy map
    int maps_per_inst;  // maps per instance in the plan's map array
};

constexpr size_t TS_MAP_BYTES = 128;   // one CUtensorMap, 64-byte aligned

// The driver's tensor-map encoder could be found.
bool tstream_available();
size_t tstream_smem_bytes(bool tab);
TsPass tstream_pass_geometry(const StreamPass& P, int map, int emap, int maps_per_inst);
// Encode the tensor maps of pass P (any pass of the same kind and chunk gives the same maps) for
// a state at psi and its energies at E (both 16-byte aligned; E NULL: none) into psi_map / e_map (host,
// 64-byte aligned).
bool tstream_encode_maps(const StreamPass& P, void* psi, void* E, void* psi_map, void* e_map);
// A plan group's passes (forward or adjoint) for launches that hold passes of several groups: the
// numbers stream_plan made them from, from which the kernels form the pass they are at.
struct TsGroup {
    int n, p, k, tb, S;          // S: passes
    int W, cs[4], ch[4];         // windows of a layer: the contiguous one, then chunks [cs, cs + ch)
    int adjoint, keep_frame, no_store, maps_per_inst;
    const StreamInst<float>* insts;
    const void* maps;
};
// One group's pass in a launch: its tiles are [tile0, the next segment's tile0).
struct TsSeg {
    uint32_t tile0;
    uint16_t group, pass;
};
constexpr int TS_MAX_GROUPS = 65535;
// Fill the windows of g (n, tb set) from its pass list.
void tstream_group_windows(const StreamPass* passes, int S, TsGroup* g);
// A launch over `nseg` segments (device array, `total` tiles in all) of the groups at `groups`, whose
// phases come from Q (tab) or from the energies in HBM; runs (with tab): each CTA takes tiles in a row
// instead of every grid-th; a bounded wait that ran out sets bit 0 of *status.
cudaError_t launch_tstream_pass(bool tab, const TsGroup* groups, const TsSeg* segs, int nseg, uint32_t total, int grid,
                                bool runs, unsigned* status, cudaStream_t st);

// Adjoint passes (tiles of TSA_TB bits, kind-B chunks of h <= 8 high qubits): per pass shape
// three maps (state psi, adjoint state lam, energies) at indices T.map, T.map + 1, T.map + 2.
size_t tstream_adj_smem_bytes();
TsPass tstream_adj_geometry(const StreamPass& P, int map, int maps_per_inst);
bool tstream_encode_adj_maps(const StreamPass& P, void* psi, void* lam, void* E, void* maps3);
cudaError_t launch_tstream_adj_pass(const TsGroup* groups, const TsSeg* segs, int nseg, uint32_t total, int grid,
                                    unsigned* status, cudaStream_t st);

}  // namespace qaoa
