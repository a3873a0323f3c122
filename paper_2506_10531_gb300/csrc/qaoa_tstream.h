// qaoa_tstream.h -- internal interface of the TMA streaming passes (k_tstream.cu): the forward
// and adjoint passes of the HBM tier for complex64, with tiles moved by TMA.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "qaoa_stream.h"

namespace qaoa {

// Tile bits of the adjoint passes (the adjoint plan of stream_plan with stream_adj_tile_bits).
constexpr int TSA_TB = 12;

constexpr size_t TS_MAP_BYTES = 128;   // one CUtensorMap, 64-byte aligned

// The driver's tensor-map encoder could be found.
bool tstream_available();
size_t tstream_smem_bytes(bool tab);
// Encode the tensor maps of pass P (any pass of the same kind and chunk gives the same maps) for
// a state at psi and its energies at E (both 16-byte aligned; E NULL: none) into psi_map / e_map (host,
// 64-byte aligned).
bool tstream_encode_maps(const StreamPass& P, void* psi, void* E, void* psi_map, void* e_map);
// The maps of an instance, of the W windows of a layer (the contiguous one, then the chunks by start qubit):
// forward the W state maps, then the W energy maps; adjoint three per window (tstream_encode_adj_maps).
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
// three maps in a row (state psi, adjoint state lam, energies).
size_t tstream_adj_smem_bytes();
bool tstream_encode_adj_maps(const StreamPass& P, void* psi, void* lam, void* E, void* maps3);
cudaError_t launch_tstream_adj_pass(const TsGroup* groups, const TsSeg* segs, int nseg, uint32_t total, int grid,
                                    unsigned* status, cudaStream_t st);

}  // namespace qaoa
