// Internal interfaces of the tensor-core path (shared by pf_tc.cu and pf_tc_flow.cu).
#pragma once

#include <cuda.h>

#include "pf_common.cuh"

namespace pf {

struct TcGeo {
    int L, d_k, d_v, r, C, n, NC;          // NC = chunks per sequence
    int rm;                                // strict-mask group size (Problem::mask_group)
    const float* b32;                      // null, or fp32 step sizes used in place of beta (Problem::beta32)
    uint32_t e_bytes, q_bytes, xi_bytes;   // per-chunk workspace record sizes
};

struct TcWs {
    int* err;       // device status word: 0, or the code of the first bounded wait that expired
    uint8_t* E;     // [G][e_bytes]
    uint8_t* Qt;    // [G][q_bytes]
    uint8_t* Xi;    // [G][xi_bytes]
};

// Tensor map of a bf16 tensor [seqs][rows][cols], zero fill out of bounds (pf_tc.cu).  The columns are seen as slabs of
// slab_cols (64 or 32: the swizzle spans a slab's row), so that one copy brings box_slabs slabs of box_rows rows, one slab
// after another: coordinates (column within the slab, row, slab, sequence).
bool make_slab_map(CUtensorMap* m, const void* base, uint64_t seqs, uint64_t rows, uint64_t cols, uint32_t slab_cols, uint32_t box_rows,
                   uint32_t box_slabs);
// The same as a three-dimensional map with boxes of 64 columns x box_rows rows: coordinates (column, row, sequence).
bool make_tile_map(CUtensorMap* m, const void* base, uint64_t seqs, uint64_t rows, uint64_t cols, uint32_t box_rows);

TcGeo tc_geo(const Problem& p);
size_t tc_ws_carve(const Problem& p, void* base, TcWs* out);

// pf_tc_flow.cu
bool tc_flow_available();
int tc_flow_launch(const Problem& p, const TcWs& ws, int dvs);

// pf_tc.cu
int tc_scan_launch(const Problem& p, const TcWs& ws);
int tc_forward_refflow(const Problem& p, void* workspace);
size_t tc_refflow_workspace_bytes(const Problem& p);

// pf_fused.cu: flow builders and state scan in one cooperative launch
bool fused_supported(const Problem& p);
double fused_estimate_us(const Problem& p);
size_t fused_workspace_bytes(const Problem& p);
int fused_forward(const Problem& p, void* workspace);

// pf_simt.cu: runs the gram/solve/wu kernels only and returns where W, Uh and P were left.
int simt_prepare(const Problem& p, void* workspace, float** W, float** U, float** P);

}  // namespace pf
