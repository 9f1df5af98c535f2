// Shared-memory staged axion-U(1) launches (u1_staged.cu).
#pragma once

#include "cl_internal.cuh"

namespace clk {

// what 0 = plaquette fields (and cos P into args cP when that is non-null), 1 = stage (or
// energies with P_ENERGY_ONLY), 2 = the fused stage (plaquette fields in shared memory, no
// plaquette launch), 3 = the E-dependent plaquette fields from a saved cos P (args cP).  Stage
// launches: blocks of args tx x ty tiles (at most 512 sites in FP32, 256 in FP64), each marching
// through args dz planes; plaquette launches: blocks of args ptx x pty tiles (at most twice the
// sites) through args pdz planes, their magnetic-energy partials in args pl_partials (pl_n of
// them, read by the stage).  Needs u1_staged_ok (2: N a multiple of 32).
bool u1_staged_ok(int precision, int N);
struct U1Tile {
    int tx, ty, dz;  // sites of a tile in x and y, planes of a z chunk
};
int u1_staged_blocks(const U1Tile& t, int N);
// The library's tile for the stage or the plaquette launches (fixed: 32 columns, the fused form's).
U1Tile u1_staged_tile(int precision, int N, int nsm, bool plaquettes, bool fixed);
cudaError_t launch_u1_staged(int precision, const void* args, int what, cudaStream_t s);

}  // namespace clk
