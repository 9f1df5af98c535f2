// Shared-memory staged axion-U(1) launches (u1_staged.cu).
#pragma once

#include "cl_internal.cuh"

namespace clk {

// what 0 = plaquette fields (and cos P into args cP when that is non-null), 1 = stage (or
// energies with P_ENERGY_ONLY), 2 = the fused stage (plaquette fields in shared memory, no
// plaquette launch), 3 = the E-dependent plaquette fields from a saved cos P (args cP).  Stage
// launches: u1_staged_blocks(.., false) blocks of 32 x 16 (FP32) or 32 x 8 (FP64) tiles, each
// marching through args dz planes; plaquette launches: u1_staged_blocks(.., true) blocks of tiles
// twice as tall through args pdz planes, their magnetic-energy partials in args pl_partials
// (pl_n of them, read by the stage).  Needs u1_staged_ok (2: N a multiple of 32).
bool u1_staged_ok(int precision, int N);
int u1_staged_blocks(int precision, int N, int dz, bool plaquettes);
// The library's z chunk: one block per SM at a time, waves x (planes + 2) minimised.
int u1_staged_dz(int precision, int N, int nsm, bool plaquettes);
cudaError_t launch_u1_staged(int precision, const void* args, int what, cudaStream_t s);

}  // namespace clk
