// Host helpers of the batched step shared by the ensemble and the server.
#pragma once

#include <vector>

#include "batch_kernels.cuh"
#include "internal.h"

namespace lbfd {

// Sites per work item: 2 when vx_max >= 2 and Lx is even, and for odd Lx in
// FP32 arithmetic but for D3Q19, whose twins measured slower than one site
// (32.3 against 36.0 GLUPS; the pairs' registers and scalar loads together).
inline int batch_vx(int lattice, int32_t Lx, int vx_max, int precision) {
  return vx_max >= 2 && (Lx % 2 == 0 || (precision != kStoreF64 && lattice != kD3Q19)) ? 2 : 1;
}

// A member of a batched launch (vx by batch_vx); the two population blocks start at value offsets off0 and off1 of
// the batch buffer; t0 is the batch clock value at which its t is 0.
BatchMember make_batch_member(int lattice, const int64_t dims[3], double tau, double rho_mean, uint64_t seed, uint32_t lattice_id,
                              int64_t off0, int64_t off1, uint64_t t0, int vx_max, int precision);

// Groups of at most kParamMembers consecutive members of about equal sites
// with their t-independent arguments, for the parameter-space launches (tile
// order 3), at least `parts` of them where there are as many members; tile0 of
// every member must be assigned.  Returns the number of groups.
int batch_build_params(const BatchMember *members, int n, int64_t ntiles, int noise_mode, int noise_dist, int parts,
                       std::vector<BatchParams> &groups);

// Parts of a set of members that step on streams of their own: while one's
// launch ends, the other's blocks take the SMs.  Measured on GB300, GLUPS with
// one part and two (three and four are no better): 60 D2Q9 members of 96..512
// a side 77.9 and 82.6, 4 of 300..500 71.4 and 76.9, 40 of 60..100 57.8 and
// 64.9, D3Q19 40 of 32..128 37.7 and 39.5, 8 of 30..60 31.2 and 36.1; but 20
// D2Q9 members of 30..80 (51000 sites) 24.6 and 24.2.  The server keeps one
// (24 mixed requests 59.5 and 59.0 ms: its types already overlap).
inline int batch_parts(int64_t sites) { return sites >= (int64_t(1) << 17) ? 2 : 1; }

// Tile passes for a launch of the members: at most `passes`, fewer where the
// tiles would not fill the GPU's `slots` resident blocks four times (a last
// wave that is nearly empty costs more than longer tiles save).
int batch_passes(const BatchMember *members, int n, int passes, int64_t slots);

// Assigns consecutive tiles of passes x 128 items to members[0..n) in order
// (tile0 and tile_start[m]); returns the number of tiles.
int64_t batch_assign_tiles(BatchMember *members, int n, int passes, int64_t *tile_start);

}  // namespace lbfd
