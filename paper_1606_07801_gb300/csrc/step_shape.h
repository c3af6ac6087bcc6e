// Launch shape of the one-launch-per-step register-pull kernels (k_step,
// k_step_vec): sites per thread and the block/grid over the lattice.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdlib>

#include "device.cuh"

namespace lbfd {

// Values per vector access at most (4, 2 or 1) that the addresses of a
// lattice's two buffers allow: a vector lies on a multiple of its size, and
// with Lx a multiple of the vector every row and population starts as the
// buffer does.
inline int vec_most(const void *a, const void *b, int value_bytes) {
  const uintptr_t at = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b);
  const uintptr_t bytes = static_cast<uintptr_t>(value_bytes);
  return at % (4 * bytes) == 0 ? 4 : (at % (2 * bytes) == 0 ? 2 : 1);
}

// Sites per thread of the register-pull step kernel (k_step_vec; 1 is
// k_step), where Lx allows: several share the address and load instructions,
// but are updated one after the other, which a lattice of few warps per SM
// pays in full.  Measured on GB300, microseconds per step:
//   4 (16-byte loads and stores of FP32) for all but D3Q19 in FP32 from 2^19
//     sites: D1Q3 FP32 2^24 63.9 against 68.2 with two (10^5 sites 2.7 against
//     2.0), D3Q19 FP16 128^3 47.8 against 50.3 with two, 256^3 367 against 401,
//     but 64^3 13.4 against 6.3; D2Q9 FP16 1024^2 12.1 against 12.9, but D2Q9
//     FP32 320^2 6.0 against 3.3.  D3Q19 in FP32 needs too many registers for
//     four (256^3 477 against 392).  D2Q5, whose sites are short, takes four
//     from the start (moment-space 400^2 2.9 against 3.4, 2048^2 26.2 against
//     27.2).
//   2 otherwise, but 1 for the smallest: D2Q9 200^2 2.8 against 3.7 with two,
//     D3Q19 24^3 3.1 against 6.7, 32^3 6.3 against 6.8.  The line was drawn
//     with k_step_vec; two sites in k_step_ahead take 2.0 and 2.1 at these two
//     sizes, so that it lies too high for the lattices that kernel steps.
//   1 in FP64, whose narrow pipe hides the extra instructions: D2Q9 512 x 384
//     47.0 against 50.3 with two, 60 x 50 6.1 against 10.3.
// A tuning knob only; results do not depend on it.  LBFD_STEP_VX = 1, 2 or 4
// overrides the choice where Lx allows.  At most `most` sites (vec_most of the
// buffers).
inline int step_vec_width(int lattice, int precision, int32_t Lx, int64_t sites = INT64_MAX, int most = 4) {
  static int forced = [] {
    const char *e = getenv("LBFD_STEP_VX");
    const int r = e ? atoi(e) : 0;
    return (r == 1 || r == 2 || r == 4) ? r : 0;
  }();
  int vx = forced;
  if (vx == 0) {
    const int64_t few = lattice != kD3Q19 ? 48 << 10 : (precision == kStoreF32 ? 40 << 10 : 24 << 10);
    const bool four = lattice != kD3Q19 || precision != kStoreF32;
    vx = precision == kStoreF64 || sites <= few ? 1 : (lattice == kD2Q5 || (four && sites >= (1 << 19)) ? 4 : 2);
  }
  if (vx == 4 && precision == kStoreF64) vx = 2;
  while (vx > most || Lx % vx != 0) vx /= 2;
  return vx;
}

// Threads of a block of the one-launch-per-step kernels.  FP64: one warp, so
// that the blocks spread evenly over the SMs' narrow FP64 pipes (D2Q9 60 x 50:
// 18.8 us with 256 threads and two sites each, 6.1 with 32 and one; D3Q19
// 64^3 168.8 and 147.4).  FP32 arithmetic: 128 for the lattices whose
// registers fill the SM, a finer last wave at the same occupancy (D3Q19 FP32
// 64^3 9.3 -> 8.3 us, 128^3 54.5 -> 53.6, FP16 128^3 51.3 -> 49.1), but 256
// where they do not (`few`): without noise (D2Q9 FP32 623 x 1187 7.1 against
// 7.6, D3Q19 FP32 50^3 3.9 against 4.2), but for D3Q19 in a 16-bit format
// (100^3 11.4 against 9.8 with 128).
inline int step_threads(int lattice, int precision, bool few = false) {
  return precision == kStoreF64 ? 32 : (lattice == kD1Q3 || few ? 256 : 128);
}

// Block and grid of the one-launch-per-step kernels for vx sites per thread:
// blocks of `threads` threads, x fastest (at least one warp along x), one grid plane
// per z.
inline void step_shape(int32_t Lx, int32_t Ly, int32_t Lz, dim3 &grid, dim3 &block, int vx = 1, int threads = 256) {
  const int cols = Lx / vx;
  int bx = threads;
  while (bx > 32 && bx / 2 >= cols) bx /= 2;
  int by = threads / bx;
  while (by > 1 && by / 2 >= Ly) by /= 2;
  block = dim3(bx, by, 1);
  grid = dim3((cols + bx - 1) / bx, (Ly + by - 1) / by, Lz);
}

}  // namespace lbfd
