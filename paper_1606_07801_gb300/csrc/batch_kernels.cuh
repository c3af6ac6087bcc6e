// Batched step: many independent lattices of one lattice type, each with its
// own size, relaxation time, mean density, seed, Philox lattice id and step
// counter, advanced by one launch per time step.  Used by the ensemble
// (members that start together) and by the server (members admitted at
// different times).
//
// Memory.  All members live in one device buffer `base`; member m keeps its
// two population blocks at value offsets off[0] and off[1].  Its own step
// counter is t = clock - t0, where clock counts the launches of the batch;
// the stored state is in block t & 1 and the step writes block (t & 1) ^ 1.
//
// Work.  Member m owns tiles [tile_start[m], tile_start[m + 1]) of a flat
// tile list; a tile is `passes` x 128 consecutive work items of one member,
// and an item is vx sites of a row: neighbours where Lx is even, a site of the
// row's first half and its twin in the second where it is odd (twin_update;
// D3Q19 takes one site there).
// Every item runs the per-site code of the single-lattice kernels, so a member
// evolves bit-identically to the same lattice stepped alone.  The step arguments
// (relaxation constants and the Philox words of the member's t) are written
// once per launch and member by k_batch_prep.  Three kernels take the tiles:
//   k_batch_tile   one block per tile; warp 0 finds the member by a 32-way
//                  search of tile_start and copies its arguments to shared
//                  memory;
//   k_batch_param  one block per tile, one launch per group of up to
//                  kParamMembers members whose t-independent arguments are a
//                  kernel parameter (uniform operands, fewer registers); the
//                  t words are formed in the block, without k_batch_prep;
//   k_batch_step   a persistent grid whose blocks take every grid-th tile or
//                  one run of consecutive tiles, reloading the arguments when
//                  the member changes.
#pragma once

#include "fastdiv.cuh"
#include "step_kernels.cuh"

namespace lbfd {

// Threads of a block: small blocks end a launch more evenly.  128 against 256
// in the parameter-space launches on GB300, GLUPS: 60 D2Q9 members of 96..512
// a side 78.5 and 75.7 (FP16 78.1 and 76.8), 20 of 30..80 24.8 and 21.1, 40
// D3Q19 members of 32..128 38.5 and 37.8, 8 of 30..60 32.0 and 30.2 (with a
// noise transform of fewer operations; 37.7 and 31.2 with the present one), 600
// D2Q9 members 83.7 and 83.2.  In the other orders, default plan, against
// blocks of 256 and the kernels of the time: 60 D2Q9 62.9 and 60.1, 40 D3Q19
// 36.1 and 33.5, 60 lines 66.3 and 62.3, 20 FP64 D2Q9 members 3.3 and 0.7.
constexpr int kBatchThreads = 128;
// Order in which blocks take tiles: a persistent grid whose blocks take every
// grid-th tile (strided) or one run of consecutive tiles (contiguous), one
// block per tile, or one block per tile with the members' arguments in the
// kernel parameters (one launch per group of members).
constexpr int kWalkStrided = 0, kWalkContiguous = 1, kWalkPerTile = 2, kWalkParam = 3;

// One member, as the host builds it (constant while the member is listed).
struct BatchMember {
  int32_t Lx, Ly, Lz, vx;  // vx: sites per work item, 1 or 2 (batch_vx)
  int64_t N;               // sites
  int64_t off[2];          // first value of population block 0 / 1 in the batch buffer
  int64_t tile0;           // first tile of the member in the launch's tile list
  uint64_t t0;             // clock value at which the member's own step counter is 0
  uint64_t seed;
  uint32_t lattice_id, pad;
  double tau, rho_mean;
};

// What one launch needs of one member (written by k_batch_prep).
struct alignas(16) BatchStep {
  StepArgs a;          // sizes, relaxation and noise constants, Philox words of this step
  int64_t src, dst;    // value offsets of the blocks read and written
  int64_t tile0;
  int32_t items, cols; // work items and items per row
  int32_t vx, pad;
  FastDiv div_cols, div_Ly;  // division by cols and by Ly
};
static_assert(sizeof(BatchStep) % 16 == 0, "BatchStep is copied as int4 words");

// What one launch needs of member mb at clock value `now` (its own step
// counter is now - t0).  Host and device share it, so the arguments a launch
// takes from kernel parameters and the ones k_batch_prep writes agree bit for
// bit.
__host__ __device__ inline BatchStep batch_step_of(const BatchMember &mb, uint64_t now, int noise_mode,
                                                   int noise_dist) {
  BatchStep s{};
  s.a.Lx = mb.Lx;
  s.a.Ly = mb.Ly;
  s.a.Lz = mb.Lz;
  s.a.N = mb.N;
  fill_step_params(s.a, mb.tau, mb.rho_mean);
  s.a.noise_mode = noise_mode;
  s.a.noise_dist = noise_dist;
  const uint64_t t = now - mb.t0;  // the member's own step counter
  s.a.ph = make_philox_step(mb.seed, mb.lattice_id, t);
  const int p = static_cast<int>(t & 1);
  s.src = mb.off[p];
  s.dst = mb.off[p ^ 1];
  s.tile0 = mb.tile0;
  s.vx = mb.vx;
  s.cols = (mb.Lx + mb.vx - 1) / mb.vx;
  s.items = static_cast<int32_t>(static_cast<int64_t>(s.cols) * mb.Ly * mb.Lz);
  s.div_cols = make_fastdiv(static_cast<uint32_t>(s.cols));
  s.div_Ly = make_fastdiv(static_cast<uint32_t>(mb.Ly));
  return s;
}

// Step arguments of every member for the clock value *clock_dev (or `clock`
// when clock_dev is null).
__global__ void k_batch_prep(const BatchMember *__restrict__ members, int n, const uint64_t *__restrict__ clock_dev,
                             uint64_t clock, int noise_mode, int noise_dist, BatchStep *__restrict__ out);

// Index m with tile_start[m] <= tile < tile_start[m + 1] (tile_start strictly
// increasing, tile_start[0] = 0 <= tile), found by warp 0: each round tests
// 32 evenly spaced splitters and keeps the segment of the last one passed.
__device__ __forceinline__ int batch_find_member(const int64_t *__restrict__ tile_start, int n, int64_t tile) {
  const int lane = threadIdx.x & 31;
  int lo = 0, len = n;
  while (len > 1) {
    const int stride = (len + 31) >> 5;
    const int idx = lo + lane * stride;
    const bool pass = idx < lo + len && __ldg(tile_start + idx) <= tile;
    const unsigned b = __ballot_sync(0xffffffffu, pass);
    const int k = 31 - __clz(b);
    const int nlo = lo + k * stride;
    len = min(stride, lo + len - nlo);
    lo = nlo;
  }
  return lo;
}

// Minimum resident blocks per SM asked of the register allocator: occupancy
// variant 0 is 8 blocks (64 registers; D3Q19 with its arguments in shared
// memory, which the compiler cannot keep as uniform operands, 6; FP64 4),
// variant 1 two blocks fewer; the tuner picks between them.
template <int LAT, typename S, int OCC, bool PARAM>
constexpr int batch_min_blocks() {
  return (sizeof(typename Store<S>::R) != 4 ? 4 : (LAT == kD3Q19 && !PARAM ? 6 : 8)) - 2 * OCC;
}

// The collision of pairs without the packed form (FP64, no noise): one site
// at a time.
template <int LAT, typename S, int NOISE>
struct BatchCollide : SrtCollideFor<LAT, S, NOISE> {
  static constexpr bool kPairs = false;
};

// Shared memory of the pair items' noise (NoiseColumn) of one block.
template <int LAT, typename S, int NOISE, int VXMAX>
__host__ __device__ constexpr int batch_column() {
  return VXMAX == 2 && NOISE != kStepNoiseOff && sizeof(typename Store<S>::R) == 4
             ? SrtCollideFor<LAT, S, NOISE>::kAhead * kBatchThreads
             : 1;
}

// The work items of one tile of member b (rel: the tile's index within the
// member).  VXMAX = 1: every member takes one site per item (the two-site
// path is not compiled in).  A pair of sites is updated at once on the packed
// FP32 instructions with its noise parked in `column`, in FP64 and without
// noise one site at a time.  Measured on GB300 in the parameter-space
// launches, against one site at a time from registers with the arguments
// prepared by a launch of its own (blocks of 256 threads, one launch a step; for
// the present figures see kBatchThreads and batch_parts): 60 D2Q9 members of
// 96..512 a side 62.8 -> 80.0 GLUPS with even rows, 59.4 -> 73.3 odd; 40 D3Q19
// members of 32..128 a side 36.9 -> 42.1 even, 33.4 -> 36.0 odd (with a noise
// transform of fewer operations).  In two parts now: D2Q9 88.3 with even rows,
// 82.6 as they are, D3Q19 42.3 and 39.5.
// ready() is called before an item's first load.
template <int LAT, typename S, int NOISE, int VXMAX, class F>
__device__ __forceinline__ void batch_tile_items(S *base, const BatchStep &b, int rel, int passes, float2 *column,
                                                 F &&ready) {
  using C = SrtCollideFor<LAT, S, NOISE>;
  constexpr bool kPacked = NOISE != kStepNoiseOff && sizeof(typename Store<S>::R) == 4;
  const C collide;
  const S *src = base + b.src;
  S *dst = base + b.dst;
  const int first = rel * passes * kBatchThreads + threadIdx.x;
  for (int p = 0; p < passes; ++p) {
    const int item = first + p * kBatchThreads;
    if (item < b.items) {
      const int row = static_cast<int>(fastdiv(static_cast<uint32_t>(item), b.div_cols));
      const int col = item - row * b.cols;
      const int z = static_cast<int>(fastdiv(static_cast<uint32_t>(row), b.div_Ly));
      const int y = row - z * b.a.Ly;
      // a member's value offsets fit 32 bits (checked when it is listed)
      if (VXMAX == 2 && b.vx == 2) {
        if constexpr (kPacked) {
          const NoiseColumn<C::kAhead, kBatchThreads> nc(column, static_cast<int>(threadIdx.x));
          if (LAT != kD3Q19 && (b.a.Lx & 1)) {  // (D3Q19: batch_vx)
            twin_update<LAT, S, uint32_t>(src, dst, b.a, col, y, z, collide, nc, ready);
          } else {
            float2 t[C::kAhead];
            collide.ahead(t, site_index(b.a, 2 * col, y, z), b.a.ph);
#pragma unroll
            for (int k = 0; k < C::kAhead; ++k) nc.put(k, t[k]);
            ready();
            float f[2][Lattice<LAT>::Q];
            const uint32_t at = vec_pull<LAT, S, 2, uint32_t>(src, b.a, 2 * col, y, z, f);
            collide_parked(collide, f[0], f[1], nc, 0, b.a);
            vec_store<LAT, S, 2, uint32_t>(dst, b.a, at, 2 * col, f);
          }
        } else if (b.a.Lx & 1) {
          ready();
          const int apart = b.cols;
          step_scalar_body<LAT, S, NOISE, C, uint32_t>(src, dst, b.a, col, y, z);
          if (col + apart < b.a.Lx) step_scalar_body<LAT, S, NOISE, C, uint32_t>(src, dst, b.a, col + apart, y, z);
        } else {
          ready();
          step_vec_body<LAT, S, 2, NOISE, BatchCollide<LAT, S, NOISE>, uint32_t>(src, dst, b.a, col * 2, y, z);
        }
      } else {
        using R = typename Store<S>::R;
        R t[C::kAhead];
        collide.ahead(t, site_index(b.a, col, y, z), b.a.ph);
        ready();
        R f[Lattice<LAT>::Q];
        const uint32_t s = scalar_pull<LAT, S, uint32_t>(src, b.a, col, y, z, f);
        collide.given(f, [&](int k) -> R { return t[k]; }, b.a);
        scalar_store<LAT, S, uint32_t>(dst, b.a, s, f);
      }
    }
  }
}

// Warp 0 finds the member of `tile`, copies its arguments to *sb and its
// first tile to *lo (and the end of its tiles to *hi when hi is not null).
__device__ __forceinline__ void batch_load_member(const BatchStep *__restrict__ steps,
                                                  const int64_t *__restrict__ tile_start, int nmembers, int ntiles,
                                                  int tile, BatchStep *sb, int *lo, int *hi) {
  if (threadIdx.x < 32) {
    const int m = batch_find_member(tile_start, nmembers, tile);
    const int4 *g = reinterpret_cast<const int4 *>(steps + m);
    int4 *s = reinterpret_cast<int4 *>(sb);
    for (int k = threadIdx.x; k < int(sizeof(BatchStep) / 16); k += 32) s[k] = g[k];
    if (threadIdx.x == 0) {
      *lo = static_cast<int>(__ldg(tile_start + m));
      if (hi) *hi = m + 1 < nmembers ? static_cast<int>(__ldg(tile_start + m + 1)) : ntiles;
    }
  }
}

// Persistent grid: the tiles of this block are every gridDim.x-th tile from
// blockIdx.x (strided walk) or one run of consecutive tiles (contiguous
// walk), in which the member changes only where the run crosses a member
// boundary.
template <int LAT, typename S, int NOISE, int OCC, int VXMAX>
__global__ void __launch_bounds__(kBatchThreads, batch_min_blocks<LAT, S, OCC, false>())
    k_batch_step(S *__restrict__ base, const BatchStep *__restrict__ steps, const int64_t *__restrict__ tile_start,
                 int nmembers, int ntiles, int passes, int walk) {
  int tile, stop, stride;
  if (walk == kWalkContiguous) {
    tile = static_cast<int>(int64_t(blockIdx.x) * ntiles / gridDim.x);
    stop = static_cast<int>(int64_t(blockIdx.x + 1) * ntiles / gridDim.x);
    stride = 1;
  } else {
    tile = blockIdx.x;
    stop = ntiles;
    stride = gridDim.x;
  }
  // two copies of the member's arguments and tile range: the copy for the
  // next member is written while no thread reads the copy before the current
  // one any more (one barrier per change of member)
  __shared__ BatchStep sb[2];
  __shared__ int srange[2][2];
  __shared__ float2 column[batch_column<LAT, S, NOISE, VXMAX>()];
  int buf = 1, lo = 0, hi = 0;
  for (; tile < stop; tile += stride) {
    if (tile < lo || tile >= hi) {
      buf ^= 1;
      batch_load_member(steps, tile_start, nmembers, ntiles, tile, &sb[buf], &srange[buf][0], &srange[buf][1]);
      __syncthreads();
      lo = srange[buf][0];
      hi = srange[buf][1];
    }
    batch_tile_items<LAT, S, NOISE, VXMAX>(base, sb[buf], tile - lo, passes, column, [] {});
  }
}

// One tile per block (grid = number of tiles): no loop state is carried
// across tiles, which leaves the per-site code the registers it has in the
// single-lattice kernels.
template <int LAT, typename S, int NOISE, int OCC, int VXMAX>
__global__ void __launch_bounds__(kBatchThreads, batch_min_blocks<LAT, S, OCC, false>())
    k_batch_tile(S *__restrict__ base, const BatchStep *__restrict__ steps, const int64_t *__restrict__ tile_start,
                 int nmembers, int ntiles, int passes) {
  __shared__ BatchStep sb;
  __shared__ int lo;
  __shared__ float2 column[batch_column<LAT, S, NOISE, VXMAX>()];
  batch_load_member(steps, tile_start, nmembers, ntiles, static_cast<int>(blockIdx.x), &sb, &lo, nullptr);
  __syncthreads();
  batch_tile_items<LAT, S, NOISE, VXMAX>(base, sb, static_cast<int>(blockIdx.x) - lo, passes, column, [] {});
}

// Members of one parameter-space launch (tile order LBFD_WALK_PARAM): the
// t-independent arguments of at most kParamMembers consecutive members travel
// as a kernel parameter (30.9 KB of the 32 KB parameter space), so the
// per-site code reads them as uniform operands, as the single-lattice kernels
// read theirs.  The Philox words of the member's t and the parity of its
// blocks are formed by every block from the clock (a dozen instructions per
// thread and tile), so nothing has to be prepared between two steps of a
// group: its launches follow each other as dependent launches.
constexpr int kParamMembers = 112;
struct BatchParams {
  int32_t n, first;                      // members first .. first + n - 1 of the batch
  int32_t tile_start[kParamMembers + 1];  // first tile of each, relative to the launch; [n] = tiles
  BatchStep mem[kParamMembers];          // arguments at t = 0; a.ph.e[0..1] hold t0 and a.ph.f the lattice id
};
static_assert(sizeof(BatchParams) + 64 <= 32764, "kernel parameters are limited to 32764 bytes");

// clock: the batch clock of this step is *clock_dev (0 where null) + clock.
template <int LAT, typename S, int NOISE, int OCC, int VXMAX>
__global__ void __launch_bounds__(kBatchThreads, batch_min_blocks<LAT, S, OCC, true>())
    k_batch_param(S *base, const __grid_constant__ BatchParams p, const uint64_t *clock_dev, uint64_t clock,
                  int passes) {
  __shared__ float2 column[batch_column<LAT, S, NOISE, VXMAX>()];
  pdl_launch_dependents();
  const int tile = static_cast<int>(blockIdx.x);
  // the member of this block: a search of uniform (parameter) words
  int lo = 0, hi = p.n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (p.tile_start[mid] <= tile)
      lo = mid;
    else
      hi = mid;
  }
  // (the clock does not change while launches that read it may run)
  BatchStep b = p.mem[lo];
  const uint64_t t0 = static_cast<uint64_t>(b.a.ph.e[1]) << 32 | b.a.ph.e[0];
  const uint64_t t = (clock_dev ? *clock_dev : 0) + clock - t0;  // the member's own step counter
  philox_step_set_t(b.a.ph, b.a.ph.f, t);
  if (t & 1) {
    const int64_t src = b.src;
    b.src = b.dst;
    b.dst = src;
  }
  batch_tile_items<LAT, S, NOISE, VXMAX>(base, b, tile - p.tile_start[lo], passes, column, [] { pdl_wait(); });
}

// When a launch happens: batch clock, and whether it may start before the
// previous launch of its stream has ended (its blocks wait for it).
struct BatchWhen {
  const uint64_t *clock_dev;
  uint64_t clock;
  bool dependent;
};

template <int LAT, typename S, int NOISE, int OCC, int VXMAX>
cudaError_t batch_param_k(S *b, const BatchParams *groups, int ngroups, const BatchWhen &when, int passes,
                          cudaStream_t stream) {
  for (int g = 0; g < ngroups; ++g) {
    const int tiles = groups[g].tile_start[groups[g].n];
    if (tiles <= 0) continue;
    StepLaunch launch(dim3(tiles), dim3(kBatchThreads), stream);
    if (!when.dependent) launch.cfg.numAttrs = 0;
    const cudaError_t e = cudaLaunchKernelEx(&launch.cfg, k_batch_param<LAT, S, NOISE, OCC, VXMAX>, b, groups[g],
                                             when.clock_dev, when.clock, passes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int LAT, typename S, int OCC, int VXMAX>
cudaError_t batch_param_occ(S *b, const BatchParams *groups, int ngroups, const BatchWhen &when, int passes,
                            int noise_mode, int noise_dist, cudaStream_t stream) {
  if (noise_mode == kNoiseOff)
    return batch_param_k<LAT, S, kStepNoiseOff, OCC, VXMAX>(b, groups, ngroups, when, passes, stream);
  if (noise_dist == kGaussian)
    return batch_param_k<LAT, S, kStepNoiseGauss, OCC, VXMAX>(b, groups, ngroups, when, passes, stream);
  return batch_param_k<LAT, S, kStepNoiseFlat, OCC, VXMAX>(b, groups, ngroups, when, passes, stream);
}

// One launch per group of at most kParamMembers members.
template <int LAT, typename S>
cudaError_t batch_param_t(void *base, const BatchParams *groups, int ngroups, const BatchWhen &when, int passes,
                          int occ, int vx_max, int noise_mode, int noise_dist, cudaStream_t stream) {
  S *b = static_cast<S *>(base);
  if (vx_max == 1)
    return occ == 1 ? batch_param_occ<LAT, S, 1, 1>(b, groups, ngroups, when, passes, noise_mode, noise_dist, stream)
                    : batch_param_occ<LAT, S, 0, 1>(b, groups, ngroups, when, passes, noise_mode, noise_dist, stream);
  return occ == 1 ? batch_param_occ<LAT, S, 1, 2>(b, groups, ngroups, when, passes, noise_mode, noise_dist, stream)
                  : batch_param_occ<LAT, S, 0, 2>(b, groups, ngroups, when, passes, noise_mode, noise_dist, stream);
}

template <int LAT, typename S, int NOISE, int OCC, int VXMAX>
cudaError_t batch_step_k(S *b, const BatchStep *steps, const int64_t *tile_start, int nmembers, int ntiles, int passes,
                         int walk, int grid, cudaStream_t stream) {
  if (walk == kWalkPerTile)
    k_batch_tile<LAT, S, NOISE, OCC, VXMAX><<<ntiles, kBatchThreads, 0, stream>>>(b, steps, tile_start, nmembers,
                                                                                  ntiles, passes);
  else
    k_batch_step<LAT, S, NOISE, OCC, VXMAX><<<grid, kBatchThreads, 0, stream>>>(b, steps, tile_start, nmembers, ntiles,
                                                                                passes, walk);
  return cudaGetLastError();
}

template <int LAT, typename S, int OCC, int VXMAX>
cudaError_t batch_step_occ(S *b, const BatchStep *steps, const int64_t *tile_start, int nmembers, int ntiles,
                           int passes, int walk, int noise_mode, int noise_dist, int grid, cudaStream_t stream) {
  if (noise_mode == kNoiseOff)
    return batch_step_k<LAT, S, kStepNoiseOff, OCC, VXMAX>(b, steps, tile_start, nmembers, ntiles, passes, walk, grid,
                                                           stream);
  if (noise_dist == kGaussian)
    return batch_step_k<LAT, S, kStepNoiseGauss, OCC, VXMAX>(b, steps, tile_start, nmembers, ntiles, passes, walk, grid,
                                                             stream);
  return batch_step_k<LAT, S, kStepNoiseFlat, OCC, VXMAX>(b, steps, tile_start, nmembers, ntiles, passes, walk, grid,
                                                          stream);
}

// vx_max: the largest sites per item of any member (1 or 2).
template <int LAT, typename S>
cudaError_t batch_step_t(void *base, const BatchStep *steps, const int64_t *tile_start, int nmembers, int64_t ntiles,
                         int passes, int occ, int walk, int vx_max, int noise_mode, int noise_dist, int grid,
                         cudaStream_t stream) {
  S *b = static_cast<S *>(base);
  if (ntiles >= (int64_t(1) << 31)) return cudaErrorInvalidValue;
  const int nt = static_cast<int>(ntiles);
  if (vx_max == 1) {
    if (occ == 1)
      return batch_step_occ<LAT, S, 1, 1>(b, steps, tile_start, nmembers, nt, passes, walk, noise_mode, noise_dist,
                                          grid, stream);
    return batch_step_occ<LAT, S, 0, 1>(b, steps, tile_start, nmembers, nt, passes, walk, noise_mode, noise_dist, grid,
                                        stream);
  }
  if (occ == 1)
    return batch_step_occ<LAT, S, 1, 2>(b, steps, tile_start, nmembers, nt, passes, walk, noise_mode, noise_dist, grid,
                                        stream);
  return batch_step_occ<LAT, S, 0, 2>(b, steps, tile_start, nmembers, nt, passes, walk, noise_mode, noise_dist, grid,
                                      stream);
}

template <int LAT, typename S, int NOISE, int OCC, int VXMAX>
int batch_blocks_k(int walk) {
  int nb = 0;
  cudaError_t e;
  if (walk == kWalkParam)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch_param<LAT, S, NOISE, OCC, VXMAX>, kBatchThreads, 0);
  else if (walk == kWalkPerTile)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch_tile<LAT, S, NOISE, OCC, VXMAX>, kBatchThreads, 0);
  else
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch_step<LAT, S, NOISE, OCC, VXMAX>, kBatchThreads, 0);
  return e == cudaSuccess && nb > 0 ? nb : 1;
}

template <int LAT, typename S, int OCC, int VXMAX>
int batch_blocks_occ(int walk, int noise_mode, int noise_dist) {
  if (noise_mode == kNoiseOff) return batch_blocks_k<LAT, S, kStepNoiseOff, OCC, VXMAX>(walk);
  if (noise_dist == kGaussian) return batch_blocks_k<LAT, S, kStepNoiseGauss, OCC, VXMAX>(walk);
  return batch_blocks_k<LAT, S, kStepNoiseFlat, OCC, VXMAX>(walk);
}

// Resident blocks per SM of the batch kernel (sizes the persistent grid).
template <int LAT, typename S>
int batch_blocks_per_sm(int occ, int vx_max, int walk, int noise_mode, int noise_dist) {
  if (vx_max == 1)
    return occ == 1 ? batch_blocks_occ<LAT, S, 1, 1>(walk, noise_mode, noise_dist)
                    : batch_blocks_occ<LAT, S, 0, 1>(walk, noise_mode, noise_dist);
  return occ == 1 ? batch_blocks_occ<LAT, S, 1, 2>(walk, noise_mode, noise_dist)
                  : batch_blocks_occ<LAT, S, 0, 2>(walk, noise_mode, noise_dist);
}

}  // namespace lbfd
