// Deterministic FP64 reductions over the lattice: the total mass and the
// sampled observables of the paper's equilibrium tests (Sec. IV):
//   sum_x rho, sum_x rho^2              (density variance, eq. rhoth)
//   sum_x f_i, sum_x f_i f_j            (<f_i>, d_ij of eqs. dij / dijexp)
//   |sum_x (rho - rho_mean) e^{-2 pi i k.x / L}|^2 for chosen k
//                                       (structure factor, eq. fkfk)
// Stage 1: a fixed grid of kReduceBlocks x kReduceThreads threads walks the
// sites in a fixed order, reduces in registers, by warp shuffles and through
// shared memory, and writes one partial per block.  Stage 2: one block adds
// the partials in block order.  The result does not depend on timing.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "device.cuh"
#include "fastdiv.cuh"
#include "internal.h"

namespace lbfd {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// Mass
// ---------------------------------------------------------------------------
template <int LAT, typename S>
__global__ void __launch_bounds__(kReduceThreads) k_mass_partials(const S *__restrict__ f, int64_t N, int64_t stride,
                                                                 double rho_mean, double *__restrict__ partials) {
  using L = Lattice<LAT>;
  __shared__ double warp_tot[kReduceThreads / 32];
  double acc = 0.0;
  for (int64_t s = blockIdx.x * static_cast<int64_t>(kReduceThreads) + threadIdx.x; s < N;
       s += static_cast<int64_t>(gridDim.x) * kReduceThreads) {
    double r = 0.0;
    static_for<L::Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      r += Store<S>::getd(f[i * stride + s], L::w(i) * rho_mean);
    });
    acc += r;
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) warp_tot[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kReduceThreads / 32; ++w) t += warp_tot[w];
    partials[blockIdx.x] = t;
  }
}

__global__ void k_sum_partials(const double *__restrict__ partials, int nblocks, double *__restrict__ out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double t = 0.0;
    for (int b = 0; b < nblocks; ++b) t += partials[b];
    *out = t;
  }
}

cudaError_t launch_mass(int lattice, int precision, const void *f, int64_t N, double rho_mean, double *partials,
                        double *out, cudaStream_t stream, int64_t stride) {
  if (stride == 0) stride = N;
  return dispatch_lattice_storage(lattice, precision, [&](auto lat, auto tag) {
    constexpr int LAT = decltype(lat)::value;
    using S = typename decltype(tag)::type;
    k_mass_partials<LAT, S><<<kReduceBlocks, kReduceThreads, 0, stream>>>(static_cast<const S *>(f), N, stride,
                                                                          rho_mean, partials);
    k_sum_partials<<<1, 32, 0, stream>>>(partials, kReduceBlocks, out);
    return cudaGetLastError();
  });
}

// ---------------------------------------------------------------------------
// Observables
// ---------------------------------------------------------------------------
struct ModeArgs {
  int32_t n;
  int32_t k[LBFD_MAX_MODES_DEV][3];
};

// partial layout per block: [rho, rho2, f_0..f_{Q-1}, re_0, im_0, .., re_{K-1}, im_{K-1}, ff pairs (i <= j)]
int obs_quantities(int Q, int n_modes) { return 2 + Q + 2 * n_modes + Q * (Q + 1) / 2; }

// The observables of FP64 storage, FP64 throughout, straight from the stored
// post-collision state (population i at site x is g_i(x - v_i), as the step
// pulls it).  The FP64 pipe bounds it (2 lanes per clock and SM), so the pair
// sums are the work: a thread keeps them in registers for its own sites where
// they fit (D1Q3, D2Q5, D2Q9: Q (Q + 1)/2 multiply-adds per site), else a
// block takes tiles of sites through shared memory in 4 x 4 blocks of pairs
// (D3Q19).  The phases of the modes are FP32 as evaluated from the FP64 sum of
// (k x mod L)/L over the axes; each quotient is rounded correctly by one
// Newton correction with the rounded reciprocal (Markstein 1990), without a
// division.  Measured on GB300 per sample with 3 modes: D2Q9 512 x 384 173 -> 55
// us, 2048^2 2234 -> 757, D3Q19 128^3 1790 -> 1135, against 45 threads of a block adding pairs while the others waited, on a
// streamed copy, with 64-bit remainders and divisions for the phases.
struct Obs64 {
  int32_t Lx, Ly, Lz;
  FastDiv div_x, div_y, div_z;
  uint64_t rec_x, rec_y, rec_z;  // floor((2^64 - 1) / L)
  double inv_x, inv_y, inv_z;    // 1 / L, rounded
  double rho_mean;
  int32_t big;  // some side >= 46341: k x may not fit 31 bits
};

// (k x) mod L for 0 <= k, x < L.  On a side of 46341 or more k x may not fit
// 31 bits: its quotient by the reciprocal rec = floor((2^64 - 1) / L) is at
// most one too small (a general 64-bit remainder for every mode and axis took
// 97 us of a sample of D1Q3 4 10^6 sites with two modes on GB300).
__device__ __forceinline__ uint32_t obs_mulmod(uint32_t k, uint32_t x, uint32_t L, FastDiv dv, uint64_t rec, bool big) {
  if (k == 0) return 0;
  if (big) {
    const uint64_t n = static_cast<uint64_t>(k) * x;
    const uint64_t r = n - __umul64hi(n, rec) * L;
    return static_cast<uint32_t>(r >= L ? r - L : r);
  }
  const uint32_t n = k * x;
  return n - fastdiv(n, dv) * L;
}

// p / L for 0 <= p < L < 2^31, correctly rounded (inv = 1 / L rounded; every p
// below 4000 and 2e8 random pairs checked).
__device__ __forceinline__ double quotient(uint32_t p, int32_t L, double inv) {
  const double P = static_cast<double>(p), q = P * inv;
  return __fma_rn(__fma_rn(-q, static_cast<double>(L), P), inv, q);
}

// The pulled populations of site s, its density (returned) and its
// structure-factor terms: re[m] += d cos, im[m] -= d sin of the phase of mode
// m < modes.n, d = rho - rho_mean.
template <int LAT, int KMAX>
__device__ __forceinline__ double obs64_site(const double *g, uint32_t s, const Obs64 &o, const ModeArgs &modes,
                                           double (&f)[Lattice<LAT>::Q], double (&re)[KMAX], double (&im)[KMAX]) {
  using L = Lattice<LAT>;
  constexpr int Q = L::Q;
  const uint32_t Lx = static_cast<uint32_t>(o.Lx), Ly = static_cast<uint32_t>(o.Ly), Lz = static_cast<uint32_t>(o.Lz);
  const uint32_t r = fastdiv(s, o.div_x), x = s - r * Lx, z = fastdiv(r, o.div_y), y = r - z * Ly;
  const uint32_t xm = (x == 0 ? Lx : x) - 1, xp = x + 1 == Lx ? 0 : x + 1;
  const uint32_t ym = (y == 0 ? Ly : y) - 1, yp = y + 1 == Ly ? 0 : y + 1;
  const uint32_t zm = (z == 0 ? Lz : z) - 1, zp = z + 1 == Lz ? 0 : z + 1;
  const size_t N = static_cast<size_t>(Lx) * Ly * Lz;
  double rho = 0.0;
  static_for<Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    constexpr int vx = L::v(i, 0), vy = L::v(i, 1), vz = L::v(i, 2);
    const uint32_t xs = vx == 0 ? x : (vx > 0 ? xm : xp);
    const uint32_t ys = vy == 0 ? y : (vy > 0 ? ym : yp);
    const uint32_t zs = vz == 0 ? z : (vz > 0 ? zm : zp);
    f[i] = g[static_cast<size_t>(i) * N + xs + static_cast<size_t>(Lx) * (ys + static_cast<size_t>(Ly) * zs)];
    rho += f[i];
  });
  const double d = rho - o.rho_mean;
#pragma unroll
  for (int m = 0; m < KMAX; ++m)
    if (m < modes.n) {
      const double px = modes.k[m][0] == 0 ? 0.0 : quotient(obs_mulmod(modes.k[m][0], x, Lx, o.div_x, o.rec_x, o.big), o.Lx, o.inv_x);
      const double py = modes.k[m][1] == 0 ? 0.0 : quotient(obs_mulmod(modes.k[m][1], y, Ly, o.div_y, o.rec_y, o.big), o.Ly, o.inv_y);
      const double pz = modes.k[m][2] == 0 ? 0.0 : quotient(obs_mulmod(modes.k[m][2], z, Lz, o.div_z, o.rec_z, o.big), o.Lz, o.inv_z);
      float sn, cs;
      sincospif(2.0f * static_cast<float>(px + py + pz), &sn, &cs);
      re[m] += d * static_cast<double>(cs);
      im[m] -= d * static_cast<double>(sn);
    }
  return rho;
}

// One block's partial set: its threads' values pass through shared memory and
// thread q adds value q of all of them in a fixed order.  Layout: [sum rho, sum rho^2, sum f_i, (re, im) of the modes, pairs i <= j].
constexpr int kObs64Threads = 128;
template <int LAT, int KMAX>
__global__ void __launch_bounds__(kObs64Threads, 2)
    k_obs64_registers(const double *g, const Obs64 o, const ModeArgs modes, double *__restrict__ partials) {
  constexpr int Q = Lattice<LAT>::Q, NP = Q * (Q + 1) / 2, T = kObs64Threads;
  extern __shared__ double obs64_smem[];
  const uint32_t N = static_cast<uint32_t>(o.Lx) * static_cast<uint32_t>(o.Ly) * static_cast<uint32_t>(o.Lz);
  double sr = 0.0, sr2 = 0.0, sf[Q], sp[NP], re[KMAX], im[KMAX];
#pragma unroll
  for (int i = 0; i < Q; ++i) sf[i] = 0.0;
#pragma unroll
  for (int p = 0; p < NP; ++p) sp[p] = 0.0;
#pragma unroll
  for (int m = 0; m < KMAX; ++m) re[m] = im[m] = 0.0;
  // the warps of all blocks take 32 sites each in turn, warp 0 of every block
  // first, so that an incomplete last round loads the SMs evenly
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t step = static_cast<uint64_t>(gridDim.x) * T;
  for (uint64_t s = (static_cast<uint64_t>(warp) * gridDim.x + blockIdx.x) * 32 + lane; s < N; s += step) {
    double f[Q];
    const double rho = obs64_site<LAT, KMAX>(g, static_cast<uint32_t>(s), o, modes, f, re, im);
    sr += rho;
    sr2 = __fma_rn(rho, rho, sr2);
    int p = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      sf[i] += f[i];
#pragma unroll
      for (int j = i; j < Q; ++j, ++p) sp[p] = __fma_rn(f[i], f[j], sp[p]);
    }
  }
  // values [sum f_i, pairs, rho, rho^2, re, im] through shared memory
  constexpr int NS = Q + NP;
  double *const v = obs64_smem + threadIdx.x;
#pragma unroll
  for (int i = 0; i < Q; ++i) v[i * (T + 1)] = sf[i];
#pragma unroll
  for (int p = 0; p < NP; ++p) v[(Q + p) * (T + 1)] = sp[p];
  v[NS * (T + 1)] = sr;
  v[(NS + 1) * (T + 1)] = sr2;
#pragma unroll
  for (int m = 0; m < KMAX; ++m)
    if (m < modes.n) {
      v[(NS + 2 + 2 * m) * (T + 1)] = re[m];
      v[(NS + 3 + 2 * m) * (T + 1)] = im[m];
    }
  __syncthreads();
  const int K = modes.n, nv = NS + 2 + 2 * K;
  double *const out = partials + static_cast<size_t>(blockIdx.x) * (2 + Q + 2 * K + NP);
  for (int q = threadIdx.x; q < nv; q += T) {
    double a[4] = {0.0, 0.0, 0.0, 0.0};  // four chains
    for (int t = 0; t < T; t += 4)
#pragma unroll
      for (int c = 0; c < 4; ++c) a[c] += obs64_smem[q * (T + 1) + t + c];
    const int at = q < Q ? 2 + q : (q < NS ? 2 + Q + 2 * K + (q - Q) : (q < NS + 2 ? q - NS : 2 + Q + (q - NS - 2)));
    out[at] = (a[0] + a[1]) + (a[2] + a[3]);
  }
}

// D3Q19: the rows f_0 .. f_18 and a row of ones in five groups of four; a
// thread owns the 4 x 4 pairs of two groups (I <= J) and one of 16 slices of
// the tile's sites.
constexpr int kObs64Tile = 256, kObs64Groups = 5, kObs64Pairs = 15, kObs64Slices = 16;
template <int LAT, int KMAX>
__global__ void __launch_bounds__(kObs64Tile)
    k_obs64_tiles(const double *g, const Obs64 o, const ModeArgs modes, double *__restrict__ partials) {
  constexpr int Q = Lattice<LAT>::Q, NP = Q * (Q + 1) / 2, QP = 4 * kObs64Groups;
  static_assert(Q + 1 == QP, "the groups hold the populations and the ones");
  extern __shared__ double obs64_smem[];  // [site][QP + 2], then the sums
  constexpr int LD = QP + 2;              // rows 16 bytes apart in the banks
  const uint32_t N = static_cast<uint32_t>(o.Lx) * static_cast<uint32_t>(o.Ly) * static_cast<uint32_t>(o.Lz);
  const int tid = static_cast<int>(threadIdx.x);
  const bool has = tid < kObs64Pairs * kObs64Slices;
  const int blk = has ? tid / kObs64Slices : 0, slice = tid % kObs64Slices;
  int I = 0, b = blk;
  while (b >= kObs64Groups - I) b -= kObs64Groups - I++;
  const int J = I + b;
  double sr = 0.0, sr2 = 0.0, pa[16], re[KMAX], im[KMAX];
#pragma unroll
  for (int e = 0; e < 16; ++e) pa[e] = 0.0;
#pragma unroll
  for (int m = 0; m < KMAX; ++m) re[m] = im[m] = 0.0;
  for (uint64_t base = static_cast<uint64_t>(blockIdx.x) * kObs64Tile; base < N;
       base += static_cast<uint64_t>(gridDim.x) * kObs64Tile) {
    double f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = 0.0;
    const bool in = base + tid < N;
    if (in) {
      const double rho = obs64_site<LAT, KMAX>(g, static_cast<uint32_t>(base + tid), o, modes, f, re, im);
      sr += rho;
      sr2 = __fma_rn(rho, rho, sr2);
    }
    double *const row = obs64_smem + tid * LD;
#pragma unroll
    for (int i = 0; i < Q; ++i) row[i] = f[i];
    row[Q] = in ? 1.0 : 0.0;
    __syncthreads();
    if (has) {
      for (int k = slice; k < kObs64Tile; k += kObs64Slices) {
        const double2 *const u = reinterpret_cast<const double2 *>(obs64_smem + k * LD + 4 * I);
        const double2 *const w = reinterpret_cast<const double2 *>(obs64_smem + k * LD + 4 * J);
        const double2 u0 = u[0], u1 = u[1], w0 = w[0], w1 = w[1];
        const double uu[4] = {u0.x, u0.y, u1.x, u1.y}, ww[4] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) pa[4 * r + c] = __fma_rn(uu[r], ww[c], pa[4 * r + c]);
      }
    }
    __syncthreads();
  }
  // the slices of every pair in order; the modes over the block
  double *const red = obs64_smem;                                      // [16 * blk + e][slices + 1]
  double *const tot = red + kObs64Pairs * 16 * (kObs64Slices + 1);     // [blk][16]
  if (has) {
#pragma unroll
    for (int e = 0; e < 16; ++e) red[(16 * blk + e) * (kObs64Slices + 1) + slice] = pa[e];
  }
  __syncthreads();
  if (tid < kObs64Pairs * 16) {
    double t = 0.0;
    for (int k = 0; k < kObs64Slices; ++k) t += red[tid * (kObs64Slices + 1) + k];
    tot[tid] = t;
  }
  __syncthreads();
  const int K = modes.n;
  double *const out = partials + static_cast<size_t>(blockIdx.x) * (2 + Q + 2 * K + NP);
  auto pair_at = [](int i, int j) {  // i <= j < QP
    const int gi = i >> 2, gj = j >> 2;
    return (gi * kObs64Groups - gi * (gi - 1) / 2 + (gj - gi)) * 16 + (i & 3) * 4 + (j & 3);
  };
  if (tid < NP) {
    int p = tid, i = 0;
    while (p >= Q - i) p -= Q - i++;
    out[2 + Q + 2 * K + tid] = tot[pair_at(i, i + p)];
  }
  if (tid < Q) out[2 + tid] = tot[pair_at(tid, Q)];
  // rho, rho^2 and the modes over the block's warps
  const int lane = tid & 31, warp = tid >> 5;
  auto put = [&](int q, double v) {
    v = warp_sum(v);
    if (lane == 0) red[q * 8 + warp] = v;
  };
  put(0, sr);
  put(1, sr2);
#pragma unroll
  for (int m = 0; m < KMAX; ++m)
    if (m < K) {
      put(2 + 2 * m, re[m]);
      put(3 + 2 * m, im[m]);
    }
  __syncthreads();
  if (tid < 2 + 2 * K) {
    double t = 0.0;
    for (int w = 0; w < kObs64Tile / 32; ++w) t += red[tid * 8 + w];
    out[tid < 2 ? tid : Q + tid] = t;
  }
}

template <int LAT, int KMAX>
static cudaError_t obs64_t(const double *g, const Obs64 &o, const ModeArgs &ma, double *partials, cudaStream_t stream) {
  constexpr int Q = Lattice<LAT>::Q;
  if constexpr (Q <= 9) {
    const size_t smem = sizeof(double) * size_t(Q + Q * (Q + 1) / 2 + 2 + 2 * ma.n) * (kObs64Threads + 1);
    cudaError_t e = cudaFuncSetAttribute(k_obs64_registers<LAT, KMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(sizeof(double) * size_t(Q + Q * (Q + 1) / 2 + 2 + 2 * KMAX) * (kObs64Threads + 1)));
    if (e != cudaSuccess) return e;
    k_obs64_registers<LAT, KMAX><<<kReduceBlocks, kObs64Threads, smem, stream>>>(g, o, ma, partials);
  } else {
    const size_t smem = sizeof(double) * std::max<size_t>(size_t(kObs64Tile) * (4 * kObs64Groups + 2),
                                                          size_t(kObs64Pairs) * 16 * (kObs64Slices + 2));
    cudaError_t e = cudaFuncSetAttribute(k_obs64_tiles<LAT, KMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    k_obs64_tiles<LAT, KMAX><<<kReduceBlocks, kObs64Tile, smem, stream>>>(g, o, ma, partials);
  }
  return cudaGetLastError();
}

template <int LAT>
static cudaError_t pull_finalize_t(const double *partials, int nblocks, int n_modes, int64_t N, float rho_f,
                                   double *fin, double *acc, cudaStream_t stream);

cudaError_t launch_observables64(int lattice, const double *g, int32_t Lx, int32_t Ly, int32_t Lz, double rho_mean,
                                 int n_modes, const int32_t *modes, double *partials, double *fin, double *acc,
                                 cudaStream_t stream) {
  const int64_t N = int64_t(Lx) * Ly * Lz;
  if (n_modes < 0 || n_modes > LBFD_MAX_MODES_DEV || N >= (int64_t(1) << 31)) return cudaErrorInvalidValue;
  const int32_t L3[3] = {Lx, Ly, Lz};
  ModeArgs ma{};
  ma.n = n_modes;
  for (int m = 0; m < n_modes; ++m)
    for (int k = 0; k < 3; ++k)
      ma.k[m][k] = static_cast<int32_t>(((int64_t(modes[3 * m + k]) % L3[k]) + L3[k]) % L3[k]);
  Obs64 o{Lx, Ly, Lz, make_fastdiv(uint32_t(Lx)), make_fastdiv(uint32_t(Ly)), make_fastdiv(uint32_t(Lz)),
          ~uint64_t(0) / uint32_t(Lx), ~uint64_t(0) / uint32_t(Ly), ~uint64_t(0) / uint32_t(Lz),
          1.0 / Lx, 1.0 / Ly, 1.0 / Lz, rho_mean, (Lx >= 46341 || Ly >= 46341 || Lz >= 46341) ? 1 : 0};
  return dispatch_lattice(lattice, [&](auto lat) -> cudaError_t {
    constexpr int LAT = decltype(lat)::value;
    const cudaError_t e = n_modes <= 4 ? obs64_t<LAT, 4>(g, o, ma, partials, stream)
                                       : obs64_t<LAT, LBFD_MAX_MODES_DEV>(g, o, ma, partials, stream);
    // stage 2 of the FP32 pass with offsets c_i = 0: the sums themselves
    return e != cudaSuccess ? e : pull_finalize_t<LAT>(partials, kReduceBlocks, n_modes, N, 0.0f, fin, acc, stream);
  });
}

// ---------------------------------------------------------------------------
// Observables of a lattice in FP32 arithmetic (FP32, FP16 and BF16 storage),
// straight from the stored post-collision state g: population i at site x
// is f_i(x, t) = g_i(x - v_i), pulled as the step pulls it, so no streamed
// copy of the state is made.  The GPU has few FP64 units, so per site the
// kernel works in FP32 on deviations e_i = f_i - c_i from the constants
// c_i = w_i rho_mean (what the 16-bit formats store), delta = sum_i e_i, and
// d = rho - rho_mean.  A block takes tiles of 256 sites.  A mode's terms are
// rounded five times in FP32 (up to four modes; a warp's sites) or thirteen
// times (more; the tile) on their way to FP64.  A thread adds its slice of the pair products and of the e_i (the
// pairs with a row of ones) in FP32 over at most 256 terms before it goes to
// FP64, so the relative error is at most 256 x 2^-24 of the sum of the terms'
// magnitudes.  The final pass restores the sums of f and rho from the
// deviations in FP64.
// ---------------------------------------------------------------------------
constexpr int kObsThreads = 256;


__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sizes of the lattice with their fast divisions and FP32 inverses.
struct ObsDims {
  int32_t Lx, Ly, Lz;
  uint32_t s0, count;           // the sites sampled: s0 .. s0 + count - 1
  FastDiv div_x, div_y, div_z;  // exact for numerators below 2^31
  float inv_x, inv_y, inv_z;
  uint64_t rec_x, rec_y, rec_z; // floor((2^64 - 1) / side)
  int32_t big;                  // some side >= 46341: k x may not fit 31 bits
};

// Pair sums sum_x e_i e_j by register blocks: the rows i are padded to QP =
// 4 G and grouped by four; a thread owns one block (I, J), I <= J, of 4 x 4
// pairs and one slice of the tile's sites (sites sl, sl + SL, ...), and reads
// each site's two row groups as two 16-byte shared loads for 16 FMAs.  Its
// FP32 block sums cover SL tiles (256 products each) before they go to FP64.
// Row Q (always padding) holds 1 at every site, so the pairs (i, Q) give
// sum_x e_i, and sum delta = sum_i sum_x e_i, sum delta^2 = sum_ij sum_x e_i e_j
// follow without per-site reductions.
template <int Q>
struct ObsPairPlan {
  static constexpr int QP = (Q / 4 + 1) * 4;
  static constexpr int G = QP / 4;
  static constexpr int NB = G * (G + 1) / 2;
  static constexpr int SL = NB <= 1 ? 256 : NB <= 2 ? 128 : NB <= 4 ? 64 : NB <= 8 ? 32 : NB <= 16 ? 16 : 8;
  static constexpr int SPS = kObsThreads / SL;  // sites of a slice in one tile
  static_assert(NB * SL <= kObsThreads && NB * 16 <= kObsThreads, "pair plan exceeds the block");
};

// FEW: at most four modes.  Their eight sums over a warp's sites take nine
// exchanges a tile, each of which halves the sums that a lane holds; lane l ends
// with sum l / 4 and adds it to FP64 (five roundings in FP32).  With more modes
// a warp adds every mode's two terms at once (ten exchanges a mode and site)
// and the block its warps' sums, in FP32.  D3Q19 200^3 with 4 modes on GB300:
// 304 -> 264 us a sample, with the packed pair sums and the parallel end of the
// block.
constexpr int kFewModes = 4;

template <int LAT, typename S, bool FEW>
__global__ void __launch_bounds__(kObsThreads) k_obs_pull(const S *__restrict__ g, const ObsDims dm, float rho_f,
                                                         float d_off, const ModeArgs modes,
                                                         const float2 *__restrict__ phase,
                                                         double *__restrict__ partials) {
  using L = Lattice<LAT>;
  constexpr int Q = L::Q;
  constexpr int NPAIR = Q * (Q + 1) / 2;
  constexpr int NW = kObsThreads / 32;
  using P = ObsPairPlan<Q>;
  constexpr int QP = P::QP, SL = P::SL, SPS = P::SPS;
  __shared__ __align__(16) float tile[kObsThreads][QP];
  __shared__ float red[P::NB * SL][16];
  __shared__ float wsum[NW][2 * LBFD_MAX_MODES_DEV];
  __shared__ double slot_sum[P::NB * 16];
  const int32_t Lx = dm.Lx, Ly = dm.Ly, Lz = dm.Lz;
  const uint32_t N = static_cast<uint32_t>(Lx) * static_cast<uint32_t>(Ly) * static_cast<uint32_t>(Lz);
  const int K = modes.n;
  const int nq1 = 2 + Q + 2 * K;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // this thread's pair block (I, J) and slice, when it has one
  const bool has_block = threadIdx.x < P::NB * SL;
  const int blk = threadIdx.x / SL, sl = threadIdx.x % SL;
  int bI = 0, bJ = 0;
  {
    int b = has_block ? blk : 0, i = 0;
    while (b >= P::G - i) {
      b -= P::G - i;
      ++i;
    }
    bI = i;
    bJ = i + b;
  }
  float pa[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) pa[e] = 0.0f;
  // mode sum threadIdx.x (< 2 K), or FEW: this warp's mode sum lane / 4; pair slot threadIdx.x (< NB * 16)
  double acc_q = 0.0, acc_pair = 0.0;
  int tiles = 0;
  // FEW: the warp's sums of the terms v[0 .. 7] of its sites, sum lane / 4 into acc_q
  auto few_modes = [&](float (&v)[2 * kFewModes]) {
    static_assert(kFewModes == 4, "three halvings");
#pragma unroll
    for (int n = kFewModes, o = 16; n > 0; n /= 2, o /= 2) {  // n sums stay
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const float other = __shfl_xor_sync(0xffffffffu, up ? v[k] : v[k + n], o);
        v[k] = (up ? v[k + n] : v[k]) + other;
      }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    acc_q += static_cast<double>(v[0]);
  };

  // FP32 block sums of the last tiles into the FP64 slot sums (in slice order)
  auto flush_pairs = [&]() {
    if (has_block) {
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        red[threadIdx.x][e] = pa[e];
        pa[e] = 0.0f;
      }
    }
    __syncthreads();
    if (threadIdx.x < P::NB * 16) {
      const int b = threadIdx.x >> 4, e = threadIdx.x & 15;
      double t = 0.0;
      for (int k = 0; k < SL; ++k) t += static_cast<double>(red[b * SL + k][e]);
      acc_pair += t;
    }
    __syncthreads();
  };

  for (uint32_t base = blockIdx.x * kObsThreads; base < dm.count; base += gridDim.x * kObsThreads) {
    const bool valid = base + threadIdx.x < dm.count;
    const uint32_t s = dm.s0 + base + threadIdx.x;
    float e[QP];
#pragma unroll
    for (int i = 0; i < QP; ++i) e[i] = 0.0f;
    float delta = 0.0f;
    uint32_t x = 0, y = 0, z = 0;
    if (valid) {
      const uint32_t r = fastdiv(s, dm.div_x);
      x = s - r * static_cast<uint32_t>(Lx);
      z = fastdiv(r, dm.div_y);
      y = r - z * static_cast<uint32_t>(Ly);
      const uint32_t xm = (x == 0 ? Lx : x) - 1, xp = (x + 1 == static_cast<uint32_t>(Lx)) ? 0 : x + 1;
      const uint32_t ym = (y == 0 ? Ly : y) - 1, yp = (y + 1 == static_cast<uint32_t>(Ly)) ? 0 : y + 1;
      const uint32_t zm = (z == 0 ? Lz : z) - 1, zp = (z + 1 == static_cast<uint32_t>(Lz)) ? 0 : z + 1;
      const uint32_t Lxu = static_cast<uint32_t>(Lx), Lxy = Lxu * static_cast<uint32_t>(Ly);
      static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int vx = L::v(i, 0), vy = L::v(i, 1), vz = L::v(i, 2);
        const uint32_t xs = vx == 0 ? x : (vx > 0 ? xm : xp);
        const uint32_t ys = vy == 0 ? y : (vy > 0 ? ym : yp);
        const uint32_t zs = vz == 0 ? z : (vz > 0 ? zm : zp);
        const S v = g[static_cast<size_t>(i) * N + xs + Lxu * ys + Lxy * zs];
        // 16-bit formats store the deviation itself; FP32 stores f
        e[i] = Store<S>::kDeviation ? Store<S>::get(v, 0.0f)
                                    : sub_rn(Store<S>::get(v, 0.0f), obs_offset<LAT>(i, rho_f));
        delta += e[i];
      });
      e[Q] = 1.0f;
    }
#pragma unroll
    for (int i = 0; i < QP; i += 4)
      *reinterpret_cast<float4 *>(&tile[threadIdx.x][i]) = make_float4(e[i], e[i + 1], e[i + 2], e[i + 3]);
    // per-tile FP32 sums of the mode quantities, one warp total each
    auto put = [&](int q, float v) {
      v = warp_sum_f(v);
      if (lane == 0) wsum[warp][q] = v;
    };
    if (K > 0) {
      const float d = valid ? delta + d_off : 0.0f;
      auto term = [&](int m) {
        float cs, sn;
        if (phase) {
          // e^{-2 pi i k.x / L} as the product of its three per-axis factors
          const float2 fx = phase[m * Lx + x];
          const float2 fy = phase[K * Lx + m * Ly + y];
          const float2 fz = phase[K * (Lx + Ly) + m * Lz + z];
          const float ar = fx.x * fy.x - fx.y * fy.y, ai = fx.x * fy.y + fx.y * fy.x;
          cs = ar * fz.x - ai * fz.y;
          sn = -(ar * fz.y + ai * fz.x);
        } else {
          const uint32_t px = obs_mulmod(static_cast<uint32_t>(modes.k[m][0]), x, Lx, dm.div_x, dm.rec_x, dm.big);
          const uint32_t py = obs_mulmod(static_cast<uint32_t>(modes.k[m][1]), y, Ly, dm.div_y, dm.rec_y, dm.big);
          const uint32_t pz = obs_mulmod(static_cast<uint32_t>(modes.k[m][2]), z, Lz, dm.div_z, dm.rec_z, dm.big);
          // each term is below 1 and exact to FP32 rounding; sincospif reduces exactly
          const float frac = fmaf(static_cast<float>(px), dm.inv_x,
                                  fmaf(static_cast<float>(py), dm.inv_y, static_cast<float>(pz) * dm.inv_z));
          sincospif(2.0f * frac, &sn, &cs);
        }
        return make_float2(mul_rn(d, cs), mul_rn(-d, sn));
      };
      if constexpr (FEW) {
        float v[2 * kFewModes];
        static_for<kFewModes>([&](auto M) {
          constexpr int m = decltype(M)::value;
          const float2 t = m < K ? term(m) : make_float2(0.0f, 0.0f);
          v[2 * m] = t.x;
          v[2 * m + 1] = t.y;
        });
        few_modes(v);
      } else {
        for (int m = 0; m < K; ++m) {
          const float2 t = term(m);
          put(2 * m, t.x);
          put(2 * m + 1, t.y);
        }
      }
    }
    __syncthreads();
    // this tile's mode sums of the warps into FP64
    if (!FEW && threadIdx.x < 2 * K) {
      float t = 0.0f;
#pragma unroll
      for (int w = 0; w < NW; ++w) t += wsum[w][threadIdx.x];
      acc_q += static_cast<double>(t);
    }
    if (has_block) {
#pragma unroll 4
      for (int kk = 0; kk < SPS; ++kk) {
        const int k = sl + kk * SL;
        const float4 u = *reinterpret_cast<const float4 *>(&tile[k][4 * bI]);
        const float4 v = *reinterpret_cast<const float4 *>(&tile[k][4 * bJ]);
        const float uu[4] = {u.x, u.y, u.z, u.w};
        const float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
#pragma unroll
        for (int a = 0; a < 4; ++a) {  // two pairs an instruction
          const float2 ua = make_float2(uu[a], uu[a]);
          const float2 r0 = fma_rn(ua, v0, make_float2(pa[4 * a], pa[4 * a + 1]));
          const float2 r1 = fma_rn(ua, v1, make_float2(pa[4 * a + 2], pa[4 * a + 3]));
          pa[4 * a] = r0.x;
          pa[4 * a + 1] = r0.y;
          pa[4 * a + 2] = r1.x;
          pa[4 * a + 3] = r1.y;
        }
      }
    }
    __syncthreads();
    if (++tiles == SL) {
      flush_pairs();
      tiles = 0;
    }
  }
  if (tiles > 0) flush_pairs();
  // gather the slot sums, then write the block's partials in the layout of
  // the stage-2 pass: [sum delta, sum delta^2, sum e_i, modes, pairs i <= j]
  if (threadIdx.x < P::NB * 16) slot_sum[threadIdx.x] = acc_pair;
  __shared__ double mode_sum[NW][2 * kFewModes];
  if (FEW && lane % 4 == 0) mode_sum[warp][lane / 4] = acc_q;
  __syncthreads();
  if (FEW && threadIdx.x < 2 * K) {
    acc_q = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) acc_q += mode_sum[w][threadIdx.x];
  }
  auto slot_of = [](int i, int j) {  // i <= j < QP
    const int I = i >> 2, J = j >> 2;
    return (I * P::G - I * (I - 1) / 2 + (J - I)) * 16 + (i & 3) * 4 + (j & 3);
  };
  double *out = partials + static_cast<size_t>(blockIdx.x) * (nq1 + NPAIR);
  if (threadIdx.x < NPAIR) {
    int p = threadIdx.x, i = 0;
    while (p >= Q - i) {
      p -= Q - i;
      ++i;
    }
    out[nq1 + threadIdx.x] = slot_sum[slot_of(i, i + p)];
  }
  if (threadIdx.x < Q) out[2 + threadIdx.x] = slot_sum[slot_of(threadIdx.x, Q)];
  if (threadIdx.x < 2 * K) out[2 + Q + threadIdx.x] = acc_q;
  if (threadIdx.x < 32)
    obs_delta_sums<Q>([&](int i) { return slot_sum[slot_of(i, Q)]; },
                      [&](int i, int j, int) { return slot_sum[slot_of(i, j)]; }, out, lane);
}

// Stage 2 of the FP32 pass, spread over the GPU (its FP64 units are few, so
// one block summing every quantity would take ~0.1 ms): warp w sums
// quantity w over the block partials (lane l adds blocks l, l + 32, ... in
// order, then a fixed butterfly), and the last block to finish (a ticket in
// fin[nq_max]) restores the sums of rho, f and f f from the deviation sums
// with c_i = w_i rho_mean (the kernels' own FP32 constants) and adds them to
// acc:
//   sum rho   = S_delta + N C,            C = sum_i c_i
//   sum rho^2 = S_delta2 + 2 C S_delta + N C^2
//   sum f_i   = E_i + N c_i
//   sum f_i f_j = P_ij + c_j E_i + c_i E_j + N c_i c_j
// Every sum has a fixed order, so the result does not depend on timing.
constexpr int kFinWarps = 8;
template <int LAT>
__global__ void __launch_bounds__(kFinWarps * 32)
    k_obs_pull_finalize(const double *__restrict__ partials, int nblocks, int K, double Nd, float rho_f,
                        double *__restrict__ tot, unsigned int *__restrict__ ticket, double *__restrict__ acc) {
  constexpr int Q = Lattice<LAT>::Q;
  const int nq = 2 + Q + 2 * K + Q * (Q + 1) / 2;
  const int lane = threadIdx.x & 31, q = blockIdx.x * kFinWarps + (threadIdx.x >> 5);
  if (q < nq) {
    double t = 0.0;
    for (int b = lane; b < nblocks; b += 32) t += partials[static_cast<size_t>(b) * nq + q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) tot[q] = t;
  }
  __threadfence();
  __syncthreads();
  __shared__ bool last;
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  // the last block: the totals into shared memory (from L2: the other blocks
  // wrote them), then one accumulator entry per thread
  __threadfence();
  __shared__ double tt[2 + LBFD_MAX_Q_DEV + 2 * LBFD_MAX_MODES_DEV + LBFD_MAX_Q_DEV * (LBFD_MAX_Q_DEV + 1) / 2];
  __shared__ double cs[LBFD_MAX_Q_DEV + 1];
  const volatile double *vt = tot;
  for (int k = threadIdx.x; k < nq; k += blockDim.x) tt[k] = vt[k];
  if (threadIdx.x < Q) cs[threadIdx.x] = static_cast<double>(obs_offset<LAT>(static_cast<int>(threadIdx.x), rho_f));
  __syncthreads();
  if (threadIdx.x == 0) {
    double C = 0.0;
    for (int i = 0; i < Q; ++i) C += cs[i];
    cs[Q] = C;
    *ticket = 0u;  // for the next launch (stream-ordered after this one)
  }
  __syncthreads();
  const double C = cs[Q];
  const int nacc = 2 + Q + Q * Q + K;
  for (int k = threadIdx.x; k < nacc; k += blockDim.x) acc[k] += obs_restore<Q>(k, tt, cs, C, Nd, K);
}

template <int LAT>
static cudaError_t pull_finalize_t(const double *partials, int nblocks, int n_modes, int64_t N, float rho_f,
                                   double *fin, double *acc, cudaStream_t stream) {
  constexpr int Q = Lattice<LAT>::Q;
  const int nq = obs_quantities(Q, n_modes);
  unsigned int *ticket = reinterpret_cast<unsigned int *>(fin + obs_quantities(Q, LBFD_MAX_MODES_DEV));
  // a plain launch: as a dependent launch it let the next step's blocks take
  // the SMs while it still waited for the sampled step, which cost D3Q19
  // 256^3 0.5 ms per sample on GB300
  k_obs_pull_finalize<LAT><<<(nq + kFinWarps - 1) / kFinWarps, kFinWarps * 32, 0, stream>>>(
      partials, nblocks, n_modes, double(N), rho_f, fin, ticket, acc);
  return cudaGetLastError();
}

// Stage 2 of the FP32-arithmetic observables for partials written by a
// fused sampling step (sample_kernels.cuh), in the layout of k_obs_pull.
cudaError_t launch_obs_pull_finalize(int lattice, const double *partials, int nblocks, int n_modes, int64_t N,
                                     double rho_mean, double *fin, double *acc, cudaStream_t stream) {
  const float rho_f = static_cast<float>(rho_mean);
  return dispatch_lattice(lattice, [&](auto lat) -> cudaError_t {
    constexpr int LAT = decltype(lat)::value;
    return pull_finalize_t<LAT>(partials, nblocks, n_modes, N, rho_f, fin, acc, stream);
  });
}

int obs_pull_blocks(int64_t N) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kObsBlocks, (N + kObsThreads - 1) / kObsThreads)));
}

cudaError_t launch_observables_pull_partials(int lattice, int precision, const void *g, int32_t Lx, int32_t Ly,
                                             int32_t Lz, int64_t s0, int64_t count, double rho_mean, int n_modes,
                                             const int32_t *modes, const void *phase, double *partials, int *nblocks,
                                             cudaStream_t stream) {
  if (n_modes < 0 || n_modes > LBFD_MAX_MODES_DEV || precision == kStoreF64) return cudaErrorInvalidValue;
  const int64_t N = int64_t(Lx) * Ly * Lz;
  if (N >= (int64_t(1) << 31) || s0 < 0 || count < 0 || s0 + count > N) return cudaErrorInvalidValue;
  const int32_t L3[3] = {Lx, Ly, Lz};
  ModeArgs ma{};
  ma.n = n_modes;
  for (int m = 0; m < n_modes; ++m)
    for (int k = 0; k < 3; ++k)
      ma.k[m][k] = static_cast<int32_t>(((int64_t(modes[3 * m + k]) % L3[k]) + L3[k]) % L3[k]);
  ObsDims dm{};
  dm.Lx = Lx;
  dm.Ly = Ly;
  dm.Lz = Lz;
  dm.s0 = static_cast<uint32_t>(s0);
  dm.count = static_cast<uint32_t>(count);
  dm.div_x = make_fastdiv(uint32_t(Lx));
  dm.div_y = make_fastdiv(uint32_t(Ly));
  dm.div_z = make_fastdiv(uint32_t(Lz));
  dm.inv_x = 1.0f / float(Lx);
  dm.inv_y = 1.0f / float(Ly);
  dm.inv_z = 1.0f / float(Lz);
  dm.rec_x = ~uint64_t(0) / uint32_t(Lx);
  dm.rec_y = ~uint64_t(0) / uint32_t(Ly);
  dm.rec_z = ~uint64_t(0) / uint32_t(Lz);
  dm.big = (Lx >= 46341 || Ly >= 46341 || Lz >= 46341) ? 1 : 0;
  const float rho_f = static_cast<float>(rho_mean);
  *nblocks = obs_pull_blocks(count);
  return dispatch_lattice_storage(lattice, precision, [&](auto lat, auto tag) {
    constexpr int LAT = decltype(lat)::value;
    using S = typename decltype(tag)::type;
    if constexpr (std::is_same_v<S, double>) {
      return cudaErrorInvalidValue;
    } else {
      constexpr int Q = Lattice<LAT>::Q;
      // d = rho - rho_mean = delta + (C - rho_mean), C from the same FP32 constants
      double C = 0.0;
      for (int i = 0; i < Q; ++i) C += static_cast<double>(static_cast<float>(Lattice<LAT>::w(i)) * rho_f);
      const float d_off = static_cast<float>(C - rho_mean);
      auto kern = n_modes <= kFewModes ? k_obs_pull<LAT, S, true> : k_obs_pull<LAT, S, false>;
      kern<<<*nblocks, kObsThreads, 0, stream>>>(static_cast<const S *>(g), dm, rho_f, d_off, ma,
                                                 static_cast<const float2 *>(phase), partials);
      return cudaGetLastError();
    }
  });
}

cudaError_t launch_observables_pull(int lattice, int precision, const void *g, int32_t Lx, int32_t Ly, int32_t Lz,
                                    double rho_mean, int n_modes, const int32_t *modes, const void *phase,
                                    double *partials, double *fin, double *acc, cudaStream_t stream) {
  const int64_t N = int64_t(Lx) * Ly * Lz;
  int nblocks = 0;
  cudaError_t e = launch_observables_pull_partials(lattice, precision, g, Lx, Ly, Lz, 0, N, rho_mean, n_modes, modes,
                                                   phase, partials, &nblocks, stream);
  if (e != cudaSuccess) return e;
  return launch_obs_pull_finalize(lattice, partials, nblocks, n_modes, N, rho_mean, fin, acc, stream);
}

size_t obs_phase_values(int n_modes, int32_t Lx, int32_t Ly, int32_t Lz) {
  return size_t(n_modes) * (size_t(Lx) + size_t(Ly) + size_t(Lz));
}

void obs_phase_fill(int n_modes, const int32_t *modes, int32_t Lx, int32_t Ly, int32_t Lz, float *out,
                    const int64_t *period, const int64_t *offset) {
  // per axis d and mode m: e^{-2 pi i r / P_d}, r = (k_d ((o_d + u) mod P_d)) mod P_d, u < L_d, in FP64 then
  // rounded (P_d = L_d and o_d = 0 unless a slab gives its global period and its first stored plane)
  const int32_t L3[3] = {Lx, Ly, Lz};
  size_t at = 0;
  for (int d = 0; d < 3; ++d)
    for (int m = 0; m < n_modes; ++m) {
      const int64_t P = period ? period[d] : L3[d], o = offset ? offset[d] : 0;
      const int64_t k = ((int64_t(modes[3 * m + d]) % P) + P) % P;
      for (int64_t u = 0; u < L3[d]; ++u, ++at) {
        const int64_t x = ((o + u) % P + P) % P;
        const double a = 2.0 * 3.14159265358979323846 * double((k * x) % P) / double(P);
        out[2 * at] = static_cast<float>(std::cos(a));
        out[2 * at + 1] = static_cast<float>(-std::sin(a));
      }
    }
}

}  // namespace lbfd
