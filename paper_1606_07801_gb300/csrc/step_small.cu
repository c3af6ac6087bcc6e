// Many steps of a small lattice in one launch: which lattices take the
// resident kernel (resident_kernels.cuh), and the single-relaxation launches.
#include <algorithm>
#include <cuda_runtime.h>

#include "resident_kernels.cuh"

namespace lbfd {

// CTAs of a lattice (1: a single block, else a cluster), 0 where the resident
// kernel is not taken.  One site per thread bounds the lattice: 16 CTAs of
// resident_threads, or less where that many sites do not fit the shared
// memory.  Measured on GB300, microseconds per step:
//   - a cluster is faster than one launch per step up to that bound (D2Q9 FP32
//     128 x 128: 1.76 resident, 1.81 launched; D3Q19 20^3 2.14 and 2.83, D1Q3
//     16000 sites 0.82 and 1.62), and several sites per thread above it were
//     not (D2Q9 128 x 170: 3.8 and 3.6 with the kernels of the time);
//   - one block, whose barrier is cheaper, wins while its warps are few
//     (D2Q9 91 sites 0.30 against 0.53 on 16 CTAs, 256 sites 0.50 and 0.53,
//     400 sites 0.86 and 0.53; D1Q3 300 sites 0.32 and 0.43, 600 sites 0.45 and
//     0.42; D3Q19 125 sites 0.76 and 0.75, 216 sites 1.11 and 0.75);
//   - beyond that, more CTAs are never slower (D2Q9 40 x 30: 1.18 on 2, 0.86
//     on 4, 0.63 on 8, 0.58 on 16).
// FP64 arithmetic, 2 lanes per clock and SM, takes a CTA per 32 sites (D2Q9 480
// sites 2.67 resident, 3.55 launched; D3Q19 216 sites 6.7 and 7.4; D1Q3 2048
// sites 1.86 and 2.38), and up to 128 sites on each, a line from when launched
// FP64 steps were slower: above about 50 sites a CTA D2Q9 and D3Q19 now step
// faster launched (D2Q9 1600 sites 4.49 against 3.61, D3Q19 1728 sites 13.9
// against 7.5).
int small_path_ctas(int lattice, int precision, int64_t N) {
  if (N < 1) return 0;
  const int elem = storage_bytes(precision);
  const bool f64 = precision == kStoreF64;
  const int Q = lattice == kD1Q3 ? 3 : (lattice == kD2Q9 ? 9 : (lattice == kD2Q5 ? 5 : 19));
  const int64_t by_smem = int64_t(kSmallMaxBytes) / (2 * int64_t(Q) * elem);
  if (N > kResidentCtas * std::min<int64_t>(by_smem, resident_threads(lattice, f64))) return 0;
  if (f64) return int(std::min<int64_t>(kResidentCtas, (N + 31) / 32));
  const int64_t one = lattice == kD1Q3 ? 512 : (lattice == kD3Q19 ? 128 : 256);
  return N <= one ? 1 : (N <= 512 ? 8 : kResidentCtas);
}

namespace {

template <int LAT>
cudaError_t resident_lat(int precision, const void *src, void *dst, const StepArgs &a, const ResidentArgs &ra,
                         cudaStream_t stream) {
  return dispatch_storage(precision, [&](auto tag) -> cudaError_t {
    using S = typename decltype(tag)::type;
    if (a.noise_mode == kNoiseOff)
      return resident_t<LAT, S>(src, dst, a, ra, SrtCollideFor<LAT, S, kStepNoiseOff>{}, precision, stream);
    if (a.noise_dist == kGaussian)
      return resident_t<LAT, S>(src, dst, a, ra, SrtCollideFor<LAT, S, kStepNoiseGauss>{}, precision, stream);
    return resident_t<LAT, S>(src, dst, a, ra, SrtCollideFor<LAT, S, kStepNoiseFlat>{}, precision, stream);
  });
}

}  // namespace

// Single-relaxation lattices (moment-space runs: launch_step_small_mrt).
cudaError_t launch_step_small(int lattice, int precision, const void *src, void *dst, const StepArgs &a,
                              uint32_t lattice_id, uint64_t t0, int nsteps, cudaStream_t stream) {
  if (nsteps < 1 || a.N < 1) return cudaErrorInvalidValue;
  ResidentArgs ra{};
  ra.lattice_id = lattice_id;
  ra.nsteps = nsteps;
  ra.t0 = t0;
  switch (lattice) {
    case kD1Q3: return resident_lat<kD1Q3>(precision, src, dst, a, ra, stream);
    case kD2Q9: return resident_lat<kD2Q9>(precision, src, dst, a, ra, stream);
    case kD3Q19: return resident_lat<kD3Q19>(precision, src, dst, a, ra, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbfd
