// Many steps of a small lattice in one launch: which lattices take the
// resident kernel (resident_kernels.cuh), and the single-relaxation launches.
#include <algorithm>
#include <cuda_runtime.h>

#include "resident_kernels.cuh"

namespace lbfd {

// The largest lattice in FP32 arithmetic that one block steps.
static int64_t one_block_sites(int lattice) { return lattice == kD1Q3 ? 512 : (lattice == kD3Q19 ? 128 : 256); }

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
  return N <= one_block_sites(lattice) ? 1 : (N <= 512 ? 8 : kResidentCtas);
}

// A launch of the resident kernel costs 3 to 16 us before its steps count (the
// cluster's start, the address and noise set-up, the state in and out), where
// a launched step of such a lattice costs 1.7 us (FP64 2 to 12) and no set-up.
// Microseconds for n steps on GB300, resident / launched, back to back:
//   - D1Q3, D2Q5 on one block: n = 2 3.5 / 4.3, 3 4.2 / 5.9;
//     on a cluster (4000 sites): 2 6.2 / 4.3, 3 6.2 / 5.9, 4 6.2 / 7.5;
//   - D2Q9 on one block (256 sites): 3 6.2 / 5.8, 4 6.2 / 7.4; on a cluster (64 x 48):
//     3 8.2 / 5.9, 4 8.3 / 7.7, 5 9.1 / 9.2; 91 x 91, where a step is slower
//     too: 5 12.4 / 9.3, 8 16.4 / 14.0, D2Q5 127 x 127 8 14.4 / 14.3;
//   - D3Q19 6^3: 3 10.6 / 6.1, 5 12.4 / 10.2, 6 13.4 / 12.3, 8 14.4 / 16.4;
//   - FP64: D1Q3 300 sites 5 12.4 / 12.0, 6 14.4 / 14.4; D2Q9 20 x 20
//     6 24.6 / 22.5, 8 30.4 / 30.0; D3Q19 8^3 6 47.2 / 45.1, 8 60.6 / 60.1.
int small_path_least(int lattice, int precision, int64_t N) {
  if (precision == kStoreF64) return lattice == kD1Q3 ? 6 : 8;
  if (lattice == kD3Q19) return 6;
  if (lattice != kD1Q3 && N > 8192) return 8;
  const bool one = N <= one_block_sites(lattice);
  return lattice == kD2Q9 ? (one ? 4 : 5) : (one ? 2 : 4);
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
