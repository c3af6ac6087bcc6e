// Many steps of a small lattice in one launch with the moment-space collision
// (mrt_kernels.cuh in resident_kernels.cuh).
#include <cmath>

#include "mrt_kernels.cuh"
#include "resident_kernels.cuh"

namespace lbfd {

cudaError_t launch_step_small_mrt(int lattice, int precision, const void *src, void *dst, const StepArgs &a,
                                  const double *m, const double *w, const double *tau, uint32_t lattice_id,
                                  uint64_t t0, int nsteps, cudaStream_t stream) {
  if (nsteps < 1 || a.N < 1 || (precision != kStoreF32 && precision != kStoreF64)) return cudaErrorInvalidValue;
  ResidentArgs ra{};
  ra.lattice_id = lattice_id;
  ra.nsteps = nsteps;
  ra.t0 = t0;
  return dispatch_lattice(lattice, [&](auto lat) -> cudaError_t {
    constexpr int LAT = decltype(lat)::value;
    if (precision == kStoreF64)
      return mrt_collide_t<LAT, double>(a, m, w, tau, [&](auto c) -> cudaError_t {
        return resident_t<LAT, double>(src, dst, a, ra, c, precision, stream);
      });
    return mrt_collide_t<LAT, float>(a, m, w, tau, [&](auto c) -> cudaError_t {
      return resident_t<LAT, float>(src, dst, a, ra, c, precision, stream);
    });
  });
}

}  // namespace lbfd
