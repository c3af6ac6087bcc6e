// Host evaluation of the FP64 Box-Muller pairs' parts over all 2^24
// arguments against long double.
#include <cmath>
#include <cstdint>

#include "bm64.cuh"

using namespace lbfd::bm64;

static const Tables kHost = make_tables();

// out: largest relative error of the radius, its root mean square, the largest
// error of the angle's cosine and sine
extern "C" void bmc_errors(double *out) {
  long double worst = 0, sum = 0, angle = 0;
  const long double two_pi = 6.283185307179586476925286766559005768L;
  for (uint32_t k = 0; k < (1u << 24); ++k) {
    const long double u = (k + 0.5L) * 0x1p-24L;
    const long double want = sqrtl(-2.0L * (u > 0.5L ? log1pl(u - 1.0L) : logl(u)));
    const long double e = fabsl(radius28(k << 8, kHost) * 0x1p-28L / want - 1.0L);
    worst = e > worst ? e : worst;
    sum += e * e;
    if (k % 7 == 0 || (k + 1) % 2048 < 2) {
      const CosSin a = angle28(k << 8, kHost);
      const long double c = fabsl(a.c * 0x1p28L - cosl(two_pi * u)), s = fabsl(a.s * 0x1p28L - sinl(two_pi * u));
      angle = c > angle ? c : angle;
      angle = s > angle ? s : angle;
    }
  }
  out[0] = static_cast<double>(worst);
  out[1] = static_cast<double>(sqrtl(sum / (1 << 24)));
  out[2] = static_cast<double>(angle);
}
