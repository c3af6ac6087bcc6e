// Host evaluation of the FP64 Box-Muller pairs' parts over all 2^24
// arguments against long double.
#include <cmath>
#include <cstdint>

#include "bm64.cuh"

using namespace lbfd::bm64;

static const Tables kHost = make_tables();

// out: largest relative error of the radius and its root mean square; the
// same of the angle's cosine and sine; their largest absolute error
extern "C" void bmc_errors(double *out) {
  long double worst = 0, sum = 0, angle = 0, relative = 0, squares = 0;
  const long double pi = 3.14159265358979323846264338327950288L;
  long n = 0;
  for (uint32_t k = 0; k < (1u << 24); ++k) {
    const long double u = (k + 0.5L) * 0x1p-24L;
    const long double want = sqrtl(-2.0L * (u > 0.5L ? log1pl(u - 1.0L) : logl(u)));
    const long double e = fabsl(radius28(k << 8, kHost) * 0x1p-28L / want - 1.0L);
    worst = e > worst ? e : worst;
    sum += e * e;
    // every seventh angle, those next to base angles' edges, and all near an axis
    const uint32_t q = k & 0x3fffff;
    if (k % 7 && (k + 1) % 2048 > 1 && q > 8192 && q < 0x3fffff - 8192) continue;
    // reduced exactly to the nearest axis
    const long double turn = rintl(4.0L * u), rest = 2.0L * pi * (u - 0.25L * turn);
    const long double c0 = cosl(rest), s0 = sinl(rest);
    const int t = static_cast<int>(turn) & 3;
    const long double cw = t == 0 ? c0 : (t == 1 ? -s0 : (t == 2 ? -c0 : s0));
    const long double sw = t == 0 ? s0 : (t == 1 ? c0 : (t == 2 ? -s0 : -c0));
    const CosSin a = angle28(k << 8, kHost);
    const long double dc = fabsl(a.c * 0x1p28L - cw), ds = fabsl(a.s * 0x1p28L - sw);
    angle = fmaxl(angle, fmaxl(dc, ds));
    relative = fmaxl(relative, fmaxl(dc / fabsl(cw), ds / fabsl(sw)));
    squares += dc / cw * (dc / cw) + ds / sw * (ds / sw);
    n += 2;
  }
  out[0] = static_cast<double>(worst);
  out[1] = static_cast<double>(sqrtl(sum / (1 << 24)));
  out[2] = static_cast<double>(relative);
  out[3] = static_cast<double>(sqrtl(squares / n));
  out[4] = static_cast<double>(angle);
}
