// Host check of the rule for sites per thread of the register-pull kernels.
#include "step_shape.h"

using namespace lbfd;

extern "C" int vwc_width(int lattice, int precision, int Lx, long long sites, unsigned long long a,
                         unsigned long long b, int value_bytes) {
  return step_vec_width(lattice, precision, Lx, sites,
                        vec_most(reinterpret_cast<const void *>(a), reinterpret_cast<const void *>(b), value_bytes));
}
