// Host check of the D3Q19 noise transform's order of operations: each value
// against the same sum written out from the basis, bit for bit.
#include <math.h>
#include <string.h>

#include "device.cuh"

using namespace lbfd;

namespace {

constexpr int LAT = kD3Q19, Q = Lattice<LAT>::Q;

// sum over the rows a = 1 .. Q - 1 of parity `par` (-1: all) in ascending
// order of w_i m_i^a z^a: the first term a product, the others multiply-adds.
float row_sum(int i, int par, const float *z, int *terms) {
  float acc = 0.0f;
  *terms = 0;
  for (int a = 1; a < Q; ++a) {
    const double c = kBasisTable<LAT>.m[a][i] * Lattice<LAT>::w(i);
    if (c == 0.0 || (par >= 0 && row_parity<LAT>(a) != par)) continue;
    const float k = static_cast<float>(c);
    acc = *terms == 0 ? k * z[a - 1] : fmaf(k, z[a - 1], acc);
    ++*terms;
  }
  return acc;
}

}  // namespace

// z: n sets of Q - 1 variates.  Returns the number of values that differ.
extern "C" int toc_d3q19_mismatches(const float *z, int n) {
  int bad = 0;
  for (int k = 0; k < n; ++k, z += Q - 1) {
    float zz[Q - 1], T[Q];
    memcpy(zz, z, sizeof zz);
    NoiseTransform<LAT, float>::apply(zz, T);
    for (int i = 0; i < Q; ++i) {
      const int ip = partner<LAT>(i);
      float want;
      int ne, no;
      if (ip == i) {
        want = row_sum(i, -1, zz, &ne);
      } else {
        const int first = i < ip ? i : ip;
        const float E = row_sum(first, 0, zz, &ne), O = row_sum(first, 1, zz, &no);
        if (no < 2) return -1;  // (a single odd term would be a multiply-add onto E; D3Q19 has none)
        want = i == first ? E + O : E - O;
      }
      bad += memcmp(&want, &T[i], sizeof(float)) != 0;
    }
  }
  return bad;
}
