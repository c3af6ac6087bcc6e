// Box-Muller pairs in FP64 from two 24-bit uniforms, for a GPU whose FP64
// pipe is narrow (GB300: 2 lanes per clock and SM, a sixty-fourth of FP32).
//
// What bounds it: the general log, sincospi and sqrt take about 105 FP64
// operations per pair, which is two thirds of all FP64 work of a D2Q9 step
// (512 x 384: 165 us per step, the FP64 pipe saturated) and most of the
// dependent chain of a small lattice's step.  The arguments are special: u0
// and u1 are odd multiples of 2^-25, so
//   - -2 ln u0 is formed in 64-bit integers: with K = u0 2^25 normalised to M
//     = K 2^(24 - e) in [2^24, 2^25), a table of 1024 cells of M gives c = C
//     2^-14 near 2^24 / M and 2 ln c, and r = M c 2^-24 - 1 is the exact
//     32-bit integer product M C modulo 2^32 (|r| < 2^-10.8); then
//       -2 ln u0 = (25 - e) 2 ln 2 + 2 ln c - 2 ln(1 + r),
//       -2 ln(1 + r) = -2 r + r^2 - (2/3) r^3 + r^4/2 - (2/5) r^5 + O(2^-66),
//     fixed point with 2^-57 below u0 = 1/2, where the value is above 1.38, and
//     with 2^-62 and 2^-65 (the last sixteenth) above, so that its relative
//     error stays below a quarter of FP64's rounding; the terms from r^4 on are
//     FP32.  One conversion makes it FP64.  Next to u0 = 1 (the last 2^-11, one
//     draw in 2048) the logarithm's series in 1 - u0 takes its place;
//   - the square root is rsqrt.approx.ftz.f64 and sqrt_seeded;
//   - the angle 2 pi u1 is a quadrant, the nearest of 2049 base angles and an
//     odd multiple of 2 pi 2^-25 below 2^-11.35, each from a table, joined by
//     the addition formulas (6 operations).
// 16 FP64 operations per pair.  The tables (96 KB) are evaluated by the
// compiler in double-double arithmetic and read through L1.  Over all 2^24
// arguments on the host the radius is within a relative 1.78e-16, root mean
// square 5.27e-17 (the C library 1.66e-16 and 5.27e-17), and the cosine and sine
// within a relative 1.88e-16, root mean square 4.3e-17.  On GB300, against
// CUDA's functions: radius times the first angle's cosine 2.79e-16, root mean
// square 7.14e-17 (2.81e-16 and 7.14e-17); one radius times all angles 3.05e-16
// and 8.59e-17 (3.59e-16 and 9.24e-17).
// Measured on GB300: D2Q9 512 x 384, a step, 159.4 -> 46.9 us; D1Q3 256 sites,
// resident, 3.95 -> 1.48 us (both with the kernels around it).
#pragma once

#include <stdint.h>

#ifndef __CUDA_ARCH__
#include <cmath>
#endif

namespace lbfd {
namespace bm64 {

// ---- double-double arithmetic at compile time (Dekker 1971, Knuth) ----------
struct DD {
  double h, l;
};
__host__ __device__ constexpr DD two_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return DD{s, (a - (s - t)) + (b - t)};
}
__host__ __device__ constexpr DD quick(double a, double b) {
  const double s = a + b;
  return DD{s, b - (s - a)};
}
__host__ __device__ constexpr DD add(DD a, DD b) {
  const DD s = two_sum(a.h, b.h);
  return quick(s.h, s.l + (a.l + b.l));
}
__host__ __device__ constexpr DD two_prod(double a, double b) {
  const double A = 134217729.0 * a, B = 134217729.0 * b;
  const double ah = A - (A - a), bh = B - (B - b), al = a - ah, bl = b - bh;
  const double p = a * b;
  return DD{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
__host__ __device__ constexpr DD mul(DD a, DD b) {
  const DD p = two_prod(a.h, b.h);
  return quick(p.h, p.l + (a.h * b.l + a.l * b.h));
}
__host__ __device__ constexpr DD neg(DD a) { return DD{-a.h, -a.l}; }
__host__ __device__ constexpr DD div(DD a, double b) {
  const double q = a.h / b;
  const DD r = add(a, neg(two_prod(q, b)));
  return quick(q, r.h / b);
}

inline constexpr DD kPi{3.141592653589793116, 1.2246467991473532072e-16};
inline constexpr DD kLn2{0.69314718055994528623, 2.3190468138462995584e-17};

constexpr int kLogCells = 1024, kBase = 2048, kFine = 1024;
constexpr double kScale = 72057594037927936.0;  // 2^56, the fixed point of -2 ln u
// u0 >= 1/2: log cells from which 9 more bits are kept instead of 6 (u0 > 15/16:
// -2 ln u0 < 2^-2.9), and from which the series is taken (u0 > 1 - 2^-11)
constexpr int kFineCell = 896, kSeriesCell = 1023;
__host__ __device__ constexpr int more_bits(int j) { return j >= kFineCell ? 9 : 6; }

// C of log cell j (M / 2^24 in [1 + j/1024, 1 + (j+1)/1024)); the last cell
// takes exactly 1/2, so that the terms cancel next to u0 = 1.
__host__ __device__ constexpr int64_t cell_c(int j) {
  return j == kLogCells - 1 ? 8192 : (static_cast<int64_t>(16384) * 2048 + (2049 + 2 * j) / 2) / (2049 + 2 * j);
}
__host__ __device__ constexpr int64_t to_fixed(DD a, int more = 0) {  // a 2^(56 + more), rounded once
  const double scale = kScale * static_cast<double>(1 << more), h = a.h * scale;
  const double l = a.l * scale + (h - static_cast<double>(static_cast<int64_t>(h)));
  return static_cast<int64_t>(h) + static_cast<int64_t>(l + (l < 0 ? -0.5 : 0.5));
}
inline constexpr int64_t kTwoLn2 = to_fixed(DD{2 * kLn2.h, 2 * kLn2.l});
// what 2 ln 2 has beyond kTwoLn2 in 6 more bits
inline constexpr int kTwoLn2More = static_cast<int>(to_fixed(DD{2 * kLn2.h, 2 * kLn2.l}, 6) - (kTwoLn2 << 6));

struct alignas(16) LogCell {
  int64_t a;  // 2 ln(C 2^-14) 2^56
  uint32_t c;
  int32_t more;  // u0 >= 1/2: what 2 ln 2 + 2 ln(C 2^-14) has beyond (kTwoLn2 + a) in more_bits
};
struct alignas(16) CosSin {
  double c, s;
};
struct Tables {
  LogCell log[kLogCells];
  CosSin base[kBase + 1];  // 2^-28 (cos, sin) of a pi / 4096
  CosSin low[kBase + 1];   // what they are beyond FP64
  CosSin fine[kFine];  // (cos - 1, sin) of (2 k + 1) 2 pi 2^-25
};

// cos and sin of a small angle by Taylor's series.
__host__ __device__ constexpr DD series(DD x, bool sine) {
  const DD x2 = mul(x, x);
  DD term = sine ? x : DD{1.0, 0.0}, sum = term;
  for (int k = sine ? 2 : 1; k < 16; k += 2) {
    term = neg(div(mul(term, x2), static_cast<double>(k) * (k + 1)));
    sum = add(sum, term);
  }
  return sum;
}
__host__ __device__ constexpr Tables make_tables() {
  Tables T{};
  // 2 ln(C 2^-14) upwards from ln(1/2): ln(C'/C) = 2 atanh((C' - C)/(C' + C))
  DD L = neg(kLn2);
  for (int j = kLogCells - 1; j >= 0; --j) {
    if (j < kLogCells - 1) {
      const double d = static_cast<double>(cell_c(j) - cell_c(j + 1)), s = static_cast<double>(cell_c(j) + cell_c(j + 1));
      const DD x = div(DD{d, 0.0}, s), x2 = mul(x, x);
      DD p = x, at = x;
      for (int k = 3; k <= 11; k += 2) {
        p = mul(p, x2);
        at = add(at, div(p, static_cast<double>(k)));
      }
      L = add(L, add(at, at));
    }
    const int64_t a = j == kLogCells - 1 ? -kTwoLn2 : to_fixed(DD{2 * L.h, 2 * L.l});
    const DD whole = add(DD{2 * L.h, 2 * L.l}, DD{2 * kLn2.h, 2 * kLn2.l});
    const int64_t more = to_fixed(whole, more_bits(j)) - (kTwoLn2 + a) * (int64_t(1) << more_bits(j));
    T.log[j] = LogCell{a, static_cast<uint32_t>(cell_c(j)), static_cast<int32_t>(more)};
  }
  // base angles by rotation by pi / 4096
  const DD d{kPi.h / 4096.0, kPi.l / 4096.0};
  DD c{1.0, 0.0}, s{0.0, 0.0};
  const DD dc = series(d, false), ds = series(d, true);
  for (int a = 0; a < kBase; ++a) {
    T.base[a] = CosSin{c.h * 3.7252902984619140625e-09, s.h * 3.7252902984619140625e-09};
    T.low[a] = CosSin{c.l * 3.7252902984619140625e-09, s.l * 3.7252902984619140625e-09};
    const DD c2 = add(mul(c, dc), neg(mul(s, ds))), s2 = add(mul(s, dc), mul(c, ds));
    c = c2;
    s = s2;
  }
  T.base[kBase] = CosSin{0.0, 3.7252902984619140625e-09};
  T.low[kBase] = CosSin{0.0, 0.0};
  // fine angles likewise, from 2 pi 2^-25 by 2 pi 2^-24; cos - 1 = -2 sin^2(x/2)
  for (int k = 0; k < kFine; ++k) {
    const double n = 2.0 * k + 1.0, u = 1.0 / 16777216.0;
    DD x = mul(kPi, DD{n * u, 0.0});  // the angle
    DD half{x.h * 0.5, x.l * 0.5};
    const DD x2 = mul(x, x), y2 = mul(half, half);
    DD sx = x, t = x, sh = half, v = half;
    for (int j = 2; j <= 6; j += 2) {
      t = neg(div(mul(t, x2), static_cast<double>(j) * (j + 1)));
      sx = add(sx, t);
      v = neg(div(mul(v, y2), static_cast<double>(j) * (j + 1)));
      sh = add(sh, v);
    }
    const DD q = mul(sh, sh);
    T.fine[k] = CosSin{-2.0 * q.h, sx.h};
  }
  return T;
}

// 1/sqrt(x) to about 2^-20: the special-function unit's instruction on the
// device, FP32 on the host (unit tests of this header only).
__host__ __device__ __forceinline__ double rsqrt_seed(double x) {
#ifdef __CUDA_ARCH__
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
#else
  return 1.0f / ::sqrtf(static_cast<float>(x));
#endif
}
__host__ __device__ __forceinline__ double fma64(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return __fma_rn(a, b, c);
#else
  return ::fma(a, b, c);
#endif
}
__host__ __device__ __forceinline__ int leading_zeros(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __clz(static_cast<int>(x));
#else
  return __builtin_clz(x);
#endif
}
__host__ __device__ __forceinline__ double add_hi(double x, int32_t hi) {  // adds to the high word
#ifdef __CUDA_ARCH__
  return __hiloint2double(__double2hiint(x) + hi, __double2loint(x));
#else
  int64_t u;
  __builtin_memcpy(&u, &x, 8);
  u += static_cast<int64_t>(static_cast<uint64_t>(static_cast<uint32_t>(hi)) << 32);
  __builtin_memcpy(&x, &u, 8);
  return x;
#endif
}

// sqrt(x) from the seed by Goldschmidt's iteration (1964), for x in [2^-900,
// 2^900]: g -> sqrt(x) and h -> 1 / (2 sqrt(x)) to about 2^-39 in one step, then
// the correction h (x - g^2), of an exact remainder, added with one rounding.
// What is added is off by less than 2^-78 of g, so the result is the nearest
// number but for one argument in about 2^25.  Five dependent FP64 operations,
// about three fewer than the general square root (each some 50 clocks on the
// small lattices' chain).
__host__ __device__ __forceinline__ double sqrt_seeded(double x) {
  const double y = rsqrt_seed(x), h = add_hi(y, -(1 << 20));  // y / 2
  const double g = x * y, r = fma64(-g, h, 0.5);
  const double g1 = fma64(g, r, g), h1 = fma64(h, r, h);
  return fma64(fma64(-g1, g1, x), h1, g1);
}
#ifdef __CUDACC__
// sqrt(x) for any x.
__device__ __forceinline__ double sqrt_any(double x) {
  const int hi = __double2hiint(x);  // the sign and exponent: 1023 - 900 .. 1023 + 900
  return hi >= (123 << 20) && hi < (1923 << 20) ? sqrt_seeded(x) : ::sqrt(x);
}
#endif
__host__ __device__ __forceinline__ uint32_t mul_high(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return static_cast<uint32_t>((static_cast<uint64_t>(a) * b) >> 32);
#endif
}

// 2^56 (-2 ln u0), u0 = ((r >> 8) + 1/2) 2^-24, to half a unit in the last
// place and a quarter of one.
__host__ __device__ __forceinline__ double log28(uint32_t r, const Tables &T) {
  const uint32_t K = (r >> 7) | 1u;  // u0 2^25
  const int nz = leading_zeros(K);   // 31 - e, e = floor(log2 K): 7 .. 31
  const uint32_t M = K << (nz - 7);  // in [2^24, 2^25)
  const int j = static_cast<int>((M >> 14) & (kLogCells - 1));
  if (nz == 7 && j >= kSeriesCell) {
    // -2 ln(1 - e) = 2 e + 2 e^2 (1/2 + e/3 + ...), e < 2^-11: the first term
    // exact, the rest added with one rounding
    const double n = static_cast<double>((1u << 25) - K);
    const double e = n * 2.98023223876953125e-08, e2 = n * 4294967296.0;  // n 2^-25, 2^56 2 e
    const double p = fma64(e, fma64(e, fma64(e, fma64(e, 1.0 / 6, 0.2), 0.25), 1.0 / 3), 0.5);
    return fma64(e2 * e, p, e2);
  }
  const LogCell cell = T.log[j];
  const int sh = nz == 7 ? more_bits(j) : 1;  // X has 56 + sh bits after the point
  // (25 - e) 2 ln 2 + 2 ln c; below u0 = 1/2 what it has beyond 56 bits goes into the one more bit
  const int beyond = (cell.more >> (more_bits(j) - 6)) + (nz - 7) * kTwoLn2More;
  const int64_t A = ((static_cast<int64_t>(nz - 6) * kTwoLn2 + cell.a) << sh) +
                    (nz == 7 ? cell.more : (beyond + 16) >> 5);
  // -2 ln(1 + r) with 65 bits, then with 56 + sh
  const int32_t ri = static_cast<int32_t>(M * cell.c);                             // r 2^38
  const float rf = static_cast<float>(ri) * 3.637978807091713e-12f, rf2 = rf * rf;
  const float tail = rf2 * rf2 * (0.5f - 0.4f * rf) * 3.6893488147419103e19f;
  const int64_t r2 = static_cast<int64_t>(ri) * ri;                                // 2^-76
  const uint32_t q = mul_high(static_cast<uint32_t>(r2 >> 23), 0xAAAAAAABu);       // (2/3) r^2, 2^-53
  const int64_t r3 = static_cast<int64_t>(ri) * static_cast<int64_t>(q);           // (2/3) r^3, 2^-91
  int64_t Y = ((r2 + (1 << 10)) >> 11) - (static_cast<int64_t>(ri) << 28) - ((r3 + (1 << 25)) >> 26);
#ifdef __CUDA_ARCH__
  Y += __float2int_rn(tail);
  const int64_t X = A + ((Y + ((1 << (9 - sh)) >> 1)) >> (9 - sh));
  return add_hi(__ll2double_rn(X), -(sh << 20));
#else
  Y += static_cast<int64_t>(::rintf(tail));
  const int64_t X = A + ((Y + ((1 << (9 - sh)) >> 1)) >> (9 - sh));
  return add_hi(static_cast<double>(X), -(sh << 20));
#endif
}

// 2^28 sqrt(-2 ln u0).
__host__ __device__ __forceinline__ double radius28(uint32_t r, const Tables &T) { return sqrt_seeded(log28(r, T)); }

// 2^-28 (cos, sin) of 2 pi u1, u1 = ((r >> 8) + 1/2) 2^-24.
__host__ __device__ __forceinline__ CosSin angle28(uint32_t r, const Tables &T) {
  const uint32_t K = (r >> 7) | 1u;
  const uint32_t m = K & 0x7fffffu, a = (m + 2048u) >> 12;  // in the quadrant; the nearest base angle, 0 .. 2048
  const int b = static_cast<int>(m) - static_cast<int>(a << 12);  // odd, -2047 .. 2047
  const CosSin A = T.base[a];
  const CosSin B = T.fine[(b < 0 ? -b : b) >> 1];
  const double sb = add_hi(B.s, b < 0 ? static_cast<int32_t>(0x80000000u) : 0);  // odd in b (B.s > 0)
  // the small part first, with what the base is beyond FP64, so that the result
  // is rounded about once
  const CosSin low = T.low[a];
  const double c = A.c + fma64(A.c, B.c, fma64(-A.s, sb, low.c));
  const double s = A.s + fma64(A.s, B.c, fma64(A.c, sb, low.s));
  // the quadrant: (c, s), (-s, c), (-c, -s), (s, -c)
  const uint32_t q = K >> 23;
  CosSin out;
  out.c = (q & 1u) ? s : c;
  out.s = (q & 1u) ? c : s;
  // a sign flip adds 2^31 to the high word modulo 2^32
  out.c = add_hi(out.c, (q == 1u || q == 2u) ? static_cast<int32_t>(0x80000000u) : 0);
  out.s = add_hi(out.s, (q & 2u) ? static_cast<int32_t>(0x80000000u) : 0);
  return out;
}

__host__ __device__ __forceinline__ void pair(uint32_t r0, uint32_t r1, const Tables &T, double &z0, double &z1) {
  const double rad = radius28(r0, T);
  const CosSin a = angle28(r1, T);
  z0 = rad * a.c;
  z1 = rad * a.s;
}

#ifdef __CUDACC__
static __device__ const Tables kTables = make_tables();
#endif

}  // namespace bm64
}  // namespace lbfd
