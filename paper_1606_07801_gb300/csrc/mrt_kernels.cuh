// Multiple-relaxation-time collision and lattices with run-time tables.
//
// The paper relaxes each moment with its own time (Sec. III: the isotropic
// collision matrix is diag(tau^rho, tau^j, tau^j, tau^n, tau^s) in moment
// space for D2Q5) and gives each non-conserved moment the noise variance
// rho (2 tau^a - 1) / (tau^a)^2 (eqs. xiglobal, xilocal).  Per site:
//   M^a   = sum_i m_i^a f_i                      (a >= 1; M^0 = rho)
//   M^a*  = (1 - 1/tau^a) M^a + sqrt(rho_n) amp_a z^a,  amp_a^2 = (2 tau^a - 1)/(tau^a)^2
//   f*_i  = w_i rho + w_i sum_{a>=1} m_i^a M^a*    (i >= 1; n_i^a = m_i^a w_i)
//   f*_0  = rho - sum_{i>=1} f*_i                  (mass conservation)
// The basis and weights are compiled in for D1Q3, D2Q9 and D3Q19; D2Q5, whose
// weights w_0 = 1 - 2 theta, w_1..4 = theta/2 depend on theta (Sec. II), takes
// its few distinct entries from the kernel arguments.  The forward transform
// uses the basis' symmetry (the D2Q9 product form; for D3Q19 the even rows on
// f_i + f_-i, the odd ones on f_i - f_-i), the back transform is the noise
// transform of the single-relaxation kernels, and the pull, the noise keys,
// the paired form and the store are theirs too, as are the dependent launch,
// the alternating sweep and the resident kernel for small lattices.
//
// What bounds it: the FMA pipe (D3Q19 FP32: both transforms and the noise, 73%
// busy) and, for small lattices, the resident kernel's chain.  Measured on
// GB300, microseconds per step, against dense transforms launched plainly:
// D3Q19 FP32 128 x 120 x 96 55.3 -> 39.9 (0.83 of the copy bandwidth on its 224
// MB), D2Q9 1024^2 18.5 -> 12.6, D2Q5 2048^2 32.8 -> 25.7, and D2Q5 81^2,
// resident, 4.1 -> 0.66.
#pragma once

#include "step_kernels.cuh"

namespace lbfd {

template <typename R, int Q>
struct MrtParams {
  R omega[Q];  // 1 - 1/tau^a for a >= 1
  R amp[Q];    // sqrt((2 tau^a - 1) / (tau^a)^2) for a >= 1
  // D2Q5: m^1 of v = (1, 0), m^2 of (0, 1), m^3 of (1, 0), m^4 of 0 and of (1, 0); the weight of i >= 1
  R m1, m2, m3, m40, m41, w;
};

// M^a = sum_i m_i^a f_i into M[a - 1] for a >= 1.
template <int LAT, typename R, typename V>
__device__ __forceinline__ void mrt_forward(const V (&f)[Lattice<LAT>::Q], V (&M)[Lattice<LAT>::Q - 1],
                                            const MrtParams<R, Lattice<LAT>::Q> &p) {
  constexpr int Q = Lattice<LAT>::Q;
  if constexpr (LAT == kD2Q5) {
    const V sx = add_rn(f[1], f[2]), sy = add_rn(f[3], f[4]);
    M[0] = mul_rn(splat<V>(p.m1), sub_rn(f[1], f[2]));
    M[1] = mul_rn(splat<V>(p.m2), sub_rn(f[3], f[4]));
    M[2] = mul_rn(splat<V>(p.m3), sub_rn(sx, sy));
    M[3] = fma_rn(splat<V>(p.m41), add_rn(sx, sy), mul_rn(splat<V>(p.m40), f[0]));
  } else if constexpr (LAT == kD3Q19) {
    V e[Q], o[Q];  // of the first velocity of each pair (i, -i)
    static_for<Q>([&](auto I) {
      constexpr int i = decltype(I)::value, ip = partner<LAT>(i);
      if constexpr (i < ip) {
        e[i] = add_rn(f[i], f[ip]);
        o[i] = sub_rn(f[i], f[ip]);
      }
    });
    static_for<Q - 1>([&](auto A) {
      constexpr int a = decltype(A)::value + 1;
      V acc = splat<V>(R(0));
      bool first = true;
      static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value, ip = partner<LAT>(i);
        constexpr double c = kBasis<LAT, a, i>;
        if constexpr (i <= ip && c != 0.0) {
          const V x = i == ip ? f[i] : (row_parity<LAT>(a) ? o[i] : e[i]);
          acc = first ? mul_rn(cst<V>(c), x) : fma_rn(cst<V>(c), x, acc);
          first = false;
        }
      });
      M[a - 1] = acc;
    });
  } else {
    // one axis of the product basis: (f_0, f_+, f_-) to (mu^0, mu^1, mu^2);
    // products: the inputs are products
    auto axis = [](auto products, const V &f0, const V &fp, const V &fm, V &m0, V &m1, V &m2) {
      constexpr bool apart = decltype(products)::value;
      const V s = apart ? add_apart(fp, fm) : add_rn(fp, fm);
      m0 = apart ? add_apart(f0, s) : add_rn(f0, s);
      m1 = mul_rn(cst<V>(kSqrt3), apart ? sub_apart(fp, fm) : sub_rn(fp, fm));
      m2 = fma_rn(cst<V>(kSqrt2), s, mul_rn(cst<V>(-kInvSqrt2), f0));
    };
    constexpr std::false_type sums{};
    constexpr std::true_type products{};
    if constexpr (LAT == kD1Q3) {
      V m0;
      axis(sums, f[0], f[1], f[2], m0, M[0], M[1]);
    } else {
      V G[3][3];  // [cx][q]
      axis(sums, f[0], f[2], f[4], G[0][0], G[0][1], G[0][2]);
      axis(sums, f[1], f[5], f[8], G[1][0], G[1][1], G[1][2]);
      axis(sums, f[3], f[6], f[7], G[2][0], G[2][1], G[2][2]);
      V m00;
      axis(sums, G[0][0], G[1][0], G[2][0], m00, M[2], M[5]);
      axis(products, G[0][1], G[1][1], G[2][1], M[0], M[3], M[6]);
      axis(sums, G[0][2], G[1][2], G[2][2], M[1], M[4], M[7]);
    }
  }
}

// The update given the site's variates z(a - 1).
template <int LAT, typename R, int NOISE, typename V, class ZF>
__device__ __forceinline__ void mrt_given(V (&f)[Lattice<LAT>::Q], const ZF &z, const StepArgs &a,
                                          const MrtParams<R, Lattice<LAT>::Q> &p) {
  using L = Lattice<LAT>;
  constexpr int Q = L::Q;
  V rho = f[0];
  static_for<Q - 1>([&](auto I) { rho = add_rn(rho, f[decltype(I)::value + 1]); });
  V M[Q - 1];
  mrt_forward<LAT, R>(f, M, p);
  // relaxation and noise, moment by moment
  if constexpr (NOISE != kStepNoiseOff) {
    const V rho_eq = splat<V>(step_param<R>(a.rho_eq, a.rho_eq_f));
    const V rho_n = a.noise_mode == kNoiseLocal ? positive_part(rho) : rho_eq;
    const V sr = noise_amplitude<V>(rho_n);
    static_for<Q - 1>([&](auto A) {
      constexpr int k = decltype(A)::value;
      M[k] = fma_rn(splat<V>(p.omega[k + 1]), M[k], mul_rn(mul_rn(sr, splat<V>(p.amp[k + 1])), z(k)));
    });
  } else {
    static_for<Q - 1>([&](auto A) {
      constexpr int k = decltype(A)::value;
      M[k] = mul_rn(splat<V>(p.omega[k + 1]), M[k]);
    });
  }
  // back transform, the weighted density added last with one rounding (a sum
  // of the density and the moments, weighted after it, rounds at the density's
  // size: its bias over hundreds of steps was several times the error of a
  // step); the rest population from mass conservation
  V moved = splat<V>(R(0));
  auto keep = [&](int i, const V &x) {
    f[i] = x;
    moved = i == 1 ? x : add_rn(moved, x);
  };
  if constexpr (LAT == kD2Q5) {
    const V w = splat<V>(p.w), wr = mul_rn(w, rho), e = mul_rn(splat<V>(p.m41), M[3]);
    const V ex = fma_rn(splat<V>(p.m3), M[2], e), ey = fma_rn(splat<V>(-p.m3), M[2], e);
    keep(1, fma_rn(w, fma_rn(splat<V>(p.m1), M[0], ex), wr));
    keep(2, fma_rn(w, fma_rn(splat<V>(-p.m1), M[0], ex), wr));
    keep(3, fma_rn(w, fma_rn(splat<V>(p.m2), M[1], ey), wr));
    keep(4, fma_rn(w, fma_rn(splat<V>(-p.m2), M[1], ey), wr));
  } else {
    V T[Q];
    NoiseTransform<LAT, R>::apply(M, T);
    static_for<Q - 1>([&](auto I) {
      constexpr int i = decltype(I)::value + 1;
      const V w = cst<V>(L::w(i));
      if constexpr (NoiseTransform<LAT, R>::kWeighted)
        keep(i, fma_rn(w, rho, T[i]));
      else
        keep(i, fma_rn(w, T[i], mul_rn(w, rho)));
    });
  }
  f[0] = sub_rn(rho, moved);
}

// The moment-space collision as a function object, with the interface of
// SrtCollide.
template <int LAT, typename R, int NOISE>
struct MrtCollide {
  static constexpr int Q = Lattice<LAT>::Q;
  static constexpr bool kPairs = std::is_same<R, float>::value;
  static constexpr int kAhead = Q - 1, kNoise = NOISE;
  MrtParams<R, Q> p;
  template <typename V>
  __device__ __forceinline__ void ahead(V (&z)[kAhead], uint32_t s, const PhiloxStep &ph, uint32_t apart = 1u) const {
    if constexpr (NOISE != kStepNoiseOff) {
      if constexpr (LaneOf<V>::kLanes == 2)
        draw_variates_pair<Q - 1, NOISE == kStepNoiseGauss>(z, s, ph, apart);
      else
        draw_variates_t<R, Q - 1, NOISE == kStepNoiseGauss>(z, s, ph);
    }
  }
  __device__ __forceinline__ void shape(R (&t)[kAhead], const R (&z)[kAhead]) const {
#pragma unroll
    for (int k = 0; k < kAhead; ++k) t[k] = z[k];
  }
  template <typename V, class ZF>
  __device__ __forceinline__ void given(V (&f)[Q], const ZF &z, const StepArgs &a) const {
    mrt_given<LAT, R, NOISE>(f, z, a, p);
  }
  template <typename V>
  __device__ __forceinline__ void whole(V (&f)[Q], uint32_t s, const StepArgs &a) const {
    V z[kAhead];
    ahead(z, s, a.ph);
    given(f, [&](int k) -> V { return z[k]; }, a);
  }
  __device__ __forceinline__ void operator()(R (&f)[Q], uint32_t s, const StepArgs &a) const { whole(f, s, a); }
  __device__ __forceinline__ void pair(R (&fa)[Q], R (&fb)[Q], uint32_t s, const StepArgs &a) const {
    if constexpr (kPairs) {
      float2 f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = make_float2(fa[i], fb[i]);
      whole(f, s, a);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        fa[i] = f[i].x;
        fb[i] = f[i].y;
      }
    }
  }
};

template <int LAT, typename S, int VX, int NOISE>
__global__ void __launch_bounds__(128, 2 * step_min_blocks<LAT, S, VX>())
    k_step_mrt(const S *src, S *dst, const StepArgs a,
               const MrtCollide<LAT, typename Store<S>::R, NOISE> c) {
  using C = MrtCollide<LAT, typename Store<S>::R, NOISE>;
  pdl_launch_dependents();
  const uint3 b = sweep_block(a.sweep);
  const int x0 = (b.x * blockDim.x + threadIdx.x) * VX;
  const int y = b.y * blockDim.y + threadIdx.y;
  const int z = b.z;
  pdl_wait();
  if (x0 >= a.Lx || y >= a.Ly) return;
  // value offsets fit 32 bits (checked by the API)
  step_vec_body<LAT, S, VX, NOISE, C, uint32_t>(src, dst, a, x0, y, z, c);
}

// Calls go(c) with the collision of a lattice and precision: m (Q*Q, [a][i])
// and w (Q) are the basis and weights (read for D2Q5, whose are not compiled
// in), tau holds tau^a for a = 0..Q-1 (entry 0 unused).
template <int LAT, typename S, class F>
cudaError_t mrt_collide_t(const StepArgs &a, const double *m, const double *w, const double *tau, F &&go) {
  using R = typename Store<S>::R;
  constexpr int Q = Lattice<LAT>::Q;
  MrtParams<R, Q> p{};
  for (int b = 1; b < Q; ++b) {
    p.omega[b] = static_cast<R>(1.0 - 1.0 / tau[b]);
    p.amp[b] = static_cast<R>(std::sqrt((2.0 * tau[b] - 1.0) / (tau[b] * tau[b])));
  }
  if constexpr (LAT == kD2Q5) {
    p.m1 = static_cast<R>(m[1 * Q + 1]);
    p.m2 = static_cast<R>(m[2 * Q + 3]);
    p.m3 = static_cast<R>(m[3 * Q + 1]);
    p.m40 = static_cast<R>(m[4 * Q + 0]);
    p.m41 = static_cast<R>(m[4 * Q + 1]);
    p.w = static_cast<R>(w[1]);
  }
  if (a.noise_mode == kNoiseOff) return go(MrtCollide<LAT, R, kStepNoiseOff>{p});
  if (a.noise_dist == kGaussian) return go(MrtCollide<LAT, R, kStepNoiseGauss>{p});
  return go(MrtCollide<LAT, R, kStepNoiseFlat>{p});
}

// One step of one lattice and storage type (FP32 or FP64).
template <int LAT, typename S>
cudaError_t step_mrt_t(const void *src, void *dst, const StepArgs &a, const double *m, const double *w,
                       const double *tau, cudaStream_t stream) {
  constexpr int precision = sizeof(S) == 8 ? kStoreF64 : kStoreF32;
  return mrt_collide_t<LAT, S>(a, m, w, tau, [&](auto c) -> cudaError_t {
    using C = decltype(c);
    constexpr int NOISE = C::kNoise;
    const int vx = step_vec_width(LAT, precision, a.Lx, a.N, vec_most(src, dst, sizeof(S)));
    dim3 grid, block;
    step_shape(a.Lx, a.Ly, a.Lz, grid, block, vx, std::min(step_threads(LAT, precision), 128));
    StepLaunch launch(grid, block, stream);
    const S *s = static_cast<const S *>(src);
    S *d = static_cast<S *>(dst);
    if (vx == 1) return cudaLaunchKernelEx(&launch.cfg, k_step<LAT, S, NOISE, uint32_t, C>, s, d, a, c);
    if constexpr (sizeof(S) == 4) {
      if constexpr (NOISE != kStepNoiseOff)
        if (vx == 2) return cudaLaunchKernelEx(&launch.cfg, k_step_ahead<LAT, S, 2, NOISE, uint32_t, C>, s, d, a, c);
      if (vx == 4) return cudaLaunchKernelEx(&launch.cfg, k_step_mrt<LAT, S, 4, NOISE>, s, d, a, c);
    }
    if constexpr (sizeof(S) == 8 || NOISE == kStepNoiseOff)
      return cudaLaunchKernelEx(&launch.cfg, k_step_mrt<LAT, S, 2, NOISE>, s, d, a, c);
    else
      return cudaErrorInvalidValue;  // (the widths are 1, 2 and 4)
  });
}

}  // namespace lbfd
