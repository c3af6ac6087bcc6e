// Many steps of a small lattice in one launch, its two population buffers
// resident in shared memory (see step_small.cu for the rule that sends a
// lattice here).  One CTA holds the lattice, or a thread-block cluster does:
// CTA r owns sites [r chunk, (r + 1) chunk) and keeps that slice of both
// buffers in its own shared memory; a site's pull reads each neighbour from
// the CTA that owns it (distributed shared memory), and one barrier separates
// the steps.
//
// What bounds it is the dependent chain of one step on a few SMs, not bytes
// (the state never leaves the chip).  So every thread has one site, and what
// does not depend on the state is taken off the chain:
//   - the site's Q neighbour addresses are formed once per launch;
//   - the noise of the next step, which depends on the site and the step
//     alone, is drawn between the barrier's arrival and its wait;
//   - each thread advances the step's Philox words itself;
//   - where the threads allow, the variates are drawn by threads of their own,
//     one per site and Philox call, two steps ahead (SPLIT): D1Q3 FP64 256
//     sites 2.25 -> 1.35 us per step (1.48 with the present FP64 pairs), D2Q9
//     FP64 24 x 20 5.23 -> 2.67, D2Q9 FP32 64 x 48 0.85 -> 0.69, D3Q19 FP32 6^3
//     1.05 -> 0.76.
// Measured on GB300, microseconds per step, against several sites per thread
// on as few CTAs as hold the state, with addresses, noise and divisions on
// the chain: D2Q9 FP32 64 x 48 5.77 -> 0.83, 100 x 100 9.42 -> 1.21, D3Q19
// FP32 16^3 8.24 -> 1.37, D1Q3 FP64 256 sites 2.75 -> 2.26.
#pragma once

#include <algorithm>
#include <cuda_runtime.h>

#include "fastdiv.cuh"
#include "step_kernels.cuh"

namespace lbfd {

constexpr int kResidentCtas = 16;  // CTAs of a cluster at most (above 8: opt-in)
// Threads of a CTA at most, by the registers of the update (FP64: by its
// narrow pipe).
__host__ __device__ constexpr int resident_threads(int lattice, bool f64) {
  return f64 ? 128 : (lattice == kD3Q19 ? 576 : 1024);
}

// Threads of a CTA at most where noise threads draw the variates (SPLIT), by
// the registers of the update; a site takes 1 + split_calls threads.
__host__ __device__ constexpr int split_calls(int lattice) {
  return lattice == kD3Q19 ? 5 : (lattice == kD2Q9 ? 2 : 1);
}
// (more noise threads than that slow the barrier and the updates down: D2Q5
// 81 x 81, 832 threads, 0.77 against 0.72 us per step without them)
__host__ __device__ constexpr int split_threads(int lattice, bool f64) {
  return f64 || lattice == kD3Q19 ? 512 : 640;
}

// The launch bound that goes with it: at most 64 registers measured faster
// than the 102 that 640 threads allow (D2Q9 FP32 64 x 48 0.72 against 0.80 us).
__host__ __device__ constexpr int split_bound(int lattice, bool f64) {
  return f64 || lattice == kD3Q19 ? 512 : 1024;
}

// What the kernel needs besides the step arguments.
struct ResidentArgs {
  uint32_t lattice_id;
  int32_t nsteps, chunk;
  int32_t sites;     // SPLIT: threads that update (chunk rounded up to warps)
  uint32_t noise_at;  // SPLIT: byte offset of the variates in shared memory
  uint64_t t0;
  FastDiv div_x, div_y, div_chunk;
};

// The stored value at a shared-memory address, of this CTA or of a CTA of
// its cluster.
template <bool CL, typename S>
__device__ __forceinline__ S ld_resident(uint32_t addr) {
  S v;
  if constexpr (sizeof(S) == 8) {
    double u;
    if constexpr (CL)
      asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(u) : "r"(addr) : "memory");
    else
      asm volatile("ld.shared.f64 %0, [%1];" : "=d"(u) : "r"(addr) : "memory");
    v = u;
  } else if constexpr (sizeof(S) == 4) {
    float u;
    if constexpr (CL)
      asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(u) : "r"(addr) : "memory");
    else
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(u) : "r"(addr) : "memory");
    v = u;
  } else {
    unsigned short u;
    if constexpr (CL)
      asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(u) : "r"(addr) : "memory");
    else
      asm volatile("ld.shared.u16 %0, [%1];" : "=h"(u) : "r"(addr) : "memory");
    v = *reinterpret_cast<const S *>(&u);
  }
  return v;
}

// Address of local address `addr` in CTA `rank` of the cluster.
template <bool CL>
__device__ __forceinline__ uint32_t resident_of(uint32_t addr, uint32_t rank) {
  if constexpr (CL) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
  } else {
    return addr;
  }
}
template <bool CL>
__device__ __forceinline__ void resident_arrive() {
  if constexpr (CL) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
template <bool CL>
__device__ __forceinline__ void resident_wait() {
  if constexpr (CL)
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  else
    // (not __syncthreads(), which all threads have to reach at one place of the
    // program: the noise threads wait in a loop of their own)
    asm volatile("barrier.sync 0;" ::: "memory");
}

// src and dst may be the same buffer (lbfd_step runs an even number of steps
// in place), so neither is __restrict__: every read of src happens before the
// first barrier and every write of dst after it.
template <int LAT, typename S, class C, bool CL, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? split_bound(LAT, sizeof(typename Store<S>::R) == 8)
                                        : resident_threads(LAT, sizeof(typename Store<S>::R) == 8))
    k_step_resident(const S *src, S *dst, const StepArgs a, const ResidentArgs ra, const C collide) {
  using L = Lattice<LAT>;
  using R = typename Store<S>::R;
  constexpr int Q = L::Q;
  extern __shared__ __align__(16) unsigned char resident_smem[];
  const int chunk = ra.chunk, N = static_cast<int>(a.N);
  uint32_t rank = 0;
  if constexpr (CL) asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int s0 = static_cast<int>(rank) * chunk, cnt = max(0, min(chunk, N - s0));
  S *const own = reinterpret_cast<S *>(resident_smem);
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(own));
  const uint32_t flip = static_cast<uint32_t>(Q) * static_cast<uint32_t>(chunk) * sizeof(S);  // to the other buffer
  for (int i = 0; i < Q; ++i)
    for (int l = threadIdx.x; l < cnt; l += blockDim.x) own[i * chunk + l] = src[static_cast<int64_t>(i) * N + s0 + l];

  // SPLIT: the first `sites` threads update a site each, the others draw: call
  // j of site l is thread sites (1 + j) + l, and the variates of three steps
  // rotate through shared memory: while step k is updated, step k + 2 is
  // drawn and step k + 1 shaped
  const int sites = SPLIT ? ra.sites : static_cast<int>(blockDim.x);
  R *const zbuf = reinterpret_cast<R *>(resident_smem + ra.noise_at);
  if constexpr (SPLIT) {
    if (static_cast<int>(threadIdx.x) >= sites) {
      const int n = static_cast<int>(threadIdx.x) - sites, j = n / sites, l = n - j * sites;
      const uint32_t site = static_cast<uint32_t>(s0 + l);
      const uint64_t sp = static_cast<uint64_t>(site) * Philox::M0;
      PhiloxStep ph = a.ph;
      auto draw = [&](int step) {
        if (l >= cnt || step >= ra.nsteps) return;
        philox_step_set_t(ph, ra.lattice_id, ra.t0 + static_cast<uint64_t>(step));
        // (words e[j] = e[0] ^ j, so that j need not be a compile-time index)
        const uint32_t e0 = ph.e[0];
        ph.e[0] = e0 ^ static_cast<uint32_t>(j);
        const uint4 r = philox_site(static_cast<uint32_t>(sp >> 32), static_cast<uint32_t>(sp), ph, 0);
        R *const to = zbuf + ((step % 3) * (Q - 1) + 4 * j) * sites + l;
        R z[4];
        call_variates<R, (Q - 1 < 4 ? Q - 1 : 4), C::kNoise == kStepNoiseGauss>(z, r, 0);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * j + k < Q - 1) to[k * sites] = z[k];
      };
      draw(0);
      draw(1);
      resident_arrive<CL>();
      resident_wait<CL>();
      for (int step = 0; step < ra.nsteps; ++step) {
        draw(step + 2);
        if (!CL && step + 1 == ra.nsteps) break;
        resident_arrive<CL>();
        resident_wait<CL>();
      }
      return;
    }
  }

  // this thread's site, and the address (in the first buffer) of the source
  // of each of its populations
  const int l = static_cast<int>(threadIdx.x);
  const bool mine = l < cnt;
  auto shape = [&](int step, R (&t)[C::kAhead]) {
    R z[Q - 1];
#pragma unroll
    for (int k = 0; k < Q - 1; ++k) z[k] = zbuf[((step % 3) * (Q - 1) + k) * sites + l];
    collide.shape(t, z);
  };
  const uint32_t s = static_cast<uint32_t>(s0 + (mine ? l : 0));
  uint32_t at[Q];
  {
    const uint32_t Lx = static_cast<uint32_t>(a.Lx), Ly = static_cast<uint32_t>(a.Ly);
    const uint32_t r = fastdiv(s, ra.div_x), z = fastdiv(r, ra.div_y);
    const uint32_t x = s - r * Lx, y = r - z * Ly;
    const uint32_t Lxy = Lx * Ly, Lxyz = static_cast<uint32_t>(N);
    // periodic neighbours as offsets from s (modulo 2^32)
    const uint32_t dxm = x == 0 ? Lx - 1u : 0u - 1u, dxp = x + 1u == Lx ? 1u - Lx : 1u;
    const uint32_t dym = y == 0 ? Lxy - Lx : 0u - Lx, dyp = y + 1u == Ly ? Lx - Lxy : Lx;
    const uint32_t dzm = z == 0 ? Lxyz - Lxy : 0u - Lxy;
    const uint32_t dzp = z + 1u == static_cast<uint32_t>(a.Lz) ? Lxy - Lxyz : Lxy;
    static_for<Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      constexpr int vx = L::v(i, 0), vy = L::v(i, 1), vz = L::v(i, 2);
      const uint32_t so = s + (vx == 0 ? 0u : (vx > 0 ? dxm : dxp)) + (vy == 0 ? 0u : (vy > 0 ? dym : dyp)) +
                          (vz == 0 ? 0u : (vz > 0 ? dzm : dzp));
      const uint32_t owner = CL ? fastdiv(so, ra.div_chunk) : 0u;
      const uint32_t lo = so - owner * static_cast<uint32_t>(chunk);
      at[i] = resident_of<CL>(base + (static_cast<uint32_t>(i * chunk) + lo) * static_cast<uint32_t>(sizeof(S)), owner);
    });
  }
  PhiloxStep ph = a.ph;
  R ahead[C::kAhead];
  if (!SPLIT && mine) {
    philox_step_set_t(ph, ra.lattice_id, ra.t0);
    collide.ahead(ahead, s, ph);
  }
  resident_arrive<CL>();
  resident_wait<CL>();  // every slice loaded, the first variates drawn
  if (SPLIT && mine) shape(0, ahead);
  for (int step = 0; step < ra.nsteps; ++step) {
    const uint32_t from = (step & 1) ? flip : 0u;
    S *const to = own + ((step & 1) ? 0 : Q * chunk) + l;
    const bool last = step + 1 == ra.nsteps;
    if (mine) {
      R f[Q];
      static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        f[i] = Store<S>::load(ld_resident<CL, S>(at[i] + from));
      });
      collide.given(f, [&](int k) -> R { return ahead[k]; }, a);
      static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if (last)
          dst[static_cast<int64_t>(i) * N + s] = Store<S>::store(f[i]);
        else
          to[i * chunk] = Store<S>::store(f[i]);
      });
    }
    if (!CL && last) break;
    // the step's writes are visible to the cluster, and its reads done, before
    // the next step's; after the last step no CTA leaves while another reads
    // its slice
    resident_arrive<CL>();
    if (!last && mine) {
      if constexpr (SPLIT) {
        shape(step + 1, ahead);
      } else {
        philox_step_set_t(ph, ra.lattice_id, ra.t0 + static_cast<uint64_t>(step + 1));
        collide.ahead(ahead, s, ph);
      }
    }
    resident_wait<CL>();
  }
}

template <int LAT, typename S, class C, bool CL, bool SPLIT>
cudaError_t resident_launch(const void *src, void *dst, const StepArgs &a, const ResidentArgs &ra, const C &c, int ctas,
                            int threads, size_t bytes, cudaStream_t stream) {
  auto kern = k_step_resident<LAT, S, C, CL, SPLIT>;
  // the opt-ins above 48 KB of dynamic shared memory and above 8 CTAs, on the current device
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmallMaxBytes));
  if (e == cudaSuccess && CL && ctas > 8)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CL ? 1 : 0;
  if (CL) {
    // a cluster that the GPU cannot place is reported, not launched
    int placeable = 0;
    e = cudaOccupancyMaxActiveClusters(&placeable, kern, &cfg);
    if (e != cudaSuccess) return e;
    if (placeable < 1) return cudaErrorNotSupported;
  }
  return cudaLaunchKernelEx(&cfg, kern, static_cast<const S *>(src), static_cast<S *>(dst), a, ra, c);
}

template <int LAT, typename S, class C>
cudaError_t resident_t(const void *src, void *dst, const StepArgs &a, ResidentArgs ra, const C &c, int precision,
                       cudaStream_t stream) {
  using R = typename Store<S>::R;
  constexpr int Q = Lattice<LAT>::Q;
  const int ctas = small_path_ctas(LAT, precision, a.N);
  if (ctas == 0) return cudaErrorInvalidValue;
  ra.chunk = int((a.N + ctas - 1) / ctas);
  ra.div_x = make_fastdiv(uint32_t(a.Lx));
  ra.div_y = make_fastdiv(uint32_t(a.Ly));
  ra.div_chunk = make_fastdiv(uint32_t(ra.chunk));
  const int threads = (ra.chunk + 31) / 32 * 32;
  const size_t state = 2 * size_t(Q) * size_t(ra.chunk) * sizeof(S);
  if constexpr (C::kNoise != kStepNoiseOff) {
    ra.sites = threads;
    ra.noise_at = uint32_t((state + 15) / 16 * 16);
    const size_t bytes = ra.noise_at + 3 * size_t(Q - 1) * size_t(threads) * sizeof(R);
    const int all = threads * (1 + split_calls(LAT));
    if (all <= split_threads(LAT, sizeof(R) == 8) && bytes <= kSmallMaxBytes)
      return ctas > 1 ? resident_launch<LAT, S, C, true, true>(src, dst, a, ra, c, ctas, all, bytes, stream)
                      : resident_launch<LAT, S, C, false, true>(src, dst, a, ra, c, 1, all, bytes, stream);
  }
  return ctas > 1 ? resident_launch<LAT, S, C, true, false>(src, dst, a, ra, c, ctas, threads, state, stream)
                  : resident_launch<LAT, S, C, false, false>(src, dst, a, ra, c, 1, threads, state, stream);
}

}  // namespace lbfd
