// resident.cuh -- many time steps of a small lattice in one launch, the populations kept in
// the shared memory of one thread-block cluster. Included by kernels.cuh.
//
// A step of a lattice of a few thousand nodes is bound by what surrounds it: a launch per
// step, and the round trip of every population through L2, 6.3 us together (4 x 4 x 256
// FP32), of which the arithmetic is a fraction. Here one cluster of up to 16 CTAs holds
// both population arrays in shared memory (38 values per node), each thread keeps one
// node for all steps, reads its 19 pull sources from its own or another CTA's shared
// memory (their addresses are formed once), and a cluster barrier separates the steps.
// The node code is the sweep's, so the bits are.
//
// A cluster has 16 SMs of the chip's 152, so the rule ends where their arithmetic takes
// as long as the launches they replace: RESIDENT_NODES.
#pragma once

namespace lbm {

// Loads and stores of stored values through shared-window addresses (own or remote CTA).
__device__ __forceinline__ double ld_cluster(uint32_t at, double) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ float ld_cluster(uint32_t at, float) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ float ld_cluster(uint32_t at, __half) {
  unsigned short v;
  asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(at) : "memory");
  return __half2float(__ushort_as_half(v));
}
__device__ __forceinline__ uint32_t cluster_address(uint32_t local, uint32_t rank) {
  uint32_t at;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(local), "r"(rank));
  return at;
}
// Hardware barrier over the cluster's threads (release / acquire at cluster scope); every
// CTA of a cluster is resident, so it ends as soon as the slowest arrives.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// `per`: nodes per CTA (the block's threads). SWAPPED state (an AA lattice between step
// pairs): population k lies in slot -k of the global array, at both ends. The new state
// goes to dst.
template <typename S, bool GEOM>
__global__ void __launch_bounds__(RESIDENT_THREADS, 1)
    resident_kernel(const __grid_constant__ SweepArgs a, int steps, bool swapped) {
  using T = typename ComputeOf<S>::T;
  extern __shared__ __align__(16) unsigned char resident_smem[];
  S* const buf = reinterpret_cast<S*>(resident_smem);  // [2][19][per]
  const uint32_t per = blockDim.x, tid = threadIdx.x;
  const uint32_t cell = blockIdx.x * per + tid;
  uint32_t lm = 0;
  if (GEOM && a.links && cell < a.N) lm = __ldg(a.links + cell);
  // solid nodes keep their populations, in both global arrays, and nobody reads them
  const bool active = cell < a.N && !(lm & SOLID_NODE);
  const uint32_t array_bytes = Q * per * uint32_t(sizeof(S));
  uint32_t from[Q];  // shared-window addresses of the pull sources in array 0
  uint32_t x = 0, y = 0, z = 0;
  int code = 0;
  if (active) {
    const uint32_t q1 = fdiv(a.div_nx, cell);
    x = cell - q1 * a.nx;
    z = fdiv(a.div_ny, q1);
    y = q1 - z * a.ny;
    const bool px = a.periodic & 1u, py = a.periodic & 2u, pz = a.periodic & 4u;
    const uint32_t xm = x ? x - 1 : (px ? a.nx - 1 : 0), xp = (x + 1 < a.nx) ? x + 1 : (px ? 0 : a.nx - 1);
    const uint32_t ym = y ? y - 1 : (py ? a.ny - 1 : 0), yp = (y + 1 < a.ny) ? y + 1 : (py ? 0 : a.ny - 1);
    const uint32_t zm = z ? z - 1 : (pz ? a.nz - 1 : 0), zp = (z + 1 < a.nz) ? z + 1 : (pz ? 0 : a.nz - 1);
    const int fx = px ? 0 : (x == 0 ? 1 : (x == a.nx - 1 ? 2 : 0));
    const int fy = py ? 0 : (y == 0 ? 1 : (y == a.ny - 1 ? 2 : 0));
    const int fz = pz ? 0 : (z == 0 ? 1 : (z == a.nz - 1 ? 2 : 0));
    code = fx + 3 * fy + 9 * fz;
    const bool links = GEOM && (lm & ~(RULE_BITS << RULE_SHIFT)) != 0u;
    static_for<0, Q>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      const uint32_t sx = cx(k) > 0 ? xm : (cx(k) < 0 ? xp : x);
      const uint32_t sy = cy(k) > 0 ? ym : (cy(k) < 0 ? yp : y);
      const uint32_t sz = cz(k) > 0 ? zm : (cz(k) < 0 ? zp : z);
      uint32_t source = chk((sz * a.ny + sy) * a.nx + sx, a.N);
      uint32_t slot = k;
      if (links && ((lm >> k) & 1u)) source = cell, slot = opp(k);  // a solid source sends the node's own back
      const uint32_t rank = source / per;
      from[k] = cluster_address(smem_u32(buf + slot * per + (source - rank * per)), rank);
      const S* own = static_cast<const S*>(a.src_pop[swapped ? opp(k) : k]);
      buf[k * per + tid] = own[cell];
    });
  }
  cluster_barrier();
  for (int s = 0; s < steps; ++s) {
    const bool last = s + 1 == steps;
    if (active) {
      const uint32_t array = (s & 1) ? array_bytes : 0u;
      T h[Q];
      auto load = [&](T (&v)[Q]) {
        static_for<0, Q>([&](auto kc) { v[decltype(kc)::value] = ld_cluster(from[decltype(kc)::value] + array, S()); });
      };
      NodeTerms<T> unused;
      update_node<S, false, GEOM>(a, lm, code, x, y, z, cell, load, h, unused);
      if (last) {
        static_for<0, Q>([&](auto kc) {
          constexpr int k = decltype(kc)::value;
          static_cast<S*>(a.dst_pop[swapped ? opp(k) : k])[cell] = Storage<S>::store(h[k]);
        });
      } else {
        S* to = buf + ((s & 1) ? 0u : Q * per) + tid;
        static_for<0, Q>([&](auto kc) { to[decltype(kc)::value * per] = Storage<S>::store(h[decltype(kc)::value]); });
      }
    }
    // separates the steps, and keeps a CTA's shared memory until the last reader is done
    cluster_barrier();
  }
}

template <typename S, bool GEOM>
cudaError_t launch_resident_geom(const SweepArgs& a, int steps, bool swapped, cudaStream_t s) {
  const void* fn = reinterpret_cast<const void*>(resident_kernel<S, GEOM>);
  // as many CTAs as a cluster has, whole warps each
  const uint32_t per = ((a.N + RESIDENT_CTAS - 1) / RESIDENT_CTAS + 31u) / 32u * 32u;
  const uint32_t ctas = (a.N + per - 1) / per;
  const size_t smem = size_t(2) * Q * per * sizeof(S);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(per);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  e = cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg);
  if (e != cudaSuccess || clusters < 1) {
    cudaGetLastError();
    return cudaErrorNotSupported;
  }
  return cudaLaunchKernelEx(&cfg, resident_kernel<S, GEOM>, a, steps, swapped);
}

// `steps` steps from src to dst (which may be the same array); cudaErrorNotSupported where
// the device has no room for the cluster.
template <typename S>
cudaError_t launch_resident_impl(const SweepArgs& a, int steps, bool swapped, cudaStream_t s) {
  if (a.links || a.forced) return launch_resident_geom<S, true>(a, steps, swapped, s);
  return launch_resident_geom<S, false>(a, steps, swapped, s);
}

}  // namespace lbm
