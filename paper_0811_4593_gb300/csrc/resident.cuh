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
// A cluster has 16 SMs of the chip's 152, so it ends where the whole chip between grid
// barriers (below) is as fast: 8,192 nodes, FP64 4,096. Per step, cluster against grid:
// FP32 periodic 8,192 nodes 1.5 against 2.0 us; FP64 4,096 nodes 2.9 against 3.1, 8,192
// nodes 5.1 against 3.2.
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

// Box boundary code of a node: fx + 3 fy + 9 fz as apply_boundary takes it.
__device__ __forceinline__ int boundary_code(const SweepArgs& a, uint32_t x, uint32_t y, uint32_t z) {
  const bool px = a.periodic & 1u, py = a.periodic & 2u, pz = a.periodic & 4u;
  const int fx = px ? 0 : (x == 0 ? 1 : (x == a.nx - 1 ? 2 : 0));
  const int fy = py ? 0 : (y == 0 ? 1 : (y == a.ny - 1 ? 2 : 0));
  const int fz = pz ? 0 : (z == 0 ? 1 : (z == a.nz - 1 ? 2 : 0));
  return fx + 3 * fy + 9 * fz;
}

// Which of a CTA's nodes each of its threads takes (NO_NODE: none). Either in node order,
// or nodes of one closure side by side (each in node order), a new warp for each group
// where the block has the threads. The slowest warp sets the pace of every step, and in
// node order the warps at the ends of a narrow channel run the bodies of an x face, a z
// face and two edges one after the other (4 x 4 x 256 FP32: 1.73 us per step, grouped 1.2).
// Grouped, that is, where some warp has two closures to run, or where fewer closures are
// run without more warps -- unless nx is a multiple of 8: the nodes of an x face then lie
// in the same few banks, which costs more (16 x 16 x 16 FP32 channel: 1.64 against 1.40 us;
// a gap word every 32 spreads them but slows all others). `key`: the group of the thread's
// own node (0: no closure).
constexpr uint32_t NODE_GROUPS = 28, NO_NODE = 0xffffu;
__device__ __forceinline__ uint32_t grouped_node(uint32_t key, uint32_t nx) {
  constexpr uint32_t WARPS = RESIDENT_THREADS / 32;
  __shared__ uint32_t before[NODE_GROUPS][WARPS], start[NODE_GROUPS], count[NODE_GROUPS];
  __shared__ uint32_t bodies[WARPS];
  __shared__ uint16_t order[RESIDENT_THREADS];
  __shared__ bool grouped;
  const uint32_t tid = threadIdx.x, warp = tid >> 5;
  const uint32_t same = __match_any_sync(0xffffffffu, key);
  const uint32_t rank = __popc(same & ((1u << (tid & 31u)) - 1u));
  for (uint32_t i = tid; i < NODE_GROUPS * WARPS; i += blockDim.x) before[i / WARPS][i % WARPS] = 0;
  order[tid] = NO_NODE;
  const uint32_t own = __popc(__ballot_sync(0xffffffffu, rank == 0 && key != 0u && key != NO_NODE));
  const bool used = __any_sync(0xffffffffu, key != NO_NODE);
  if ((tid & 31u) == 0) bodies[warp] = used ? own + 0x10000u : 0u;  // and one warp
  __syncthreads();
  if (key != NO_NODE && rank == 0) before[key][warp] = __popc(same);
  __syncthreads();
  if (tid < NODE_GROUPS) {
    uint32_t sum = 0;
    for (uint32_t w = 0; w < WARPS; ++w) {
      const uint32_t n = before[tid][w];
      before[tid][w] = sum;
      sum += n;
    }
    count[tid] = sum;
  }
  __syncthreads();
  if (tid == 0) {
    uint32_t now = 0, most = 0, whole = 0, next = 0;
    for (uint32_t w = 0; w < blockDim.x / 32u; ++w) {
      now += bodies[w];
      most = most > (bodies[w] & 0xffffu) ? most : bodies[w] & 0xffffu;
    }
    for (uint32_t g = 0; g < NODE_GROUPS; ++g) whole += (count[g] + 31u) / 32u;
    const uint32_t closures = whole - (count[0] + 31u) / 32u;
    grouped = most > 1u || ((nx & 7u) != 0 && closures < (now & 0xffffu) && whole <= now >> 16);
    const uint32_t mask = whole * 32u <= blockDim.x ? 31u : 0u;
    for (uint32_t g = 0; g < NODE_GROUPS; ++g) {
      start[g] = next;
      next += (count[g] + mask) & ~mask;
    }
  }
  __syncthreads();
  if (!grouped) return key != NO_NODE ? tid : NO_NODE;
  if (key != NO_NODE) order[start[key] + before[key][warp] + rank] = uint16_t(tid);
  __syncthreads();
  return order[tid];
}

// `per`: nodes per CTA, at most the block's threads. SWAPPED state (an AA lattice between
// step pairs): population k lies in slot -k of the global array, at both ends. The new
// state goes to dst.
template <typename S, bool GEOM>
__global__ void __launch_bounds__(RESIDENT_THREADS, 1)
    resident_kernel(const __grid_constant__ SweepArgs a, int steps, uint32_t per, bool swapped) {
  using T = typename ComputeOf<S>::T;
  extern __shared__ __align__(16) unsigned char resident_smem[];
  S* const buf = reinterpret_cast<S*>(resident_smem);  // [2][19][per]
  auto place = [&](uint32_t cell, uint32_t& x, uint32_t& y, uint32_t& z) {
    const uint32_t q1 = fdiv(a.div_nx, cell);
    x = cell - q1 * a.nx;
    z = fdiv(a.div_ny, q1);
    y = q1 - z * a.ny;
  };
  uint32_t x = 0, y = 0, z = 0, key = NO_NODE, lm = 0;
  uint32_t cell = blockIdx.x * per + threadIdx.x;
  if (threadIdx.x < per && cell < a.N) {
    place(cell, x, y, z);
    if (GEOM) lm = geometry_word(a, cell);
    const uint32_t c = uint32_t(boundary_code(a, x, y, z));
    // both x faces share a body; solid nodes keep their populations, in both global
    // arrays, and nobody reads them
    key = ((lm >> RULE_SHIFT) & RULE_BITS) ? NODE_GROUPS - 1 : (c == 2u ? 1u : c);
    if (lm & SOLID_NODE) key = NO_NODE;
  }
  const uint32_t node = grouped_node(key, a.nx);
  const bool active = node != NO_NODE;
  const uint32_t array_bytes = Q * per * uint32_t(sizeof(S));
  uint32_t from[Q];  // shared-window addresses of the pull sources in array 0
  int code = 0;
  if (active) {
    cell = blockIdx.x * per + node;
    place(cell, x, y, z);
    lm = GEOM ? geometry_word(a, cell) : 0u;
    code = boundary_code(a, x, y, z);
    const bool px = a.periodic & 1u, py = a.periodic & 2u, pz = a.periodic & 4u;
    const uint32_t xm = x ? x - 1 : (px ? a.nx - 1 : 0), xp = (x + 1 < a.nx) ? x + 1 : (px ? 0 : a.nx - 1);
    const uint32_t ym = y ? y - 1 : (py ? a.ny - 1 : 0), yp = (y + 1 < a.ny) ? y + 1 : (py ? 0 : a.ny - 1);
    const uint32_t zm = z ? z - 1 : (pz ? a.nz - 1 : 0), zp = (z + 1 < a.nz) ? z + 1 : (pz ? 0 : a.nz - 1);
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
      buf[k * per + node] = own[cell];
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
      update_node<S, false, GEOM, true>(a, lm, code, x, y, z, cell, load, h, unused);
      if (last) {
        static_for<0, Q>([&](auto kc) {
          constexpr int k = decltype(kc)::value;
          static_cast<S*>(a.dst_pop[swapped ? opp(k) : k])[cell] = Storage<S>::store(h[k]);
        });
      } else {
        S* to = buf + ((s & 1) ? 0u : Q * per) + node;
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
  // more warps than the nodes fill, so that the groups of grouped_node can start at warp
  // boundaries: eight, or for FP64, whose steps are bound by the warps on a scheduler, no
  // more than fill up a set of four
  const uint32_t more = std::is_same<S, double>::value ? (per + 127u) / 128u * 128u : per + 256u;
  const uint32_t threads = more < RESIDENT_THREADS ? more : RESIDENT_THREADS;
  const size_t smem = size_t(2) * Q * per * sizeof(S);
  // The limit belongs to the kernel, not to the launch, and other threads may be launching it
  // for lattices of other sizes: always the largest lattice's (77,824 bytes; binary16 half).
  constexpr uint32_t most = (std::is_same<S, double>::value ? RESIDENT_NODES_F64 : RESIDENT_NODES) / RESIDENT_CTAS;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(2 * Q * most * sizeof(S)));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(threads);
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
  return cudaLaunchKernelEx(&cfg, resident_kernel<S, GEOM>, a, steps, per, swapped);
}

// `steps` steps from src to dst (which may be the same array); cudaErrorNotSupported where
// the device has no room for the cluster.
template <typename S>
cudaError_t launch_resident_impl(const SweepArgs& a, int steps, bool swapped, cudaStream_t s) {
  if (a.links || a.forced) return launch_resident_geom<S, true>(a, steps, swapped, s);
  return launch_resident_geom<S, false>(a, steps, swapped, s);
}

// ---------------------------------------------------------------------------------
// Many steps of a lattice that one block per SM covers, in one launch: each thread keeps
// its node, the arrays stay in global memory (L2), and a grid barrier separates the steps.
// A launch per step of such a lattice pays for the launch, for the fetch of its
// instructions into every SM's cache and for the drain of the wave; the barrier is one
// atomic per block and a poll through L2. The node code is the sweep's. One block per SM
// and no more, so that few arrive at the barrier (with 256-node blocks, several per SM, a
// step of 64 x 64 x 32 FP32 took 4.8 us, with one block 3.7, by launches 5.0).
// ---------------------------------------------------------------------------------

// Nodes a block holds at most, and so the largest lattice (152 SMs: 155,648 nodes, FP64
// 77,824): the threads that its registers allow without spills. Beyond, launches are as
// fast: 64 x 64 x 32 FP32 with a body force 5.4 against 5.6 us, 99 x 33 x 33 FP64 (with
// 768 threads and spills) 10.2 against 9.3 us.
template <typename S> constexpr int grid_step_threads() { return std::is_same<S, double>::value ? 512 : 1024; }

// Grid barrier: every block arrives and waits for `target` arrivals; false once the wait
// has taken STAGE_WAIT_LIMIT_NS. A cooperative grid is placed as a whole: beside a kernel
// that kept one SM for 3 s, and beside a second such grid, blocks that fill an SM each
// started together when there was room for all, and no wait ran out. So a wait lasts as
// long as the slowest block's step; the limit bounds it all the same. Every thread of the
// block takes part.
__device__ __forceinline__ bool grid_barrier(uint32_t* arrivals, uint32_t target, const SweepArgs& a) {
  __shared__ bool ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!(a.drop_copies && blockIdx.x == 0))  // test hook: the wait runs out
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrivals) : "memory");
    uint32_t seen;
    uint64_t t0 = 0;
    bool in_time = true;
    for (uint32_t spins = 0;; ++spins) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(arrivals) : "memory");
      if (seen >= target) break;
      if ((spins & 1023u) == 1023u) {
        const uint64_t now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > STAGE_WAIT_LIMIT_NS) {
          if (a.err) atomicOr(a.err, ERR_GRID_WAIT);
          in_time = false;
          break;
        }
      }
    }
    ok = in_time;
  }
  __syncthreads();
  return ok;
}

// `a` goes from array 0 to array 1, `b` back.
template <typename S, bool GEOM>
__global__ void __launch_bounds__((grid_step_threads<S>()), 1)
    grid_steps_kernel(const __grid_constant__ SweepArgs a, const __grid_constant__ SweepArgs b, int steps,
                      uint32_t* arrivals) {
  uint32_t cell = blockIdx.x * blockDim.x + threadIdx.x, lm = 0;
  if constexpr (GEOM) {
    const uint2 node = geometry_node(a, cell);
    cell = node.x;
    lm = node.y;
  }
  NodeTerms<typename ComputeOf<S>::T> unused;
  for (int s = 0;;) {
    sweep_node<S, false, STREAM_AB, GEOM, true, true>((s & 1) ? b : a, cell, lm, unused);
    if (++s == steps) break;
    if (!grid_barrier(arrivals, uint32_t(s) * gridDim.x, a)) break;
  }
}

template <typename S, bool GEOM>
cudaError_t launch_grid_steps_geom(const SweepArgs& a, int steps, uint32_t* arrivals, cudaStream_t s) {
  const void* fn = reinterpret_cast<const void*>(grid_steps_kernel<S, GEOM>);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const uint32_t nodes = GEOM ? plain_step_nodes(a) : a.N;
  const uint32_t per = ((nodes + uint32_t(sms) - 1) / uint32_t(sms) + 31u) / 32u * 32u;
  if (per == 0) return cudaErrorNotSupported;
  const uint32_t blocks = (nodes + per - 1) / per;
  if (per > uint32_t(grid_step_threads<S>()) || uint64_t(steps) * blocks >= (1ull << 32)) return cudaErrorNotSupported;
  e = cudaMemsetAsync(arrivals, 0, sizeof(uint32_t), s);
  if (e != cudaSuccess) return e;
  SweepArgs b = a;
  b.src = a.dst;
  b.dst = const_cast<void*>(a.src);
  for (int k = 0; k < Q; ++k) {
    b.src_pop[k] = a.dst_pop[k];
    b.dst_pop[k] = const_cast<void*>(a.src_pop[k]);
  }
  SweepArgs first = a;
  void* args[] = {&first, &b, &steps, &arrivals};
  e = cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(per), args, 0, s);
  // fewer SMs are free for this process than the device has, or no such launches at all
  if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) return e;
  cudaGetLastError();
  return cudaErrorNotSupported;
}

// `steps` steps from src, alternating the two arrays; cudaErrorNotSupported where one block
// per SM does not cover the lattice. `arrivals`: a device word of the caller's.
template <typename S>
cudaError_t launch_grid_steps_impl(const SweepArgs& a, int steps, uint32_t* arrivals, cudaStream_t s) {
  if (a.links || a.forced) return launch_grid_steps_geom<S, true>(a, steps, arrivals, s);
  return launch_grid_steps_geom<S, false>(a, steps, arrivals, s);
}

}  // namespace lbm
