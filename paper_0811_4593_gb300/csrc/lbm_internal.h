// lbm_internal.h -- interface between the C-ABI runtime (runtime.cu) and the kernel
// translation units (sweep_f64.cu, sweep_f32.cu, sweep_f16.cu).
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cmath>
#include <cstdint>

namespace lbm {

// Unsigned 32-bit division by an invariant divisor with one multiply-high, after
// Granlund & Montgomery, "Division by invariant integers using multiplication"
// (PLDI 1994), Fig. 4.1: q = (t + ((n - t) >> s1)) >> s2 with t = mulhi(m, n).
struct FastDiv {
  uint32_t d, m, s1, s2;
};

inline FastDiv make_fastdiv(uint32_t d) {
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;  // l = ceil(log2 d)
  FastDiv f;
  f.d = d;
  f.m = uint32_t(((1ull << 32) * ((1ull << l) - d)) / d + 1);
  f.s1 = l < 1 ? l : 1;
  f.s2 = l > 1 ? l - 1 : 0;
  return f;
}

#ifdef __CUDACC__
__device__ __forceinline__ uint32_t fdiv(const FastDiv& f, uint32_t n) {
  uint32_t t = __umulhi(f.m, n);
  return (t + ((n - t) >> f.s1)) >> f.s2;
}
#endif

// Largest float not above -rho0: for a float drho, rho0 + drho > 0 exactly if drho > it.
inline float floor_neg(double rho0) {
  const float f = float(-rho0);
  return double(f) > -rho0 ? std::nextafter(f, -INFINITY) : f;
}

// One boundary-face node as the sweep reads it: the first half for FP64 arithmetic, the
// second for float sweeps, or in an FP64 lattice for its fixed-point closures. Velocity face: the prescribed velocity and 1 / (1 - u.n) for the density
// relation (n = inward normal), formed in double on the host, for float sweeps as a pair
// hi + lo. Pressure face: the tangential velocity (normal part zero), the prescribed
// density in `inv`, and for float sweeps its reciprocal as a pair, the density and its
// difference from rho0.
struct __align__(16) FaceNode {
  double u[3];
  double inv;
  union {
    struct {
      float uf[3];
      float inv_hi, inv_lo;
      float rho, drho;
      float pad;
    };
    int64_t fx[4];  // FixedFace: u[0], u[1], r, ok (make_fixed_face)
  };
};

// Boundary data of one face for the sweep.
struct FaceBC {
  const FaceNode* tab;  // device [n2][n1] or nullptr (uniform: `uni`)
  FaceNode uni;
};

// Parameters of the fixed-point relaxation of FP64 lattices (fixed64.cuh), with S = 2^E.
// Factors are (high, low) limbs of value 2^62.
struct FixedArgs {
  uint32_t on;        // 0: this lattice relaxes in double only
  uint32_t e_in;      // biased exponent of S 2^-12
  uint32_t e_out;     // (991 + E) << 20
  int32_t keep[2];    // 1 - omega
  int32_t w3[2];      // omega / 3
  int32_t w[2];       // omega / 36
  int64_t force[3];   // tau F in units of S 2^-64
  double unit_in, unit_out;  // S 2^-64, S 2^-63
  double rest[2];     // axis and diagonal populations at rest: rho0 / 18, rho0 / 36
};

// The parameters for density scale rho0, omega and tau F. Off where a scale has no
// normal double, where omega is below 2^-61 or where the force is not small.
inline FixedArgs make_fixed(double rho0, double omega, const double (&tforce)[3]) {
  FixedArgs fx{};
  int e = 0;
  const double m = std::frexp(rho0, &e);  // rho0 = m 2^e, 1/2 <= m < 1
  e += m == 0.5 ? 1 : 2;                  // rho0 / 2^e in (1/8, 1/4]
  if (e < -900 || e > 900 || !(omega > 0.0) || !(omega < 2.0)) return fx;
  const int64_t w = int64_t(std::ldexp(omega, 62));
  if (w < 2) return fx;
  auto limbs = [](int64_t b, int32_t (&to)[2]) {
    to[0] = int32_t(b >> 31);
    to[1] = int32_t(b & 0x7fffffff);
  };
  limbs((int64_t(1) << 62) - w, fx.keep);
  limbs((w + 1) / 3, fx.w3);
  limbs((w + 18) / 36, fx.w);
  for (int i = 0; i < 3; ++i) {
    const double f = std::ldexp(tforce[i], 64 - e);
    if (!(std::fabs(f) < 0x1p56)) return fx;  // tau F below S / 256
    fx.force[i] = std::llrint(f);
  }
  fx.e_in = uint32_t(1011 + e);
  fx.e_out = uint32_t(991 + e) << 20;
  fx.unit_in = std::ldexp(1.0, e - 64);
  fx.unit_out = std::ldexp(1.0, e - 63);
  fx.rest[0] = rho0 / 18.0;
  fx.rest[1] = rho0 / 36.0;
  fx.on = 1u;
  return fx;
}

// The fixed-point record of a face node on axis `axis` with inward normal component un and
// velocity u (velocity face), or density rho (pressure face). Marked unfit (0) where the
// velocity is not below 1/4 or the density not near the lattice's, and in lattices that
// relax in double.
inline void make_fixed_face(const FixedArgs& fx, int axis, const double* u, double un, bool pressure, double rho,
                            int64_t (&out)[4]) {
  out[0] = out[1] = out[2] = out[3] = 0;
  if (!fx.on) return;
  int n = 0;
  for (int i = 0; i < 3; ++i) {
    if (i == axis) continue;
    if (!(std::fabs(u[i]) < 0.25)) return;
    out[n++] = std::llrint(std::ldexp(u[i] * 2.0 / 3.0, 62));
  }
  if (pressure) {
    const double r = rho / fx.unit_in;  // S is a power of two
    if (!(r > 0x1p60) || !(r < 0x1p63)) return;
    out[2] = int64_t(r);
  } else {
    if (!(std::fabs(un) < 0.25)) return;
    out[2] = std::llrint(std::ldexp(un / (1.0 - un), 62));  // 1 / (1 - un) - 1
  }
  out[3] = 1;
}

// Everything one sweep launch needs, passed by value.
struct SweepArgs {
  const void* src;   // storage [19][N], post-collision state of the previous step
  void* dst;         // storage [19][N], post-collision state after this step
  const void* src_pop[19];  // src + k N: the start of population k (set with src / dst
  void* dst_pop[19];        // so that each access is one add and one wide multiply-add)
  uint32_t nx, ny, nz, N;
  FastDiv div_nx, div_ny;
  FastDiv div_nxh;    // nx / 2 (the paired binary16 sweep, even nx)
  uint32_t periodic;  // bit a set: axis a is periodic
  uint32_t pressure;  // bit f set: face f is a pressure face
  double rho0;
  double omega;       // 1 / tau
  float rho0f, omegaf;
  float rho0_lo;      // rho0 - rho0f
  float neg_rho0;     // floor_neg(rho0)
  float mom_coef[2][2];  // omegaf / 6 and omegaf / 12 as hi + lo float pairs
  FaceBC face[6];
  void* snap;         // residual steps: [3][N] velocity snapshot in the compute type
  double* partials;   // residual steps: [blocks][4] per-block sums, then [groups][4] of the fold
  const uint32_t* links;  // optional [N] geometry words (nullptr: no geometry), see below
  // optional list of the fluid nodes (cell, geometry word) in cell order: plain steps then
  // visit them only, in warps without idle lanes
  const uint2* fluid;
  uint32_t nfluid;
  uint32_t forced;        // nonzero: a body force acts (eq. gravity)
  double force[3];        // F: momentum the collision adds per step
  double tforce[3];       // tau F: the equilibrium velocity shift times rho
  float forcef[3], tforcef[3];
  FixedArgs fx;           // FP64 lattices: the relaxation in fixed point
  // Device word a sweep sets (bit 0) when it gave up waiting for its staged loads (a
  // bounded wait ran out); the host reads and clears it at its synchronisation points.
  uint32_t* err;
  // Failure injection for tests of the bounded waits: nonzero makes the row-staged
  // sweep's first CTA announce the copies of its first row group but not issue them,
  // so its waits run out (no fault, no unbounded wait).
  uint32_t drop_copies;
};

// Error bits of SweepArgs::err.
constexpr uint32_t ERR_STAGE_WAIT = 1u;  // the row-staged sweep
constexpr uint32_t ERR_GRID_WAIT = 2u;   // the grid barrier of the multi-step kernel

// Geometry word of a node: bits 0..18 (nodes without a rule): the pull source of
// population k is solid (mid-grid bounce-back); bits 24..29: the node's on-site rule
// (0: none; 1..50: the C ABI codes of planes, concave edges, corners and junctions;
// 51..62: the convex edges -7..-18 as 44 - code); bit 31: the node is solid.
constexpr uint32_t SOLID_NODE = 1u << 31;
constexpr int RULE_SHIFT = 24;
constexpr uint32_t RULE_BITS = 0x3fu;

// One lattice of a batch, as the batched sweep reads it from device memory.
struct BatchEntry {
  SweepArgs a;           // src/dst are taken from buf[] and the step parity
  const void* buf[2];    // the lattice's two population buffers
  uint32_t cur;          // index into buf[] of the current state at step parity 0
  uint32_t block_begin;  // first global block of this lattice in the batch
  uint32_t nblocks;      // 256-node blocks of this lattice
  uint32_t slot;         // row of the batch's result table
};

struct BatchHeader {
  uint32_t nentries;      // entries in use, ordered by block_begin
  uint32_t total_blocks;  // sum of nblocks
  uint32_t nchunks;       // work units of the batched sweep (chunk table rows - 1)
  uint32_t pad;
};

// One work unit of the batched sweep: the global blocks from `start` up to the next
// chunk's start, the first of them in entry `entry`. The table ends with a sentinel
// row {total_blocks, nentries}. CTAs take chunks in order from a device counter, so
// a CTA that met expensive blocks (boundary-heavy lattices) takes fewer chunks.
struct BatchChunk {
  uint32_t start;
  uint32_t entry;
};

constexpr int SWEEP_THREADS = 256;
// Final fold of the partial sums: one block of FOLD_THREADS folds FOLD_ROWS rows.
constexpr int FOLD_THREADS = 256;
constexpr uint32_t FOLD_ROWS = 1024;

inline uint32_t sweep_blocks(uint32_t N) { return (N + SWEEP_THREADS - 1) / SWEEP_THREADS; }
// groups of the fold of `nblocks` rows (19 N < 2^32, so nblocks < 2^20 and one more level
// of FOLD_ROWS rows folds the groups)
__host__ __device__ inline uint32_t fold_groups(uint32_t nblocks) { return (nblocks + FOLD_ROWS - 1) / FOLD_ROWS; }
// rows of a partial-sum buffer: the sweep's blocks, then the fold's groups
inline uint32_t partial_rows(uint32_t nblocks) { return nblocks + fold_groups(nblocks); }

// The multi-step kernel of small lattices (resident.cuh): nodes a CTA holds at most, the
// largest (non-portable) cluster, and the shortest run of steps it is taken for (below,
// loading and storing the state costs as much as the launches).
constexpr uint32_t RESIDENT_THREADS = 512;
constexpr uint32_t RESIDENT_CTAS = 16;
constexpr uint32_t RESIDENT_NODES = RESIDENT_THREADS * RESIDENT_CTAS, RESIDENT_NODES_F64 = RESIDENT_NODES / 2;
constexpr int RESIDENT_MIN_STEPS = 16;
// Steps of one launch at most, even: about 5 to 20 ms, after which work of other streams
// gets the SMs, as it does between the launches of single steps.
constexpr int MULTI_STEPS_MAX = 4096;
// Nodes beyond which no A/B lattice takes its steps in one launch of a block per SM (the
// launch itself knows the SMs).
constexpr uint32_t GRID_STEPS_NODES = 262144;

// Nodes a plain step visits.
inline uint32_t plain_step_nodes(const SweepArgs& a) { return a.fluid ? a.nfluid : a.N; }

// mode: 0 A/B pull, 1 AA gather-scatter step, 2 AA in-place step (see kernels.cuh)
template <typename S> cudaError_t launch_sweep(const SweepArgs& a, bool resid, int mode, cudaStream_t s);
// `steps` steps of a small lattice in one launch (resident.cuh), from src to dst
template <typename S> cudaError_t launch_resident(const SweepArgs& a, int steps, bool swapped, cudaStream_t s);
// `steps` A/B steps of a lattice that one block per SM covers, in one launch; arrivals: a
// device word for its grid barrier
template <typename S> cudaError_t launch_grid_steps(const SweepArgs& a, int steps, uint32_t* arrivals, cudaStream_t s);
template <typename S> cudaError_t launch_init(void* dst, uint32_t N, double rho0, cudaStream_t s);
// swapped: the state holds f_k in slot -k (an AA lattice between step pairs)
template <typename S> cudaError_t launch_macros(const void* src, uint32_t N, double rho0, void* rho,
                                                void* u, bool swapped, cudaStream_t s);
template <typename S> cudaError_t launch_state_reduce(const void* src, uint32_t N, double rho0,
                                                      void* snap, double* partials, bool swapped, cudaStream_t s);
// partials: partial_rows(nblocks) rows, the first nblocks of them summed into out[4];
// ticket: a device word that is zero between folds
cudaError_t launch_final_reduce(double* partials, uint32_t nblocks, double* out, uint32_t* ticket, cudaStream_t s);
// next_chunk: a device counter that is zero when the launch starts (the caller clears
// it in stream order before every launch); each CTA draws chunks from it until the
// table is exhausted
template <typename S> cudaError_t launch_sweep_batched(const BatchHeader* hdr, const BatchEntry* ents,
                                                       const BatchChunk* chunks, uint32_t* next_chunk, uint32_t parity,
                                                       bool resid, int mode, int grid, cudaStream_t s);
// persistent grid of a batched variant: SMs x its resident blocks per SM (0 on error)
template <typename S> int batched_grid(bool resid, int mode);
template <typename S> uint32_t bounds_errors();  // debug build: indices out of range (read resets)
cudaError_t launch_batch_final_reduce(const BatchHeader* hdr, const BatchEntry* ents, int capacity, double* results,
                                      cudaStream_t s);

// Sets the calling thread's context-free error message (lbm_last_error(NULL)).
void record_error(const char* msg);

}  // namespace lbm
