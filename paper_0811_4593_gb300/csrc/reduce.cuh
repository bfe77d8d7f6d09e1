// reduce.cuh -- fixed-order sums of the residual reductions (mass, |du|^2, |u|^2 and a
// bad-node count), shared by the sweeps, the single-lattice and the batched final folds
// so that a lattice reduces to the same bits in all of them.
//
// The FP64 pipe issues one warp instruction in about 19 SM cycles (527 G thread
// operations per second on 152 SMs), so the sums are arranged to issue few of them.
#pragma once
#include "lbm_internal.h"

namespace lbm {

// An unevaluated float sum hi + lo (lo below half an ulp of hi after each accumulation
// of hi; about 48 bits).
struct fpair {
  float hi, lo;
};

// The same with a third part (about 72 bits): the rounding of the second part of a pair, which
// left sums of squares 4 to 20 units of 2^-53 from the exact ones (27 to 65,536 nodes; in
// double 0.3 to 1), is kept.
struct ftriple {
  float hi, lo, rest;
};

__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ fpair shfl_xor(fpair v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ ftriple shfl_xor(ftriple v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o),
          __shfl_xor_sync(0xffffffffu, v.rest, o)};
}
__device__ __forceinline__ double sum_of(double a, double b) { return __dadd_rn(a, b); }
// a + b as the rounded sum and its error (Knuth's TwoSum, error-free).
__device__ __forceinline__ fpair two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
// Sum of two pairs: the high parts error-free, the low parts and the error by rounded float
// additions.
__device__ __forceinline__ fpair sum_of(fpair a, fpair b) {
  const fpair s = two_sum(a.hi, b.hi);
  return {s.hi, __fadd_rn(__fadd_rn(a.lo, b.lo), s.lo)};
}
// Of two triples: the low parts and the error of the high ones error-free too.
__device__ __forceinline__ ftriple sum_of(ftriple a, ftriple b) {
  const fpair s = two_sum(a.hi, b.hi), t = two_sum(a.lo, b.lo), l = two_sum(t.hi, s.lo);
  return {s.hi, l.hi, __fadd_rn(__fadd_rn(a.rest, b.rest), __fadd_rn(t.lo, l.lo))};
}

// Warp totals of four quantities: lane l returns the total of quantity l / 8. The first
// two steps halve what a lane still carries instead of reducing four values over five
// steps each, so a warp issues 6 additions in place of 20.
template <typename V>
__device__ __forceinline__ V warp_sum4(V q0, V q1, V q2, V q3) {
  const bool up = threadIdx.x & 16, up2 = threadIdx.x & 8;
  const V k0 = sum_of(up ? q2 : q0, shfl_xor(up ? q0 : q2, 16));
  const V k1 = sum_of(up ? q3 : q1, shfl_xor(up ? q1 : q3, 16));
  V k = sum_of(up2 ? k1 : k0, shfl_xor(up2 ? k0 : k1, 8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) k = sum_of(k, shfl_xor(k, o));
  return k;
}

// Totals over the 8 warps of a 256-thread block from one row of four doubles per warp
// (lane l of the first warp holds row l / 4, quantity l % 4); valid in its lanes 0..3.
__device__ __forceinline__ double block_sum_rows(double v) {
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) v = sum_of(v, shfl_xor(v, o));
  return v;
}

// FOLD_THREADS threads fold `count` <= FOLD_ROWS rows of four doubles into out[4]:
// thread t adds rows t, t + FOLD_THREADS, ... in ascending order, then the warp and
// block sums above. The order depends only on `count`. Ends with a block barrier behind
// the write of out.
__device__ __forceinline__ void fold_rows(const double* rows, uint32_t count, double* out) {
  __shared__ double warp_rows[FOLD_THREADS / 32][4];
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (uint32_t b = threadIdx.x; b < count; b += FOLD_THREADS) {
    const double2 x = __ldcg(reinterpret_cast<const double2*>(rows) + 2ull * b);
    const double2 y = __ldcg(reinterpret_cast<const double2*>(rows) + 2ull * b + 1);
    v[0] += x.x;
    v[1] += x.y;
    v[2] += y.x;
    v[3] += y.y;
  }
  const double k = warp_sum4(v[0], v[1], v[2], v[3]);
  const int lane = threadIdx.x & 31;
  if ((lane & 7) == 0) warp_rows[threadIdx.x >> 5][lane >> 3] = k;
  __syncthreads();
  if (threadIdx.x < 32) {
    const double s = block_sum_rows(warp_rows[lane >> 2][lane & 3]);
    if (lane < 4) out[lane] = s;
  }
  __syncthreads();
}

}  // namespace lbm
