// fixed64.cuh -- moments and BGK relaxation of FP64 populations in 64-bit fixed point.
//
// The FP64 pipe of this GPU issues one warp instruction in about 19 SM cycles; the
// relaxation of a node takes 130 of them, 2,470 cycles per warp against about 450 for its
// memory traffic. The same work in integers is about 850 instructions of the 32-bit
// integer pipes, which issue several per cycle.
//
// A node's populations are converted, summed, relaxed and converted back:
//   in    F = f 2^64 / S          exactly (a shift of the 53-bit significand),
//   sums  R = sum F, J = sum c F  exactly,
//   out   v = f' 2^63 / S         then rounded to the nearest double,
// with S = 2^E and rho0 / S in (1/8, 1/4]. Every product is rounded to one unit of v, that
// is S 2^-63: for rho0 = 1 one eighth of the last place of a diagonal population (1/36)
// and less of the others'. Products and sums are centred (no drift from truncation).
//
// The error is absolute, so relative to a population far below its weight it is large; but
// so it is in double, whose equilibrium is rounded in the last place of larger numbers, by
// omega of it. Rms in units of 2^-53 of the population, fixed point beside double, the
// largest over density scales (rho0 / 36 is 2^-8.2 to 2^-7.2 S):
//   size, S         tau = 0.6    tau = 3      tau = 10     tau = 1000
//   2^-8 to 2^-7    0.5   4.8    0.6   0.9    0.6   0.7    0.5   0.6
//   2^-9 to 2^-8    0.8   9.5    0.7   1.3    0.7   0.7    0.7   0.6
//   2^-10 to 2^-9   1.5  19      0.9   1.2    1.2   0.9    1.3   0.6
//   2^-12 to 2^-11  2.9  41      -     -      2.3   1.0    4.0   0.6
// Up to tau = 3 the result is the more exact one for any size; at longer relaxation times
// populations below 2^-8 S lose up to three bits against double (they are kept here all the
// same: telling them apart cost FP64 steps of any tau 1 to 2 %). The largest error of a whole
// node is two thirds (long relaxation times) to a tenth (short ones) of double's; rms 3.7e-18
// to 4.8e-18 rho0 per population, mass drift of a node and step at most 1.7e-17 rho0.
//
// A node takes this path when its populations lie where a lattice flow keeps them
// (positive; diagonal and axis ones below 2.25 to 4.5 times their weight times rho0, the
// rest population between 0.38 and 3 times; all above S 2^-12); the windows bound every
// intermediate below. Any other node -- negative, tiny, huge or not finite -- is relaxed
// in double. The choice depends on the node's values only, so every sweep variant makes
// the same one.
#pragma once
#include <cstdint>
#include <cstring>

#include "lbm_internal.h"

namespace lbm {

#if defined(__CUDA_ARCH__)
__device__ __forceinline__ uint32_t hi_word(double v) { return uint32_t(__double2hiint(v)); }
__device__ __forceinline__ uint32_t lo_word(double v) { return uint32_t(__double2loint(v)); }
__device__ __forceinline__ double from_words(uint32_t hi, uint32_t lo) { return __hiloint2double(int(hi), int(lo)); }
__device__ __forceinline__ uint32_t funnel_l(uint32_t lo, uint32_t hi, uint32_t s) { return __funnelshift_l(lo, hi, s); }
__device__ __forceinline__ uint32_t funnel_r(uint32_t lo, uint32_t hi, uint32_t s) { return __funnelshift_r(lo, hi, s); }
__device__ __forceinline__ uint32_t msb_index(uint32_t v) { return 31u - uint32_t(__clz(int(v))); }
// about 2^56 / v for v in [2^26, 2^31), to 22 bits
__device__ __forceinline__ uint32_t reciprocal_seed(uint32_t v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint2float_rn(v)));
  return __float2uint_rn(r * 0x1p56f);
}
#else  // the same on the host, for the tests of the arithmetic
inline uint64_t word_bits(double v) { uint64_t b; std::memcpy(&b, &v, 8); return b; }
inline uint32_t hi_word(double v) { return uint32_t(word_bits(v) >> 32); }
inline uint32_t lo_word(double v) { return uint32_t(word_bits(v)); }
inline double from_words(uint32_t hi, uint32_t lo) { const uint64_t b = (uint64_t(hi) << 32) | lo; double v; std::memcpy(&v, &b, 8); return v; }
inline uint32_t funnel_l(uint32_t lo, uint32_t hi, uint32_t s) { s &= 31; return s ? (hi << s) | (lo >> (32 - s)) : hi; }
inline uint32_t funnel_r(uint32_t lo, uint32_t hi, uint32_t s) { s &= 31; return s ? (hi << (32 - s)) | (lo >> s) : lo; }
inline uint32_t msb_index(uint32_t v) { return 31u - uint32_t(__builtin_clz(v)); }
inline uint32_t reciprocal_seed(uint32_t v) { return uint32_t(1.0f / float(v) * 0x1p56f + 0.5f); }
#endif

// A factor as high and low limb: value = h 2^31 + l, 0 <= l < 2^31.
struct Limbs {
  int32_t h, l;
};
__host__ __device__ __forceinline__ Limbs limbs_of(int64_t b) {
  return {int32_t(b >> 31), int32_t(uint32_t(b) & 0x7fffffffu)};
}
__host__ __device__ __forceinline__ Limbs limbs_of(const int32_t (&b)[2]) { return {b[0], b[1]}; }
// a b / 2^63 to about one unit: the products of the low limbs are left out and their
// mean (1/4), together with half a unit for rounding, is added as CENTRED 2^-31 (the mean
// error is then zero; zero times anything is zero). |a|, |b| < 2^62, or |a| < 2^63
// beside |b| <= 2^63 / 3.
constexpr uint32_t CENTRED = 3u << 29;
__host__ __device__ __forceinline__ int64_t mul63(int64_t a, Limbs b) {
  const int32_t ah = int32_t(a >> 32), al = int32_t(uint32_t(a) >> 1);
  const int64_t mid = int64_t(al) * b.h + (int64_t(ah) * b.l + int64_t(CENTRED));
  return int64_t(ah) * b.h + (mid >> 31);
}

// Sums of a node in units of S 2^-64.
struct FixedSums {
  int64_t r, x, y, z;
};

// Population windows by exponent: s = exponent - (exponent of S 2^-12).
__host__ __device__ __forceinline__ bool fixed_in_range(const double (&h)[19], const FixedArgs& fx) {
  auto s = [&](int k) { return (hi_word(h[k]) >> 20) - fx.e_in; };  // a sign bit makes it huge
  uint32_t axis = 0, diag = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) axis = axis > s(k) ? axis : s(k);
#pragma unroll
  for (int k = 6; k < 18; ++k) diag = diag > s(k) ? diag : s(k);
  // sum < (6/32 + 12/64 + 1/8) S = S / 2; rest >= S / 64
  return axis < 7u && diag < 6u && s(18) - 6u < 3u;
}

// The same windows for closed populations (S 2^-12 is 2^52): positive, and no larger.
__host__ __device__ __forceinline__ bool fixed_closed_in_range(const int64_t (&f)[19]) {
  auto top = [&](int k) { return uint32_t(uint64_t(f[k]) >> 32) - (1u << 20); };
  uint32_t axis = 0, diag = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) axis = axis > top(k) ? axis : top(k);
#pragma unroll
  for (int k = 6; k < 18; ++k) diag = diag > top(k) ? diag : top(k);
  const uint32_t rest = uint32_t(uint64_t(f[18]) >> 32) - (1u << 26);
  return axis < (1u << 27) - (1u << 20) && diag < (1u << 26) - (1u << 20) && rest < (1u << 29) - (1u << 26);
}

__host__ __device__ __forceinline__ int64_t fixed_in(double v, const FixedArgs& fx) {
  const uint32_t hi = hi_word(v), lo = lo_word(v);
  const uint32_t s = (hi >> 20) - fx.e_in;
  const uint32_t m = (hi & 0xfffffu) | 0x100000u;
  return int64_t((uint64_t(funnel_l(lo, m, s)) << 32) | (lo << s));
}

// 33 additions: the populations with c_x = +1, -1 and 0 share their partial sums.
__host__ __device__ __forceinline__ FixedSums fixed_sums(const int64_t (&f)[19]) {
  const int64_t p = f[0] + (f[6] + f[7]) + (f[8] + f[9]);
  const int64_t m = f[1] + (f[10] + f[11]) + (f[12] + f[13]);
  const int64_t yp = f[2] + (f[14] + f[15]), ym = f[3] + (f[16] + f[17]);
  FixedSums q;
  q.r = (p + m) + (yp + ym) + (f[4] + f[5] + f[18]);
  q.x = p - m;
  q.y = (yp - ym) + (f[6] - f[7]) + (f[10] - f[11]);
  q.z = (f[4] - f[5]) + (f[14] - f[15]) + (f[16] - f[17]) + (f[8] - f[9]) + (f[12] - f[13]);
  return q;
}

// 3/2 S/rho in units of 2^-55, from R in [2^58, 2^63): a seed of 22 bits, then
// y (1 + e + e^2) with e = 1 - R y (Newton's iteration with its second term).
__host__ __device__ __forceinline__ int64_t fixed_three_halves_over(int64_t r) {
  const uint32_t rh = uint32_t(uint64_t(r) >> 32), rl = uint32_t(r);
  const uint32_t y = reciprocal_seed(rh);  // 2^24 S/rho
  // e 2^72 = -(R y 2^-16) modulo 2^64
  int64_t e = -int64_t(((uint64_t(rh) * y) << 16) + ((uint64_t(rl) * y) >> 16));
  const int32_t eh = int32_t(e >> 32);
  e += (int64_t(eh) * eh) >> 8;
  const uint64_t low = (uint64_t(y) * uint32_t(e)) >> 32;
  const int64_t corr = int64_t(int32_t(y)) * int32_t(e >> 32) + int64_t(low);  // y e 2^64
  const int64_t inv = (int64_t(y) << 31) + (corr >> 9);
  return inv + (inv >> 1);
}

// Nearest double of v S 2^-63 (ties up) for v >= 2^53.
__host__ __device__ __forceinline__ double fixed_out(int64_t v, const FixedArgs& fx) {
  const uint32_t i = msb_index(uint32_t(uint64_t(v) >> 32));  // >= 21
  const uint32_t s = i - 20u;                                 // bits below the significand
  const uint64_t u = uint64_t(v) + ((1u << s) >> 1);
  const uint32_t lo = uint32_t(u), hi = uint32_t(u >> 32);
  return from_words((hi >> s) + (i << 20) + fx.e_out, funnel_r(lo, hi, s));
}

// Density and momentum in double from the sums (each rounded once).
__host__ __device__ __forceinline__ void fixed_to_double(const FixedSums& q, const FixedArgs& fx, double (&m)[4]) {
  m[0] = double(q.r) * fx.unit_in;
  m[1] = double(q.x) * fx.unit_in;
  m[2] = double(q.y) * fx.unit_in;
  m[3] = double(q.z) * fx.unit_in;
}

// BGK relaxation of a node whose populations passed fixed_in_range, from F to the new
// populations in double; `q` holds the momentum the equilibrium takes (with a body force
// the node's plus tau F). In units of v, with w = omega / 36, o = w rho - w j.v,
// v = 3/2 u, a = 3 w j and q_i = a_i v_i (so w j.v = (q_x + q_y + q_z) / 3):
//   rest 12 o,   axis +-x: 2 (o + q_x +- a_x),
//   diagonals of the x-y plane (b = o + q_x + q_y, c = a_x v_y):
//     (+,+) (b + a_x) + (2 c + a_y)      (+,-) (b + a_x) - (2 c + a_y)
//     (-,-) (b - a_x) + (2 c - a_y)      (-,+) (b - a_x) - (2 c - a_y)
// added to (1 - omega) f; the same relaxation as `collide` writes for double. KEEP false:
// omega = 1 (tau = 1, where a step replaces the populations by their equilibrium), without
// the 19 products with zero, 9 % of a node's instructions; the bits are the same.
template <bool KEEP>
__host__ __device__ __forceinline__ void fixed_relax_to(const int64_t (&f)[19], const FixedSums& q, const FixedArgs& fx,
                                                     double (&h)[19]) {
  const Limbs y = limbs_of(fixed_three_halves_over(q.r));
  const Limbs w3 = limbs_of(fx.w3), keep = limbs_of(fx.keep);
  // v in units of 2^-61 (from 2^-56), |v| < 3/2
  const Limbs vx = limbs_of(mul63(q.x, y) << 5), vy = limbs_of(mul63(q.y, y) << 5), vz = limbs_of(mul63(q.z, y) << 5);
  const int64_t ax4 = mul63(q.x, w3), ay4 = mul63(q.y, w3), az4 = mul63(q.z, w3);  // 4 a
  auto quarter = [](int64_t b) { return (b + 1 + int64_t((uint32_t(b) >> 2) & 1u)) >> 2; };  // ties to even
  const int64_t ax = quarter(ax4), ay = quarter(ay4), az = quarter(az4);
  const int64_t qx = mul63(ax4, vx), qy = mul63(ay4, vy), qz = mul63(az4, vz);
  const int64_t sq = qx + qy + qz;
  const int64_t o = mul63(q.r, limbs_of(fx.w)) - mul63(sq, limbs_of(int64_t(0x2aaaaaaaaaaaaaab)));
  int32_t least = INT32_MAX;
  int64_t v[19];
  auto set = [&](int k, int64_t eq) {
    v[k] = KEEP ? mul63(f[k], keep) + eq : eq;
    const int32_t top = int32_t(v[k] >> 32);
    least = top < least ? top : least;
  };
  const int64_t o2 = o + o;
  // rounding half up to a double adds half a unit to each of the 19 populations on
  // average; the rest population, whose last place is 128 units, gives it back
  set(18, 6 * o2 - 9);
  const int64_t ex = o2 + (qx + qx), ey = o2 + (qy + qy), ez = o2 + (qz + qz);
  set(0, ex + (ax + ax));
  set(1, ex - (ax + ax));
  set(2, ey + (ay + ay));
  set(3, ey - (ay + ay));
  set(4, ez + (az + az));
  set(5, ez - (az + az));
  const int64_t all = o + sq;
  auto plane = [&](int pp, int pm, int mp, int mm, int64_t b, int64_t a1, int64_t a2, int64_t c) {
    const int64_t p = b + a1, m = b - a1, r = (c + c) + a2, s = (c + c) - a2;
    set(pp, p + r);
    set(pm, p - r);
    set(mm, m + s);
    set(mp, m - s);
  };
  plane(6, 7, 10, 11, all - qz, ax, ay, mul63(ax4, vy));
  plane(8, 9, 12, 13, all - qy, ax, az, mul63(ax4, vz));
  plane(14, 15, 16, 17, all - qx, ay, az, mul63(ay4, vz));
  if (least >= (1 << 21)) {  // every v at least 2^53
#pragma unroll
    for (int k = 0; k < 19; ++k) h[k] = fixed_out(v[k], fx);
  } else {
#pragma unroll
    for (int k = 0; k < 19; ++k) h[k] = double(v[k]) * fx.unit_out;
  }
}

// UNIT: ask whether omega is 1. A kernel then holds two bodies, which is free in the plain
// single-lattice A/B steps (256 x 64 x 64 at tau = 0.6 65.0 us with and without, at tau = 1
// 56.9 against 65.0), but not in those that spill or hold more beside it: AA steps at other
// tau 1,109 against 1,101 us (256^3), batches 466 against 453 us a step (ten lattices of 40
// to 150 nodes a side); they go without.
template <bool UNIT = true>
__host__ __device__ __forceinline__ void fixed_relax(const int64_t (&f)[19], const FixedSums& q, const FixedArgs& fx,
                                                     double (&h)[19]) {
  if (UNIT && (fx.keep[0] | fx.keep[1]) == 0) fixed_relax_to<false>(f, q, fx, h);
  else fixed_relax_to<true>(f, q, fx, h);
}

}  // namespace lbm
