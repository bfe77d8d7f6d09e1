// fixed_close.cuh -- the boundary closures of FP64 nodes in 64-bit fixed point, on the
// populations of fixed64.cuh (units of S 2^-64). Included by kernels.cuh.
//
// A face closure in double is 49 FP64 instructions, 930 SM cycles for every warp that
// holds a face node, and an edge or corner as much again: in short-row and small lattices
// more than the relaxation itself (32 x 32 x 16 with four walled faces: 23 us per step
// against 6 with periodic ones). Here a face is about 80 integer instructions. Sums are
// exact; each product is rounded to a unit of S 2^-63. A node whose known populations
// or closed ones leave the windows, or whose prescribed values are not small
// (make_fixed_face), is closed and relaxed in double instead.
#pragma once

namespace lbm {

// 2/3 and 2/n as factors (value 2^62): mul63 with them gives a third, a n-th
constexpr int64_t fixed_part(int n) { return int64_t(((uint64_t(1) << 63) + uint64_t(n) / 2) / uint64_t(n)); }

// Prescribed values of a face node, as make_fixed_face lays them down.
struct FixedFace {
  int64_t u[2];  // 2/3 of the tangential velocities (axes in increasing order), factors
  int64_t r;     // velocity face: 1 / (1 - u.n) - 1 as a factor; pressure face: rho_p
  bool ok;
};

// Plane with inward normal SG e_A. With S the relation's sum and d = rho - S = rho u.n,
// g_t = s_t - rho u_t for the two tangential axes (s_t the in-plane sum of c_t h, the
// transverse correction N_t = (s_t - 2/3 rho u_t) / 2):
//   velocity face  rho = S / (1 - u.n), pressure face  rho = rho_p,
//   h_n = h_-n + d / 3,   h_(n +- t) = h_-(n +- t) + (d / 3 -+ g_t) / 2,
// which is the rule of close_face and close_face_pressure with its terms gathered. The
// two halves of d / 3 add up exactly.
// False where rho does not fit (the sums of populations at the upper ends of their windows).
template <int A, int SG>
__device__ __forceinline__ bool fixed_close_face(int64_t (&f)[Q], const FixedFace& v, bool pressure) {
  int64_t in = 0, out = 0;
  static_for<0, Q>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    constexpr int cn = SG * ca(k, A);
    if constexpr (cn == 0) in += f[k];
    else if constexpr (cn < 0) out += f[k];
  });
  const int64_t s = in + (out + out);
  const int64_t d = pressure ? v.r - s : mul63(s, limbs_of(v.r)) * 2;
  const int64_t rho = int64_t(uint64_t(s) + uint64_t(d));  // below 2^64: negative where it does not fit
  const int64_t third = mul63(d, limbs_of(fixed_part(3)));
  auto tangent = [&](auto tc, int64_t factor) {
    constexpr int T = decltype(tc)::value;
    constexpr int n[3] = {A == 0 ? SG : 0, A == 1 ? SG : 0, A == 2 ? SG : 0};
    constexpr int kp = vel_index(n[0] + (T == 0), n[1] + (T == 1), n[2] + (T == 2));
    constexpr int km = vel_index(n[0] - (T == 0), n[1] - (T == 1), n[2] - (T == 2));
    int64_t st = 0;
    static_for<0, Q>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (ca(k, A) == 0 && ca(k, T) > 0) st += f[k];
      else if constexpr (ca(k, A) == 0 && ca(k, T) < 0) st -= f[k];
    });
    const int64_t g = st - 3 * mul63(rho, limbs_of(factor));
    const int64_t half = (third - g) >> 1;
    f[kp] = f[opp(kp)] + half;
    f[km] = f[opp(km)] + (third - half);
  };
  tangent(std::integral_constant<int, (A == 0 ? 1 : 0)>{}, v.u[0]);
  tangent(std::integral_constant<int, (A == 2 ? 1 : 2)>{}, v.u[1]);
  constexpr int kn = vel_index(A == 0 ? SG : 0, A == 1 ? SG : 0, A == 2 ? SG : 0);
  f[kn] = f[opp(kn)] + third;
  return rho > 0;
}

// As close_edge and close_corner: bounce-back, the along-edge correction, buried links
// and rest population from the other moving populations (beside a pressure plane from
// the prescribed density rho_p).
template <int A1, int S1, int A2, int S2>
__device__ __forceinline__ void fixed_close_edge(int64_t (&f)[Q], bool pressure, int64_t rho_p) {
  using R = EdgeRule<A1, S1, A2, S2>;
  static_for<0, Q>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    if constexpr (R::unknown(k) && !R::buried(k)) f[k] = f[opp(k)];
  });
  const int64_t ne = (f[R::PE] - f[R::ME] + 2) >> 2;
  int64_t s = 0;
  static_for<0, Q - 1>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    if constexpr (R::unknown(k) && !R::buried(k) && R::along(k) != 0) f[k] -= R::along(k) * ne;
    if constexpr (!R::buried(k)) s += f[k];
  });
  const int64_t fb = pressure ? mul63(rho_p - s, limbs_of(fixed_part(14))) : mul63(s, limbs_of(fixed_part(22)));
  static_for<0, Q - 1>([&](auto kc) {
    if constexpr (R::buried(decltype(kc)::value)) f[decltype(kc)::value] = fb;
  });
  f[Q - 1] = 12 * fb;
}

template <int SX, int SY, int SZ>
__device__ __forceinline__ void fixed_close_corner(int64_t (&f)[Q], bool pressure, int64_t rho_p) {
  using R = CornerRule<SX, SY, SZ>;
  int64_t s = 0;
  static_for<0, Q - 1>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    if constexpr (R::unknown(k) && !R::buried(k)) f[k] = f[opp(k)];
    if constexpr (!R::buried(k)) s += R::unknown(k) ? f[opp(k)] : f[k];
  });
  const int64_t fb = mul63(pressure ? rho_p - s : s, limbs_of(fixed_part(18)));
  static_for<0, Q - 1>([&](auto kc) {
    if constexpr (R::buried(decltype(kc)::value)) f[decltype(kc)::value] = fb;
  });
  f[Q - 1] = 12 * fb;
}

// As close_convex and close_junction.
template <int DX, int DY, int DZ>
__device__ __forceinline__ void fixed_close_convex(int64_t (&f)[Q]) {
  using R = ConvexRule<DX, DY, DZ>;
  f[R::KD] = f[opp(R::KD)];
  int64_t p = 0;
  static_for<0, Q>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    if constexpr (R::along(k) != 0) p += R::along(k) * f[k];
  });
  const int64_t q = (p + 2) >> 2;
  static_for<0, Q>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    if constexpr (R::into_bulk(k) && R::along(k) != 0) f[k] -= R::along(k) * q;
  });
}

template <int A, int SG, int DX, int DY, int DZ>
__device__ __forceinline__ void fixed_close_junction(int64_t (&f)[Q]) {
  constexpr int KD = vel_index(DX, DY, DZ);
  static_for<0, Q>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    if constexpr (SG * ca(k, A) > 0 || k == KD) f[k] = f[opp(k)];
  });
  int64_t s = 0;
  static_for<0, Q - 1>([&](auto kc) { s += f[decltype(kc)::value]; });
  f[Q - 1] = (s + 1) >> 1;
}

// Rule R of the geometry word, as rule_case.
template <int R>
__device__ __forceinline__ void fixed_rule_case(int64_t (&f)[Q]) {
  if constexpr (R >= 1 && R <= 6) {
    constexpr int k = R - 1;
    fixed_close_face<axis_of(k), sign_of(k)>(f, FixedFace{{0, 0}, 0, true}, false);
  } else if constexpr (R >= 7 && R <= 18) {
    constexpr int k = R - 1;
    constexpr int A1 = cx(k) != 0 ? 0 : 1;
    constexpr int S1 = A1 == 0 ? cx(k) : cy(k);
    constexpr int A2 = cz(k) != 0 ? 2 : 1;
    constexpr int S2 = A2 == 2 ? cz(k) : cy(k);
    fixed_close_edge<A1, S1, A2, S2>(f, false, 0);
  } else if constexpr (R >= 19 && R <= 26) {
    constexpr int b = R - 19;
    fixed_close_corner<(b & 1) ? -1 : 1, (b & 2) ? -1 : 1, (b & 4) ? -1 : 1>(f, false, 0);
  } else if constexpr (R >= 27 && R <= 50) {
    constexpr int p = (R - 27) / 4;
    constexpr int d = junction_diagonal(p, (R - 27) % 4);
    fixed_close_junction<axis_of(p), sign_of(p), cx(d), cy(d), cz(d)>(f);
  } else if constexpr (R >= 51 && R <= 62) {
    constexpr int k = R - 45;
    fixed_close_convex<cx(k), cy(k), cz(k)>(f);
  }
}

template <int LO, int HI>
__device__ __forceinline__ void fixed_apply_rule(uint32_t r, int64_t (&f)[Q]) {
  if constexpr (LO == HI) {
    fixed_rule_case<LO>(f);
  } else {
    constexpr int MID = (LO + HI) / 2;
    if (r <= uint32_t(MID)) fixed_apply_rule<LO, MID>(r, f);
    else fixed_apply_rule<MID + 1, HI>(r, f);
  }
}

template <int A>
__device__ __forceinline__ FixedFace fixed_face_values(const SweepArgs& a, int face, uint32_t x, uint32_t y, uint32_t z) {
  const FaceBC& fb = a.face[face];
  int64_t v[4];
  if (fb.tab) {
    const uint32_t t1 = (A == 0) ? y : x;
    const uint32_t t2 = (A == 2) ? y : z;
    const uint32_t n1 = (A == 0) ? a.ny : a.nx;
    const uint32_t n2 = (A == 2) ? a.ny : a.nz;
    const longlong2* p = reinterpret_cast<const longlong2*>(fb.tab + chk(t2 * n1 + t1, n1 * n2)) + 2;
    const longlong2 p0 = __ldg(p), p1 = __ldg(p + 1);
    v[0] = p0.x;
    v[1] = p0.y;
    v[2] = p1.x;
    v[3] = p1.y;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = fb.uni.fx[i];
  }
  return {{v[0], v[1]}, v[2], v[3] != 0};
}

template <int A, int SG>
__device__ __forceinline__ bool fixed_face_case(const SweepArgs& a, uint32_t x, uint32_t y, uint32_t z, int64_t (&f)[Q]) {
  const FixedFace v = fixed_face_values<A>(a, face_id<A, SG>(), x, y, z);
  return fixed_close_face<A, SG>(f, v, a.pressure & (1u << face_id<A, SG>())) && v.ok;
}

// Both x faces in one body, as x_face_case.
__device__ __forceinline__ bool fixed_x_face_case(const SweepArgs& a, bool high, uint32_t x, uint32_t y, uint32_t z,
                                                  int64_t (&f)[Q]) {
  auto mirror = [&] {
    static_for<0, Q>([&](auto kc) {
      constexpr int k = decltype(kc)::value, m = mirror_x(k);
      if constexpr (cx(k) > 0) {
        const int64_t t = high ? f[m] : f[k];
        f[m] = high ? f[k] : f[m];
        f[k] = t;
      }
    });
  };
  const FixedFace v = fixed_face_values<0>(a, high ? 1 : 0, x, y, z);
  mirror();
  const bool fits = fixed_close_face<0, +1>(f, v, a.pressure & (high ? 2u : 1u));
  mirror();
  return fits && v.ok;
}

template <int A1, int S1, int A2, int S2>
__device__ __forceinline__ bool fixed_edge_case(const SweepArgs& a, uint32_t x, uint32_t y, uint32_t z, int64_t (&f)[Q]) {
  constexpr uint32_t b1 = 1u << face_id<A1, S1>(), b2 = 1u << face_id<A2, S2>();
  FixedFace v = {{0, 0}, 0, true};
  const bool pressure = a.pressure & (b1 | b2);
  if (pressure) v = (a.pressure & b1) ? fixed_face_values<A1>(a, face_id<A1, S1>(), x, y, z)
                                      : fixed_face_values<A2>(a, face_id<A2, S2>(), x, y, z);
  fixed_close_edge<A1, S1, A2, S2>(f, pressure, v.r);
  return v.ok;
}

template <int SX, int SY, int SZ>
__device__ __forceinline__ bool fixed_corner_case(const SweepArgs& a, uint32_t x, uint32_t y, uint32_t z, int64_t (&f)[Q]) {
  constexpr uint32_t bx = 1u << face_id<0, SX>(), by = 1u << face_id<1, SY>(), bz = 1u << face_id<2, SZ>();
  FixedFace v = {{0, 0}, 0, true};
  const bool pressure = a.pressure & (bx | by | bz);
  if (pressure) v = (a.pressure & bx)   ? fixed_face_values<0>(a, face_id<0, SX>(), x, y, z)
                    : (a.pressure & by) ? fixed_face_values<1>(a, face_id<1, SY>(), x, y, z)
                                        : fixed_face_values<2>(a, face_id<2, SZ>(), x, y, z);
  fixed_close_corner<SX, SY, SZ>(f, pressure, v.r);
  return v.ok;
}

// Cases as apply_boundary; false where the prescribed values are not fit for fixed point.
__device__ __forceinline__ bool fixed_apply_boundary(int code, const SweepArgs& a, uint32_t x, uint32_t y, uint32_t z,
                                                     int64_t (&f)[Q]) {
  switch (code) {
    case 1:
    case 2: return fixed_x_face_case(a, code == 2, x, y, z, f);
    case 3: return fixed_face_case<1, +1>(a, x, y, z, f);
    case 6: return fixed_face_case<1, -1>(a, x, y, z, f);
    case 9: return fixed_face_case<2, +1>(a, x, y, z, f);
    case 18: return fixed_face_case<2, -1>(a, x, y, z, f);
    case 4: return fixed_edge_case<0, +1, 1, +1>(a, x, y, z, f);
    case 5: return fixed_edge_case<0, -1, 1, +1>(a, x, y, z, f);
    case 7: return fixed_edge_case<0, +1, 1, -1>(a, x, y, z, f);
    case 8: return fixed_edge_case<0, -1, 1, -1>(a, x, y, z, f);
    case 10: return fixed_edge_case<0, +1, 2, +1>(a, x, y, z, f);
    case 11: return fixed_edge_case<0, -1, 2, +1>(a, x, y, z, f);
    case 19: return fixed_edge_case<0, +1, 2, -1>(a, x, y, z, f);
    case 20: return fixed_edge_case<0, -1, 2, -1>(a, x, y, z, f);
    case 12: return fixed_edge_case<1, +1, 2, +1>(a, x, y, z, f);
    case 15: return fixed_edge_case<1, -1, 2, +1>(a, x, y, z, f);
    case 21: return fixed_edge_case<1, +1, 2, -1>(a, x, y, z, f);
    case 24: return fixed_edge_case<1, -1, 2, -1>(a, x, y, z, f);
    case 13: return fixed_corner_case<+1, +1, +1>(a, x, y, z, f);
    case 14: return fixed_corner_case<-1, +1, +1>(a, x, y, z, f);
    case 16: return fixed_corner_case<+1, -1, +1>(a, x, y, z, f);
    case 17: return fixed_corner_case<-1, -1, +1>(a, x, y, z, f);
    case 22: return fixed_corner_case<+1, +1, -1>(a, x, y, z, f);
    case 23: return fixed_corner_case<-1, +1, -1>(a, x, y, z, f);
    case 25: return fixed_corner_case<+1, -1, -1>(a, x, y, z, f);
    case 26: return fixed_corner_case<-1, -1, -1>(a, x, y, z, f);
    default: return true;
  }
}

// Closure of one node in fixed point: false where it has to be done in double. `f` holds
// the converted populations, the unknown ones any value.
template <bool GEOM>
__device__ __forceinline__ bool fixed_close_node(const SweepArgs& a, uint32_t lm, int code, uint32_t x, uint32_t y,
                                                 uint32_t z, int64_t (&f)[Q]) {
  const uint32_t rule = GEOM ? (lm >> RULE_SHIFT) & RULE_BITS : 0u;
  if (rule == 0u && code == 0) return true;
  bool ok = true;
  if (GEOM && rule != 0u) fixed_apply_rule<1, 62>(rule, f);
  else ok = fixed_apply_boundary(code, a, x, y, z, f);
  return ok && fixed_closed_in_range(f);
}

// The populations a box boundary node cannot stream hold whatever the clamped load gave:
// values inside the windows take their place, so that the node is judged by what it has.
__device__ __forceinline__ void fixed_fill_unknown(const SweepArgs& a, int code, double (&h)[Q]) {
  const int fx = code % 3, fy = code / 3 % 3, fz = code / 9;
  const bool xl = fx == 1, xh = fx == 2, yl = fy == 1, yh = fy == 2, zl = fz == 1, zh = fz == 2;
  static_for<0, Q - 1>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    const bool unknown = (cx(k) > 0 && xl) || (cx(k) < 0 && xh) || (cy(k) > 0 && yl) || (cy(k) < 0 && yh) ||
                         (cz(k) > 0 && zl) || (cz(k) < 0 && zh);
    if (unknown) h[k] = a.fx.rest[k < 6 ? 0 : 1];
  });
}

}  // namespace lbm
