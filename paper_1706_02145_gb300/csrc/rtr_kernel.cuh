// Coupling matvec y_i = sum_{j != i} W^{ij} x_j by rotation-translation-
// rotation (see rtr_tables.cuh for the factorisation W = D^H W_z D).
//
// Per ordered pair (i, j), one thread (the receiver's), with the sources held
// in the cosine / sine basis of rtr_tables.cuh (c_M and s_M of each tau):
//   1. geometry: k|d| and its phase (FP32 kernel: float-float arithmetic;
//      FP64 kernel: FP64), h_p(k|d|), cos / sin of q theta and m phi
//   2. (c_M, s_M) turned by M phi, then c'_mu = sum_M C_{mu M} c_M and
//      s'_mu = sum_M S_{mu M} s_M per degree l and tau
//   3. the axial products: for mu > 0 the sums c1 +- s2 and c2 +- s1 see only
//      A + iB or A - iB, so each entry is one complex number per sum
//   4. the same C and S (symmetric, their own inverses), turned back by M phi,
//      added to the receiver's sums
// All coefficients (rotation blocks, axial a5/b5 terms) are compile-time
// immediates; one code stream serves every warp.  Per pair the thread does
// O(L^3) work instead of the O(L^4) of the direct per-entry evaluation.  The
// real basis halves the rotations' products (2 l^2 + 2 l + 1 per degree
// against (2 l + 1)^2) and makes every number of steps 2 and 4 real, so that
// (re, im) travel together through the packed two-lane FMA.
//
// Bound by FP32 (FP64) issue; memory traffic is a few MB per product.  In the
// cosine / sine basis a pair costs 4 448 flops at lmax 4 (5 728 with complex
// rotations of all 2 l + 1 orders), 2 248 at lmax 3, 7 780 at lmax 5, and the
// entries of the rotation blocks need no half-angle powers.  Measured on
// GB300, master product, before -> after: FP32 N = 10 000 lmax 4 9.87 -> 7.71
// ms (error against 64 bits 6.0e-7 -> 3.2e-7), N = 777 lmax 5 with 8 right-hand
// sides 2.27 -> 1.11 ms, N = 100 000 lmax 3 492 -> 404 ms; FP64 N = 2001 lmax 4
// 22.9 -> 17.5 ms (16.9 ms with the shape below).
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "coupling_kernel.cuh"
#include "rtr_tables.cuh"
#include "kernels.h"

namespace celes {
namespace rtr {

template <typename R>
struct alignas(4 * sizeof(R)) Quad4 {
  R x, y, z, w;
};

// a complex value whose two parts take the same real factors
template <typename R>
struct C2 {
  R x, y;
};
// w b + c and w b for a real w: FP32 on the packed two-lane FMA of sm_100+
// (per lane the rounding of fmaf), which halves the issue slots of the
// rotations while the scalar FMAs of the axial step fill the other half of the
// FP32 lanes
__device__ __forceinline__ C2<float> fma2(float w, C2<float> b, C2<float> c) {
  const float2 r = __ffma2_rn(make_float2(w, w), make_float2(b.x, b.y), make_float2(c.x, c.y));
  return C2<float>{r.x, r.y};
}
__device__ __forceinline__ C2<float> mul2(float w, C2<float> b) {
  const float2 r = __fmul2_rn(make_float2(w, w), make_float2(b.x, b.y));
  return C2<float>{r.x, r.y};
}
__device__ __forceinline__ C2<double> fma2(double w, C2<double> b, C2<double> c) {
  return C2<double>{fma_(w, b.x, c.x), fma_(w, b.y, c.y)};
}
__device__ __forceinline__ C2<double> mul2(double w, C2<double> b) { return C2<double>{w * b.x, w * b.y}; }

// the scalars of one pair that every table derives from
template <typename R>
struct GeomS {
  R ix, sn, cs;        // 1/(k d), sin(k d), cos(k d)
  R ct, st, cph, sph;  // cos/sin theta, cos/sin phi of d
};

// ---- FP32 pair geometry without FP64 arithmetic ----------------------------
// Positions are scaled by k and split into float pairs (hi + lo, 48
// significant bits).  Per pair, k|d| is formed with error-free float
// transformations (two-sum and fma-based two-product, Knuth / Dekker) to about
// 2^-44 relative, then reduced mod pi/2 with an exact fma (the product of an
// integer quadrant count and the float nearest pi/2 has no bits below 2^-23),
// so the phase e^{i k|d|} keeps FP32 accuracy at any cluster size while the
// FP64 pipe (1/64 of the FP32 rate on this part) stays idle.
struct alignas(16) PosFF {
  float xh, yh, zh, ph;
  float xl, yl, zl, pl;
};

static_assert(sizeof(PosFF) == sizeof(Pos4), "the source tile holds either form");

__device__ __forceinline__ PosFF split_pos(const Pos4& p, double k) {
  const double x = k * p.x, y = k * p.y, z = k * p.z;
  PosFF o;
  o.xh = static_cast<float>(x);
  o.yh = static_cast<float>(y);
  o.zh = static_cast<float>(z);
  o.xl = static_cast<float>(x - static_cast<double>(o.xh));
  o.yl = static_cast<float>(y - static_cast<double>(o.yh));
  o.zl = static_cast<float>(z - static_cast<double>(o.zh));
  o.ph = o.pl = 0.0f;
  return o;
}

// s + e == a - b exactly (two-sum of a and -b)
__device__ __forceinline__ void two_diff(float a, float b, float& s, float& e) {
  s = __fsub_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
}
// s + e == a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// sin and cos of q pi/2 + y, |y| <= pi/4 (+ rounding): Taylor series to y^9 /
// y^10 (truncation below 2e-9), quadrant q mod 4 selects signs and the swap
__device__ __forceinline__ void sincos_quadrant(float y, int iq, float& s, float& c) {
  const float y2 = y * y;
  float ps = fma_(y2, 1.0f / 362880.0f, -1.0f / 5040.0f);
  ps = fma_(y2, ps, 1.0f / 120.0f);
  ps = fma_(y2, ps, -1.0f / 6.0f);
  const float sr = fma_(y * y2, ps, y);
  float pc = fma_(y2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
  pc = fma_(y2, pc, -1.0f / 720.0f);
  pc = fma_(y2, pc, 1.0f / 24.0f);
  pc = fma_(y2, pc, -0.5f);
  const float cr = fma_(y2, pc, 1.0f);
  const float s0 = (iq & 1) ? cr : sr;
  const float c0 = (iq & 1) ? sr : cr;
  s = (iq & 2) ? -s0 : s0;
  c = ((iq + 1) & 2) ? -c0 : c0;
}

// h_p(k d), p = 0..2L (closed forms of h_0, h_1 and upward recurrence)
template <int L, typename R>
struct Hankel {
  R re[2 * L + 1], im[2 * L + 1];
  __device__ __forceinline__ explicit Hankel(const GeomS<R>& q) {
    const R ix = q.ix, sn = q.sn, cs = q.cs;
    re[0] = sn * ix;
    im[0] = -cs * ix;
    re[1] = -ix * fma_(-sn, ix, cs);
    im[1] = -ix * fma_(cs, ix, sn);
#pragma unroll
    for (int p = 1; p < 2 * L; ++p) {
      const R c = static_cast<R>(2 * p + 1) * ix;
      re[p + 1] = fma_(c, re[p], -re[p - 1]);
      im[p + 1] = fma_(c, im[p], -im[p - 1]);
    }
  }
};

// cos / sin of q theta and m phi, q, m = 0..L
template <int L, typename R>
struct Angles {
  R ct[L + 1], st[L + 1], cf[L + 1], sf[L + 1];
  __device__ __forceinline__ Angles(R c, R s, R cp, R sp) {
    ct[0] = cf[0] = static_cast<R>(1);
    st[0] = sf[0] = static_cast<R>(0);
    ct[1] = c;
    st[1] = s;
    cf[1] = cp;
    sf[1] = sp;
#pragma unroll
    for (int m = 2; m <= L; ++m) {
      ct[m] = fma_(ct[m - 1], c, -st[m - 1] * s);
      st[m] = fma_(ct[m - 1], s, st[m - 1] * c);
      cf[m] = fma_(cf[m - 1], cp, -sf[m - 1] * sp);
      sf[m] = fma_(cf[m - 1], sp, sf[m - 1] * cp);
    }
  }
};

__device__ __forceinline__ GeomS<float> geometry_ff(const PosFF& a, const PosFF& b) {
  // k (r_a - r_b) per axis as s + e (unnormalised; |e| << |s| or s == 0)
  float sx, ex, sy, ey, sz, ez;
  two_diff(a.xh, b.xh, sx, ex);
  two_diff(a.yh, b.yh, sy, ey);
  two_diff(a.zh, b.zh, sz, ez);
  ex = __fadd_rn(ex, __fsub_rn(a.xl, b.xl));
  ey = __fadd_rn(ey, __fsub_rn(a.yl, b.yl));
  ez = __fadd_rn(ez, __fsub_rn(a.zl, b.zl));
  // (k d)^2 = sum (s + e)^2 = sum s^2 (exact two-products) + e (2 s + e)
  const float px = __fmul_rn(sx, sx), py = __fmul_rn(sy, sy), pz = __fmul_rn(sz, sz);
  float lo = __fadd_rn(__fadd_rn(__fmaf_rn(sx, sx, -px), __fmaf_rn(sy, sy, -py)), __fmaf_rn(sz, sz, -pz));
  lo = __fmaf_rn(ex, __fmaf_rn(2.0f, sx, ex), lo);
  lo = __fmaf_rn(ey, __fmaf_rn(2.0f, sy, ey), lo);
  lo = __fmaf_rn(ez, __fmaf_rn(2.0f, sz, ez), lo);
  float S, E1, S2, E2;
  two_sum(px, py, S, E1);
  two_sum(S, pz, S2, E2);
  lo = __fadd_rn(lo, __fadd_rn(E1, E2));
  // k d = r + delta: one Newton correction of the FP32 square root
  const float rinv = rsqrtf(S2);
  const float r = __fmul_rn(S2, rinv);
  const float rr = __fmul_rn(r, r);
  const float rre = __fmaf_rn(r, r, -rr);
  const float resid = __fadd_rn(__fsub_rn(__fsub_rn(S2, rr), rre), lo);
  const float delta = __fmul_rn(resid, 0.5f * rinv);
  // phase: k d = n pi/2 + y
  constexpr double HALF_PI = 1.5707963267948966192313216916398;
  constexpr float H1 = static_cast<float>(HALF_PI);
  constexpr float H2 = static_cast<float>(HALF_PI - static_cast<double>(H1));
  const float n = rintf(__fmul_rn(r, static_cast<float>(1.0 / HALF_PI)));
  float y = __fmaf_rn(-n, H1, r);  // exact
  y = __fadd_rn(y, __fmaf_rn(-n, H2, delta));
  GeomS<float> q;
  sincos_quadrant(y, static_cast<int>(n) & 3, q.sn, q.cs);
  // reciprocals from the approximate reciprocal square roots, each with one
  // Newton step (an error of about half an ulp, without the branches of an
  // exact division or square root)
  const float kd = __fadd_rn(r, delta);
  q.ix = fma_(rinv, fma_(-kd, rinv, 1.0f), rinv);
  const float dxf = __fadd_rn(sx, ex), dyf = __fadd_rn(sy, ey), dzf = __fadd_rn(sz, ez);
  const float rho2 = fma_(dxf, dxf, dyf * dyf);
  const float w = rsqrtf(rho2);
  const float t = rho2 * w;  // rho
  const float e = 0.5f * fma_(-t, w, 1.0f);
  const bool off_axis = rho2 > 0.0f;  // on the z axis phi does not matter
  const float ir = fma_(w, e, w);
  q.ct = dzf * q.ix;
  q.st = off_axis ? fma_(t, e, t) * q.ix : 0.0f;
  q.cph = off_axis ? dxf * ir : 1.0f;
  q.sph = off_axis ? dyf * ir : 0.0f;
  return q;
}

// FP64 pair geometry (the FP64 kernel)
__device__ __forceinline__ GeomS<double> geometry(double dx, double dy, double dz, double k) {
  const double d = sqrt(fma_(dx, dx, fma_(dy, dy, dz * dz)));
  const double kd = k * d;
  const double TWO_PI = 6.283185307179586476925286766559;
  const double ph = fma_(-rint(kd * (1.0 / TWO_PI)), TWO_PI, kd);
  GeomS<double> q;
  sincos(ph, &q.sn, &q.cs);
  q.ix = 1.0 / kd;
  const double id = 1.0 / d;
  const double rho = sqrt(fma_(dx, dx, dy * dy));
  q.ct = dz * id;
  q.st = rho * id;
  const double ir = rho > 0.0 ? 1.0 / rho : 0.0;
  q.cph = rho > 0.0 ? dx * ir : 1.0;
  q.sph = dy * ir;
  return q;
}

// ---- rotation blocks C and S of degree l -----------------------------------
template <int L, int l, int KIND, int MU, int M, int Q, typename R>
__device__ __forceinline__ void rot_term(const Angles<L, R>& g, R& acc) {
  using E = RotCoef<l, KIND, MU, M, Q>;
  if constexpr (E::v != 0.0) {
    constexpr R c = static_cast<R>(E::v);
    const R f = E::sine ? g.st[Q] : g.ct[Q];
    if constexpr (Q == 0) acc = c;
    else acc = E::before() == 0 ? c * f : fma_(c, f, acc);
  }
}
template <int L, int l, int KIND, int MU, int M, typename R, int... QI>
__device__ __forceinline__ R rot_value(const Angles<L, R>& g, std::integer_sequence<int, QI...>) {
  R acc = static_cast<R>(0);
  (rot_term<L, l, KIND, MU, M, QI>(g, acc), ...);
  return acc;
}
template <int L, int l, int KIND, int MU, typename R, int... MI>
__device__ __forceinline__ void rot_table_row(const Angles<L, R>& g, R* v, std::integer_sequence<int, MI...>) {
  ((v[rot_id(KIND, MU, MI + KIND)] = rot_value<L, l, KIND, MU, MI + KIND>(g, std::make_integer_sequence<int, l + 1>{})),
   ...);
}
template <int L, int l, typename R, int... MUI>
__device__ __forceinline__ void rot_table(const Angles<L, R>& g, R* vc, R* vs, std::integer_sequence<int, MUI...>) {
  (rot_table_row<L, l, 0, MUI>(g, vc, std::make_integer_sequence<int, MUI + 1>{}), ...);
  (rot_table_row<L, l, 1, MUI>(g, vs, std::make_integer_sequence<int, MUI>{}), ...);
}

// row index of (l, m) inside one polarisation block
template <int l, int m>
struct Row {
  static constexpr int r = l * (l + 1) - 1 + m;
};

// row mu of block KIND times in[tau][.] (C: columns 0..l, S: 1..l, stored from 0)
template <int l, int KIND, int MU, typename R, int... MI>
__device__ __forceinline__ C2<R> rot_row(const R* v, const C2<R>* in, std::integer_sequence<int, MI...>) {
  if constexpr (RotEntry<l, KIND, KIND, KIND>::unit()) {
    if constexpr (RotCoef<l, KIND, KIND, KIND, 0>::v > 0.0) return in[0];
    else return C2<R>{-in[0].x, -in[0].y};
  } else {
    C2<R> a = mul2(v[rot_id(KIND, MU + KIND, KIND)], in[0]);
    ((a = fma2(v[rot_id(KIND, MU + KIND, MI + 1 + KIND)], in[MI + 1], a)), ...);
    return a;
  }
}
template <int l, int KIND, typename R, int... MUI>
__device__ __forceinline__ void rot_apply(const R* v, const C2<R>* in, C2<R>* out,
                                          std::integer_sequence<int, MUI...>) {
  constexpr int n = KIND == 0 ? l + 1 : l;
  ((out[MUI] = rot_row<l, KIND, MUI>(v, in, std::make_integer_sequence<int, n - 1>{})), ...);
}

// ---- step 2: x' = (C, S) (x turned by phi), degree l ------------------------
template <int L, int l, typename R, typename XV>
__device__ __forceinline__ void rot_fwd_block(const Angles<L, R>& g, const Quad4<R>* __restrict__ xs, XV& xp) {
  C2<R> c[2][l + 1], s[2][l], oc[2][l + 1], os[2][l];
  {
    const Quad4<R> q = xs[Row<l, 0>::r];
    c[0][0] = C2<R>{q.x, q.y};
    c[1][0] = C2<R>{q.z, q.w};
  }
#pragma unroll
  for (int m = 1; m <= l; ++m) {
    const Quad4<R> qc = xs[l * (l + 1) - 1 + m], qs = xs[l * (l + 1) - 1 - m];
    const R cf = g.cf[m], sf = g.sf[m];
    c[0][m] = fma2(cf, C2<R>{qc.x, qc.y}, mul2(sf, C2<R>{qs.x, qs.y}));
    s[0][m - 1] = fma2(cf, C2<R>{qs.x, qs.y}, mul2(-sf, C2<R>{qc.x, qc.y}));
    c[1][m] = fma2(cf, C2<R>{qc.z, qc.w}, mul2(sf, C2<R>{qs.z, qs.w}));
    s[1][m - 1] = fma2(cf, C2<R>{qs.z, qs.w}, mul2(-sf, C2<R>{qc.z, qc.w}));
  }
  R vc[RotCount<l>::nc], vs[RotCount<l>::ns];
  rot_table<L, l>(g, vc, vs, std::make_integer_sequence<int, l + 1>{});
  rot_apply<l, 0>(vc, c[0], oc[0], std::make_integer_sequence<int, l + 1>{});
  rot_apply<l, 0>(vc, c[1], oc[1], std::make_integer_sequence<int, l + 1>{});
  rot_apply<l, 1>(vs, s[0], os[0], std::make_integer_sequence<int, l>{});
  rot_apply<l, 1>(vs, s[1], os[1], std::make_integer_sequence<int, l>{});
#pragma unroll
  for (int t = 0; t < 2; ++t) {
#pragma unroll
    for (int m = 0; m <= l; ++m) {
      xp(4 * (l * (l + 1) - 1 + m) + 2 * t) = oc[t][m].x;
      xp(4 * (l * (l + 1) - 1 + m) + 2 * t + 1) = oc[t][m].y;
    }
#pragma unroll
    for (int m = 0; m < l; ++m) {
      xp(4 * (l * (l + 1) - 2 - m) + 2 * t) = os[t][m].x;
      xp(4 * (l * (l + 1) - 2 - m) + 2 * t + 1) = os[t][m].y;
    }
  }
}
template <int L, typename R, typename XV, int... LI>
__device__ __forceinline__ void rot_fwd(const Angles<L, R>& g, const Quad4<R>* __restrict__ xs, XV& xp,
                                        std::integer_sequence<int, LI...>) {
  (rot_fwd_block<L, LI + 1>(g, xs, xp), ...);
}

// ---- step 3: axial translation, in place (y' overwrites x') -----------------
// (MU > 0: times 1/2, the factor of going to the sums and back)
template <int L, int MU, int LO, int LI, int T, typename R>
__device__ __forceinline__ void ax_a(const Hankel<L, R>& h, R& ar, R& ai) {
  using A = AxialA<L, MU, LO, LI, T>;
  constexpr R C = static_cast<R>(MU > 0 ? 0.5 * A::c : A::c);
  ar = T == 0 ? C * h.re[A::p] : fma_(C, h.re[A::p], ar);
  ai = T == 0 ? C * h.im[A::p] : fma_(C, h.im[A::p], ai);
}
template <int L, int MU, int LO, int LI, int T, typename R>
__device__ __forceinline__ void ax_b(const Hankel<L, R>& h, R& br, R& bi) {
  using B = AxialB<L, MU, LO, LI, T>;
  constexpr R C = static_cast<R>(MU > 0 ? 0.5 * B::c : B::c);
  br = T == 0 ? C * h.re[B::p] : fma_(C, h.re[B::p], br);
  bi = T == 0 ? C * h.im[B::p] : fma_(C, h.im[B::p], bi);
}
template <int L, int MU, int LO, int LI, typename R, int... KA, int... KB>
__device__ __forceinline__ void ax_entry(const Hankel<L, R>& h, R& ar, R& ai, R& br, R& bi,
                                         std::integer_sequence<int, KA...>, std::integer_sequence<int, KB...>) {
  (ax_a<L, MU, LO, LI, KA>(h, ar, ai), ...);
  (ax_b<L, MU, LO, LI, KB>(h, br, bi), ...);
}

// The axial products of mu > 0 on the packed FMA as well, both sums of one
// factor together: at lmax 4 the scalar half of the FP32 lanes is the fuller
// one without it (N = 10 000: 7.84 -> 7.68 ms; 1.77 -> 1.83 ms at lmax 2, 403 ->
// 407 ms at N = 100 000 and lmax 3, 16.4 -> 16.5 ms at lmax 5)
template <int L, typename R>
constexpr bool kPackedAxial = sizeof(R) == 4 && L == 4;

// y += w x for two complex values of one factor: y, x = (re, im, re, im)
__device__ __forceinline__ void cmac_pair(float* y, float wr, float wi, const float* x) {
  const C2<float> xr{x[0], x[2]}, xi{x[1], x[3]};
  const C2<float> yr = fma2(wr, xr, fma2(-wi, xi, C2<float>{y[0], y[2]}));
  const C2<float> yi = fma2(wr, xi, fma2(wi, xr, C2<float>{y[1], y[3]}));
  y[0] = yr.x;
  y[1] = yi.x;
  y[2] = yr.y;
  y[3] = yi.y;
}

// y += S w x for one (row, column) entry, S = +-1 at compile time
template <int S, typename R>
__device__ __forceinline__ void cmac_s(R* y, R wr, R wi, const R* x) {
  if constexpr (S > 0) {
    y[0] = fma_(wr, x[0], fma_(-wi, x[1], y[0]));
    y[1] = fma_(wr, x[1], fma_(wi, x[0], y[1]));
  } else {
    y[0] = fma_(-wr, x[0], fma_(wi, x[1], y[0]));
    y[1] = fma_(-wr, x[1], fma_(-wi, x[0], y[1]));
  }
}

// Transpose symmetry of the axial block: for a translation along +z the entry
// (l', l) of every |mu| equals (-1)^{l + l'} times the entry (l, l') (A and B
// alike; it follows from the inversion parity of the SVWFs, and is checked
// against the dense coupling matrix).  So each entry with LO <= LI is formed
// once and applied to row LO (column LI) and, with that sign, to row LI
// (column LO).  u[l - 1], y[l - 1]: the sums of degree l, MU > 0
// (c1 + s2, c2 - s1 | c1 - s2, c2 + s1), MU = 0 (c1, c2), re and im each.
template <int L, int MU, int LO, int LI, typename R>
__device__ __forceinline__ void ax_sym_pair(const Hankel<L, R>& h, const R (&u)[L][8], R (&y)[L][8]) {
  if constexpr (LO >= MU && LI >= MU && LO <= LI) {
    R ar = 0, ai = 0, br = 0, bi = 0;
    ax_entry<L, MU, LO, LI>(h, ar, ai, br, bi, std::make_integer_sequence<int, AxialN<L, MU, LO, LI>::na>{},
                            std::make_integer_sequence<int, AxialN<L, MU, LO, LI>::nb>{});
    constexpr int S = ((LO + LI) & 1) ? -1 : 1;
    if constexpr (MU == 0) {
      cmac_s<1>(y[LO - 1], ar, ai, u[LI - 1]);
      cmac_s<1>(y[LO - 1] + 2, ar, ai, u[LI - 1] + 2);
      if constexpr (LO != LI) {
        cmac_s<S>(y[LI - 1], ar, ai, u[LO - 1]);
        cmac_s<S>(y[LI - 1] + 2, ar, ai, u[LO - 1] + 2);
      }
    } else {
      // W+ = A + i B', W- = A - i B'
      const R wpr = ar - bi, wpi = ai + br, wmr = ar + bi, wmi = ai - br;
      if constexpr (kPackedAxial<L, R>) {
        cmac_pair(y[LO - 1], wpr, wpi, u[LI - 1]);
        cmac_pair(y[LO - 1] + 4, wmr, wmi, u[LI - 1] + 4);
        if constexpr (LO != LI) {
          constexpr R SS = static_cast<R>(S);
          cmac_pair(y[LI - 1], SS * wpr, SS * wpi, u[LO - 1]);
          cmac_pair(y[LI - 1] + 4, SS * wmr, SS * wmi, u[LO - 1] + 4);
        }
        return;
      }
      cmac_s<1>(y[LO - 1], wpr, wpi, u[LI - 1]);
      cmac_s<1>(y[LO - 1] + 2, wpr, wpi, u[LI - 1] + 2);
      cmac_s<1>(y[LO - 1] + 4, wmr, wmi, u[LI - 1] + 4);
      cmac_s<1>(y[LO - 1] + 6, wmr, wmi, u[LI - 1] + 6);
      if constexpr (LO != LI) {
        cmac_s<S>(y[LI - 1], wpr, wpi, u[LO - 1]);
        cmac_s<S>(y[LI - 1] + 2, wpr, wpi, u[LO - 1] + 2);
        cmac_s<S>(y[LI - 1] + 4, wmr, wmi, u[LO - 1] + 4);
        cmac_s<S>(y[LI - 1] + 6, wmr, wmi, u[LO - 1] + 6);
      }
    }
  }
}
template <int L, int MU, int LO, typename R, int... LII>
__device__ __forceinline__ void ax_sym_row(const Hankel<L, R>& h, const R (&u)[L][8], R (&y)[L][8],
                                           std::integer_sequence<int, LII...>) {
  (ax_sym_pair<L, MU, LO, LII + 1>(h, u, y), ...);
}
template <int L, int MU, int l, typename R, typename XV>
__device__ __forceinline__ void ax_load(XV& xp, R (&u)[L][8], R (&y)[L][8]) {
  if constexpr (l >= MU) {
    constexpr int rc = 4 * Row<l, MU>::r, rs = 4 * Row<l, -MU>::r;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const R c1 = xp(rc + q), c2 = xp(rc + 2 + q);
      if constexpr (MU == 0) {
        u[l - 1][q] = c1;
        u[l - 1][2 + q] = c2;
      } else {
        const R s1 = xp(rs + q), s2 = xp(rs + 2 + q);
        u[l - 1][q] = c1 + s2;
        u[l - 1][2 + q] = c2 - s1;
        u[l - 1][4 + q] = c1 - s2;
        u[l - 1][6 + q] = c2 + s1;
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) y[l - 1][q] = static_cast<R>(0);
  }
}
template <int L, int MU, int l, typename R, typename XV>
__device__ __forceinline__ void ax_store(XV& xp, const R (&y)[L][8]) {
  if constexpr (l >= MU) {
    constexpr int rc = 4 * Row<l, MU>::r, rs = 4 * Row<l, -MU>::r;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if constexpr (MU == 0) {
        xp(rc + q) = y[l - 1][q];
        xp(rc + 2 + q) = y[l - 1][2 + q];
      } else {
        xp(rc + q) = y[l - 1][q] + y[l - 1][4 + q];
        xp(rc + 2 + q) = y[l - 1][2 + q] + y[l - 1][6 + q];
        xp(rs + q) = y[l - 1][6 + q] - y[l - 1][2 + q];
        xp(rs + 2 + q) = y[l - 1][q] - y[l - 1][4 + q];
      }
    }
  }
}
template <int L, int MU, typename R, typename XV, int... LOI>
__device__ __forceinline__ void ax_mu(const Hankel<L, R>& h, XV& xp, std::integer_sequence<int, LOI...>) {
  R u[L][8], y[L][8];
  (ax_load<L, MU, LOI + 1>(xp, u, y), ...);
  (ax_sym_row<L, MU, LOI + 1>(h, u, y, std::make_integer_sequence<int, L>{}), ...);
  (ax_store<L, MU, LOI + 1>(xp, y), ...);
}
template <int L, typename R, typename XV, int... MUS>
__device__ __forceinline__ void axial(const Hankel<L, R>& h, XV& xp, std::integer_sequence<int, MUS...>) {
  (ax_mu<L, MUS>(h, xp, std::make_integer_sequence<int, L>{}), ...);
}

// ---- step 4: y += ((C, S) y') turned back by phi, degree l ------------------
template <int L, int l, typename R, typename XV, typename Acc>
__device__ __forceinline__ void rot_bwd_block(const Angles<L, R>& g, XV& xp, Acc& acc) {
  C2<R> c[2][l + 1], s[2][l], oc[2][l + 1], os[2][l];
#pragma unroll
  for (int t = 0; t < 2; ++t) {
#pragma unroll
    for (int m = 0; m <= l; ++m) {
      const int rc = 4 * (l * (l + 1) - 1 + m) + 2 * t;
      c[t][m] = C2<R>{xp(rc), xp(rc + 1)};
    }
#pragma unroll
    for (int m = 0; m < l; ++m) {
      const int rs = 4 * (l * (l + 1) - 2 - m) + 2 * t;
      s[t][m] = C2<R>{xp(rs), xp(rs + 1)};
    }
  }
  R vc[RotCount<l>::nc], vs[RotCount<l>::ns];
  rot_table<L, l>(g, vc, vs, std::make_integer_sequence<int, l + 1>{});
  rot_apply<l, 0>(vc, c[0], oc[0], std::make_integer_sequence<int, l + 1>{});
  rot_apply<l, 0>(vc, c[1], oc[1], std::make_integer_sequence<int, l + 1>{});
  rot_apply<l, 1>(vs, s[0], os[0], std::make_integer_sequence<int, l>{});
  rot_apply<l, 1>(vs, s[1], os[1], std::make_integer_sequence<int, l>{});
  C2<R> a[2];
  acc.load(Row<l, 0>::r, a);
  a[0] = C2<R>{a[0].x + oc[0][0].x, a[0].y + oc[0][0].y};
  a[1] = C2<R>{a[1].x + oc[1][0].x, a[1].y + oc[1][0].y};
  acc.store(Row<l, 0>::r, a);
#pragma unroll
  for (int m = 1; m <= l; ++m) {
    const int rc = l * (l + 1) - 1 + m, rs = l * (l + 1) - 1 - m;
    const R cf = g.cf[m], sf = g.sf[m];
    acc.load(rc, a);
#pragma unroll
    for (int t = 0; t < 2; ++t) a[t] = fma2(cf, oc[t][m], fma2(-sf, os[t][m - 1], a[t]));
    acc.store(rc, a);
    acc.load(rs, a);
#pragma unroll
    for (int t = 0; t < 2; ++t) a[t] = fma2(cf, os[t][m - 1], fma2(sf, oc[t][m], a[t]));
    acc.store(rs, a);
  }
}
template <int L, typename R, typename XV, typename Acc, int... LI>
__device__ __forceinline__ void rot_bwd(const Angles<L, R>& g, XV& xp, Acc& acc, std::integer_sequence<int, LI...>) {
  (rot_bwd_block<L, LI + 1>(g, xp, acc), ...);
}

// x' and y' of one pair: compile-time indices, in registers as far as they go
template <typename R>
struct AccReg {
  R* a;
  __device__ __forceinline__ R& operator()(int q) const { return a[q]; }
};

// receiver sums, one 4-vector (tau 1 re, im, tau 2 re, im) per row (l, m):
// c_m for m >= 0, s_|m| for m < 0; registers [NH][4], or shared memory
// [NH][BLOCK] of 4-vectors (one 16- or 32-byte access per row)
template <typename R>
struct RowAccReg {
  R* a;
  __device__ __forceinline__ void load(int r, C2<R> (&c)[2]) const {
    c[0] = C2<R>{a[4 * r], a[4 * r + 1]};
    c[1] = C2<R>{a[4 * r + 2], a[4 * r + 3]};
  }
  __device__ __forceinline__ void store(int r, const C2<R> (&c)[2]) const {
    a[4 * r] = c[0].x;
    a[4 * r + 1] = c[0].y;
    a[4 * r + 2] = c[1].x;
    a[4 * r + 3] = c[1].y;
  }
};
template <typename R, int BLOCK>
struct RowAccSmem {
  Quad4<R>* a;  // this thread's element of row 0
  __device__ __forceinline__ void load(int r, C2<R> (&c)[2]) const {
    const Quad4<R> v = a[r * BLOCK];
    c[0] = C2<R>{v.x, v.y};
    c[1] = C2<R>{v.z, v.w};
  }
  __device__ __forceinline__ void store(int r, const C2<R> (&c)[2]) const {
    a[r * BLOCK] = Quad4<R>{c[0].x, c[0].y, c[1].x, c[1].y};
  }
};

// the sums of one receiver from the cosine / sine basis to (y+, y-) =
// (y_1 + y_2, y_1 - y_2) per row, in place, once per tile
template <int L, typename R, typename Acc>
__device__ __forceinline__ void to_plus_minus(Acc& acc) {
  constexpr R H = static_cast<R>(0.5), Q = static_cast<R>(0.70710678118654752440);
#pragma unroll
  for (int l = 1; l <= L; ++l) {
    const int r0 = l * (l + 1) - 1;
    C2<R> a[2], b[2];
    acc.load(r0, a);  // y_1 = c1 / sqrt 2, y_2 = i c2 / sqrt 2
    b[0] = C2<R>{Q * (a[0].x - a[1].y), Q * (a[0].y + a[1].x)};
    b[1] = C2<R>{Q * (a[0].x + a[1].y), Q * (a[0].y - a[1].x)};
    acc.store(r0, b);
#pragma unroll
    for (int m = 1; m <= l; ++m) {
      acc.load(r0 + m, a);  // c1, c2
      acc.load(r0 - m, b);  // s1, s2
      const C2<R> u{a[0].x + b[1].x, a[0].y + b[1].y}, v{a[0].x - b[1].x, a[0].y - b[1].y};
      const C2<R> p{a[1].x - b[0].x, a[1].y - b[0].y}, q{a[1].x + b[0].x, a[1].y + b[0].y};
      // y+_m = (u + i p)/2, y-_m = (v - i q)/2, y+_{-m} = (v + i q)/2, y-_{-m} = (u - i p)/2
      a[0] = C2<R>{H * (u.x - p.y), H * (u.y + p.x)};
      a[1] = C2<R>{H * (v.x + q.y), H * (v.y - q.x)};
      b[0] = C2<R>{H * (v.x - q.y), H * (v.y + q.x)};
      b[1] = C2<R>{H * (u.x + p.y), H * (u.y - p.x)};
      acc.store(r0 + m, a);
      acc.store(r0 - m, b);
    }
  }
}

// Row r of source vector x ([2][NH] complex) in the cosine / sine basis
template <typename R>
__device__ __forceinline__ Quad4<R> stage_row(const Pair2<R>* __restrict__ x, int NH, int r) {
  // degree l holds rows l^2 - 1 .. (l+1)^2 - 2, m = 0 at l (l + 1) - 1
  const int l = 1 + (r >= 3) + (r >= 8) + (r >= 15) + (r >= 24);
  const int m = r - (l * (l + 1) - 1);
  const Pair2<R> a1 = x[r], a2 = x[NH + r];
  if (m == 0) {
    constexpr R Q = static_cast<R>(1.41421356237309504880);
    return Quad4<R>{Q * a1.re, Q * a1.im, Q * a2.im, -Q * a2.re};
  }
  const Pair2<R> b1 = x[r - 2 * m], b2 = x[NH + r - 2 * m];
  if (m > 0) return Quad4<R>{a1.re + b1.re, a1.im + b1.im, a2.im + b2.im, -(a2.re + b2.re)};
  // b is x_|m| here: s1 = i (b1 - a1), s2 = b2 - a2
  return Quad4<R>{a1.im - b1.im, b1.re - a1.re, b2.re - a2.re, b2.im - a2.im};
}

// One pair.  The angle tables are rebuilt for the backward rotation from the
// pair's scalars, read through an optimizer barrier, so that they are not kept
// alive across the axial step (fewer live registers per thread).
template <int L, typename R, typename XV, typename Acc>
__device__ __forceinline__ void pair(const GeomS<R>& q, const Quad4<R>* __restrict__ xs, XV& xp, Acc& acc) {
  {
    const Angles<L, R> g(q.ct, q.st, q.cph, q.sph);
    rot_fwd<L>(g, xs, xp, std::make_integer_sequence<int, L>{});
  }
  {
    const Hankel<L, R> h(q);
    axial<L>(h, xp, std::make_integer_sequence<int, L + 1>{});
  }
  R ct = q.ct, st = q.st, cph = q.cph, sph = q.sph;
  if constexpr (sizeof(R) == 4) asm volatile("" : "+f"(ct), "+f"(st), "+f"(cph), "+f"(sph));
  else asm volatile("" : "+d"(ct), "+d"(st), "+d"(cph), "+d"(sph));
  {
    const Angles<L, R> g(ct, st, cph, sph);
    rot_bwd<L>(g, xp, acc, std::make_integer_sequence<int, L>{});
  }
}

// Launch shape per (lmax, precision).  FP64: the FP64 pipe takes a warp
// instruction every 76 clocks, so every scheduler needs a warp and nothing else
// matters: x' stays in thread-local memory (spilled registers) where a second
// shared-memory array would leave schedulers without one (N = 2000, lmax 5: 56.8
// ms with x' in shared memory and two warps per SM, 33.8 ms with four; lmax 4
// 17.6 -> 16.8 ms with four-warp CTAs, lmax 3 9.09 -> 8.92 ms).  FP32: 64
// receivers a CTA, which idle fewer lanes on a small or ragged number of
// spheres than 128 and cost as little at large ones (lmax 4, N = 10 000: 7.88
// against 7.84 ms; a batch of 12 ensembles x 4 right-hand sides of 300-1163
// spheres 3.79 -> 3.57 ms).
template <int L, typename R>
struct Config {
  static constexpr bool FP64 = sizeof(R) == 8;
  static constexpr int BLOCK = FP64 && L == 4 ? 128 : 64;
  static constexpr int TJ = FP64 ? (L >= 5 ? 8 : 16) : 32;
  static constexpr bool ACC_SMEM = FP64 ? (L >= 2) : (L >= 3);
  static constexpr int MINB = (!FP64 && L == 3) ? 6 : 1;  // minimum resident CTAs per SM for the allocator
  static constexpr bool SYNC_PAIR = false;                // barrier per source
};

// The alternative FP32 launch shape of each lmax, the second candidate of the
// autotuner (celes_ctx tuning): 128 receivers per CTA; at lmax 5 one CTA of 256
// whose warps take every source together, since the code of a pair (about
// 3 600 instructions) is larger than the instruction cache (15.7 against 16.4
// ms).
template <int L, typename R>
struct ConfigAlt : Config<L, R> {
  static constexpr int BLOCK = L == 5 ? 256 : 128;
  static constexpr int MINB = L == 3 ? 3 : 1;
  static constexpr bool SYNC_PAIR = L == 5;
};

template <int L, typename R, typename C = Config<L, R>>
struct Layout {
  static constexpr int NH = L * (L + 2);
  static constexpr size_t col = sizeof(R) * 4 * NH * C::BLOCK;  // one [4 NH][BLOCK] array
  static constexpr size_t off_pos = 0;
  static constexpr size_t off_x = off_pos + sizeof(Pos4) * C::TJ;
  static constexpr size_t off_acc = off_x + sizeof(Quad4<R>) * NH * C::TJ;
  static constexpr size_t bytes = off_acc + (C::ACC_SMEM ? col : 0);
};

// whether `atomic` asks for the in-L2 vector reduction of the partial sums
// (FP32 only; otherwise the request is ignored)
template <typename R>
constexpr bool partial_atomic(bool atomic) {
  return atomic && sizeof(R) == 4;
}

// One tile: receivers rb*BLOCK .. +BLOCK against sources j0 .. j1 - 1; writes
// this tile's partial sums in the +- basis to out ([N][2][NH] complex, the
// slice of the tile's source chunk).  Called by every thread of the CTA.
// CRED (shared-memory accumulators only): the CTAs of one thread-block
// cluster (one receiver block, consecutive source chunks) add their sums
// through distributed shared memory and write one partial per cluster, so
// the partial-sum traffic shrinks by the cluster size.
// ATOM (FP32): the sums are added into out with vector reductions in L2
// (out zero before the launch), so all source chunks share one slice and
// only the final sums reach DRAM; the order of the additions, and so the
// last bits of the result, vary from launch to launch.
template <int L, typename R, typename C, bool CRED = false, bool ATOM = false>
__device__ __forceinline__ void rtr_tile(int N, const Pos4* __restrict__ pos, const Pair2<R>* __restrict__ x,
                                         Pair2<R>* __restrict__ outp, double k, int rb, int j0, int j1,
                                         unsigned char* smem_raw) {
  using LY = Layout<L, R, C>;
  constexpr int NH = L * (L + 2);
  constexpr int BLOCK = C::BLOCK;
  constexpr int TJ = C::TJ;
  Pos4* spos = reinterpret_cast<Pos4*>(smem_raw + LY::off_pos);
  Quad4<R>* sx = reinterpret_cast<Quad4<R>*>(smem_raw + LY::off_x);
  R* sacc = reinterpret_cast<R*>(smem_raw + LY::off_acc);

  const int tid = threadIdx.x;
  const int i = rb * BLOCK + tid;
  const bool active = i < N;
  constexpr bool FF = sizeof(R) == 4;  // FP32: float-float positions scaled by k
  Pos4 ri = Pos4{0, 0, 0, 0};
  if (active) ri = pos[i];
  const PosFF rf = split_pos(ri, k);
  PosFF* sposf = reinterpret_cast<PosFF*>(spos);

  R areg[C::ACC_SMEM ? 1 : 4 * NH];
  Quad4<R>* sacc4 = reinterpret_cast<Quad4<R>*>(sacc);
  if constexpr (C::ACC_SMEM) {
    for (int r = 0; r < NH; ++r) sacc4[r * BLOCK + tid] = Quad4<R>{0, 0, 0, 0};
  } else {
#pragma unroll
    for (int q = 0; q < 4 * NH; ++q) areg[q] = static_cast<R>(0);
  }

  for (int jt = j0; jt < j1; jt += TJ) {
    const int nj = min(TJ, j1 - jt);
    __syncthreads();
    for (int q = tid; q < nj * NH; q += BLOCK) {
      const int jj = q / NH;
      const int r = q - jj * NH;
      sx[q] = stage_row<R>(x + (size_t)(jt + jj) * (2 * NH), NH, r);
    }
    if constexpr (FF) {
      for (int q = tid; q < nj; q += BLOCK) sposf[q] = split_pos(pos[jt + q], k);
    } else {
      for (int q = tid; q < nj; q += BLOCK) spos[q] = pos[jt + q];
    }
    __syncthreads();
    for (int jj = 0; jj < nj; ++jj) {
      if constexpr (C::SYNC_PAIR) __syncthreads();
      if (!active || jt + jj == i) continue;  // no self coupling
      GeomS<R> gs;
      if constexpr (FF) {
        gs = geometry_ff(rf, sposf[jj]);
      } else {
        const Pos4 rj = spos[jj];
        gs = geometry(ri.x - rj.x, ri.y - rj.y, ri.z - rj.z, k);
      }
      const Quad4<R>* xs = sx + jj * NH;
      R xa[4 * NH];
      AccReg<R> xp{xa};
      if constexpr (C::ACC_SMEM) {
        RowAccSmem<R, BLOCK> acc{sacc4 + tid};
        pair<L, R>(gs, xs, xp, acc);
      } else {
        RowAccReg<R> acc{areg};
        pair<L, R>(gs, xs, xp, acc);
      }
    }
  }
  if constexpr (C::ACC_SMEM) {
    RowAccSmem<R, BLOCK> acc{sacc4 + tid};
    to_plus_minus<L, R>(acc);
  } else {
    RowAccReg<R> acc{areg};
    to_plus_minus<L, R>(acc);
  }
  if constexpr (CRED) {
    static_assert(C::ACC_SMEM, "the cluster reduction reads shared-memory accumulators");
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int ncl = static_cast<int>(cl.num_blocks());
    const int rk = static_cast<int>(cl.block_rank());
    cl.sync();  // every CTA of the cluster has its sums in shared memory
    if (active) {
      Pair2<R>* out = outp + (size_t)i * (2 * NH);
      // rows dealt round robin over the cluster's CTAs; ranks added in order
      for (int r = rk; r < NH; r += ncl) {
        R a0 = 0, a1 = 0, a2 = 0, a3 = 0;
        for (int q = 0; q < ncl; ++q) {
          const Quad4<R> v = cl.map_shared_rank(sacc4, q)[r * BLOCK + tid];
          a0 += v.x;
          a1 += v.y;
          a2 += v.z;
          a3 += v.w;
        }
        if constexpr (ATOM) {
          atomicAdd(reinterpret_cast<float2*>(out + r), make_float2(a0, a1));
          atomicAdd(reinterpret_cast<float2*>(out + NH + r), make_float2(a2, a3));
        } else {
          out[r] = Pair2<R>{a0, a1};
          out[NH + r] = Pair2<R>{a2, a3};
        }
      }
    }
    cl.sync();  // no CTA leaves while others read its shared memory
    return;
  }
  if constexpr (ATOM) {
    static_assert(sizeof(R) == 4, "vector reductions of the partial sums are FP32 only");
    // the 2 NH complex sums of a receiver are NH float4 (element pairs 2p,
    // 2p+1 of the flattened [2][NH] row: the + rows, then the - rows)
    auto elem = [&](int t, int e, float& re, float& im) {
      const int r = e < NH ? e : e - NH;
      if constexpr (C::ACC_SMEM) {
        const Quad4<R> v = sacc4[r * BLOCK + t];
        re = e < NH ? v.x : v.z;
        im = e < NH ? v.y : v.w;
      } else {
        re = areg[4 * r + (e < NH ? 0 : 2)];
        im = areg[4 * r + (e < NH ? 1 : 3)];
      }
    };
    if constexpr (C::ACC_SMEM) {
      // a warp's 32 receivers are contiguous in out: lane-consecutive float4
      // (512 B per warp instruction); each thread's sums are written by its
      // own thread only, so the warp's accumulators are complete here
      __syncwarp();
      const int w0 = tid & ~31;
      const int lane = tid & 31;
      float4* base = reinterpret_cast<float4*>(outp + (size_t)(rb * BLOCK + w0) * (2 * NH));
      for (int q = lane; q < 32 * NH; q += 32) {
        const int t = q / NH;
        const int p = q - t * NH;
        if (rb * BLOCK + w0 + t >= N) break;  // q ascending: later q are further receivers
        float4 v;
        elem(w0 + t, 2 * p, v.x, v.y);
        elem(w0 + t, 2 * p + 1, v.z, v.w);
        atomicAdd(base + q, v);
      }
    } else if (active) {
      float4* base = reinterpret_cast<float4*>(outp + (size_t)i * (2 * NH));
#pragma unroll
      for (int p = 0; p < NH; ++p) {
        float4 v;
        elem(tid, 2 * p, v.x, v.y);
        elem(tid, 2 * p + 1, v.z, v.w);
        atomicAdd(base + p, v);
      }
    }
    return;
  }
  if (active) {
    // partial layout [2][NH] complex: y+ rows, then y- rows
    Pair2<R>* out = outp + (size_t)i * (2 * NH);
    if constexpr (C::ACC_SMEM) {
      for (int r = 0; r < NH; ++r) {
        const Quad4<R> v = sacc4[r * BLOCK + tid];
        out[r] = Pair2<R>{v.x, v.y};
        out[NH + r] = Pair2<R>{v.z, v.w};
      }
    } else {
#pragma unroll
      for (int r = 0; r < NH; ++r) {
        out[r] = Pair2<R>{areg[4 * r], areg[4 * r + 1]};
        out[NH + r] = Pair2<R>{areg[4 * r + 2], areg[4 * r + 3]};
      }
    }
  }
}

// grid (receiver blocks of BLOCK, source chunks, right-hand sides); writes
// partial sums in the +- basis, [rhs][slices][N][2][NH] complex (per right-hand
// side the layout of the direct kernel)
// CRED: launched with clusters of `ncl` CTAs along y; cluster c writes
// partial slice c (the grid's y extent is a multiple of ncl)
// ATOM: every tile adds into slice 0 of its right-hand side (zero before the launch)
template <int L, typename R, typename C = Config<L, R>, bool CRED = false, bool ATOM = false>
__global__ void __launch_bounds__(C::BLOCK, C::MINB)
    rtr_partial_kernel(int N, const Pos4* __restrict__ pos, const Pair2<R>* __restrict__ x,
                       Pair2<R>* __restrict__ partial, double k, int chunk, int ncl) {
  extern __shared__ __align__(32) unsigned char smem_raw[];
  constexpr int NH = L * (L + 2);
  const int j0 = blockIdx.y * chunk;
  const int j1 = min(N, j0 + chunk);
  if (ATOM && !CRED && j0 >= j1) return;  // a chunk past the last source adds nothing
  const size_t slices = ATOM ? 1 : (CRED ? gridDim.y / ncl : gridDim.y);
  const size_t slice = blockIdx.z * slices + (ATOM ? 0 : (CRED ? blockIdx.y / ncl : blockIdx.y));
  rtr_tile<L, R, C, CRED, ATOM>(N, pos, x + (size_t)blockIdx.z * N * (2 * NH), partial + slice * N * (2 * NH), k,
                                blockIdx.x, j0, j1, smem_raw);
}

// ---- batched form: one persistent launch over the tiles of many systems ----
// A system is one right-hand side of one sphere ensemble (all of the same
// lmax in one launch).  Its tiles are (receiver block, source chunk) pairs
// numbered tile0 .. tile0 + nrb * chunks - 1 within the launch; CTAs take
// tiles from a global counter (dynamic scheduling, so uneven ensembles
// balance), and systems whose flag `active` is 0 are skipped.  The FP32
// launch adds all chunks of a system into its one partial slice in L2 (the
// batched epilogue reads the slice and zeroes it again); the FP64 launch
// writes one slice per chunk.
struct BatchSys {
  const Pos4* pos;
  const void* x;      // input vector [N][nmax] complex (FP32 or FP64 as launched)
  void* y;            // output [N][nmax]
  void* partial;      // [chunks][N][2][NH] scratch
  const void* tq;     // T [N][2][L] complex in the launch's precision (master operator)
  double k;
  long long tile0;
  int N, L, chunk, nrb, chunks, active;
};

template <int L, typename R, typename C = Config<L, R>, bool ATOM = partial_atomic<R>(true)>
__global__ void __launch_bounds__(C::BLOCK, C::MINB)
    rtr_batch_kernel(const BatchSys* __restrict__ sys, int nsys, long long ntiles,
                     unsigned long long* __restrict__ counter) {
  extern __shared__ __align__(32) unsigned char smem_raw[];
  constexpr int NH = L * (L + 2);
  __shared__ long long tile_s;
  for (;;) {
    if (threadIdx.x == 0) tile_s = static_cast<long long>(atomicAdd(counter, 1ULL));
    __syncthreads();
    const long long t = tile_s;
    __syncthreads();
    if (t >= ntiles) break;
    // system holding tile t (tile0 ascending)
    int lo = 0, hi = nsys - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (sys[mid].tile0 <= t) lo = mid;
      else hi = mid - 1;
    }
    const BatchSys& S = sys[lo];
    if (!S.active) continue;
    const int local = static_cast<int>(t - S.tile0);
    const int rb = local % S.nrb, ch = local / S.nrb;
    if (ch >= S.chunks) continue;  // never taken with consistent descriptors
    const int j0 = ch * S.chunk;
    const int j1 = min(S.N, j0 + S.chunk);
    rtr_tile<L, R, C, false, ATOM>(S.N, S.pos, static_cast<const Pair2<R>*>(S.x),
                                   static_cast<Pair2<R>*>(S.partial) + (ATOM ? 0 : (size_t)ch * S.N * (2 * NH)), S.k,
                                   rb, j0, j1, smem_raw);
  }
}

// one-time setup of a kernel's shared-memory limit; returns its resident CTAs
// per SM (0 on error)
template <typename K>
int kernel_setup(K* kern, int block, size_t smem) {
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
    return 0;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, block, smem) != cudaSuccess) return 0;
  return occ;
}

// resident CTAs per SM of the per-context and the batched kernel on the
// current device; the first call on each device sets the kernel's
// shared-memory limit there (0 on error)
template <int L, typename R, typename C = Config<L, R>>
int partial_occupancy() {
  static PerDevice cache;
  return cache.get(current_device,
                   [] { return kernel_setup(rtr_partial_kernel<L, R, C, false>, C::BLOCK, Layout<L, R, C>::bytes); });
}
template <int L, typename R, typename C = Config<L, R>>
int batch_occupancy() {
  static PerDevice cache;
  return cache.get(current_device,
                   [] { return kernel_setup(rtr_batch_kernel<L, R, C>, C::BLOCK, Layout<L, R, C>::bytes); });
}

// resident CTAs of the per-context kernel on the whole GPU (SMs x CTAs per SM)
template <int L, typename R, typename C = Config<L, R>>
int resident_slots() {
  const int occ = partial_occupancy<L, R, C>();
  return device_sms() * (occ > 0 ? occ : 1);
}

// cluster size of the partial-sum reduction for `chunks` source chunks: the
// largest of 8, 4, 2 that divides it (shared-memory accumulators only), else 1
template <int L, typename R, typename C = Config<L, R>>
int partial_cluster(int chunks, int maxcl) {
  if constexpr (!C::ACC_SMEM) {
    return 1;
  } else {
    for (int c = 8; c > 1; c >>= 1)
      if (c <= maxcl && chunks % c == 0) return c;
    return 1;
  }
}

// resident CTAs per SM of one reduction form of the per-context kernel (the
// first call on each device sets its shared-memory limit there)
template <int L, typename R, typename C, bool CRED, bool ATOM>
int partial_form_occupancy() {
  static PerDevice cache;
  return cache.get(current_device, [] {
    return kernel_setup(rtr_partial_kernel<L, R, C, CRED, ATOM>, C::BLOCK, Layout<L, R, C>::bytes);
  });
}

// partial-sum slices the epilogue must add after a launch with these options
template <int L, typename R, typename C = Config<L, R>>
int partial_slices(int chunks, int maxcl, bool atomic) {
  if (partial_atomic<R>(atomic)) return 1;
  return chunks / partial_cluster<L, R, C>(chunks, maxcl);
}

template <int L, typename R, typename C, bool CRED, bool ATOM>
cudaError_t launch_partial_form(int64_t N, const void* pos, const void* x, void* partial, double k, int chunks,
                                int ncl, cudaStream_t st, int nrhs) {
  using LY = Layout<L, R, C>;
  if (partial_form_occupancy<L, R, C, CRED, ATOM>() < 1) return cudaErrorInvalidConfiguration;
  const int64_t chunk = (N + chunks - 1) / chunks;
  dim3 grid(static_cast<unsigned>((N + C::BLOCK - 1) / C::BLOCK), static_cast<unsigned>(chunks),
            static_cast<unsigned>(nrhs));
  if constexpr (CRED) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(C::BLOCK);
    cfg.dynamicSmemBytes = LY::bytes;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = static_cast<unsigned>(ncl);
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, rtr_partial_kernel<L, R, C, true, ATOM>, static_cast<int>(N),
                                             static_cast<const Pos4*>(pos), static_cast<const Pair2<R>*>(x),
                                             static_cast<Pair2<R>*>(partial), k, static_cast<int>(chunk), ncl);
    note_launch();
    return e;
  } else {
    rtr_partial_kernel<L, R, C, false, ATOM><<<grid, C::BLOCK, LY::bytes, st>>>(
        static_cast<int>(N), static_cast<const Pos4*>(pos), static_cast<const Pair2<R>*>(x),
        static_cast<Pair2<R>*>(partial), k, static_cast<int>(chunk), 1);
    note_launch();
    return cudaGetLastError();
  }
}

// `chunks` source chunks, partial-sum clusters of at most `maxcl` CTAs (1:
// no cluster reduction), `atomic`: all chunks added into one slice in L2
// (FP32; the caller hands that slice over zeroed); writes, for each of nrhs
// right-hand sides, partial_slices(chunks, maxcl, atomic) partial slices (the
// count the epilogue must add)
template <int L, typename R, typename C = Config<L, R>>
cudaError_t launch_partial(int64_t N, const void* pos, const void* x, void* partial, double k, int chunks,
                           cudaStream_t st, int maxcl = 1, bool atomic = false, int nrhs = 1) {
  const int occ = partial_occupancy<L, R, C>();
  if (occ < 1) return cudaErrorInvalidConfiguration;
  if (N <= 0) return cudaSuccess;
  if (chunks < 1) chunks = 1;
  const int ncl = partial_cluster<L, R, C>(chunks, maxcl);
  constexpr bool AT_OK = partial_atomic<R>(true);
  if (ncl > 1) {
    if constexpr (C::ACC_SMEM) {
      if (AT_OK && atomic) return launch_partial_form<L, R, C, true, AT_OK>(N, pos, x, partial, k, chunks, ncl, st, nrhs);
      return launch_partial_form<L, R, C, true, false>(N, pos, x, partial, k, chunks, ncl, st, nrhs);
    }
  }
  if (AT_OK && atomic) return launch_partial_form<L, R, C, false, AT_OK>(N, pos, x, partial, k, chunks, 1, st, nrhs);
  return launch_partial_form<L, R, C, false, false>(N, pos, x, partial, k, chunks, 1, st, nrhs);
}

// persistent batched launch: one CTA per resident slot, tiles from `counter`
// (zeroed by the caller before the launch)
template <int L, typename R, typename C = Config<L, R>>
cudaError_t launch_batch(const void* sys, int nsys, long long ntiles, unsigned long long* counter, cudaStream_t st) {
  using LY = Layout<L, R, C>;
  const int occ = batch_occupancy<L, R, C>();
  if (occ < 1) return cudaErrorInvalidConfiguration;
  if (nsys <= 0 || ntiles <= 0) return cudaSuccess;
  const long long slots = static_cast<long long>(device_sms()) * occ;
  const unsigned grid = static_cast<unsigned>(ntiles < slots ? ntiles : slots);
  rtr_batch_kernel<L, R, C><<<grid, C::BLOCK, LY::bytes, st>>>(static_cast<const BatchSys*>(sys), nsys, ntiles,
                                                                counter);
  note_launch();
  return cudaGetLastError();
}

}  // namespace rtr
}  // namespace celes

namespace celes {
namespace rtr {
static_assert(Layout<5, float>::bytes <= 227 * 1024, "shared memory of the lmax 5 FP32 kernel");
static_assert(Layout<5, double>::bytes <= 227 * 1024, "shared memory of the lmax 5 FP64 kernel");
static_assert(Layout<4, float>::bytes <= 227 * 1024, "shared memory of the lmax 4 FP32 kernel");
}  // namespace rtr
}  // namespace celes
