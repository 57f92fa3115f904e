// Electric field at arbitrary points (Sec. 2.1; the near-field maps of the
// paper's examples), FP64:
//   scattered  E_s(r) = sum_i sum_n b^i_n Psi^(3)_n(r - r_i)
//   incident   plane wave E0 Phi_pol(alpha, beta; r) (App. A.1), or the
//              Gaussian beam's angular spectrum integral (App. C), evaluated
//              with the same beta range and Gauss-Legendre nodes as its
//              expansion coefficients; the integral over alpha is J_0, J_1
//              and J_2 of k rho sin(beta)
//   total      E_s + E_in
// Psi^(3) in the form of App. A.1 with the normalised Legendre functions
// P_l^m, pi_l^m = P_l^m / sin(theta) and tau_l^m = dP_l^m/dtheta (no
// Condon-Shortley phase).  The expansion about sphere i holds outside that
// sphere only, so points inside a sphere get NaN in the scattered and total
// fields (the internal field is not part of this call).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "../../include/celes.h"
#include "cmath.cuh"
#include "coupling_kernel.cuh"
#include "coupling_tables.cuh"
#include "kernels.h"

namespace celes {
namespace {

constexpr int kNfThreads = 128;  // plane wave and sums
constexpr int kNfPoints = 64;    // points of a CTA of the scattered field
constexpr int kNfTile = 16;      // spheres staged at a time
constexpr int kNfWarps = 8;      // points of a CTA of the Gaussian beam, one per warp

// one sphere's coefficients of row (l, +-m), normalised by 1/sqrt(2l(l+1)):
// c_m = b_m + b_{-m} at (l, m >= 0), s_m = i (b_m - b_{-m}) at (l, -m), both tau
struct NfRow {
  double c1r, c1i, c2r, c2i;
};

// constants of the recursions of pi_l^m (normalised Legendre functions)
constexpr double nf_diag(int m) {  // pi_m^m / sin^{m-1}
  double c = 0.70710678118654752440;
  for (int q = 1; q <= m; ++q) c *= tab::csqrt((2.0 * q + 1.0) / (2.0 * q));
  return c;
}
constexpr double nf_a(int l, int m) { return tab::csqrt((4.0 * l * l - 1.0) / (1.0 * l * l - 1.0 * m * m)); }
constexpr double nf_b(int l, int m) {
  return tab::csqrt(((l - 1.0) * (l - 1.0) - 1.0 * m * m) / (4.0 * (l - 1.0) * (l - 1.0) - 1.0));
}
constexpr double nf_f(int l, int m) {
  return tab::csqrt((2.0 * l + 1.0) * (1.0 * l * l - 1.0 * m * m) / (2.0 * l - 1.0));
}

// sums over m of one degree, both parts: tau 1: m pi V and tau U; tau 2: P U,
// tau U and m pi V, with U, V = the two sums of b_{+-m} e^{+-i m phi}
template <int L>
struct NfSums {
  double pv1[L + 1][2] = {}, tu1[L + 1][2] = {}, pu2[L + 1][2] = {}, tu2[L + 1][2] = {}, pv2[L + 1][2] = {};
};

template <int L, int m, int l>
__device__ __forceinline__ void nf_degree(const NfRow* __restrict__ rows, double ct, double st, double cm, double sm,
                                          double& p0, double& p1, NfSums<L>& S) {
  // pi_l^m from the two before it
  double pi;
  if constexpr (l == m) pi = p0;
  else if constexpr (l == m + 1) {
    constexpr double A = tab::csqrt(2.0 * m + 3.0);
    pi = A * ct * p0;
  } else {
    constexpr double A = nf_a(l, m), AB = nf_a(l, m) * nf_b(l, m);
    pi = fma(A * ct, p1, -AB * p0);
  }
  double tau = l * ct * pi;
  if constexpr (l > m) {
    constexpr double F = nf_f(l, m);
    tau = fma(-F, l == m + 1 ? p0 : p1, tau);
  }
  if constexpr (l > m) {
    if constexpr (l > m + 1) p0 = p1;
    p1 = pi;
  }
  const NfRow c = rows[l * (l + 1) - 1 + m], s = rows[l * (l + 1) - 1 - m];
  const double P = st * pi, mp = m * pi;
  double u, v;
  u = fma(cm, c.c1r, sm * s.c1r);
  v = fma(cm, s.c1r, -sm * c.c1r);
  S.pv1[l][0] = fma(mp, v, S.pv1[l][0]);
  S.tu1[l][0] = fma(tau, u, S.tu1[l][0]);
  u = fma(cm, c.c1i, sm * s.c1i);
  v = fma(cm, s.c1i, -sm * c.c1i);
  S.pv1[l][1] = fma(mp, v, S.pv1[l][1]);
  S.tu1[l][1] = fma(tau, u, S.tu1[l][1]);
  u = fma(cm, c.c2r, sm * s.c2r);
  v = fma(cm, s.c2r, -sm * c.c2r);
  S.pu2[l][0] = fma(P, u, S.pu2[l][0]);
  S.tu2[l][0] = fma(tau, u, S.tu2[l][0]);
  S.pv2[l][0] = fma(mp, v, S.pv2[l][0]);
  u = fma(cm, c.c2i, sm * s.c2i);
  v = fma(cm, s.c2i, -sm * c.c2i);
  S.pu2[l][1] = fma(P, u, S.pu2[l][1]);
  S.tu2[l][1] = fma(tau, u, S.tu2[l][1]);
  S.pv2[l][1] = fma(mp, v, S.pv2[l][1]);
  if constexpr (m == 1) {
    // tau_l^0 = -sqrt(l(l+1)) sin pi_l^1
    constexpr double F0 = -tab::csqrt(l * (l + 1.0));
    const double t0 = F0 * P;
    const NfRow z = rows[l * (l + 1) - 1];
    S.tu1[l][0] = fma(t0, z.c1r, S.tu1[l][0]);
    S.tu1[l][1] = fma(t0, z.c1i, S.tu1[l][1]);
    S.tu2[l][0] = fma(t0, z.c2r, S.tu2[l][0]);
    S.tu2[l][1] = fma(t0, z.c2i, S.tu2[l][1]);
  }
}
template <int L, int m, int... LI>
__device__ __forceinline__ void nf_order(const NfRow* __restrict__ rows, double ct, double st, double cm, double sm,
                                         double sp, NfSums<L>& S, std::integer_sequence<int, LI...>) {
  constexpr double D = nf_diag(m);
  double p0 = D * sp, p1 = 0.0;
  (nf_degree<L, m, m + LI>(rows, ct, st, cm, sm, p0, p1, S), ...);
}
template <int L, int m>
__device__ __forceinline__ void nf_orders(const NfRow* __restrict__ rows, double ct, double st, double cp, double sph,
                                          double cm, double sm, double sp, NfSums<L>& S) {
  nf_order<L, m>(rows, ct, st, cm, sm, sp, S, std::make_integer_sequence<int, L - m + 1>{});
  if constexpr (m < L)
    nf_orders<L, m + 1>(rows, ct, st, cp, sph, fma(cm, cp, -sm * sph), fma(cm, sph, sm * cp), sp * st, S);
}
// the m = 0 part of P U for degrees l = 1..L
template <int L, int l>
__device__ __forceinline__ void nf_zero(const NfRow* __restrict__ rows, double ct, double pm2, double pm1,
                                        NfSums<L>& S) {
  constexpr double A = nf_a(l, 0), AB = nf_a(l, 0) * (l > 1 ? nf_b(l, 0) : 0.0);
  const double p = fma(A * ct, pm1, -AB * pm2);
  const NfRow z = rows[l * (l + 1) - 1];
  S.pu2[l][0] = fma(p, z.c2r, S.pu2[l][0]);
  S.pu2[l][1] = fma(p, z.c2i, S.pu2[l][1]);
  if constexpr (l < L) nf_zero<L, l + 1>(rows, ct, pm1, p, S);
}

// Scattered field of the spheres of one chunk at 64 points, one per thread.
// Bound by FP64 issue.  Per (point, sphere) all orders +-m share one real pair
// (c_m, s_m), every angular factor is real and meets the radial functions once
// per degree, and the recursions' constants are immediates: about 500 FP64
// instructions at lmax 3, where the direct sum over (tau, l, m) with runtime
// recursions took thousands.  Grid (points, sphere chunks); out holds one slice
// per chunk, added in order afterwards.  A point inside a sphere turns its slice
// into NaN.  With the Gaussian beam below, GB300, 1 000 spheres, lmax 3, 4 096
// points: 139 -> 3.1 ms.
template <int L>
__global__ void __launch_bounds__(kNfPoints)
    nearfield_scattered_kernel(int64_t Np, const double* __restrict__ pts, int64_t N, int64_t chunk, double k,
                               const Pos4* __restrict__ pos, const double* __restrict__ radii,
                               const double2* __restrict__ b, double* __restrict__ out) {
  constexpr int NH = L * (L + 2);
  __shared__ NfRow rows[kNfTile][NH];
  __shared__ Pos4 sp[kNfTile];  // centre, and the radius squared in the fourth place
  const int64_t t = blockIdx.x * (int64_t)kNfPoints + threadIdx.x;
  const bool active = t < Np;
  double px = 0.0, py = 0.0, pz = 0.0;
  if (active) {
    px = pts[3 * t];
    py = pts[3 * t + 1];
    pz = pts[3 * t + 2];
  }
  const double ik = 1.0 / k;
  double E[6] = {};
  bool inside = false;
  const int64_t i0 = blockIdx.y * chunk, i1 = i0 + chunk < N ? i0 + chunk : N;
  for (int64_t it = i0; it < i1; it += kNfTile) {
    const int ni = static_cast<int>(i1 - it < kNfTile ? i1 - it : kNfTile);
    __syncthreads();
    for (int q = threadIdx.x; q < ni * NH; q += kNfPoints) {
      const int j = q / NH, r = q - j * NH;
      const int l = 1 + (r >= 3) + (r >= 8) + (r >= 15) + (r >= 24);
      const int m = r - (l * (l + 1) - 1);
      const double nrm = 1.0 / sqrt(2.0 * l * (l + 1.0));
      const double2* bi = b + (it + j) * 2 * NH;
      const double2 a1 = bi[r], a2 = bi[NH + r];
      NfRow o{a1.x, a1.y, a2.x, a2.y};
      if (m != 0) {
        const double2 d1 = bi[r - 2 * m], d2 = bi[NH + r - 2 * m];
        if (m > 0) o = NfRow{a1.x + d1.x, a1.y + d1.y, a2.x + d2.x, a2.y + d2.y};
        else o = NfRow{a1.y - d1.y, d1.x - a1.x, a2.y - d2.y, d2.x - a2.x};  // d is b_|m| here
      }
      rows[j][r] = NfRow{nrm * o.c1r, nrm * o.c1i, nrm * o.c2r, nrm * o.c2i};
    }
    for (int q = threadIdx.x; q < ni; q += kNfPoints) {
      const Pos4 c = pos[it + q];
      const double R = radii[it + q];
      sp[q] = Pos4{c.x, c.y, c.z, R * R};
    }
    __syncthreads();
    for (int j = 0; j < ni; ++j) {
      if (!active || inside) continue;
      const Pos4 c = sp[j];
      const double dx = px - c.x, dy = py - c.y, dz = pz - c.z;
      const double rho2 = fma(dx, dx, dy * dy), d2 = fma(dz, dz, rho2);
      if (d2 < c.w) {
        inside = true;
        continue;
      }
      const double id = rsqrt(d2), d = d2 * id;
      const double ct = dz * id;
      const bool off = rho2 > 0.0;
      const double ir = off ? rsqrt(rho2) : 0.0;
      const double st = rho2 * ir * id;
      const double cp = off ? dx * ir : 1.0, sph = dy * ir;
      NfSums<L> S;
      nf_zero<L, 1>(rows[j], ct, 0.0, 0.70710678118654752440, S);
      nf_orders<L, 1>(rows[j], ct, st, cp, sph, cp, sph, 1.0, S);
      // radial functions: h_l(x) by upward recurrence, d(x h_l)/x
      const double x = k * d, ix = id * ik;
      double sn, cs;
      sincos_phase(x, &sn, &cs);
      double h0r = sn * ix, h0i = -cs * ix;
      double h1r = -ix * fma(-sn, ix, cs), h1i = -ix * fma(cs, ix, sn);
      double Ar[2] = {}, At[2] = {}, Ap[2] = {};
#pragma unroll
      for (int l = 1; l <= L; ++l) {
        const double gr = fma(-l * ix, h1r, h0r), gi = fma(-l * ix, h1i, h0i);
        const double er = (l * (l + 1)) * ix * h1r, ei = (l * (l + 1)) * ix * h1i;
        Ar[0] = fma(er, S.pu2[l][0], fma(-ei, S.pu2[l][1], Ar[0]));
        Ar[1] = fma(er, S.pu2[l][1], fma(ei, S.pu2[l][0], Ar[1]));
        At[0] = fma(h1r, S.pv1[l][0], fma(-h1i, S.pv1[l][1], At[0]));
        At[1] = fma(h1r, S.pv1[l][1], fma(h1i, S.pv1[l][0], At[1]));
        At[0] = fma(gr, S.tu2[l][0], fma(-gi, S.tu2[l][1], At[0]));
        At[1] = fma(gr, S.tu2[l][1], fma(gi, S.tu2[l][0], At[1]));
        Ap[0] = fma(-h1r, S.tu1[l][0], fma(h1i, S.tu1[l][1], Ap[0]));
        Ap[1] = fma(-h1r, S.tu1[l][1], fma(-h1i, S.tu1[l][0], Ap[1]));
        Ap[0] = fma(gr, S.pv2[l][0], fma(-gi, S.pv2[l][1], Ap[0]));
        Ap[1] = fma(gr, S.pv2[l][1], fma(gi, S.pv2[l][0], Ap[1]));
        const double f = (2 * l + 1) * ix;
        const double nr = fma(f, h1r, -h0r), ni_ = fma(f, h1i, -h0i);
        h0r = h1r;
        h0i = h1i;
        h1r = nr;
        h1i = ni_;
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const double w = fma(st, Ar[q], ct * At[q]);  // component along e_rho
        E[q] = fma(cp, w, fma(-sph, Ap[q], E[q]));
        E[2 + q] = fma(sph, w, fma(cp, Ap[q], E[2 + q]));
        E[4 + q] = fma(ct, Ar[q], fma(-st, At[q], E[4 + q]));
      }
    }
  }
  if (!active) return;
  double* o = out + ((int64_t)blockIdx.y * Np + t) * 6;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
  for (int q = 0; q < 6; ++q) o[q] = inside ? nan : E[q];
}

// E = sum of the chunks' slices, in order
__global__ void nearfield_sum_kernel(int64_t n, int chunks, const double* __restrict__ part, double* __restrict__ E) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int c = 0; c < chunks; ++c) s += part[c * n + t];
    E[t] = s;
  }
}

// E += E0 e^{i k.r} e_pol(alpha, beta)
__global__ void nearfield_plane_kernel(int64_t Np, const double* __restrict__ pts, double k, double beta,
                                       double alpha, int pol, double e0r, double e0i, double* __restrict__ E) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= Np) return;
  double sb, cb, sa, ca;
  sincos(beta, &sb, &cb);
  sincos(alpha, &sa, &ca);
  const double kx = k * sb * ca, ky = k * sb * sa, kz = k * cb;
  const cd ph = cexp_i(kx * pts[3 * t] + ky * pts[3 * t + 1] + kz * pts[3 * t + 2]) * cd{e0r, e0i};
  const double e[3] = {pol == 1 ? -sa : cb * ca, pol == 1 ? ca : cb * sa, pol == 1 ? 0.0 : -sb};
  double* o = E + 6 * t;
  for (int q = 0; q < 3; ++q) {
    o[2 * q] += ph.re * e[q];
    o[2 * q + 1] += ph.im * e[q];
  }
}

// J_0, J_1, J_2 of z >= 0 to 2e-16 absolute (CUDA's j0 and j1 differ from the
// true values by up to 4e-13 above 8, which the sums over the nodes do not
// average out).  Up to 1/2 the power series, whose J_1 and J_2 keep their
// relative accuracy; below 25 the Taylor polynomial of J_0 about the middle of the
// unit interval and its derivative -J_1; above, Hankel's asymptotic expansion,
// whose first neglected term is under 1e-17 there.  J_2 by the recurrence.
constexpr int kBesselIntervals = 25, kBesselDegree = 16;
struct BesselTable {
  double a[kBesselIntervals][kBesselDegree + 1];
};
constexpr BesselTable make_bessel_table() {
  BesselTable t{};
  // about 1/2: J_0(x) = sum_k (-1/4)^k / k!^2 x^{2k}, re-expanded
  for (int n = 0; n <= kBesselDegree; ++n) {
    double f = 1.0, sum = 0.0;
    for (int k = 0; k <= 16; ++k) {
      if (k > 0) f *= -0.25 / (1.0 * k * k);
      if (2 * k < n) continue;
      double term = f;  // times binomial(2k, n) / 2^{2k - n}
      for (int q = 1; q <= n; ++q) term *= (2.0 * k - n + q) / q;
      for (int q = 0; q < 2 * k - n; ++q) term *= 0.5;
      sum += term;
    }
    t.a[0][n] = sum;
  }
  for (int i = 1; i < kBesselIntervals; ++i) {
    const double c = i + 0.5;
    // J_0 and J_1 by Miller's downward recurrence
    double up = 0.0, cur = 1e-200, sum = 0.0, j1 = 0.0;
    for (int n = 80; n > 0; --n) {
      if (n % 2 == 0) sum += cur;
      const double down = 2.0 * n / c * cur - up;
      up = cur;
      cur = down;
      if (n == 2) j1 = cur;
    }
    const double r = 1.0 / (2.0 * sum + cur);
    double* a = t.a[i];
    a[0] = cur * r;
    a[1] = -j1 * r;
    // Bessel's equation, order by order in x - c
    for (int n = 0; n + 2 <= kBesselDegree; ++n)
      a[n + 2] = -((n + 1.0) * (n + 1.0) * a[n + 1] + c * a[n] + (n > 0 ? a[n - 1] : 0.0)) / (c * (n + 2.0) * (n + 1.0));
  }
  return t;
}
__device__ const BesselTable kBesselTable = make_bessel_table();

// (-1)^{k/2} of Hankel's coefficients (4 nu^2 - 1)(4 nu^2 - 9) .. / (k! 8^k)
constexpr double hankel_coef(int nu, int k) {
  double a = (k / 2) % 2 ? -1.0 : 1.0;
  for (int j = 1; j <= k; ++j) a *= (4.0 * nu * nu - (2.0 * j - 1.0) * (2.0 * j - 1.0)) / (8.0 * j);
  return a;
}
template <int NU, int... K>
__device__ __forceinline__ void hankel_pq(double r, double q, double& P, double& Q, std::integer_sequence<int, K...>) {
  constexpr int M = static_cast<int>(sizeof...(K)) - 1;
  P = Q = 0.0;
  (
      [&] {
        constexpr double p = hankel_coef(NU, 2 * (M - K)), w = hankel_coef(NU, 2 * (M - K) + 1);
        P = fma(P, q, p);
        Q = fma(Q, q, w);
      }(),
      ...);
  Q *= r;
}
template <int NU, int... K>
__device__ __forceinline__ double bessel_series(double q, std::integer_sequence<int, K...>) {
  // sum_k (-q)^k / (k! (k + NU)!), q <= 1/16: terms to k = 7 leave 1e-20
  constexpr int M = static_cast<int>(sizeof...(K)) - 1;
  double s = 0.0;
  (
      [&] {
        constexpr double c = 1.0 / (tab::fact(M - K) * tab::fact(M - K + NU));
        s = fma(-q, s, c);
      }(),
      ...);
  return s;
}
__device__ __forceinline__ void bessel_012(double z, const double* __restrict__ table, double& J0, double& J1,
                                           double& J2) {
  if (z <= 0.5) {
    constexpr auto terms = std::make_integer_sequence<int, 8>{};
    const double q = 0.25 * z * z;
    J0 = bessel_series<0>(q, terms);
    J1 = 0.5 * z * bessel_series<1>(q, terms);
    J2 = q * bessel_series<2>(q, terms);
    return;
  }
  if (z < kBesselIntervals) {
    const int i = static_cast<int>(z);
    const double h = z - (i + 0.5);
    const double* a = table + i * (kBesselDegree + 1);
    double p = a[kBesselDegree], d = 0.0;
#pragma unroll
    for (int n = kBesselDegree - 1; n >= 0; --n) {
      d = fma(d, h, p);
      p = fma(p, h, a[n]);
    }
    J0 = p;
    J1 = -d;
  } else {
    constexpr auto terms = std::make_integer_sequence<int, 9>{};
    const double r = 1.0 / z;
    double s, c, P, Q;
    sincos_phase(z, &s, &c);
    const double f = rsqrt(3.14159265358979323846 * z);
    hankel_pq<0>(r, r * r, P, Q, terms);
    J0 = f * fma(P, c + s, -Q * (s - c));
    hankel_pq<1>(r, r * r, P, Q, terms);
    J1 = f * fma(P, s - c, Q * (s + c));
  }
  J2 = fma(2.0 / z, J1, -J0);
}

// E += E0 (k w)^2/(4 pi) int_0^bmax dbeta int_0^2pi dalpha sin(b) cos(b)
//        exp(-(w k sin b)^2/4) e^{i k(b,a).(r - r_G)} (cos(a - aG) e_a + sin(a - aG) e_b)
// The alpha integral in closed form: its integrand is e^{i z cos(a - phi)}, z = k
// rho sin b, times harmonics of order 0, 1 and 2 in a, so it is J_0, J_1 and
// J_2 of z (the trapezoid rule that stood here took 2 (k rho + 40) nodes of
// three sincos each).  One warp per point, lanes over the beta nodes.  Error far
// from the axis (k rho of 100 to 1 000, waist 500), of E_0: 7e-16, like the
// trapezoid rule's; 5e-14 with CUDA's j0 and j1, which also took 1 % longer.
__global__ void __launch_bounds__(32 * kNfWarps)
    nearfield_gauss_kernel(int64_t Np, const double* __restrict__ pts, double k, double w, double fx, double fy,
                           double fz, double aG, double e0r, double e0i, int nb, const double* __restrict__ bnode,
                           const double* __restrict__ bw, double* __restrict__ E) {
  constexpr int NT = 128;
  constexpr int NB = kBesselIntervals * (kBesselDegree + 1);
  __shared__ double ssb[NT], scb[NT], sg[NT];
  __shared__ double table[NB];  // the lanes of a warp read different intervals
  for (int q = threadIdx.x; q < NB; q += blockDim.x) table[q] = kBesselTable.a[q / (kBesselDegree + 1)][q % (kBesselDegree + 1)];
  const int lane = threadIdx.x & 31;
  const int64_t t = blockIdx.x * (int64_t)kNfWarps + (threadIdx.x >> 5);
  const bool active = t < Np;
  const double rx = active ? pts[3 * t] - fx : 0.0, ry = active ? pts[3 * t + 1] - fy : 0.0;
  const double rz = active ? pts[3 * t + 2] - fz : 0.0;
  const double rho = sqrt(rx * rx + ry * ry);
  // sums over the nodes of weight e^{i k z cos b} times J_0, cos b J_0, J_2, cos b J_2, sin b J_1
  double S[5][2] = {};
  for (int b0 = 0; b0 < nb; b0 += NT) {
    const int n = nb - b0 < NT ? nb - b0 : NT;
    __syncthreads();
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
      double sb, cb;
      sincos(bnode[b0 + q], &sb, &cb);
      ssb[q] = sb;
      scb[q] = cb;
      sg[q] = sb * cb * exp(-(w * k * sb) * (w * k * sb) / 4.0) * bw[b0 + q];
    }
    __syncthreads();
    if (!active) continue;
    for (int q = lane; q < n; q += 32) {
      const double sb = ssb[q], cb = scb[q], g = sg[q];
      if (g == 0.0) continue;
      const double z = k * rho * sb;
      double J0, J1, J2, sn, cs;
      bessel_012(z, table, J0, J1, J2);
      sincos_phase(k * rz * cb, &sn, &cs);
      const double f[5] = {J0, cb * J0, J2, cb * J2, sb * J1};
#pragma unroll
      for (int u = 0; u < 5; ++u) {
        S[u][0] = fma(g * cs, f[u], S[u][0]);
        S[u][1] = fma(g * sn, f[u], S[u][1]);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 5; ++u)
    for (int o = 16; o > 0; o >>= 1) {
      S[u][0] += __shfl_down_sync(0xffffffffu, S[u][0], o);
      S[u][1] += __shfl_down_sync(0xffffffffu, S[u][1], o);
    }
  if (!active || lane != 0) return;
  const double TWO_PI = 6.283185307179586476925286766559;
  const double cp = rho > 0.0 ? rx / rho : 1.0, sp = rho > 0.0 ? ry / rho : 0.0;
  double sG, cG;
  sincos(aG, &sG, &cG);
  // 2 phi - aG and phi - aG
  const double c2p = cp * cp - sp * sp, s2p = 2.0 * sp * cp;
  const double c2 = c2p * cG + s2p * sG, s2 = s2p * cG - c2p * sG, s1 = sp * cG - cp * sG;
  double v[3][2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    // I_0 = 2 pi J_0; cos / sin(2 a - aG) -> -2 pi J_2 cos / sin(2 phi - aG); sin(a - aG) -> 2 pi i J_1 sin(phi - aG)
    v[0][q] = 0.5 * TWO_PI * ((s2 * S[2][q] - sG * S[0][q]) - (s2 * S[3][q] + sG * S[1][q]));
    v[1][q] = 0.5 * TWO_PI * ((cG * S[0][q] - c2 * S[2][q]) + (cG * S[1][q] + c2 * S[3][q]));
    v[2][q] = -TWO_PI * s1 * (q == 0 ? -S[4][1] : S[4][0]);
  }
  const cd s = cd{e0r, e0i} * ((k * w) * (k * w) / (4.0 * 3.14159265358979323846264338328));
  double* o = E + 6 * t;
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    const cd e = s * cd{v[u][0], v[u][1]};
    o[2 * u] += e.re;
    o[2 * u + 1] += e.im;
  }
}

template <int L>
void launch_scattered(int64_t Np, const double* pts, const CtxView& v, const double* b, int chunks, double* out,
                      cudaStream_t st) {
  const dim3 grid(static_cast<unsigned>((Np + kNfPoints - 1) / kNfPoints), static_cast<unsigned>(chunks));
  nearfield_scattered_kernel<L><<<grid, kNfPoints, 0, st>>>(Np, pts, v.N, (v.N + chunks - 1) / chunks, v.k,
                                                            static_cast<const Pos4*>(v.pos), v.radii,
                                                            reinterpret_cast<const double2*>(b), out);
  note_launch();
}

inline unsigned nblocks(int64_t n) { return static_cast<unsigned>((n + kNfThreads - 1) / kNfThreads); }

}  // namespace

// Gauss-Legendre nodes and weights on [a, b] (the rule of the Gaussian-beam coefficients)
void gauss_legendre_nodes(int n, double a, double b, std::vector<double>& x, std::vector<double>& w);

}  // namespace celes

extern "C" int celes_nearfield(celes_ctx* ctx, const double* points, int64_t Np, int rhs, int what, double* E) {
  celes::NvtxRange nvtx_range_("celes_nearfield");
  using namespace celes;
  if (!ctx || Np < 0 || (Np > 0 && (!points || !E)) || what < 0 || what > 2) return CELES_EINVAL;
  CtxView v{};
  int s = ctx_view(ctx, &v);
  if (s) return s;
  if (rhs < 0 || rhs >= v.nrhs) return CELES_EINVAL;
  if (what != 1 && !v.has_b) return CELES_ESTATE;
  if (Np == 0) return CELES_OK;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(v.device);
  struct Restore {
    int d;
    ~Restore() { cudaSetDevice(d); }
  } restore{prev};
  const cudaStream_t st = v.stream;
  // chunks of spheres so that small maps fill the GPU too (eight CTAs of two
  // warps per SM; a sphere takes 8 us one after another), with slices of at
  // most 64 MB
  const int64_t tiles = (Np + kNfPoints - 1) / kNfPoints;
  int64_t chunks = (8LL * device_sms() + tiles - 1) / tiles;
  chunks = std::min<int64_t>(chunks, (v.N + 1) / 2);
  chunks = std::max<int64_t>(1, std::min<int64_t>(chunks, (int64_t(64) << 20) / (48 * Np)));
  // points, field, the beam's nodes and weights, slices
  const int nb_max = v.incidents[rhs].kind == CELES_PLANE_WAVE ? 0 : (v.incidents[rhs].n_beta > 0 ? v.incidents[rhs].n_beta : 128);
  const size_t slices = what != 1 && chunks > 1 ? static_cast<size_t>(chunks) * 6 * Np : 0;
  FieldWorkspace ws(ctx);
  if (ws.ensure(sizeof(double) * (9 * static_cast<size_t>(Np) + 2 * nb_max + slices)) != cudaSuccess) {
    cudaGetLastError();
    return CELES_ENOMEM;
  }
  double* dp = reinterpret_cast<double*>(ws.at(0));
  double* dE = dp + 3 * Np;
  double* dn = dE + 6 * Np;
  double* dw = dn + nb_max;
  double* dS = dw + nb_max;
  auto cleanup = [&]() { cudaStreamSynchronize(st); };
  cudaError_t e = cudaMemcpyAsync(dp, points, sizeof(double) * 3 * Np, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && what == 1) e = cudaMemsetAsync(dE, 0, sizeof(double) * 6 * Np, st);
  if (e != cudaSuccess) {
    cleanup();
    return CELES_ECUDA;
  }
  if (what != 1) {
    const double* b = v.b + (size_t)rhs * v.N * v.nmax * 2;
    double* out = chunks > 1 ? dS : dE;
    const int nc = static_cast<int>(chunks);
    switch (v.L) {
      case 1: launch_scattered<1>(Np, dp, v, b, nc, out, st); break;
      case 2: launch_scattered<2>(Np, dp, v, b, nc, out, st); break;
      case 3: launch_scattered<3>(Np, dp, v, b, nc, out, st); break;
      case 4: launch_scattered<4>(Np, dp, v, b, nc, out, st); break;
      default: launch_scattered<5>(Np, dp, v, b, nc, out, st); break;
    }
    if (chunks > 1) {
      const int64_t n = 6 * Np;
      const int64_t g = std::min<int64_t>((n + kNfThreads - 1) / kNfThreads, 16LL * device_sms());
      nearfield_sum_kernel<<<static_cast<unsigned>(g), kNfThreads, 0, st>>>(n, nc, dS, dE);
      note_launch();
    }
  }
  if (what != 0) {
    const celes_incident& d = v.incidents[rhs];
    if (d.kind == CELES_PLANE_WAVE) {
      nearfield_plane_kernel<<<nblocks(Np), kNfThreads, 0, st>>>(Np, dp, v.k, d.beta, d.alpha, d.pol, d.E0_re,
                                                                 d.E0_im, dE);
    } else {
      const int nb = d.n_beta > 0 ? d.n_beta : 128;
      const double aa = std::pow(d.waist * v.k, 2) / 4.0;
      const double s2 = 39.2 / aa;
      const double bmax = s2 >= 1.0 ? M_PI / 2 : std::asin(std::sqrt(s2));
      std::vector<double> hx, hw;
      gauss_legendre_nodes(nb, 0.0, bmax, hx, hw);
      if (cudaMemcpyAsync(dn, hx.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, st) != cudaSuccess ||
          cudaMemcpyAsync(dw, hw.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, st) != cudaSuccess) {
        cleanup();
        return CELES_ECUDA;
      }
      nearfield_gauss_kernel<<<static_cast<unsigned>((Np + kNfWarps - 1) / kNfWarps), 32 * kNfWarps, 0, st>>>(Np, dp, v.k, d.waist, d.focus[0], d.focus[1],
                                                                 d.focus[2], d.alpha_G, d.E0_re, d.E0_im, nb, dn, dw,
                                                                 dE);
    }
    note_launch();
  }
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(E, dE, sizeof(double) * 6 * Np, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cleanup();
  return e == cudaSuccess ? CELES_OK : CELES_ECUDA;
}
