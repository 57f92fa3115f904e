// Compile-time tables of the rotation-translation-rotation factorisation of
// the coupling block (the O(lmax^3) scheme of Sec. 5; exact, not an
// approximation):
//
//   W(d) = D^H W_z(k|d|) D,   D = blockdiag_l R^l(theta) diag(e^{i m phi})
//
// where (|d|, theta, phi) are the spherical coordinates of d = r_i - r_j,
// R^l_{mu m}(theta) = s_mu s_m d^l_{m mu}(theta) with Wigner's small-d matrix
// and s_m = (-1)^m for m >= 0, 1 for m < 0 (the sign that converts the
// Condon-Shortley convention to the normalised Legendre functions of App. A.1
// used here), and W_z is the coupling block of a translation along +z: it is
// diagonal in m, with (theta = 0, so only P_p^0(1) = sqrt((2p+1)/2) survives)
//
//   W_z[(tau,l,mu),(tau',l',mu)] = sum_p {a5 | i b5'}(l',mu|l,mu|p) sqrt((2p+1)/2) h_p(k|d|)
//
// (a5 for tau = tau', i b5' otherwise; App. A.2).  Under mu -> -mu the a5
// factor is unchanged and b5' changes sign.
//
// The rotations run in the cosine / sine basis
//   c_0 = sqrt(2) x_0,  c_M = x_M + x_{-M},  s_M = i (x_M - x_{-M})   (M > 0)
// of each tau (tau = 2 multiplied by -i).  R_{-mu,-m} = R_{mu m} and
// R_{-mu,m} = R_{mu,-m}, so R^l splits into a (l+1) x (l+1) block C on the c
// and an l x l block S on the s: 2 l^2 + 2 l + 1 products instead of
// (2 l + 1)^2, and e^{i M phi} becomes a real rotation of (c_M, s_M).  With
// the rotated row mu multiplied by (-1)^mu (which W_z does not see) both blocks
// are symmetric and orthogonal, hence their own inverses: the forward and the
// backward rotation use the same numbers.
//
// Wigner's small-d matrix from its explicit sum:
//   d^l_{m'm}(b) = sum_k (-1)^{k-m+m'} sqrt((l+m')!(l-m')!(l+m)!(l-m)!)
//                  / [(l+m-k)! k! (l-k-m')! (k-m+m')!]  c^{2l-j} s^j,
//   c = cos(b/2), s = sin(b/2), j = 2k - m + m',
// expanded here into cos(q b) or sin(q b), q = 0..l: entry (mu, m) of a block
// has two or three such terms (q of one parity) whose coefficients are at most
// one, so it loses nothing to cancellation.
#pragma once

#include "coupling_tables.cuh"

namespace celes {
namespace rtr {

using tab::csqrt;
using tab::fact;
using tab::iabs;
using tab::imax;
using tab::imin;

constexpr int sgn_pm1(int e) { return (((e % 2) + 2) % 2) ? -1 : 1; }
constexpr int sigma(int m) { return m >= 0 ? sgn_pm1(m) : 1; }

// ---------------------------------------------------------------------------
// rotation blocks of one degree l
// ---------------------------------------------------------------------------
// Fourier coefficients of one entry: sum_q v[q] cos(q b), or sin(q b) when
// `sine` (the entries with mu - m odd)
template <int l>
struct Fourier {
  double v[l + 1] = {};
  bool sine = false;
};

// d^l_{m'm} as a Fourier sum: c^{2l-j} s^j = (z + 1/z)^{2l-j} (z - 1/z)^j / (2^{2l} i^j), z = e^{i b/2}
template <int l>
constexpr Fourier<l> wigner_fourier(int mp, int m) {
  Fourier<l> F{};
  F.sine = iabs(mp - m) % 2 == 1;
  const double num = csqrt(fact(l + mp) * fact(l - mp) * fact(l + m) * fact(l - m));
  for (int k = 0; k <= 2 * l; ++k) {
    const int a1 = l + m - k, a2 = l - k - mp, a3 = k - m + mp;
    if (a1 < 0 || a2 < 0 || a3 < 0) continue;
    const int j = 2 * k - m + mp;
    const double c = sgn_pm1(k - m + mp) * num / (fact(a1) * fact(k) * fact(a2) * fact(a3));
    // coefficients of z^{2 t - 2 l}, t = 0..2l
    double w[2 * l + 1] = {1.0};
    for (int f = 0; f < 2 * l; ++f) {
      const double sg = f < j ? -1.0 : 1.0;
      for (int t = f + 1; t >= 0; --t) w[t] = (t > 0 ? w[t - 1] : 0.0) + sg * (t <= f ? w[t] : 0.0);
    }
    double scale = c;
    for (int f = 0; f < 2 * l; ++f) scale *= 0.5;
    if (!F.sine) {
      if ((j / 2) % 2) scale = -scale;  // i^{-j}, j even
      F.v[0] += scale * w[l];
      for (int q = 1; q <= l; ++q) F.v[q] += 2.0 * scale * w[l + q];
    } else {
      if (((j - 1) / 2) % 2) scale = -scale;  // i^{1-j}, j odd
      for (int q = 1; q <= l; ++q) F.v[q] += 2.0 * scale * w[l + q];
    }
  }
  return F;
}

// entry (mu, m) of block C (KIND 0, mu, m >= 0) or S (KIND 1, mu, m >= 1)
template <int l, int KIND>
constexpr Fourier<l> rot_fourier(int mu, int m) {
  // R_{mu m} = s_mu s_m d_{m mu}
  Fourier<l> F = wigner_fourier<l>(m, mu);
  const double s1 = sigma(mu) * sigma(m);
  const double f = sgn_pm1(mu) * s1 * ((mu == 0) != (m == 0) ? csqrt(2.0) : 1.0);
  Fourier<l> G{};
  double g = 0.0;
  if (mu > 0 && m > 0) {
    G = wigner_fourier<l>(-m, mu);
    g = (KIND == 0 ? 1.0 : -1.0) * sgn_pm1(mu) * sigma(mu) * sigma(-m);
  }
  for (int q = 0; q <= l; ++q) {
    F.v[q] = f * F.v[q] + g * G.v[q];
    if (F.v[q] < 1e-13 && F.v[q] > -1e-13) F.v[q] = 0.0;  // terms that cancel
  }
  return F;
}

template <int l, int KIND, int MU, int M>
struct RotEntry {
  static constexpr Fourier<l> value = rot_fourier<l, KIND>(MU, M);
  // true when the entry is the constant +-1 (S of degree 1)
  static constexpr bool unit() { return l == 1 && KIND == 1; }
  static constexpr int terms() {
    int n = 0;
    for (int q = 0; q <= l; ++q) n += value.v[q] != 0.0;
    return n;
  }
};
// coefficient of cos(q b) or sin(q b) in an entry
template <int l, int KIND, int MU, int M, int Q>
struct RotCoef {
  static constexpr double v = RotEntry<l, KIND, MU, M>::value.v[Q];
  static constexpr bool sine = RotEntry<l, KIND, MU, M>::value.sine;
  static constexpr int before() {  // terms of lower q
    int n = 0;
    for (int q = 0; q < Q; ++q) n += RotEntry<l, KIND, MU, M>::value.v[q] != 0.0;
    return n;
  }
};
// canonical position of entry (mu, m) (symmetric blocks, lower triangle)
constexpr int rot_id(int kind, int mu, int m) {
  const int a = mu > m ? mu : m, b = mu > m ? m : mu;
  return kind == 0 ? a * (a + 1) / 2 + b : (a - 1) * a / 2 + (b - 1);
}
template <int l>
struct RotCount {
  static constexpr int nc = (l + 1) * (l + 2) / 2, ns = l * (l + 1) / 2;
};

// ---------------------------------------------------------------------------
// axial coupling terms, one table per (mu >= 0, l, l')
// ---------------------------------------------------------------------------
template <int L>
struct AxialRow {
  static constexpr int MAXT = 2 * (2 * L + 2);
  int na = 0, nb = 0;
  int ap[MAXT] = {}, bp[MAXT] = {};
  double ac[MAXT] = {}, bc[MAXT] = {};
};

template <int L>
constexpr AxialRow<L> make_axial(int mu, int l, int lp) {
  AxialRow<L> T{};
  for (int p = iabs(l - lp); p <= l + lp; ++p) {
    const double w = csqrt((2.0 * p + 1.0) / 2.0);
    const double a = tab::ab5_real(0, lp, mu, l, mu, p);
    const double b = tab::ab5_real(1, lp, mu, l, mu, p);
    if (a != 0.0) {
      T.ap[T.na] = p;
      T.ac[T.na] = a * w;
      ++T.na;
    }
    if (b != 0.0) {
      T.bp[T.nb] = p;
      T.bc[T.nb] = b * w;
      ++T.nb;
    }
  }
  return T;
}

template <int L, int MU, int LO, int LI>
struct Axial {
  static constexpr AxialRow<L> value = make_axial<L>(MU, LO, LI);
};
template <int L, int MU, int LO, int LI, int T>
struct AxialA {
  static constexpr int p = Axial<L, MU, LO, LI>::value.ap[T];
  static constexpr double c = Axial<L, MU, LO, LI>::value.ac[T];
};
template <int L, int MU, int LO, int LI, int T>
struct AxialB {
  static constexpr int p = Axial<L, MU, LO, LI>::value.bp[T];
  static constexpr double c = Axial<L, MU, LO, LI>::value.bc[T];
};
template <int L, int MU, int LO, int LI>
struct AxialN {
  static constexpr int na = Axial<L, MU, LO, LI>::value.na;
  static constexpr int nb = Axial<L, MU, LO, LI>::value.nb;
};

}  // namespace rtr
}  // namespace celes
