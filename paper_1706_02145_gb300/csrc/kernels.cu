// Setup, epilogue, vector and far-field kernels of the solver.
//
//  * coupling epilogue: sum of the per-chunk partial products, change from the
//    +- basis back to (tau = 1, tau = 2), optional M x = x - T (W x) (Sec. 2.2)
//  * Mie T-matrix (App. B)
//  * incident-field coefficients: plane wave (App. A.2) and Gaussian beam (App. C)
//  * GMRES vector operations (Sec. 3.2): multi-dot, multi-axpy, norms, casts
//  * far-field amplitude g_j (App. D)
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>

#include "../../include/celes.h"
#include "cmath.cuh"
#include "coupling_kernel.cuh"
#include "coupling_tables.cuh"
#include "kernels.h"

namespace celes {

static std::atomic<int64_t> g_launch_count{0};
void note_launch(int n) { g_launch_count += n; }
int64_t kernel_launch_count() { return g_launch_count.load(); }

// degree of row r (l^2 - 1 <= r < (l+1)^2 - 1), in integers: a square root would
// go through the FP64 pipe
static __device__ __forceinline__ int row_l_rt(int r) {
  int l = 1;
  while ((l + 1) * (l + 1) - 1 <= r) ++l;
  return l;
}

// ---------------------------------------------------------------------------
// coupling epilogue
// ---------------------------------------------------------------------------
// grid (blocks, right-hand sides).  SPLIT > 1 (many slices on few spheres): that
// many threads share an element, each adds a run of the slices, and the runs
// are added in order (FP64, N = 120, 120 slices: 67 -> 15 us).  ZERO: one slice, zeroed again behind the
// read (each element by the thread that read it) for the next launch that adds
// into it
template <typename R, bool ZERO, int SPLIT>
__global__ void __launch_bounds__(256)
    coupling_epilogue_kernel(int64_t N, int L, int chunks, Pair2<R>* __restrict__ partial,
                             const Pair2<R>* __restrict__ x, const Pair2<R>* __restrict__ tq, Pair2<R>* __restrict__ y,
                             int mode) {
  const int NH = L * (L + 2);
  const int64_t total = N * NH;
  partial += (int64_t)blockIdx.y * chunks * total * 2;
  x += (int64_t)blockIdx.y * total * 2;
  y += (int64_t)blockIdx.y * total * 2;
  constexpr int PER = 256 / SPLIT;  // elements of a block at a time
  __shared__ R runs[SPLIT > 1 ? SPLIT : 1][4][PER];
  const int el = threadIdx.x % PER, part = threadIdx.x / PER;
  const int c0 = chunks * part / SPLIT, c1 = chunks * (part + 1) / SPLIT;
  for (int64_t tb = blockIdx.x * (int64_t)PER; tb < total; tb += (int64_t)gridDim.x * PER) {
    const int64_t t = tb + el;
    if (SPLIT == 1 && t >= total) break;
    const int64_t i = t / NH;
    const int r = static_cast<int>(t - i * NH);
    R pr = 0, pi = 0, mr = 0, mi = 0;
    for (int c = c0; c < (t < total ? c1 : c0); ++c) {
      Pair2<R>* pc = partial + ((int64_t)c * N + i) * (2 * NH);
      const Pair2<R> a = pc[r];
      const Pair2<R> b = pc[NH + r];
      if (ZERO) pc[r] = pc[NH + r] = Pair2<R>{0, 0};
      pr += a.re;
      pi += a.im;
      mr += b.re;
      mi += b.im;
    }
    if constexpr (SPLIT > 1) {
      __syncthreads();
      runs[part][0][el] = pr;
      runs[part][1][el] = pi;
      runs[part][2][el] = mr;
      runs[part][3][el] = mi;
      __syncthreads();
      if (part > 0 || t >= total) continue;
      for (int q = 1; q < SPLIT; ++q) {
        pr += runs[q][0][el];
        pi += runs[q][1][el];
        mr += runs[q][2][el];
        mi += runs[q][3][el];
      }
    }
    // y_1 = (y+ + y-)/2, y_2 = (y+ - y-)/2
    Pair2<R> y1{static_cast<R>(0.5) * (pr + mr), static_cast<R>(0.5) * (pi + mi)};
    Pair2<R> y2{static_cast<R>(0.5) * (pr - mr), static_cast<R>(0.5) * (pi - mi)};
    const int64_t o1 = i * 2 * NH + r, o2 = o1 + NH;
    if (mode == 1) {
      const int l = row_l_rt(r);
      const Pair2<R> q1 = tq[(i * 2 + 0) * L + (l - 1)];
      const Pair2<R> q2 = tq[(i * 2 + 1) * L + (l - 1)];
      const Pair2<R> x1 = x[o1], x2 = x[o2];
      y1 = Pair2<R>{x1.re - (q1.re * y1.re - q1.im * y1.im), x1.im - (q1.re * y1.im + q1.im * y1.re)};
      y2 = Pair2<R>{x2.re - (q2.re * y2.re - q2.im * y2.im), x2.im - (q2.re * y2.im + q2.im * y2.re)};
    }
    y[o1] = y1;
    y[o2] = y2;
  }
}

// About `waves` waves of CTAs, in chunks of at least 16 sources (FP32) or 4
// (FP64, whose pair takes forty times as long): a chunk pays for staging, its
// flush and its share of the epilogue, one or two pairs' time, and fewer,
// longer chunks leave the last wave of a mid-sized problem mostly empty (FP64
// N = 1000, lmax 3: 3.0 ms with at least 64 sources, 2.5 ms so; FP32 N = 2000,
// lmax 3: 224 and 196 us).  Where even that leaves resident slots empty, chunks
// down to 2 or 1 sources fill them: the sources of a chunk are walked one after
// another (N = 50, lmax 3, FP32: 18.5 -> 8.0 us; a refined solve at N = 120:
// 30.4 -> 5.4 ms, most of it the FP64 products).
int coupling_chunks(int64_t N, int64_t rb, int slots, double waves, int precision) {
  const bool fp64 = precision == CELES_FP64;
  int64_t ch = static_cast<int64_t>(std::ceil(waves * slots / static_cast<double>(rb)));
  ch = std::min<int64_t>(ch, std::max<int64_t>(1, N / (fp64 ? 4 : 16)));
  const int64_t fill = (slots + rb - 1) / rb;
  ch = std::max(ch, std::min(fill, std::max<int64_t>(1, N / (fp64 ? 1 : 2))));
  // a multiple of 8 (of 4 below 8): whole clusters for the cluster reduction
  if (ch >= 8) ch = (ch + 7) / 8 * 8;
  else if (ch >= 4) ch = 4;
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(ch, 512)));
}

template <typename R>
cudaError_t launch_coupling_epilogue(int64_t N, int L, int chunks, void* partial, const void* x, const void* tq,
                                     void* y, int mode, cudaStream_t st, int nrhs, bool zero) {
  const int64_t total = N * L * (L + 2);
  const bool split = chunks >= 16 && total < 64LL * device_sms() * 32;
  const int per = split ? 32 : 256;
  const int64_t blocks = (total + per - 1) / per;
  const int64_t cap = 32LL * device_sms();
  const dim3 grid(static_cast<unsigned>(blocks < cap ? (blocks > 0 ? blocks : 1) : cap), static_cast<unsigned>(nrhs));
  auto* p = static_cast<Pair2<R>*>(partial);
  auto* xv = static_cast<const Pair2<R>*>(x);
  auto* t = static_cast<const Pair2<R>*>(tq);
  auto* yv = static_cast<Pair2<R>*>(y);
  if (zero && chunks == 1) coupling_epilogue_kernel<R, true, 1><<<grid, 256, 0, st>>>(N, L, 1, p, xv, t, yv, mode);
  else if (split) coupling_epilogue_kernel<R, false, 8><<<grid, 256, 0, st>>>(N, L, chunks, p, xv, t, yv, mode);
  else coupling_epilogue_kernel<R, false, 1><<<grid, 256, 0, st>>>(N, L, chunks, p, xv, t, yv, mode);
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_coupling_epilogue<float>(int64_t, int, int, void*, const void*, const void*, void*, int,
                                                     cudaStream_t, int, bool);
template cudaError_t launch_coupling_epilogue<double>(int64_t, int, int, void*, const void*, const void*, void*, int,
                                                      cudaStream_t, int, bool);

// ---------------------------------------------------------------------------
// Mie T-matrix (App. B): one thread per sphere, all l
//   Q_1l = [j(x) dj(y) - j(y) dj(x)] / [j(y) dh(x) - h(x) dj(y)]
//   Q_2l = [j(x) dj(y) - m^2 j(y) dj(x)] / [m^2 j(y) dh(x) - h(x) dj(y)]
// x = k R, y = m k R, m = n_i / n0, dz(t) = d/dt [t z_l(t)] = t z_{l-1}(t) - l z_l(t)
// ---------------------------------------------------------------------------
__global__ void mie_kernel(int64_t N, int L, double k, const double* __restrict__ radii,
                           const double* __restrict__ n_rel, double* __restrict__ tq) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double R = radii[i];
  const cd m = mkc(n_rel[2 * i], n_rel[2 * i + 1]);
  const double x = k * R;
  const cd y = m * x;
  cd jx[16], jy[16], hx[16];
  double yx[16];
  sph_jn_c(L, mkc(x), jx);
  sph_jn_c(L, y, jy);
  sph_yn_r(L, x, yx);
  for (int l = 0; l <= L; ++l) hx[l] = jx[l] + cd{0.0, yx[l]};
  const cd m2 = m * m;
  for (int l = 1; l <= L; ++l) {
    const cd djx = x * jx[l - 1] - static_cast<double>(l) * jx[l];
    const cd djy = y * jy[l - 1] - static_cast<double>(l) * jy[l];
    const cd dhx = x * hx[l - 1] - static_cast<double>(l) * hx[l];
    const cd q1 = (jx[l] * djy - jy[l] * djx) / (jy[l] * dhx - hx[l] * djy);
    const cd q2 = (jx[l] * djy - m2 * jy[l] * djx) / (m2 * jy[l] * dhx - hx[l] * djy);
    double* o = tq + ((i * 2 + 0) * L + (l - 1)) * 2;
    o[0] = q1.re;
    o[1] = q1.im;
    o = tq + ((i * 2 + 1) * L + (l - 1)) * 2;
    o[0] = q2.re;
    o[1] = q2.im;
  }
}

cudaError_t launch_mie(int64_t N, int L, double k, const double* radii, const double* n_rel, double* tq,
                       cudaStream_t st) {
  const int threads = 128;
  mie_kernel<<<static_cast<unsigned>((N + threads - 1) / threads), threads, 0, st>>>(N, L, k, radii, n_rel, tq);
  note_launch();
  return cudaGetLastError();
}

// T-matrix as an [N][nmax] diagonal and as FP32 copies
__global__ void tq_expand_kernel(int64_t N, int L, const double* __restrict__ tq, double* __restrict__ tdiag,
                                 float* __restrict__ tq32) {
  const int NH = L * (L + 2);
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < N * 2 * L) {
    tq32[2 * t] = static_cast<float>(tq[2 * t]);
    tq32[2 * t + 1] = static_cast<float>(tq[2 * t + 1]);
  }
  if (t >= N * NH) return;
  const int64_t i = t / NH;
  const int r = static_cast<int>(t - i * NH);
  const int l = row_l_rt(r);
  for (int tau = 0; tau < 2; ++tau) {
    const double* q = tq + ((i * 2 + tau) * L + (l - 1)) * 2;
    double* o = tdiag + (i * 2 * NH + tau * NH + r) * 2;
    o[0] = q[0];
    o[1] = q[1];
  }
}

cudaError_t launch_tq_expand(int64_t N, int L, const double* tq, double* tdiag, float* tq32, cudaStream_t st) {
  const int64_t total = N * (L * (L + 2) > 2 * L ? L * (L + 2) : 2 * L);
  const int threads = 256;
  tq_expand_kernel<<<static_cast<unsigned>((total + threads - 1) / threads), threads, 0, st>>>(N, L, tq, tdiag, tq32);
  note_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// incident coefficients
// ---------------------------------------------------------------------------
static __device__ __forceinline__ void row_decode(int n, int L, int& tau, int& l, int& m) {
  const int NH = L * (L + 2);
  tau = n < NH ? 1 : 2;
  const int r = n < NH ? n : n - NH;
  l = row_l_rt(r);
  m = r - (l * (l + 1) - 1);
}

// Plane wave (App. A.2): a_n = 4 E0 e^{i k.r_i} e^{-i m alpha} B^dagger_nj(beta)
__global__ void plane_wave_kernel(int64_t N, int L, double k, const Pos4* __restrict__ pos, double beta, double alpha,
                                  int pol, double e0r, double e0i, double* __restrict__ a) {
  const int nmax = 2 * L * (L + 2);
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= N * nmax) return;
  const int64_t i = t / nmax;
  const int n = static_cast<int>(t - i * nmax);
  int tau, l, m;
  row_decode(n, L, tau, l, m);
  const int am = m < 0 ? -m : m;
  double pi[16], ta[16];
  double sb, cb;
  sincos(beta, &sb, &cb);
  pi_tau_m(L, am, cb, sb, pi, ta);
  const cd bd = b_transform(tau, l, m, pol, pi[l], ta[l], true);
  double sa, ca;
  sincos(alpha, &sa, &ca);
  const Pos4 r = pos[i];
  const double kr = k * (sb * ca * r.x + sb * sa * r.y + cb * r.z);
  const cd v = 4.0 * (mkc(e0r, e0i) * cexp_i(kr - m * alpha)) * bd;
  a[2 * t] = v.re;
  a[2 * t + 1] = v.im;
}

cudaError_t launch_plane_wave(int64_t N, int L, double k, const void* pos, double beta, double alpha, int pol,
                              double e0r, double e0i, double* a, cudaStream_t st) {
  const int64_t total = N * 2 * L * (L + 2);
  const int threads = 128;
  plane_wave_kernel<<<static_cast<unsigned>((total + threads - 1) / threads), threads, 0, st>>>(
      N, L, k, static_cast<const Pos4*>(pos), beta, alpha, pol, e0r, e0i, a);
  note_launch();
  return cudaGetLastError();
}

// Gaussian beam (App. C):
//   a_n = E0 k^2 w^2 / pi  sum_j int_0^{pi/2} dbeta sin cos exp(-w^2 k^2 sin^2/4 + i k z_G cos)
//         B^dagger_nj(beta) I_jn(beta)
//   I_jn = 2 pi e^{-i aG} i^{|m-1|} e^{-i(m-1) phi_G} J_{|m-1|}(k rho_G sin) (d_j1 - i d_j2)/2
//        + 2 pi e^{+i aG} i^{|m+1|} e^{-i(m+1) phi_G} J_{|m+1|}(k rho_G sin) (d_j1 + i d_j2)/2
// (rho_G, phi_G, z_G) cylindrical coordinates of r_i - r_G.  beta integral by
// the Gauss-Legendre nodes/weights given in (nodes, weights).
// The sums over beta that rows share: for every degree and |m| and the two
// Bessel orders |m| - 1 and |m| + 1, Z = sum w e^{i k z cos} {tau_l^m, m pi_l^m}
// J; the rows of both tau and of +-m combine them with factors that do not depend
// on beta.  A CTA holds 32 spheres (lanes); per step of 8 nodes its warps first
// form weight e^{i k z cos} and J_0 .. J_{L+1} of one node each, then add the
// products of their (l, |m|) (12 FP64 instructions per node, where a row of the
// per-row form took about 40, of 48 rows at lmax 4).  Bound by FP64 issue: about
// 310 instructions per (sphere, node).  GB300, 10 000 spheres, lmax 4, 128
// nodes: 13.9 -> 1.7 ms.  Few spheres: a cluster of up to 8 CTAs shares the
// nodes of 32 spheres and adds the sums through distributed shared memory, in
// rank order.
constexpr int kGbMaxL = 5;
constexpr int kGbSpheres = 32;
constexpr int kGbNodes = 8;  // nodes of a step, and warps of the CTA
constexpr int kGbThreads = kGbSpheres * kGbNodes;
constexpr int gb_combos(int L) { return L * (L + 3) / 2; }  // (l, |m|), l = 1..L

// index of (l, |m|): orders ascend, then degrees
__host__ __device__ __forceinline__ int gb_combo(int L, int l, int am) {
  return am == 0 ? l - 1 : L + (am - 1) * (2 * L - am + 2) / 2 + (l - am);
}

// per node: weight sin cos exp(-(w k sin)^2 / 4), sin, cos, then (tau_l^m, m pi_l^m) per (l, |m|)
__global__ void gaussian_table_kernel(int nb, int L, double k, double w, const double* __restrict__ nodes,
                                      const double* __restrict__ weights, double* __restrict__ table) {
  const int id = blockIdx.x * blockDim.x + threadIdx.x;  // (node, |m|)
  const int q = id / (L + 1), am = id - q * (L + 1);
  if (q >= nb) return;
  const int nc = gb_combos(L);
  double* t = table + (int64_t)q * (3 + 2 * nc);
  double sb, cb;
  sincos(nodes[q], &sb, &cb);
  if (am == 0) {
    t[0] = weights[q] * sb * cb * exp(-0.25 * (w * k * sb) * (w * k * sb));
    t[1] = sb;
    t[2] = cb;
  }
  double pi[16], ta[16];
  pi_tau_m(L, am, cb, sb, pi, ta);
  for (int l = am > 1 ? am : 1; l <= L; ++l) {
    t[3 + 2 * gb_combo(L, l, am)] = ta[l];
    t[4 + 2 * gb_combo(L, l, am)] = am * pi[l];
  }
}

// J_0 .. J_M at x >= 0: Miller's downward recurrence with sum J_0 + 2 J_2 + 2
// J_4 + .. = 1 below 8 (from order 34, or 16 below 1: what is left out is under
// 1e-17 of J_M), the leading terms below 1e-8 (the next one of J_0 is x^2 / 4),
// else j0, j1 and the upward recurrence, which is stable for orders below x
template <int M>
__device__ __forceinline__ void bessel_orders(double x, double (&J)[M + 1]) {
  if (x < 1e-8) {
    J[0] = 1.0;
#pragma unroll
    for (int n = 1; n <= M; ++n) J[n] = J[n - 1] * (0.5 * x / n);
    return;
  }
  if (x < 8.0) {
    const double f = 2.0 / x;
    double up = 0.0, cur = 1e-200, sum = 0.0;
    const int top = x < 1.0 ? 16 : 34;  // even
    double g = top * f;                  // 2 n / x
    for (int n = top; n > M + 1; --n) {  // cur holds order n
      if ((n & 1) == 0) sum += cur;
      const double dn = fma(g, cur, -up);
      g -= f;
      up = cur;
      cur = dn;
    }
#pragma unroll
    for (int o = M + 1; o >= 0; --o) {
      if (o <= M) J[o <= M ? o : 0] = cur;
      if (o > 0) {
        if ((o & 1) == 0) sum += cur;
        const double dn = fma(o * f, cur, -up);
        up = cur;
        cur = dn;
      }
    }
    const double r = 1.0 / fma(2.0, sum, J[0]);
#pragma unroll
    for (int o = 0; o <= M; ++o) J[o] *= r;
    return;
  }
  J[0] = j0(x);
  J[1] = j1(x);
  const double f = 2.0 / x;
#pragma unroll
  for (int n = 1; n < M; ++n) J[n + 1] = fma(n * f, J[n], -J[n - 1]);
}

template <int L>
struct GbSmem {
  static constexpr int NC = gb_combos(L);
  union {
    struct {
      double ezr[kGbNodes][kGbSpheres], ezi[kGbNodes][kGbSpheres];
      double J[kGbNodes][L + 2][kGbSpheres];
    } step;
    double Z[NC][8][kGbSpheres];  // (tau, J_-), (tau, J_+), (m pi, J_-), (m pi, J_+), re and im each
  };
  cd U[2 * L + 1][kGbSpheres], V[2 * L + 1][kGbSpheres];
};

template <int L>
__global__ void __launch_bounds__(kGbThreads)
    gaussian_beam_kernel(int64_t N, double k, const Pos4* __restrict__ pos, double w, double fx, double fy, double fz,
                         double alphaG, double e0r, double e0i, int nb, const double* __restrict__ table,
                         double* __restrict__ a) {
  extern __shared__ __align__(16) unsigned char gb_smem[];
  GbSmem<L>& sm = *reinterpret_cast<GbSmem<L>*>(gb_smem);
  constexpr int NC = gb_combos(L), PER = (NC + kGbNodes - 1) / kGbNodes, TS = 3 + 2 * NC;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int C = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t i0 = blockIdx.x / C * (int64_t)kGbSpheres;
  const Pos4 r = pos[i0 + lane < N ? i0 + lane : N - 1];
  const double dx = r.x - fx, dy = r.y - fy, kz = k * (r.z - fz);
  const double krho = k * sqrt(dx * dx + dy * dy);
  const double phiG = atan2(dy, dx);
  for (int q = wid; q <= 2 * L; q += kGbNodes) {
    const int m = q - L;
    sm.U[q][lane] = cexp_i(-alphaG - (m - 1) * phiG) * ipow(abs(m - 1));
    sm.V[q][lane] = cexp_i(alphaG - (m + 1) * phiG) * ipow(abs(m + 1));
  }
  // this warp's (l, |m|): the Bessel orders they take
  int jm[PER], jp[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    int c = wid + u * kGbNodes, am = 0;
    if (c >= L) {
      c -= L;
      am = 1;
      while (am < L && c >= L - am + 1) {  // past the last one: not used
        c -= L - am + 1;
        ++am;
      }
    }
    jm[u] = am == 0 ? 1 : am - 1;
    jp[u] = am + 1;
  }
  double acc[PER][8] = {};
  for (int q0 = rank * kGbNodes; q0 < nb; q0 += C * kGbNodes) {
    __syncthreads();
    {
      const int q = q0 + wid;
      double J[L + 2], g = 0.0, sn = 0.0, cs = 0.0;
#pragma unroll
      for (int o = 0; o <= L + 1; ++o) J[o] = 0.0;
      if (q < nb) g = table[(int64_t)q * TS];
      if (g != 0.0) {
        const double* t = table + (int64_t)q * TS;
        bessel_orders<L + 1>(krho * t[1], J);
        sincos_phase(kz * t[2], &sn, &cs);
      }
      sm.step.ezr[wid][lane] = g * cs;
      sm.step.ezi[wid][lane] = g * sn;
#pragma unroll
      for (int o = 0; o <= L + 1; ++o) sm.step.J[wid][o][lane] = J[o];
    }
    __syncthreads();
    for (int v = 0; v < kGbNodes; ++v) {
      if (q0 + v >= nb) break;
      const double er = sm.step.ezr[v][lane], ei = sm.step.ezi[v][lane];
      const double* t = table + (int64_t)(q0 + v) * TS + 3;
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int c = wid + u * kGbNodes;
        if (c < NC) {
          const double ta = t[2 * c], mp = t[2 * c + 1];
          const double Jm = sm.step.J[v][jm[u]][lane], Jp = sm.step.J[v][jp[u]][lane];
          const double tr = ta * er, ti = ta * ei, pr = mp * er, pi = mp * ei;
          acc[u][0] = fma(tr, Jm, acc[u][0]);
          acc[u][1] = fma(ti, Jm, acc[u][1]);
          acc[u][2] = fma(tr, Jp, acc[u][2]);
          acc[u][3] = fma(ti, Jp, acc[u][3]);
          acc[u][4] = fma(pr, Jm, acc[u][4]);
          acc[u][5] = fma(pi, Jm, acc[u][5]);
          acc[u][6] = fma(pr, Jp, acc[u][6]);
          acc[u][7] = fma(pi, Jp, acc[u][7]);
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int c = wid + u * kGbNodes;
    if (c < NC) {
#pragma unroll
      for (int z = 0; z < 8; ++z) sm.Z[c][z][lane] = acc[u][z];
    }
  }
  cluster.sync();
  constexpr int nmax = 2 * L * (L + 2);
  const cd scale = (k * k * w * w / 3.14159265358979323846) * mkc(e0r, e0i);
  // rows along the lanes: coalesced
  for (int q = rank * kGbThreads + threadIdx.x; q < kGbSpheres * nmax; q += C * kGbThreads) {
    const int sph = q / nmax, n = q - sph * nmax;
    if (i0 + sph >= N) continue;
    int tau, l, m;
    row_decode(n, L, tau, l, m);
    const int am = m < 0 ? -m : m, c = gb_combo(L, l, am);
    // J_{|m-1|} and J_{|m+1|}: J_- and J_+ of |m|, the other way round for m < 0
    const int zu = m >= 0 ? 0 : 2, zv = 2 - zu;
    auto Z = [&](int kind, int off) {
      cd z = mkc(0.0);
      for (int o = 0; o < C; ++o) {
        const GbSmem<L>& other = *cluster.map_shared_rank(&sm, o);
        z = z + cd{other.Z[c][4 * kind + off][sph], other.Z[c][4 * kind + off + 1][sph]};
      }
      return z;
    };
    // B_nj takes tau_l^|m| for j = tau, m pi_l^|m| otherwise
    const double sg1 = tau == 1 ? 1.0 : (m < 0 ? -1.0 : 1.0), sg2 = tau == 2 ? 1.0 : (m < 0 ? -1.0 : 1.0);
    const int k1 = tau == 1 ? 0 : 1, k2 = tau == 2 ? 0 : 1;
    const cd U = sm.U[m + L][sph], V = sm.V[m + L][sph];
    // I_1 = pi (U + V), I_2 = pi (-i U + i V)
    const cd I1 = 3.14159265358979323846 * (U * Z(k1, zu) + V * Z(k1, zv));
    const cd I2 = 3.14159265358979323846 * (cd{0, -1} * (U * Z(k2, zu)) + cd{0, 1} * (V * Z(k2, zv)));
    const cd B1 = b_transform(1, l, m, 1, 0.0, sg1, true), B2 = b_transform(2, l, m, 2, 0.0, sg2, true);
    const cd v = scale * (B1 * I1 + B2 * I2);
    a[2 * ((i0 + sph) * nmax + n)] = v.re;
    a[2 * ((i0 + sph) * nmax + n) + 1] = v.im;
  }
  cluster.sync();  // no CTA leaves while others read its sums
}

int64_t gaussian_table_entries(int L, int nb) { return (int64_t)nb * (3 + 2 * gb_combos(L)); }

template <int L>
static cudaError_t launch_gaussian_t(int64_t N, double k, const void* pos, double w, const double* focus,
                                     double alphaG, double e0r, double e0i, int nb, const double* table, double* a,
                                     cudaStream_t st) {
  static PerDevice attr;
  if (attr.get(current_device, [] {
        return cudaFuncSetAttribute(gaussian_beam_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    static_cast<int>(sizeof(GbSmem<L>))) == cudaSuccess
                   ? 1
                   : 0;
      }) == 0)
    return cudaErrorInvalidConfiguration;
  // two CTAs per SM before the nodes are shared out
  const int64_t tiles = (N + kGbSpheres - 1) / kGbSpheres;
  int C = 1;
  while (C < 8 && tiles * C * 2 <= 2 * device_sms() && C * kGbNodes < nb) C *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles * C));
  cfg.blockDim = dim3(kGbThreads);
  cfg.dynamicSmemBytes = sizeof(GbSmem<L>);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = static_cast<unsigned>(C);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, gaussian_beam_kernel<L>, N, k, static_cast<const Pos4*>(pos), w,
                                           focus[0], focus[1], focus[2], alphaG, e0r, e0i, nb, table, a);
  note_launch();
  return e;
}

// table: device scratch of gaussian_table_entries(L, nb) doubles
cudaError_t launch_gaussian_beam(int64_t N, int L, double k, const void* pos, double w, const double* focus,
                                 double alphaG, double e0r, double e0i, int nb, const double* nodes,
                                 const double* weights, double* table, double* a, cudaStream_t st) {
  if (L < 1 || L > kGbMaxL) return cudaErrorInvalidValue;
  if (N <= 0) return cudaSuccess;
  gaussian_table_kernel<<<(nb * (L + 1) + 63) / 64, 64, 0, st>>>(nb, L, k, w, nodes, weights, table);
  note_launch();
  switch (L) {
    case 1: return launch_gaussian_t<1>(N, k, pos, w, focus, alphaG, e0r, e0i, nb, table, a, st);
    case 2: return launch_gaussian_t<2>(N, k, pos, w, focus, alphaG, e0r, e0i, nb, table, a, st);
    case 3: return launch_gaussian_t<3>(N, k, pos, w, focus, alphaG, e0r, e0i, nb, table, a, st);
    case 4: return launch_gaussian_t<4>(N, k, pos, w, focus, alphaG, e0r, e0i, nb, table, a, st);
    default: return launch_gaussian_t<5>(N, k, pos, w, focus, alphaG, e0r, e0i, nb, table, a, st);
  }
}

// ---------------------------------------------------------------------------
// vector kernels (complex vectors of n elements, element type Pair2<R>)
// ---------------------------------------------------------------------------
constexpr int kVecThreads = 256;

// partial[b][j] = sum over this block's range of conj(V_j) w, sixteen vectors
// per pass (w read once per pass), two elements per loop step so that 34
// loads are in flight per thread; per-thread and warp sums in the vector's own
// precision (a few dozen terms each), block sums in FP64.  Launched with two
// CTAs per SM (vec_dot_blocks): each thread then covers enough elements per
// pass to repay the pass's reduction (measured on GB300 at 480 000 elements
// and 50 vectors: 62 us against 118 us for eight vectors per pass at four
// CTAs per SM).
template <typename R>
__global__ void __launch_bounds__(kVecThreads) multi_dotc_kernel(int64_t n, int nv, const Pair2<R>* __restrict__ V,
                                                                int64_t ldv, const Pair2<R>* __restrict__ w,
                                                                double* __restrict__ partial) {
  constexpr int JT = 16;
  __shared__ double red[2 * JT][kVecThreads / 32];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int j0 = 0; j0 < nv; j0 += JT) {
    const int nj = nv - j0 < JT ? nv - j0 : JT;
    R sr[JT], si[JT];
#pragma unroll
    for (int q = 0; q < JT; ++q) sr[q] = si[q] = static_cast<R>(0);
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; t + stride < n; t += 2 * stride) {
      const Pair2<R> b0 = w[t], b1 = w[t + stride];
#pragma unroll
      for (int q = 0; q < JT; ++q) {
        if (q < nj) {
          const Pair2<R> a0 = V[(j0 + q) * ldv + t];
          const Pair2<R> a1 = V[(j0 + q) * ldv + t + stride];
          sr[q] = fma_(a0.re, b0.re, fma_(a0.im, b0.im, sr[q]));
          si[q] = fma_(a0.re, b0.im, fma_(-a0.im, b0.re, si[q]));
          sr[q] = fma_(a1.re, b1.re, fma_(a1.im, b1.im, sr[q]));
          si[q] = fma_(a1.re, b1.im, fma_(-a1.im, b1.re, si[q]));
        }
      }
    }
    if (t < n) {
      const Pair2<R> b0 = w[t];
#pragma unroll
      for (int q = 0; q < JT; ++q) {
        if (q < nj) {
          const Pair2<R> a0 = V[(j0 + q) * ldv + t];
          sr[q] = fma_(a0.re, b0.re, fma_(a0.im, b0.im, sr[q]));
          si[q] = fma_(a0.re, b0.im, fma_(-a0.im, b0.re, si[q]));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < JT; ++q) {
      R a = sr[q], b = si[q];
      for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
      }
      if ((threadIdx.x & 31) == 0) {
        red[2 * q][threadIdx.x >> 5] = static_cast<double>(a);
        red[2 * q + 1][threadIdx.x >> 5] = static_cast<double>(b);
      }
    }
    __syncthreads();
    if (threadIdx.x < 2 * nj) {
      double s = 0.0;
      for (int q = 0; q < kVecThreads / 32; ++q) s += red[threadIdx.x][q];
      const int q = threadIdx.x >> 1;
      partial[((int64_t)blockIdx.x * nv + j0 + q) * 2 + (threadIdx.x & 1)] = s;
    }
    __syncthreads();
  }
}

__global__ void reduce_partials_kernel(int nblocks, int nv, const double* __restrict__ partial,
                                       double* __restrict__ out) {
  const int j = blockIdx.x;
  double a = 0.0, b = 0.0;
  for (int q = threadIdx.x; q < nblocks; q += blockDim.x) {
    a += partial[((int64_t)q * nv + j) * 2];
    b += partial[((int64_t)q * nv + j) * 2 + 1];
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  __shared__ double red[2][32];
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = a;
    red[1][threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sa = 0.0, sb = 0.0;
    for (int q = 0; q < (int)(blockDim.x + 31) / 32; ++q) {
      sa += red[0][q];
      sb += red[1][q];
    }
    out[2 * j] = sa;
    out[2 * j + 1] = sb;
  }
}

int device_sms() {
  static PerDevice cache;
  const int n = cache.get(current_device, [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return v;
  });
  return n > 0 ? n : 1;
}

int vec_dot_blocks(int64_t n) {
  const int64_t b = (n + kVecThreads - 1) / kVecThreads;
  const int64_t cap = 2LL * device_sms();
  return static_cast<int>(b < cap ? (b > 0 ? b : 1) : cap);
}

template <typename R>
cudaError_t launch_multi_dotc(int64_t n, int nv, const void* V, int64_t ldv, const void* w, double* partial,
                              double* out, cudaStream_t st) {
  const int nb = vec_dot_blocks(n);
  multi_dotc_kernel<R><<<nb, kVecThreads, 0, st>>>(n, nv, static_cast<const Pair2<R>*>(V), ldv,
                                                   static_cast<const Pair2<R>*>(w), partial);
  reduce_partials_kernel<<<nv, 256, 0, st>>>(nb, nv, partial, out);
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_multi_dotc<float>(int64_t, int, const void*, int64_t, const void*, double*, double*,
                                              cudaStream_t);
template cudaError_t launch_multi_dotc<double>(int64_t, int, const void*, int64_t, const void*, double*, double*,
                                               cudaStream_t);

// w <- alpha0 * w - sum_j h_j V_j   (h given as FP64 complex on the device;
// arithmetic in the vector's precision).  Two elements
// per thread step and the loads of eight vectors issued before their FMAs
// (16 loads in flight per thread), four CTAs per SM; each element's sum is
// formed in the same order as a plain loop over j (measured on GB300 at
// 480 000 elements and 50 vectors: 70 us against 110 us for one element and
// one vector at a time).
template <typename R>
__global__ void __launch_bounds__(kVecThreads) multi_axpy_kernel(int64_t n, int nv, const Pair2<R>* __restrict__ V,
                                                                int64_t ldv, const double* __restrict__ h,
                                                                double alpha0, Pair2<R>* __restrict__ w) {
  constexpr int U = 8;
  __shared__ R hs[2 * 128];
  for (int q = threadIdx.x; q < 2 * nv && q < 256; q += blockDim.x) hs[q] = static_cast<R>(h[q]);
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += 2 * stride) {
    const bool two = t + stride < n;
    const int64_t t1 = two ? t + stride : t;
    R ar0 = static_cast<R>(alpha0) * w[t].re, ai0 = static_cast<R>(alpha0) * w[t].im;
    R ar1 = static_cast<R>(alpha0) * w[t1].re, ai1 = static_cast<R>(alpha0) * w[t1].im;
    int j = 0;
    for (; j + U <= nv; j += U) {
      Pair2<R> v0[U], v1[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        v0[u] = V[(j + u) * ldv + t];
        v1[u] = V[(j + u) * ldv + t1];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int jj = j + u;
        const R hr = jj < 128 ? hs[2 * jj] : static_cast<R>(h[2 * jj]);
        const R hi = jj < 128 ? hs[2 * jj + 1] : static_cast<R>(h[2 * jj + 1]);
        ar0 = fma_(-hr, v0[u].re, fma_(hi, v0[u].im, ar0));
        ai0 = fma_(-hr, v0[u].im, fma_(-hi, v0[u].re, ai0));
        ar1 = fma_(-hr, v1[u].re, fma_(hi, v1[u].im, ar1));
        ai1 = fma_(-hr, v1[u].im, fma_(-hi, v1[u].re, ai1));
      }
    }
    for (; j < nv; ++j) {
      const Pair2<R> a = V[j * ldv + t], b = V[j * ldv + t1];
      const R hr = j < 128 ? hs[2 * j] : static_cast<R>(h[2 * j]);
      const R hi = j < 128 ? hs[2 * j + 1] : static_cast<R>(h[2 * j + 1]);
      ar0 = fma_(-hr, a.re, fma_(hi, a.im, ar0));
      ai0 = fma_(-hr, a.im, fma_(-hi, a.re, ai0));
      ar1 = fma_(-hr, b.re, fma_(hi, b.im, ar1));
      ai1 = fma_(-hr, b.im, fma_(-hi, b.re, ai1));
    }
    w[t] = Pair2<R>{ar0, ai0};
    if (two) w[t1] = Pair2<R>{ar1, ai1};
  }
}

// One Arnoldi step of a short Krylov vector in one cooperative launch: classical
// Gram-Schmidt of w against V_0 .. V_{nv-1}, twice, the norm and the normalised
// next vector.  w stays in registers (up to four elements a thread); the dots
// sum per thread and warp in the vector's precision and per block in FP64, like
// multi_dotc_kernel, and the blocks' sums are added in order.  Vectors this short
// (basis in L2) are bound by latency: five barriers here against eight launches,
// three copies and three host synchronisations (N = 120, lmax 3, refined solve:
// 5.4 -> 2.8 ms).  CL: up to eight blocks form one cluster and meet at its
// hardware barrier (23 us a step at n = 3 600, as with fifteen blocks and grid
// barriers); otherwise a cooperative launch of 33 to 64 blocks, which deals the
// dots out.
// out: nv coefficients (the sum of both passes), then the squared norm.
constexpr int kArnoldiElems = 4;
constexpr int kArnoldiCluster = 8;

template <typename R, bool CL>
__global__ void __launch_bounds__(kVecThreads)
    arnoldi_kernel(int64_t n, int nv, Pair2<R>* __restrict__ V, int64_t ldv, const Pair2<R>* __restrict__ w,
                   double* __restrict__ partial, double* __restrict__ hbuf, double* __restrict__ out) {
  constexpr int JT = 16, NW = kVecThreads / 32;
  namespace cg = cooperative_groups;
  auto sync = [] {
    if constexpr (CL) cg::this_cluster().sync();
    else cg::this_grid().sync();
  };
  __shared__ double red[2 * JT][NW];
  __shared__ R hs[2 * kArnoldiMaxVectors];
  __shared__ double hd[2 * kArnoldiMaxVectors];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nb = gridDim.x;
  const int64_t stride = (int64_t)nb * kVecThreads, t0 = blockIdx.x * (int64_t)kVecThreads + tid;
  Pair2<R> x[kArnoldiElems];
#pragma unroll
  for (int e = 0; e < kArnoldiElems; ++e) x[e] = t0 + e * stride < n ? w[t0 + e * stride] : Pair2<R>{0, 0};
  // block b's dots conj(U_j) x, j < cnt, into partial[b][j]
  auto dots = [&](const Pair2<R>* U, int cnt, bool self) {
    for (int j0 = 0; j0 < cnt; j0 += JT) {
      const int nj = cnt - j0 < JT ? cnt - j0 : JT;
      R sr[JT], si[JT];
#pragma unroll
      for (int q = 0; q < JT; ++q) sr[q] = si[q] = static_cast<R>(0);
#pragma unroll
      for (int e = 0; e < kArnoldiElems; ++e) {
        const int64_t t = t0 + e * stride;
        if (t < n) {
#pragma unroll
          for (int q = 0; q < JT; ++q) {
            if (q < nj) {
              const Pair2<R> a = self ? x[e] : U[(j0 + q) * ldv + t];
              sr[q] = fma_(a.re, x[e].re, fma_(a.im, x[e].im, sr[q]));
              si[q] = fma_(a.re, x[e].im, fma_(-a.im, x[e].re, si[q]));
            }
          }
        }
      }
#pragma unroll
      for (int q = 0; q < JT; ++q) {
        if (q < nj) {
          R a = sr[q], b = si[q];
          for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
          }
          if (lane == 0) {
            red[2 * q][wid] = static_cast<double>(a);
            red[2 * q + 1][wid] = static_cast<double>(b);
          }
        }
      }
      __syncthreads();
      if (tid < 2 * nj) {
        double s = 0.0;
        for (int q = 0; q < NW; ++q) s += red[tid][q];
        partial[((int64_t)blockIdx.x * kArnoldiMaxVectors + j0) * 2 + tid] = s;
      }
      __syncthreads();
    }
  };
  // the blocks' sums of dot j, by one warp
  auto total = [&](int j, double& re, double& im) {
    re = im = 0.0;
    for (int b = lane; b < nb; b += 32) {
      re += __ldcg(partial + ((int64_t)b * kArnoldiMaxVectors + j) * 2);
      im += __ldcg(partial + ((int64_t)b * kArnoldiMaxVectors + j) * 2 + 1);
    }
    for (int o = 16; o > 0; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
  };
  for (int pass = 0; pass < 2; ++pass) {
    dots(V, nv, false);
    sync();
    // (a cluster never has more than 16 blocks; asked all the same, since with CL alone
    // the compiler takes 76 registers instead of 64, and a refined solve of 120
    // spheres 2.80 instead of 2.71 ms)
    if (CL && nb <= 16) {
      // few blocks: every block adds up all dots, one part per thread (a warp per
      // dot would wait for its loads and FP64 shuffles dot after dot)
      for (int q = tid; q < 2 * nv; q += kVecThreads) {
        double sum = 0.0;
#pragma unroll 8
        for (int b = 0; b < nb; ++b) sum += __ldcg(partial + (int64_t)b * kArnoldiMaxVectors * 2 + q);
        hd[q] = sum;
      }
    } else {
      // the dots are dealt to the blocks; the barrier after them also lets the next
      // ones overwrite the sums
      for (int j = blockIdx.x + nb * wid; j < nv; j += nb * NW) {
        double re, im;
        total(j, re, im);
        if (lane == 0) {
          hbuf[(pass * kArnoldiMaxVectors + j) * 2] = re;
          hbuf[(pass * kArnoldiMaxVectors + j) * 2 + 1] = im;
        }
      }
      sync();
      for (int q = tid; q < 2 * nv; q += kVecThreads) hd[q] = __ldcg(hbuf + pass * kArnoldiMaxVectors * 2 + q);
    }
    __syncthreads();
    for (int q = tid; q < 2 * nv; q += kVecThreads) {
      hs[q] = static_cast<R>(hd[q]);
      if (blockIdx.x == 0) out[q] = pass == 0 ? hd[q] : out[q] + hd[q];
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < kArnoldiElems; ++e) {
      const int64_t t = t0 + e * stride;
      if (t < n) {
        R ar = x[e].re, ai = x[e].im;
#pragma unroll 8
        for (int j = 0; j < nv; ++j) {
          const Pair2<R> v = V[j * ldv + t];
          ar = fma_(-hs[2 * j], v.re, fma_(hs[2 * j + 1], v.im, ar));
          ai = fma_(-hs[2 * j], v.im, fma_(-hs[2 * j + 1], v.re, ai));
        }
        x[e] = Pair2<R>{ar, ai};
      }
    }
    if (CL && nb <= 16) sync();  // every block has read the sums that the next dots overwrite
  }
  dots(V, 1, true);
  sync();
  double n2, unused;
  total(0, n2, unused);
  if (blockIdx.x == 0 && tid == 0) out[2 * nv] = n2;
  if (n2 > 0.0) {
    const double a = 1.0 / sqrt(n2);
    Pair2<R>* next = V + (int64_t)nv * ldv;
#pragma unroll
    for (int e = 0; e < kArnoldiElems; ++e) {
      const int64_t t = t0 + e * stride;
      if (t < n)
        next[t] = Pair2<R>{static_cast<R>(a * static_cast<double>(x[e].re)), static_cast<R>(a * static_cast<double>(x[e].im))};
    }
  }
}

// blocks of the one-launch step for vectors of n elements and nv basis vectors; 0: not for these
int arnoldi_blocks(int64_t n, int max_vectors) {
  const int64_t b = (n + kVecThreads - 1) / kVecThreads;
  const int64_t cap = std::min(64, device_sms());
  if (max_vectors > kArnoldiMaxVectors || n > cap * kVecThreads * kArnoldiElems) return 0;
  if (n <= kArnoldiCluster * kVecThreads * kArnoldiElems) {  // one cluster: 1, 2, 4 or 8 blocks
    int c = 1;
    while (c < kArnoldiCluster && c < b) c *= 2;
    return c;
  }
  return static_cast<int>(std::max<int64_t>(1, std::min(b, cap)));
}
size_t arnoldi_scratch_bytes(int blocks) { return sizeof(double) * 2 * kArnoldiMaxVectors * (blocks + 2); }

// V_nv = w orthogonalised against V_0 .. V_{nv-1} and normalised; out (device):
// 2 nv + 1 doubles.  scratch: arnoldi_scratch_bytes(arnoldi_blocks(n, ..))
template <typename R>
cudaError_t launch_arnoldi(int64_t n, int nv, void* V, int64_t ldv, const void* w, void* scratch, double* out,
                           cudaStream_t st) {
  const int nb = arnoldi_blocks(n, nv);
  if (nb < 1) return cudaErrorInvalidValue;
  auto* Vp = static_cast<Pair2<R>*>(V);
  auto* wp = static_cast<const Pair2<R>*>(w);
  double* partial = static_cast<double*>(scratch);
  double* hbuf = partial + (int64_t)2 * kArnoldiMaxVectors * nb;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(nb));
  cfg.blockDim = dim3(kVecThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaError_t e;
  if (nb <= kArnoldiCluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = static_cast<unsigned>(nb);
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    e = cudaLaunchKernelEx(&cfg, arnoldi_kernel<R, true>, n, nv, Vp, ldv, wp, partial, hbuf, out);
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    e = cudaLaunchKernelEx(&cfg, arnoldi_kernel<R, false>, n, nv, Vp, ldv, wp, partial, hbuf, out);
  }
  note_launch();
  return e;
}
template cudaError_t launch_arnoldi<float>(int64_t, int, void*, int64_t, const void*, void*, double*, cudaStream_t);
template cudaError_t launch_arnoldi<double>(int64_t, int, void*, int64_t, const void*, void*, double*, cudaStream_t);

// y <- beta * y + sum_j c_j V_j    (c given on the device)
template <typename R>
__global__ void multi_combine_kernel(int64_t n, int nv, const Pair2<R>* __restrict__ V, int64_t ldv,
                                     const double* __restrict__ c, double beta, Pair2<R>* __restrict__ y) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    R ar = 0, ai = 0;
    if (beta != 0.0) {
      ar = static_cast<R>(beta) * y[t].re;
      ai = static_cast<R>(beta) * y[t].im;
    }
    for (int j = 0; j < nv; ++j) {
      const Pair2<R> v = V[j * ldv + t];
      const R cr = static_cast<R>(c[2 * j]), ci = static_cast<R>(c[2 * j + 1]);
      ar = fma_(cr, v.re, fma_(-ci, v.im, ar));
      ai = fma_(cr, v.im, fma_(ci, v.re, ai));
    }
    y[t] = Pair2<R>{ar, ai};
  }
}

static int vec_grid(int64_t n) {
  const int64_t b = (n + kVecThreads - 1) / kVecThreads;
  const int64_t cap = 16LL * device_sms();
  return static_cast<int>(b < cap ? (b > 0 ? b : 1) : cap);
}

template <typename R>
cudaError_t launch_multi_axpy(int64_t n, int nv, const void* V, int64_t ldv, const double* h, double alpha0, void* w,
                              cudaStream_t st) {
  const int64_t pairs = (n + 2 * kVecThreads - 1) / (2 * kVecThreads);
  const int64_t cap = 4LL * device_sms();
  const unsigned grid = static_cast<unsigned>(pairs < cap ? (pairs > 0 ? pairs : 1) : cap);
  multi_axpy_kernel<R><<<grid, kVecThreads, 0, st>>>(n, nv, static_cast<const Pair2<R>*>(V), ldv, h, alpha0,
                                                            static_cast<Pair2<R>*>(w));
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_multi_axpy<float>(int64_t, int, const void*, int64_t, const double*, double, void*,
                                              cudaStream_t);
template cudaError_t launch_multi_axpy<double>(int64_t, int, const void*, int64_t, const double*, double, void*,
                                               cudaStream_t);

template <typename R>
cudaError_t launch_multi_combine(int64_t n, int nv, const void* V, int64_t ldv, const double* c, double beta, void* y,
                                 cudaStream_t st) {
  multi_combine_kernel<R><<<vec_grid(n), kVecThreads, 0, st>>>(n, nv, static_cast<const Pair2<R>*>(V), ldv, c, beta,
                                                               static_cast<Pair2<R>*>(y));
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_multi_combine<float>(int64_t, int, const void*, int64_t, const double*, double, void*,
                                                 cudaStream_t);
template cudaError_t launch_multi_combine<double>(int64_t, int, const void*, int64_t, const double*, double, void*,
                                                  cudaStream_t);

// y <- a * x + b * y (real scalars), element types may differ (cast)
template <typename RX, typename RY>
__global__ void axpby_kernel(int64_t n, double a, const Pair2<RX>* x, double b, Pair2<RY>* y) {  // x may alias y
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    double r = a * static_cast<double>(x[t].re), i = a * static_cast<double>(x[t].im);
    if (b != 0.0) {
      r += b * static_cast<double>(y[t].re);
      i += b * static_cast<double>(y[t].im);
    }
    y[t] = Pair2<RY>{static_cast<RY>(r), static_cast<RY>(i)};
  }
}

// z = a x + b y with complex a, b (z may alias x or y)
template <typename R>
__global__ void caxpbyz_kernel(int64_t n, R ar, R ai, const Pair2<R>* x, R br, R bi, const Pair2<R>* y,
                               Pair2<R>* z) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const Pair2<R> u = x[t], v = y[t];
    const R re = fma_(ar, u.re, fma_(-ai, u.im, fma_(br, v.re, -bi * v.im)));
    const R im = fma_(ar, u.im, fma_(ai, u.re, fma_(br, v.im, bi * v.re)));
    z[t] = Pair2<R>{re, im};
  }
}
template <typename R>
cudaError_t launch_caxpbyz(int64_t n, double ar, double ai, const void* x, double br, double bi, const void* y,
                           void* z, cudaStream_t st) {
  caxpbyz_kernel<R><<<vec_grid(n), kVecThreads, 0, st>>>(n, static_cast<R>(ar), static_cast<R>(ai),
                                                           static_cast<const Pair2<R>*>(x), static_cast<R>(br),
                                                           static_cast<R>(bi), static_cast<const Pair2<R>*>(y),
                                                           static_cast<Pair2<R>*>(z));
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_caxpbyz<float>(int64_t, double, double, const void*, double, double, const void*, void*,
                                           cudaStream_t);
template cudaError_t launch_caxpbyz<double>(int64_t, double, double, const void*, double, double, const void*, void*,
                                            cudaStream_t);

template <typename RX, typename RY>
cudaError_t launch_axpby(int64_t n, double a, const void* x, double b, void* y, cudaStream_t st) {
  axpby_kernel<RX, RY><<<vec_grid(n), kVecThreads, 0, st>>>(n, a, static_cast<const Pair2<RX>*>(x), b,
                                                            static_cast<Pair2<RY>*>(y));
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_axpby<float, float>(int64_t, double, const void*, double, void*, cudaStream_t);
template cudaError_t launch_axpby<double, double>(int64_t, double, const void*, double, void*, cudaStream_t);
template cudaError_t launch_axpby<float, double>(int64_t, double, const void*, double, void*, cudaStream_t);
template cudaError_t launch_axpby<double, float>(int64_t, double, const void*, double, void*, cudaStream_t);

// y = T x elementwise with the [N][nmax] FP64 diagonal (RHS T a_in)
__global__ void tdiag_mul_kernel(int64_t n_per_rhs, int nrhs, const double* __restrict__ tdiag,
                                 const double* __restrict__ x, double* __restrict__ y) {
  const int64_t total = n_per_rhs * nrhs;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = t % n_per_rhs;
    const cd v = mkc(tdiag[2 * e], tdiag[2 * e + 1]) * mkc(x[2 * t], x[2 * t + 1]);
    y[2 * t] = v.re;
    y[2 * t + 1] = v.im;
  }
}

cudaError_t launch_tdiag_mul(int64_t n_per_rhs, int nrhs, const double* tdiag, const double* x, double* y,
                             cudaStream_t st) {
  tdiag_mul_kernel<<<vec_grid(n_per_rhs * nrhs), kVecThreads, 0, st>>>(n_per_rhs, nrhs, tdiag, x, y);
  note_launch();
  return cudaGetLastError();
}

// non-finite scan: flag[0] = 1 if any element is NaN or Inf
template <typename R>
__global__ void nonfinite_kernel(int64_t n, const R* __restrict__ v, int* __restrict__ flag) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    if (!isfinite(v[t])) *flag = 1;
  }
}
template <typename R>
cudaError_t launch_nonfinite(int64_t n, const void* v, int* flag, cudaStream_t st) {
  nonfinite_kernel<R><<<vec_grid(n), kVecThreads, 0, st>>>(n, static_cast<const R*>(v), flag);
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_nonfinite<float>(int64_t, const void*, int*, cudaStream_t);
template cudaError_t launch_nonfinite<double>(int64_t, const void*, int*, cudaStream_t);

// ---------------------------------------------------------------------------
// far field (App. D)
//   g_j = 1/(2 pi) sum_n B_nj(beta) e^{i m alpha} F_n,   F_n = sum_i e^{-i k.r_i} b^i_n
// The sum over spheres first: F is a (directions x spheres) phase matrix times
// the (spheres x nmax) coefficients, which both polarisations share, and the
// angular factors meet it once per direction.  Bound by FP64 issue: 3 FMAs per
// (direction, sphere, n) (complex products as three real ones) plus the phase,
// 26 instructions per (direction, sphere); one CTA per direction contracting
// with both B_nj per sphere took 8 FMAs and a full sincos.  GB300, 10 000
// spheres, lmax 4, 2 048 directions: 23.8 -> 6.1 ms.
// Its error is that of k.r, as long as that is summed like x and y first, then z
// (packings are centred in x and y: 1.2 times the error with z first), and no
// running sum is long: one takes every eighth or fourth sphere of a chunk (256
// spheres where there are many directions), then 16 chunks.  653 spheres, lmax 5, 221
// directions, against 64 bits: 1.05e-15 with one running sum per chunk and z
// first, 8.0e-16 so, 7.8e-16 with one CTA per direction (10 000 spheres: 7.3e-15).
// ---------------------------------------------------------------------------
constexpr int kFfTile = 8;      // spheres staged at a time
constexpr int kFfThreads = 256;
constexpr int kFfMaxL = 5;

// grid (direction tiles, sphere chunks): F [chunk][direction][nmax] complex.
// Thread (tx, ty) = (tid & 15, tid >> 4) holds DT directions from DT ty and rows
// tx + 16 u, u < NPT.
template <int NPT, int DT>
__global__ void __launch_bounds__(kFfThreads)
    farfield_sum_kernel(int64_t N, int64_t chunk, int nmax, double k, const Pos4* __restrict__ pos,
                        const double2* __restrict__ b, int64_t Nd, const double* __restrict__ dirs,
                        double2* __restrict__ F) {
  constexpr int kFfDirs = 16 * DT;
  __shared__ double kv[kFfDirs][3];
  __shared__ double pc[kFfTile][kFfDirs], ps[kFfTile][kFfDirs], pt[kFfTile][kFfDirs];
  __shared__ double br[kFfTile][16 * NPT], bi[kFfTile][16 * NPT], bt[kFfTile][16 * NPT];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int64_t d0 = blockIdx.x * (int64_t)kFfDirs;
  if (tid < kFfDirs) {
    const int64_t d = d0 + tid < Nd ? d0 + tid : Nd - 1;
    double sb, cb, sa, ca;
    sincos_phase(dirs[2 * d], &sb, &cb);
    sincos_phase(dirs[2 * d + 1], &sa, &ca);
    kv[tid][0] = k * sb * ca;
    kv[tid][1] = k * sb * sa;
    kv[tid][2] = k * cb;
  }
  // products P1 = c br, P2 = s bi, P3 = (c + s)(br + bi) of the phase c + i s, in NC
  // running sums that take the spheres in turn; with 64 directions, whose registers
  // are full, in one of at most 256 spheres, added up in F
  constexpr int NC = DT > 1 ? 1 : (NPT == 2 || NPT == 3 ? 8 : 4), kRun = 256;
  double p1[NC][DT][NPT] = {}, p2[NC][DT][NPT] = {}, p3[NC][DT][NPT] = {};
  bool stored = false;
  auto store = [&] {
#pragma unroll
    for (int a = 0; a < DT; ++a) {
      const int64_t d = d0 + DT * ty + a;
#pragma unroll
      for (int u = 0; u < NPT; ++u) {
#pragma unroll
        for (int w = NC / 2; w > 0; w /= 2) {
#pragma unroll
          for (int q = 0; q < w; ++q) {
            p1[q][a][u] += p1[q + w][a][u];
            p2[q][a][u] += p2[q + w][a][u];
            p3[q][a][u] += p3[q + w][a][u];
          }
        }
        const int n = tx + 16 * u;
        if (d < Nd && n < nmax) {
          double2& f = F[((int64_t)blockIdx.y * Nd + d) * nmax + n];
          double2 v = make_double2(p1[0][a][u] - p2[0][a][u], p3[0][a][u] - p1[0][a][u] - p2[0][a][u]);
          if (stored) {
            v.x += f.x;
            v.y += f.y;
          }
          f = v;
        }
        p1[0][a][u] = p2[0][a][u] = p3[0][a][u] = 0.0;
      }
    }
    stored = true;
  };
  const int64_t i0 = blockIdx.y * chunk, i1 = i0 + chunk < N ? i0 + chunk : N;
  for (int64_t it = i0; it < i1; it += kFfTile) {
    const int ni = static_cast<int>(i1 - it < kFfTile ? i1 - it : kFfTile);
    __syncthreads();
    for (int q = tid; q < kFfTile * kFfDirs; q += kFfThreads) {
      const int j = q / kFfDirs, d = q % kFfDirs;
      double s = 0.0, c = 0.0;
      if (j < ni) {
        const Pos4 r = pos[it + j];
        sincos_phase(-fma(kv[d][2], r.z, fma(kv[d][0], r.x, kv[d][1] * r.y)), &s, &c);
      }
      pc[j][d] = c;
      ps[j][d] = s;
      pt[j][d] = c + s;
    }
    for (int q = tid; q < kFfTile * 16 * NPT; q += kFfThreads) {
      const int j = q / (16 * NPT), n = q % (16 * NPT);
      const double2 v = j < ni && n < nmax ? b[(it + j) * nmax + n] : make_double2(0.0, 0.0);
      br[j][n] = v.x;
      bi[j][n] = v.y;
      bt[j][n] = v.x + v.y;
    }
    __syncthreads();
#pragma unroll(NC > 1 ? kFfTile : 2)
    for (int j = 0; j < kFfTile; ++j) {
      const int q = j % NC;
#pragma unroll
      for (int u = 0; u < NPT; ++u) {
        const double vr = br[j][tx + 16 * u], vi = bi[j][tx + 16 * u], vt = bt[j][tx + 16 * u];
#pragma unroll
        for (int a = 0; a < DT; ++a) {
          p1[q][a][u] = fma(pc[j][DT * ty + a], vr, p1[q][a][u]);
          p2[q][a][u] = fma(ps[j][DT * ty + a], vi, p2[q][a][u]);
          p3[q][a][u] = fma(pt[j][DT * ty + a], vt, p3[q][a][u]);
        }
      }
    }
    if (DT > 1 && (it + kFfTile - i0) % kRun == 0 && it + kFfTile < i1) store();
  }
  store();
}

// constants of the recursions of pi_l^m (pi_tau_m in cmath.cuh), for one m per thread
struct PiTable {
  double d[kFfMaxL + 1], a[kFfMaxL + 1][kFfMaxL + 1], ab[kFfMaxL + 1][kFfMaxL + 1], f[kFfMaxL + 1][kFfMaxL + 1];
  double norm[kFfMaxL + 1], tau0[kFfMaxL + 1];
};
constexpr PiTable make_pi_table() {
  PiTable t{};
  for (int m = 0; m <= kFfMaxL; ++m) {
    const int mm = m == 0 ? 1 : m;  // tau_l^0 comes from pi_l^1
    t.d[m] = 0.70710678118654752440;
    for (int q = 1; q <= mm; ++q) t.d[m] *= tab::csqrt((2.0 * q + 1.0) / (2.0 * q));
    for (int l = mm; l <= kFfMaxL; ++l) {
      if (l == mm + 1) t.a[m][l] = tab::csqrt(2.0 * mm + 3.0);
      if (l > mm + 1) {
        t.a[m][l] = tab::csqrt((4.0 * l * l - 1.0) / (1.0 * l * l - 1.0 * mm * mm));
        t.ab[m][l] = t.a[m][l] * tab::csqrt(((l - 1.0) * (l - 1.0) - 1.0 * mm * mm) / (4.0 * (l - 1.0) * (l - 1.0) - 1.0));
      }
      t.f[m][l] = tab::csqrt((2.0 * l + 1.0) * (1.0 * l * l - 1.0 * m * m) / (2.0 * l - 1.0));
    }
  }
  for (int l = 1; l <= kFfMaxL; ++l) {
    t.norm[l] = 1.0 / tab::csqrt(2.0 * l * (l + 1.0));
    t.tau0[l] = -tab::csqrt(l * (l + 1.0));
  }
  return t;
}
__constant__ PiTable kPiTable = make_pi_table();

// eight lanes per direction, lane |m|: the chunks of F added in order, then the
// contraction with B_nj e^{i m alpha} of both orders +-m
__global__ void __launch_bounds__(128)
    farfield_contract_kernel(int64_t Nd, int chunks, int L, const double* __restrict__ dirs,
                             const double2* __restrict__ F, double* __restrict__ g) {
  const int NH = L * (L + 2), nmax = 2 * NH;
  const int am = threadIdx.x & 7;
  const int64_t d = blockIdx.x * (int64_t)(blockDim.x >> 3) + (threadIdx.x >> 3);
  cd g1 = mkc(0.0), g2 = mkc(0.0);
  if (d < Nd && am <= L) {
    double sb, cb;
    sincos_phase(dirs[2 * d], &sb, &cb);
    cd em;
    sincos_phase(am * dirs[2 * d + 1], &em.im, &em.re);
    const int l0 = am == 0 ? 1 : am;
    double pl = kPiTable.d[am], prev = 0.0;
    for (int q = 1; q < l0; ++q) pl *= sb;
    for (int l = l0; l <= L; ++l) {
      if (l > l0) {
        const double nx = kPiTable.a[am][l] * cb * pl - kPiTable.ab[am][l] * prev;
        prev = pl;
        pl = nx;
      }
      const double tau = am == 0 ? kPiTable.tau0[l] * sb * pl : l * cb * pl - kPiTable.f[am][l] * prev;
      const double mp = am * pl;
      // sums over the chunks of the rows (tau 1, 2) of +m and -m
      cd f[4] = {};
      const int r = l * (l + 1) - 1;
      for (int c0 = 0; c0 < chunks; c0 += 16) {
        cd h[4] = {};
        const int c1 = chunks < c0 + 16 ? chunks : c0 + 16;
        for (int c = c0; c < c1; ++c) {
          const double2* Fc = F + ((int64_t)c * Nd + d) * nmax;
          const double2 v0 = Fc[r + am], v1 = Fc[NH + r + am];
          h[0] = h[0] + cd{v0.x, v0.y};
          h[1] = h[1] + cd{v1.x, v1.y};
          if (am > 0) {
            const double2 w0 = Fc[r - am], w1 = Fc[NH + r - am];
            h[2] = h[2] + cd{w0.x, w0.y};
            h[3] = h[3] + cd{w1.x, w1.y};
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) f[q] = f[q] + h[q];
      }
      // B_n1 = -(1/i^{l+1}) norm i ang, B_n2 = -(1/i^{l+1}) norm ang; ang = tau for j = tau index, else m pi
      const cd a = em * f[0], b = em * f[1], c = conj(em) * f[2], e = conj(em) * f[3];
      const cd pre = (-kPiTable.norm[l]) * ipow(-(l + 1));
      g1 = g1 + pre * (cd{0, 1} * (tau * (a + c) + mp * (b - e)));
      g2 = g2 + pre * (mp * (a - c) + tau * (b + e));
    }
  }
  double v[4] = {g1.re, g1.im, g2.re, g2.im};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    for (int o = 4; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o, 8);
    if (d < Nd && am == 0) g[4 * d + q] = v[q] / (2.0 * 3.14159265358979323846);
  }
}

// Directions of a tile and of one pass, and sphere chunks.  64 directions a CTA
// and chunks for four CTAs per SM, within 64 MB of scratch; a problem too small
// for that takes tiles of 16 and at most 0.9 MB (a device allocation above 1 MB
// costs a first call as much as the evaluation: 114 spheres, 399 directions).
struct FarfieldShape {
  int64_t tile, nd, chunks;
};
static FarfieldShape farfield_shape(int64_t N, int L, int64_t Nd) {
  const int64_t row = 16LL * 2 * L * (L + 2), most = (N + kFfTile - 1) / kFfTile;
  const bool small = (Nd + 63) / 64 * most < 4LL * device_sms();
  const int64_t cap = small ? 900000 : int64_t(64) << 20;
  FarfieldShape f;
  f.tile = small ? 16 : 64;
  f.nd = std::min(Nd, std::max<int64_t>(f.tile, (int64_t(64) << 20) / row / f.tile * f.tile));
  const int64_t tiles = (f.nd + f.tile - 1) / f.tile;
  const int64_t ch = std::min<int64_t>((4LL * device_sms() + tiles - 1) / tiles, most);
  f.chunks = std::max<int64_t>(1, std::min(ch, cap / (row * f.nd)));
  return f;
}
size_t farfield_scratch_bytes(int64_t N, int L, int64_t Nd) {
  const FarfieldShape f = farfield_shape(N, L, Nd);
  return static_cast<size_t>(f.nd * f.chunks) * 16 * 2 * L * (L + 2);
}

template <int DT>
static void launch_farfield_sum(int64_t N, int nmax, double k, const Pos4* p, const double2* b, int64_t n, int64_t ch,
                                const double* dirs, double2* F, cudaStream_t st) {
  const dim3 grid(static_cast<unsigned>((n + 16 * DT - 1) / (16 * DT)), static_cast<unsigned>(ch));
  const int64_t chunk = (N + ch - 1) / ch;
  switch ((nmax + 15) / 16) {
    case 1: farfield_sum_kernel<1, DT><<<grid, kFfThreads, 0, st>>>(N, chunk, nmax, k, p, b, n, dirs, F); break;
    case 2: farfield_sum_kernel<2, DT><<<grid, kFfThreads, 0, st>>>(N, chunk, nmax, k, p, b, n, dirs, F); break;
    case 3: farfield_sum_kernel<3, DT><<<grid, kFfThreads, 0, st>>>(N, chunk, nmax, k, p, b, n, dirs, F); break;
    default: farfield_sum_kernel<5, DT><<<grid, kFfThreads, 0, st>>>(N, chunk, nmax, k, p, b, n, dirs, F); break;
  }
}

cudaError_t launch_farfield(int64_t N, int L, double k, const void* pos, const double* b, int64_t Nd,
                            const double* dirs, double* g, void* scratch, cudaStream_t st) {
  const int nmax = 2 * L * (L + 2);
  const FarfieldShape f = farfield_shape(N, L, Nd);
  double2* F = static_cast<double2*>(scratch);
  const auto* p = static_cast<const Pos4*>(pos);
  const auto* bv = reinterpret_cast<const double2*>(b);
  for (int64_t d0 = 0; d0 < Nd; d0 += f.nd) {
    const int64_t n = std::min(f.nd, Nd - d0);
    if (f.tile == 16) launch_farfield_sum<1>(N, nmax, k, p, bv, n, f.chunks, dirs + 2 * d0, F, st);
    else launch_farfield_sum<4>(N, nmax, k, p, bv, n, f.chunks, dirs + 2 * d0, F, st);
    farfield_contract_kernel<<<static_cast<unsigned>((n + 15) / 16), 128, 0, st>>>(n, static_cast<int>(f.chunks), L,
                                                                                   dirs + 2 * d0, F, g + 4 * d0);
    note_launch(2);
  }
  return cudaGetLastError();
}

// overlap check: flag[0] = 1 if some pair overlaps (|r_i - r_j| < R_i + R_j).
// Every pair in FP32 relative to the first sphere, widened by a bound on the
// rounding of both coordinates; only pairs that this cannot clear (neighbours,
// lengths whose squares leave FP32's range) are tested in FP64.  Grid (row tiles,
// column tiles), upper triangle; one thread per row against a staged tile.
// (10 000 spheres: 4.7 ms with one FP64 thread per sphere over all later ones,
// 0.03 ms so.)
constexpr int kOvTile = 256;
// squares below this lose digits to FP32's least exponent (the test in FP64 takes those pairs)
constexpr float kOvTiny = 1e-32f;

__global__ void __launch_bounds__(kOvTile)
    overlap_kernel(int64_t N, int64_t y0, const Pos4* __restrict__ pos, const double* __restrict__ radii,
                   int* __restrict__ flag) {
  const int64_t jt = y0 + blockIdx.y;  // column tile
  if (jt < blockIdx.x) return;
  __shared__ float4 sp[kOvTile];
  __shared__ float se[kOvTile];
  const Pos4 o = pos[0];
  auto load = [&](int64_t i, float4& p, float& e) {
    const Pos4 r = pos[i];
    p = make_float4(static_cast<float>(r.x - o.x), static_cast<float>(r.y - o.y), static_cast<float>(r.z - o.z),
                    static_cast<float>(radii[i]));
    // 2^-21 of the largest coordinate and of the radius: over four times the rounding of a
    // coordinate, of the sum of radii and of the distance formed from them
    e = 4.8e-7f * (fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fabsf(p.z)) + p.w);
  };
  const int64_t i = blockIdx.x * (int64_t)kOvTile + threadIdx.x, j0 = jt * kOvTile;
  const int nj = static_cast<int>(N - j0 < kOvTile ? N - j0 : kOvTile);
  load(j0 + threadIdx.x < N ? j0 + threadIdx.x : N - 1, sp[threadIdx.x], se[threadIdx.x]);
  __syncthreads();
  if (i >= N) return;
  float4 p;
  float e;
  load(i, p, e);
  bool hit = false;
  for (int jb = 0; jb < nj; jb += 32) {
    // candidates of 32 columns as a mask first: with the FP64 test inside this
    // loop the compiler predicates it, and it takes the FP64 pipe for every pair
    unsigned near = 0;
#pragma unroll 8
    for (int u = 0; u < 32; ++u) {
      const float4 q = sp[jb + u];
      const float dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
      const float s = (p.w + q.w) + 2.0f * (e + se[jb + u]);
      near |= (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) > fmaf(s, s, kOvTiny) ? 0u : 1u) << u;
    }
    if (nj - jb < 32) near &= (1u << (nj - jb)) - 1u;
    while (near) {
      const int64_t j = j0 + jb + __ffs(near) - 1;
      near &= near - 1;
      if (j <= i) continue;
      const Pos4 a = pos[i], b = pos[j];
      const double ax = a.x - b.x, ay = a.y - b.y, az = a.z - b.z;
      const double t = radii[i] + radii[j];
      if (ax * ax + ay * ay + az * az < t * t) hit = true;
    }
  }
  if (hit) *flag = 1;
}

cudaError_t launch_overlap_check(int64_t N, const void* pos, const double* radii, int* flag, cudaStream_t st) {
  const int64_t tiles = (N + kOvTile - 1) / kOvTile;
  // the grid's second extent ends at 65 535 tiles (16.7 million spheres): bands of columns
  for (int64_t y0 = 0; y0 < tiles; y0 += 65535) {
    const int64_t ny = tiles - y0 < 65535 ? tiles - y0 : 65535;
    overlap_kernel<<<dim3(static_cast<unsigned>(tiles), static_cast<unsigned>(ny)), kOvTile, 0, st>>>(
        N, y0, static_cast<const Pos4*>(pos), radii, flag);
    note_launch();
  }
  return cudaGetLastError();
}

}  // namespace celes
