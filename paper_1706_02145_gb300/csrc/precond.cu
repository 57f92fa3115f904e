// Block-diagonal preconditioner (Sec. 3.2.1): assembly of the diagonal blocks
// M_j of M = I - T W, batched LU factorisation with partial pivoting
// (P_j M_j = L_j U_j) and the block solve x = M_j^{-1} y, all in FP64.
//
// Storage: block j holds n_j = N_j nmax unknowns (its spheres in partition
// order); its matrix is column-major at mats + mat_off[j] (complex128), LU
// factors overwrite it in place (unit lower L below the diagonal, U on and
// above), piv holds the LAPACK-style row interchanges (row k swapped with
// piv[k] at step k).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <numeric>
#include <type_traits>
#include <vector>

#include "cmath.cuh"
#include "coupling_kernel.cuh"
#include "kernels.h"

namespace celes {

// ---------------------------------------------------------------------------
// batched LU with partial pivoting, blocked by 32 columns
//
// FP64 arithmetic bounds the build: 8/3 n^3 flops for the factors of a block
// and as many for their inverses, on a pipe that does 1.7 FMAs per clock and
// SM.  Blocks differ in size by an order of magnitude, so one CTA per block
// leaves the GPU to the largest one.  All blocks go through the same panel
// step together instead: (1) the panel's 32 columns, one row per thread in
// registers, a cluster of up to 8 CTAs per block; (2) the row interchanges and
// U_12, one CTA per 32 columns; (3) the trailing update, one CTA per 32 x 32
// tile of any block, which is nearly all of the work and spreads over the whole
// GPU.  Tiles of 32 move 0.25 bytes per flop, far below what this FP64 rate
// asks of L2.  Measured on GB300, 175 blocks of up to 1 248 unknowns (77
// GFLOP): the whole build 1 090-1 260 ms with one unblocked CTA per block (859
// ms of it the factors), 133 ms now (about 65 ms of it the factors: the FP64
// pipe at its 1.05 TFLOP/s during the update).
// ---------------------------------------------------------------------------
namespace cg = cooperative_groups;

constexpr int kTile = 32;
constexpr int kPanelMaxCluster = 8;
constexpr int kTileThreads = 256;

// tile `t` of a step, of the block that holds it: blocks are listed in `order`
// and `off[s]` counts the tiles of the blocks before order[s]
__device__ __forceinline__ int tile_block(const int64_t* __restrict__ off, int nact, int64_t t) {
  int lo = 0, hi = nact - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// (1) panel of columns kb .. kb + 31 of the blocks order[0 .. grid / C - 1];
// grid: clusters of C CTAs, one per block; the panel has at most C * THREADS
// rows.  The owner of a candidate row also inverts its pivot, so that the rows
// below are scaled by a product (every row dividing for itself took as long as
// the rest of the column's work).
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
    precond_panel_kernel(int64_t kb, const int* __restrict__ order, const int64_t* __restrict__ block_off,
                         const int64_t* __restrict__ mat_off, int nmax, double2* __restrict__ mats,
                         int* __restrict__ piv, int* __restrict__ info) {
  cg::cluster_group cluster = cg::this_cluster();
  const int C = static_cast<int>(cluster.num_blocks());
  const int rank = static_cast<int>(cluster.block_rank());
  const int q = order[blockIdx.x / C];
  const int64_t n = (block_off[q + 1] - block_off[q]) * nmax;
  double2* A = mats + mat_off[q];
  int* pv = piv + block_off[q] * nmax;
  __shared__ double wval[THREADS / 32];
  __shared__ int widx[THREADS / 32];
  // candidates of every CTA and the row at the pivot position, double buffered
  __shared__ double cval[2][kPanelMaxCluster];
  __shared__ int cidx[2][kPanelMaxCluster];
  __shared__ double2 crow[2][kPanelMaxCluster][kTile];
  __shared__ double2 cinv[2][kPanelMaxCluster];
  __shared__ double2 krow[2][kTile];
  const int tid = threadIdx.x;
  const int tb = static_cast<int>(n - kb < kTile ? n - kb : kTile);
  const int i = static_cast<int>(kb) + rank * THREADS + tid;  // this thread's row
  const bool live = i < n;
  double2 a[kTile];
#pragma unroll
  for (int t = 0; t < kTile; ++t) a[t] = live && t < tb ? A[i + (kb + t) * n] : make_double2(0.0, 0.0);
  if (kb == 0 && rank == 0 && tid == 0) info[q] = 0;
  if (C > 1) cluster.sync();  // every CTA has started before any writes into another's shared memory
#pragma unroll
  for (int c = 0; c < kTile; ++c) {
    if (c < tb) {
      const int kk = static_cast<int>(kb) + c, par = c & 1;
      double best = live && i >= kk ? fabs(a[c].x) + fabs(a[c].y) : -1.0;
      if (!(best >= 0.0)) best = -1.0;  // NaN never wins
      int bi = i;
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) {
          best = ob;
          bi = oi;
        }
      }
      if ((tid & 31) == 0) {
        wval[tid >> 5] = best;
        widx[tid >> 5] = bi;
      }
      __syncthreads();
      best = wval[0];
      bi = widx[0];
#pragma unroll
      for (int w = 1; w < THREADS / 32; ++w) {
        if (wval[w] > best) {  // rows ascend with w: ties keep the first
          best = wval[w];
          bi = widx[w];
        }
      }
      if (i == bi || i == kk) {
        const cd pv_c = mkc(a[c].x, a[c].y);
        const cd rp = i == bi && abs2(pv_c) > 0.0 ? mkc(1.0) / pv_c : mkc(0.0);
        for (int dst = 0; dst < C; ++dst) {
          double2* cr = C > 1 ? cluster.map_shared_rank(&crow[par][rank][0], dst) : &crow[par][rank][0];
          double2* kr = C > 1 ? cluster.map_shared_rank(&krow[par][0], dst) : &krow[par][0];
          if (i == bi) {
            double* cv = C > 1 ? cluster.map_shared_rank(&cval[par][rank], dst) : &cval[par][rank];
            int* ci = C > 1 ? cluster.map_shared_rank(&cidx[par][rank], dst) : &cidx[par][rank];
            double2* cp = C > 1 ? cluster.map_shared_rank(&cinv[par][rank], dst) : &cinv[par][rank];
            *cv = best;
            *ci = bi;
            *cp = make_double2(rp.re, rp.im);
#pragma unroll
            for (int t = 0; t < kTile; ++t) cr[t] = a[t];
          }
          if (i == kk) {
#pragma unroll
            for (int t = 0; t < kTile; ++t) kr[t] = a[t];
          }
        }
      }
      if (C > 1) cluster.sync();
      else __syncthreads();
      int b = 0;
      for (int r = 1; r < C; ++r)
        if (cval[par][r] > cval[par][b]) b = r;
      const bool none = !(cval[par][b] > 0.0);
      const int p = cval[par][b] < 0.0 ? kk : cidx[par][b];
      const double2* prow = cval[par][b] < 0.0 ? krow[par] : crow[par][b];
      if (rank == 0 && tid == 0) {
        pv[kk] = p;
        if (none && info[q] == 0) info[q] = kk + 1;
      }
      if (p != kk) {
        if (i == kk) {
#pragma unroll
          for (int t = 0; t < kTile; ++t) a[t] = prow[t];
        } else if (i == p) {
#pragma unroll
          for (int t = 0; t < kTile; ++t) a[t] = krow[par][t];
        }
      }
      if (live && i > kk) {
        const double2 rp = cval[par][b] < 0.0 ? make_double2(0.0, 0.0) : cinv[par][b];
        const cd l = mkc(a[c].x, a[c].y) * mkc(rp.x, rp.y);
        a[c] = make_double2(l.re, l.im);
#pragma unroll
        for (int t = c + 1; t < kTile; ++t) {
          const double2 u = prow[t];
          a[t].x = fma(-l.re, u.x, fma(l.im, u.y, a[t].x));
          a[t].y = fma(-l.re, u.y, fma(-l.im, u.x, a[t].y));
        }
      }
    }
  }
  if (live) {
#pragma unroll
    for (int t = 0; t < kTile; ++t)
      if (t < tb) A[i + (kb + t) * n] = a[t];
  }
  if (C > 1) cluster.sync();  // no CTA leaves while others may still read what it wrote into them
}

// (1), panels of more rows than a cluster holds: one CTA per block, in global memory
__global__ void __launch_bounds__(1024) precond_panel_tall_kernel(int64_t kb, const int* __restrict__ order,
                                                                  const int64_t* __restrict__ block_off,
                                                                  const int64_t* __restrict__ mat_off, int nmax,
                                                                  double2* __restrict__ mats, int* __restrict__ piv,
                                                                  int* __restrict__ info) {
  const int q = order[blockIdx.x];
  const int64_t n = (block_off[q + 1] - block_off[q]) * nmax;
  double2* A = mats + mat_off[q];
  int* pv = piv + block_off[q] * nmax;
  __shared__ double sval[32];
  __shared__ int sidx[32];
  __shared__ int s_p;
  __shared__ double2 s_row[kTile];
  const int tb = static_cast<int>(n - kb < kTile ? n - kb : kTile);
  if (kb == 0 && threadIdx.x == 0) info[q] = 0;
  for (int c = 0; c < tb; ++c) {
    const int64_t kk = kb + c;
    double best = -1.0;
    int bi = static_cast<int>(kk);
    for (int64_t i = kk + threadIdx.x; i < n; i += blockDim.x) {
      const double2 v = A[i + kk * n];
      const double x = fabs(v.x) + fabs(v.y);
      if (x > best) {
        best = x;
        bi = static_cast<int>(i);
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_down_sync(0xffffffffu, best, o);
      const int oi = __shfl_down_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
    if ((threadIdx.x & 31) == 0) {
      sval[threadIdx.x >> 5] = best;
      sidx[threadIdx.x >> 5] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double b = -1.0;
      int ix = static_cast<int>(kk);
      for (int w = 0; w < static_cast<int>(blockDim.x) / 32; ++w) {
        if (sval[w] > b || (sval[w] == b && sidx[w] < ix)) {
          b = sval[w];
          ix = sidx[w];
        }
      }
      s_p = ix;
      pv[kk] = ix;
      if (b <= 0.0 && info[q] == 0) info[q] = static_cast<int>(kk) + 1;
    }
    __syncthreads();
    const int64_t p = s_p;
    if (threadIdx.x < tb) {
      const int64_t col = (kb + threadIdx.x) * n;
      const double2 u = A[p + col];
      s_row[threadIdx.x] = u;
      if (p != kk) {
        A[p + col] = A[kk + col];
        A[kk + col] = u;
      }
    }
    __syncthreads();
    const cd pvt = mkc(s_row[c].x, s_row[c].y);
    const bool ok = abs2(pvt) > 0.0;
    for (int64_t i = kk + 1 + threadIdx.x; i < n; i += blockDim.x) {
      const double2 v = A[i + kk * n];
      const cd l = ok ? mkc(v.x, v.y) / pvt : mkc(0.0);
      A[i + kk * n] = make_double2(l.re, l.im);
      for (int t = c + 1; t < tb; ++t) {
        double2 x = A[i + (kb + t) * n];
        const double2 u = s_row[t];
        x.x = fma(-l.re, u.x, fma(l.im, u.y, x.x));
        x.y = fma(-l.re, u.y, fma(-l.im, u.x, x.y));
        A[i + (kb + t) * n] = x;
      }
    }
    __syncthreads();
  }
}

// (2) the panel's row interchanges on 32 other columns of a block, and, right
// of the panel, U_12 = L_11^{-1} A_12 by forward substitution.  One CTA per
// column tile; lanes are columns, warps take the rows in turn.
__global__ void __launch_bounds__(kTileThreads)
    precond_swap_solve_kernel(int64_t kb, int nact, const int* __restrict__ order, const int64_t* __restrict__ off,
                              const int64_t* __restrict__ block_off, const int64_t* __restrict__ mat_off, int nmax,
                              double2* __restrict__ mats, const int* __restrict__ piv) {
  const int s = tile_block(off, nact, blockIdx.x);
  const int q = order[s];
  const int64_t n = (block_off[q + 1] - block_off[q]) * nmax;
  double2* A = mats + mat_off[q];
  int64_t ct = blockIdx.x - off[s];
  if (ct >= kb / kTile) ++ct;  // every column tile but the panel's own
  const int tb = static_cast<int>(n - kb < kTile ? n - kb : kTile);
  const int cb = static_cast<int>(n - ct * kTile < kTile ? n - ct * kTile : kTile);
  __shared__ double2 top[kTile][kTile + 1];  // [row][column] of rows kb ..
  __shared__ double2 far[kTile][kTile + 1];  // rows below the panel's top tile that a swap touches; then L_11
  __shared__ int prow[kTile], slot[kTile];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (wid == 0) {
    const int p = lane < tb ? piv[block_off[q] * nmax + kb + lane] : static_cast<int>(kb) + lane;
    prow[lane] = p;
    slot[lane] = __ffs(__match_any_sync(0xffffffffu, p)) - 1;  // the first interchange with the same row
  }
  __syncthreads();
  // rows along the lanes: coalesced
  for (int e = tid; e < kTile * kTile; e += kTileThreads) {
    const int c = e >> 5, r = e & 31;
    const double2* col = A + (ct * kTile + c) * n;
    if (c < cb && r < tb) {
      top[r][c] = col[kb + r];
      if (slot[r] == r && prow[r] >= kb + tb) far[r][c] = col[prow[r]];
    }
  }
  __syncthreads();
  if (wid == 0 && lane < cb) {
    for (int k = 0; k < tb; ++k) {
      const int p = prow[k];
      if (p == kb + k) continue;
      double2& x = p < kb + tb ? top[p - kb][lane] : far[slot[k]][lane];
      const double2 t = top[k][lane];
      top[k][lane] = x;
      x = t;
    }
  }
  __syncthreads();
  for (int e = tid; e < kTile * kTile; e += kTileThreads) {
    const int c = e >> 5, r = e & 31;
    if (c < cb && r < tb && slot[r] == r && prow[r] >= kb + tb) A[prow[r] + (ct * kTile + c) * n] = far[r][c];
  }
  if (ct * kTile > kb) {
    __syncthreads();
    for (int e = tid; e < kTile * kTile; e += kTileThreads) {
      const int c = e >> 5, r = e & 31;
      if (r < tb && c < tb) far[r][c] = A[(kb + r) + (kb + c) * n];
    }
    __syncthreads();
    for (int j = 0; j < tb; ++j) {
      const double2 u = top[j][lane];
      for (int r = wid; r < tb; r += kTileThreads / 32) {
        if (r > j) {
          const double2 l = far[r][j];
          double2 x = top[r][lane];
          x.x = fma(-l.x, u.x, fma(l.y, u.y, x.x));
          x.y = fma(-l.x, u.y, fma(-l.y, u.x, x.y));
          top[r][lane] = x;
        }
      }
      __syncthreads();
    }
  }
  for (int e = tid; e < kTile * kTile; e += kTileThreads) {
    const int c = e >> 5, r = e & 31;
    if (c < cb && r < tb) A[kb + r + (ct * kTile + c) * n] = top[r][c];
  }
}

// A complex 32 x 32 tile as three real ones, [col][row]: real and imaginary
// part and their sum.  Products take three real multiplications instead of
// four (Re = P1 - P2, Im = P3 - P1 - P2 with P1 = ar br, P2 = ai bi, P3 =
// (ar + ai)(br + bi)): the FP64 pipe is all that these kernels wait for (the
// two updates 119 -> 98 ms at the size above; the application's error against
// 64 bits 1.6e-15 -> 1.5e-15; the FP64 mma runs no faster than the FMA here,
// 1.04 against 1.00 TFLOP/s).
struct Tile3 {
  double re[kTile][kTile + 1], im[kTile][kTile + 1], sum[kTile][kTile + 1];
  __device__ __forceinline__ void set(int c, int r, double2 v) {
    re[c][r] = v.x;
    im[c][r] = v.y;
    sum[c][r] = v.x + v.y;
  }
};
// stage tile (ti, tk) of a column-major n x n matrix, zero outside the block
__device__ __forceinline__ void load_tile(Tile3& dst, const double2* __restrict__ M, int64_t n, int64_t ti,
                                          int64_t tk) {
  const int64_t r0 = ti * kTile, c0 = tk * kTile;
  for (int e = threadIdx.x; e < kTile * kTile; e += kTileThreads) {
    const int c = e >> 5, r = e & 31;
    dst.set(c, r, r0 + r < n && c0 + c < n ? M[(r0 + r) + (c0 + c) * n] : make_double2(0.0, 0.0));
  }
}
// the inverse of a diagonal tile (32 x 32 column-major, identity-padded)
__device__ __forceinline__ void load_tinv(Tile3& dst, const double2* __restrict__ Ti) {
  for (int e = threadIdx.x; e < kTile * kTile; e += kTileThreads) dst.set(e >> 5, e & 31, Ti[e]);
}
// acc[u] += S (as xs)[r][4 g + u], thread (r, g) = (tid & 31, tid >> 5)
template <int S>
__device__ __forceinline__ void tile_product(const Tile3& as, const Tile3& xs, double2 (&acc)[4]) {
  const int r = threadIdx.x & 31, g = threadIdx.x >> 5;
  double p1[4] = {}, p2[4] = {}, p3[4] = {};
#pragma unroll 8
  for (int m = 0; m < kTile; ++m) {
    const double ar = as.re[m][r], ai = as.im[m][r], at = as.sum[m][r];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      p1[u] = fma(ar, xs.re[4 * g + u][m], p1[u]);
      p2[u] = fma(ai, xs.im[4 * g + u][m], p2[u]);
      p3[u] = fma(at, xs.sum[4 * g + u][m], p3[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const double re = p1[u] - p2[u], im = p3[u] - p1[u] - p2[u];
    acc[u].x = S > 0 ? acc[u].x + re : acc[u].x - re;
    acc[u].y = S > 0 ? acc[u].y + im : acc[u].y - im;
  }
}

// (3) A_22 -= L_21 U_12, one CTA per 32 x 32 tile
__global__ void __launch_bounds__(kTileThreads)
    precond_update_kernel(int64_t kt, int nact, const int* __restrict__ order, const int64_t* __restrict__ off,
                          const int64_t* __restrict__ block_off, const int64_t* __restrict__ mat_off, int nmax,
                          double2* __restrict__ mats) {
  const int s = tile_block(off, nact, blockIdx.x);
  const int q = order[s];
  const int64_t n = (block_off[q + 1] - block_off[q]) * nmax;
  const int64_t rem = (n + kTile - 1) / kTile - kt - 1;
  const int64_t t = blockIdx.x - off[s];
  const int64_t ti = kt + 1 + t % rem, tj = kt + 1 + t / rem;
  double2* A = mats + mat_off[q];
  extern __shared__ Tile3 tiles3[];
  Tile3& as = tiles3[0];
  Tile3& xs = tiles3[1];
  load_tile(as, A, n, ti, kt);
  load_tile(xs, A, n, kt, tj);
  const int r = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t row = ti * kTile + r, col = tj * kTile + 4 * g;
  double2 acc[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    acc[u] = row < n && col + u < n ? A[row + (col + u) * n] : make_double2(0.0, 0.0);
  __syncthreads();
  tile_product<-1>(as, xs, acc);
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (row < n && col + u < n) A[row + (col + u) * n] = acc[u];
}

// the two staged tiles are above the default limit of 48 KB
template <typename K>
static cudaError_t tile_smem(K* kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(2 * sizeof(Tile3)));
}

// The blocks of one panel step by the rows they have left, each class with the
// smallest cluster that holds them: a launch has one cluster size, and eight
// CTAs for the small blocks too would be nine waves of mostly idle rows.  The
// classes run side by side on streams of their own (with the reciprocal pivots
// and the three-product tiles, this took the build of the 175 blocks above from
// 173 to 133 ms).
struct PanelClass {
  int64_t rows;
  int threads, cluster;
};
constexpr PanelClass kPanelClasses[] = {{128, 128, 1}, {256, 128, 2}, {512, 128, 4}, {1024, 128, 8}, {2048, 256, 8}};
constexpr int kPanelStreams = 5;

// side streams and events of one build, given back at its end
struct PanelStreams {
  cudaStream_t side[kPanelStreams] = {};
  cudaEvent_t fork = nullptr, join[kPanelStreams] = {};
  cudaError_t init() {
    cudaError_t e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
    for (int q = 0; q < kPanelStreams && e == cudaSuccess; ++q) {
      e = cudaStreamCreateWithFlags(&side[q], cudaStreamNonBlocking);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join[q], cudaEventDisableTiming);
    }
    return e;
  }
  ~PanelStreams() {
    if (fork) cudaEventDestroy(fork);
    for (int q = 0; q < kPanelStreams; ++q) {
      if (side[q]) cudaStreamDestroy(side[q]);  // its work is done first
      if (join[q]) cudaEventDestroy(join[q]);
    }
  }
};

template <int THREADS>
static cudaError_t launch_panel(int64_t kb, int nblk, int C, const int* order, const int64_t* block_off,
                                const int64_t* mat_off, int nmax, double2* M, int* piv, int* info, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(nblk * C));
  cfg.blockDim = dim3(THREADS);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = static_cast<unsigned>(C);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, precond_panel_kernel<THREADS>, kb, order, block_off, mat_off, nmax, M, piv, info);
}

cudaError_t launch_precond_lu(const PrecondPlan& plan, const int64_t* block_off, const int64_t* mat_off, int nmax,
                              double* mats, int* piv, int* info, cudaStream_t st) {
  double2* M = reinterpret_cast<double2*>(mats);
  PanelStreams ps;
  cudaError_t e = tile_smem(precond_update_kernel);
  if (e == cudaSuccess) e = ps.init();
  for (size_t k = 0; k < plan.steps.size() && e == cudaSuccess; ++k) {
    const PrecondPlan::Step& p = plan.steps[k];
    const int64_t kb = static_cast<int64_t>(k) * kTile;
    e = cudaEventRecord(ps.fork, st);
    // blocks are in descending order of size: each class is a run of them
    int side = 0;
    for (int s = 0; s < p.active && e == cudaSuccess;) {
      const int64_t rows = plan.dims[s] - kb;
      const PanelClass* pc = nullptr;
      for (const PanelClass& c : kPanelClasses)
        if (!pc && rows <= c.rows) pc = &c;
      int end = s + 1;
      const int64_t least = !pc ? kPanelClasses[4].rows : (pc == kPanelClasses ? 0 : pc[-1].rows);
      while (end < p.active && plan.dims[end] - kb > least) ++end;
      // the last class stays on the main stream
      const bool fork = end < p.active;
      const cudaStream_t to = fork ? ps.side[side] : st;
      if (fork) e = cudaStreamWaitEvent(to, ps.fork, 0);
      if (e != cudaSuccess) break;
      if (!pc) {
        precond_panel_tall_kernel<<<static_cast<unsigned>(end - s), 1024, 0, to>>>(kb, plan.order + s, block_off,
                                                                                   mat_off, nmax, M, piv, info);
        e = cudaGetLastError();
      } else if (pc->threads == 128) {
        e = launch_panel<128>(kb, end - s, pc->cluster, plan.order + s, block_off, mat_off, nmax, M, piv, info, to);
      } else {
        e = launch_panel<256>(kb, end - s, pc->cluster, plan.order + s, block_off, mat_off, nmax, M, piv, info, to);
      }
      note_launch();
      if (fork && e == cudaSuccess) e = cudaEventRecord(ps.join[side], to);
      if (fork) ++side;
      s = end;
    }
    for (int q = 0; q < side && e == cudaSuccess; ++q) e = cudaStreamWaitEvent(st, ps.join[q], 0);
    if (e != cudaSuccess) break;
    if (p.columns > 0) {
      precond_swap_solve_kernel<<<static_cast<unsigned>(p.columns), kTileThreads, 0, st>>>(
          kb, p.active, plan.order, plan.off + p.columns_off, block_off, mat_off, nmax, M, piv);
      note_launch();
    }
    if (p.tiles > 0) {
      precond_update_kernel<<<static_cast<unsigned>(p.tiles), kTileThreads, 2 * sizeof(Tile3), st>>>(
          static_cast<int64_t>(k), p.active, plan.order, plan.off + p.tiles_off, block_off, mat_off, nmax, M);
      note_launch();
    }
    e = cudaGetLastError();
  }
  return e;
}

// ---------------------------------------------------------------------------
// apply: one CTA per (block, rhs): gather, permute, forward and back
// substitution, scatter.  The block's vector lives in shared memory when it
// fits (one barrier per substitution step), else in the global work array.
// Factors in the precision F: FP64, or an FP32 copy for FP32 vectors (a
// preconditioner only has to be the same operator wherever it is applied).
// ---------------------------------------------------------------------------
template <typename F>
__device__ __forceinline__ Pair2<F> cmul_sub(Pair2<F> a, Pair2<F> l, Pair2<F> y) {
  return Pair2<F>{a.re - (l.re * y.re - l.im * y.im), a.im - (l.re * y.im + l.im * y.re)};
}

// acc - sum_{j < tb} A[i, kb + j] v[kb + j]; a full 32-column tile is
// unrolled so that a thread's 32 factor loads are all in flight at once
template <typename F>
__device__ __forceinline__ Pair2<F> tile_gemv(const Pair2<F>* __restrict__ A, int64_t n, int64_t i, int64_t kb,
                                              int tb, const Pair2<F>* v, Pair2<F> acc) {
  const Pair2<F>* col = A + i + kb * n;
  if (tb == 32) {
    Pair2<F> a[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) a[j] = col[j * n];
#pragma unroll
    for (int j = 0; j < 32; ++j) acc = cmul_sub(acc, a[j], v[kb + j]);
  } else {
    for (int j = 0; j < tb; ++j) acc = cmul_sub(acc, col[j * n], v[kb + j]);
  }
  return acc;
}

template <typename F>
__device__ __forceinline__ Pair2<F> shfl_pair(Pair2<F> v, int src) {
  return Pair2<F>{__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src)};
}

// Blocked substitution: warp 0 resolves each 32-row diagonal tile with
// shuffles (no block barrier inside a tile), then the whole CTA applies the
// tile's columns to the remaining rows (a GEMV over contiguous column
// segments).  Two barriers per 32 unknowns instead of one or two per unknown.
// The row permutation of partial pivoting is folded into the gather (pivperm:
// position i of the permuted vector holds original entry pivperm[i]).
template <typename R, typename F, bool SMEM>
__global__ void __launch_bounds__(256) precond_apply_kernel(const int64_t* __restrict__ block_off,
                                                            const int64_t* __restrict__ mat_off, int nmax,
                                                            const int* __restrict__ perm,
                                                            const Pair2<F>* __restrict__ mats,
                                                            const int* __restrict__ pivperm, int64_t N,
                                                            const Pair2<R>* __restrict__ x, Pair2<R>* __restrict__ y,
                                                            Pair2<F>* __restrict__ work) {
  extern __shared__ __align__(16) unsigned char pa_smem[];
  const int64_t q = blockIdx.x;
  const int rhs = blockIdx.y;
  const int64_t s0 = block_off[q];
  const int64_t ns = block_off[q + 1] - s0;
  const int64_t n = ns * nmax;
  const Pair2<F>* A = mats + mat_off[q];
  const int* pp = pivperm + s0 * nmax;
  Pair2<F>* v = SMEM ? reinterpret_cast<Pair2<F>*>(pa_smem) : work + (int64_t)rhs * N * nmax + s0 * nmax;
  const Pair2<R>* xr = x + (int64_t)rhs * N * nmax;
  Pair2<R>* yr = y + (int64_t)rhs * N * nmax;
  const int lane = threadIdx.x & 31;
  for (int64_t t = threadIdx.x; t < n; t += blockDim.x) {
    const int64_t src = pp[t];
    const int64_t a = src / nmax;
    const int r = static_cast<int>(src - a * nmax);
    const Pair2<R> e = xr[(int64_t)perm[s0 + a] * nmax + r];
    v[t] = Pair2<F>{static_cast<F>(e.re), static_cast<F>(e.im)};
  }
  __syncthreads();
  // the diagonal tile is staged in shared memory by the whole CTA (one
  // memory latency) before warp 0 walks its 32 dependent steps
  __shared__ Pair2<F> dt[32][33];
  auto stage = [&](int64_t kb, int tb) {
    for (int t = threadIdx.x; t < 32 * 32; t += blockDim.x) {
      const int j = t >> 5, i = t & 31;  // column j, row i: coalesced along i
      dt[j][i] = (i < tb && j < tb) ? A[(kb + i) + (kb + j) * n] : Pair2<F>{0, 0};
    }
  };
  // forward substitution with the unit lower factor
  for (int64_t kb = 0; kb < n; kb += 32) {
    const int tb = static_cast<int>(n - kb < 32 ? n - kb : 32);
    stage(kb, tb);
    __syncthreads();
    if (threadIdx.x < 32) {
      Pair2<F> yl = lane < tb ? v[kb + lane] : Pair2<F>{0, 0};
      for (int j = 0; j < tb; ++j) {
        const Pair2<F> yj = shfl_pair(yl, j);
        if (lane > j && lane < tb) yl = cmul_sub(yl, dt[j][lane], yj);
      }
      if (lane < tb) v[kb + lane] = yl;
    }
    __syncthreads();
    for (int64_t i = kb + tb + threadIdx.x; i < n; i += blockDim.x) v[i] = tile_gemv(A, n, i, kb, tb, v, v[i]);
    __syncthreads();
  }
  // back substitution with the upper factor (tiles from the bottom)
  const int64_t ntile = (n + 31) / 32;
  for (int64_t tt = ntile - 1; tt >= 0; --tt) {
    const int64_t kb = tt * 32;
    const int tb = static_cast<int>(n - kb < 32 ? n - kb : 32);
    stage(kb, tb);
    __syncthreads();
    if (threadIdx.x < 32) {
      Pair2<F> yl = lane < tb ? v[kb + lane] : Pair2<F>{0, 0};
      for (int j = tb - 1; j >= 0; --j) {
        if (lane == j) {
          const Pair2<F> u = dt[j][j];
          const F den = u.re * u.re + u.im * u.im;
          yl = Pair2<F>{(yl.re * u.re + yl.im * u.im) / den, (yl.im * u.re - yl.re * u.im) / den};
        }
        const Pair2<F> xj = shfl_pair(yl, j);
        if (lane < j) yl = cmul_sub(yl, dt[j][lane], xj);
      }
      if (lane < tb) v[kb + lane] = yl;
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < kb; i += blockDim.x) v[i] = tile_gemv(A, n, i, kb, tb, v, v[i]);
    __syncthreads();
  }
  for (int64_t t = threadIdx.x; t < n; t += blockDim.x) {
    const int64_t a = t / nmax;
    const int r = static_cast<int>(t - a * nmax);
    yr[(int64_t)perm[s0 + a] * nmax + r] = Pair2<R>{static_cast<R>(v[t].re), static_cast<R>(v[t].im)};
  }
}

// ---------------------------------------------------------------------------
// apply, cluster form: each block's triangular solves are spread over a
// thread-block cluster of C CTAs (distributed shared memory).  CTA s of the
// cluster owns a contiguous run of the block's 32-row tiles.  Per tile step
// the owner multiplies its (updated) tile by the explicit inverse of the
// 32 x 32 diagonal tile of L (forward) or U (backward), both formed at build
// time, and writes the 32 solved values into every CTA's copy of the block
// vector; after one cluster barrier every CTA applies that tile column to its
// own rows.  The serial chain of a block is then one barrier and one short
// GEMV per tile, the factor traffic is spread over C SMs, and blocks much
// fewer than SMs still fill the GPU.
// ---------------------------------------------------------------------------

// explicit inverses of the diagonal tiles of each block's LU (unit lower L,
// upper U), column-major 32 x 32 each, tiles beyond the block padded with the
// identity; one CTA of 64 threads per tile (32 columns of Linv, 32 of Uinv)
__global__ void __launch_bounds__(64) precond_tile_inverse_kernel(const int64_t* __restrict__ block_off,
                                                                  const int64_t* __restrict__ mat_off,
                                                                  const int64_t* __restrict__ tile_off, int nmax,
                                                                  const double2* __restrict__ mats,
                                                                  double2* __restrict__ tinv) {
  const int64_t q = blockIdx.y;
  const int64_t n = (block_off[q + 1] - block_off[q]) * nmax;
  const int64_t ntile = (n + 31) / 32;
  const int64_t k = blockIdx.x;
  if (k >= ntile) return;
  const int64_t kb = k * 32;
  const int tb = static_cast<int>(n - kb < 32 ? n - kb : 32);
  const double2* A = mats + mat_off[q];
  __shared__ double2 t[32][33];  // t[c][r] = A[kb + r, kb + c]
  for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
    const int c = e >> 5, r = e & 31;
    t[c][r] = (r < tb && c < tb) ? A[(kb + r) + (kb + c) * n] : make_double2(r == c ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  double2* Li = tinv + tile_off[q] + k * 2048;
  double2* Ui = Li + 1024;
  const int j = threadIdx.x & 31;
  cd x[32];
  if (threadIdx.x < 32) {
    // column j of L^{-1}: L x = e_j, unit diagonal
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      cd acc = mkc(r == j ? 1.0 : 0.0);
#pragma unroll
      for (int c = 0; c < r; ++c) {
        if (r < tb && c < tb) acc = acc - mkc(t[c][r].x, t[c][r].y) * x[c];
      }
      x[r] = acc;
    }
#pragma unroll
    for (int r = 0; r < 32; ++r) Li[j * 32 + r] = make_double2(x[r].re, x[r].im);
  } else {
    // column j of U^{-1}: U x = e_j
#pragma unroll
    for (int r = 31; r >= 0; --r) {
      cd acc = mkc(r == j ? 1.0 : 0.0);
#pragma unroll
      for (int c = r + 1; c < 32; ++c) acc = acc - mkc(t[c][r].x, t[c][r].y) * x[c];
      x[r] = acc / mkc(t[r][r].x, t[r][r].y);
    }
#pragma unroll
    for (int r = 0; r < 32; ++r) Ui[j * 32 + r] = make_double2(x[r].re, x[r].im);
  }
}

cudaError_t launch_precond_tile_inverse(int64_t nblocks, int64_t max_tiles, const int64_t* block_off,
                                        const int64_t* mat_off, const int64_t* tile_off, int nmax, const double* mats,
                                        double* tinv, cudaStream_t st) {
  if (nblocks <= 0 || max_tiles <= 0) return cudaSuccess;
  dim3 grid(static_cast<unsigned>(max_tiles), static_cast<unsigned>(nblocks));
  precond_tile_inverse_kernel<<<grid, 64, 0, st>>>(block_off, mat_off, tile_off, nmax,
                                                   reinterpret_cast<const double2*>(mats),
                                                   reinterpret_cast<double2*>(tinv));
  note_launch();
  return cudaGetLastError();
}

constexpr int kApplyThreads = 256;
constexpr int kApplyClusterMaxSmem = 160 * 1024;  // largest block vector of the cluster form

// FP64 vectors: the CTA of cluster rank s owns tiles [s * per, min(ntile, (s + 1) * per))
template <typename R, typename F>
__global__ void __launch_bounds__(kApplyThreads) precond_apply_cluster_kernel(
    const int64_t* __restrict__ block_off, const int64_t* __restrict__ mat_off, const int64_t* __restrict__ tile_off,
    int nmax, const int* __restrict__ perm, const Pair2<F>* __restrict__ mats, const Pair2<F>* __restrict__ tinv,
    const int* __restrict__ pivperm, int64_t N, const Pair2<R>* __restrict__ x, Pair2<R>* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char pc_smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = static_cast<int>(cluster.num_blocks());
  const int s = static_cast<int>(cluster.block_rank());
  const int64_t q = blockIdx.x / C;
  const int rhs = blockIdx.y;
  const int64_t s0 = block_off[q];
  const int64_t n = (block_off[q + 1] - s0) * nmax;
  const int64_t ntile = (n + 31) / 32;
  const int64_t per = (ntile + C - 1) / C;
  const int64_t t_lo = s * per < ntile ? s * per : ntile;
  const int64_t t_hi = (s + 1) * per < ntile ? (s + 1) * per : ntile;
  const int64_t r_lo = t_lo * 32, r_hi = t_hi * 32 < n ? t_hi * 32 : n;
  const Pair2<F>* A = mats + mat_off[q];
  const Pair2<F>* TI = tinv + tile_off[q];
  const int* pp = pivperm + s0 * nmax;
  const Pair2<R>* xr = x + (int64_t)rhs * N * nmax;
  Pair2<R>* yr = y + (int64_t)rhs * N * nmax;
  Pair2<F>* v = reinterpret_cast<Pair2<F>*>(pc_smem);  // [n]: own rows (partial sums) + solved tiles
  __shared__ Pair2<F> dt[32][33];
  __shared__ Pair2<F> w[32];
  // gather own rows (the pivot permutation folded in)
  for (int64_t t = r_lo + threadIdx.x; t < r_hi; t += blockDim.x) {
    const int64_t src = pp[t];
    const int64_t a = src / nmax;
    const int r = static_cast<int>(src - a * nmax);
    const Pair2<R> e = xr[(int64_t)perm[s0 + a] * nmax + r];
    v[t] = Pair2<F>{static_cast<F>(e.re), static_cast<F>(e.im)};
  }
  __syncthreads();
  cluster.sync();  // every CTA of the cluster has started before any writes into another's shared memory
  const int lane = threadIdx.x & 31;
  // one triangular sweep; fwd: tiles 0..ntile-1 with L, else ntile-1..0 with U
  auto sweep = [&](bool fwd) {
    for (int64_t step = 0; step < ntile; ++step) {
      const int64_t k = fwd ? step : ntile - 1 - step;
      const int64_t kb = k * 32;
      const int tb = static_cast<int>(n - kb < 32 ? n - kb : 32);
      const bool owner = k >= t_lo && k < t_hi;
      if (owner) {
        const Pair2<F>* Ti = TI + k * 2048 + (fwd ? 0 : 1024);
        for (int e = threadIdx.x; e < 1024; e += blockDim.x) dt[e >> 5][e & 31] = Ti[e];
        __syncthreads();
        if (threadIdx.x < 32) {
          F re = 0, im = 0;
#pragma unroll 8
          for (int c = 0; c < 32; ++c) {
            if (c < tb) {
              const Pair2<F> a = dt[c][lane], u = v[kb + c];
              re += a.re * u.re - a.im * u.im;
              im += a.re * u.im + a.im * u.re;
            }
          }
          w[lane] = Pair2<F>{re, im};
        }
        __syncthreads();
        // the solved tile into every CTA's copy of the block vector
        for (int e = threadIdx.x; e < C * 32; e += blockDim.x) {
          const int dst = e >> 5, r = e & 31;
          if (r < tb) cluster.map_shared_rank(v, dst)[kb + r] = w[r];
        }
      }
      cluster.sync();
      // apply tile column k to own rows below (fwd) / above (back) the tile
      const int64_t a0 = fwd ? (r_lo > kb + tb ? r_lo : kb + tb) : r_lo;
      const int64_t a1 = fwd ? r_hi : (r_hi < kb ? r_hi : kb);
      for (int64_t i = a0 + threadIdx.x; i < a1; i += blockDim.x) v[i] = tile_gemv(A, n, i, kb, tb, v, v[i]);
      __syncthreads();
    }
  };
  sweep(true);
  sweep(false);
  for (int64_t t = r_lo + threadIdx.x; t < r_hi; t += blockDim.x) {
    const int64_t a = t / nmax;
    const int r = static_cast<int>(t - a * nmax);
    yr[(int64_t)perm[s0 + a] * nmax + r] = Pair2<R>{static_cast<R>(v[t].re), static_cast<R>(v[t].im)};
  }
  // no CTA leaves while others may still write its shared memory
  cluster.sync();
}

// ---------------------------------------------------------------------------
// The block solve as two triangular products with explicit inverses.  At
// build time each block's FP64 factors are turned into L^{-1} (strictly lower
// part; unit diagonal implied) and U^{-1} (upper part with the diagonal), in
// FP64, stored in the same n x n column-major slot (an FP32 copy serves FP32
// vectors).  The
// apply x = U^{-1} (L^{-1} (P y)) is then two matrix-vector products with no
// serial chain: a cluster of C CTAs per block deals the 32-row tiles round
// robin, computes its rows of t = L^{-1} P y, writes them into every CTA's
// copy of t, meets the others at one cluster barrier and computes its rows of
// x = U^{-1} t.  It reads the same bytes as a substitution (one entry per
// factor element) and is bound by memory bandwidth.  A preconditioner only
// has to be a fixed linear operator close to the block inverse; forming the
// inverses in FP64 keeps the FP32 copy within FP32 rounding of the FP64 one.
// ---------------------------------------------------------------------------

// Inverses of L and U of every block, in step k for row tile k of L^{-1}
// (from the top) and row tile T - 1 - k of U^{-1} (from the bottom), all blocks
// together.  With S_ij = sum_k T_ik X_kj over the finished rows k, a step first
// forms X_kj = -inv(T_kk) S_kj, then adds T_ik X_kj to the S_ij of the rows to
// come: every tile of a step is one CTA and one tile product, so the work of
// the largest block spreads over the whole GPU (163 ms with one CTA per column
// tile, 58 ms now; 175 blocks of up to 1 248 unknowns).  S and X
// share the slot of the result; the diagonal tile keeps the strictly lower part
// of L^{-1} and the upper part of U^{-1}.
__global__ void __launch_bounds__(kTileThreads)
    precond_inverse_row_kernel(int64_t k, int nact, const int* __restrict__ order, const int64_t* __restrict__ off,
                               const int64_t* __restrict__ block_off, const int64_t* __restrict__ mat_off,
                               const int64_t* __restrict__ tile_off, int nmax, const double2* __restrict__ tinv,
                               double2* __restrict__ inv) {
  const int s = tile_block(off, nact, blockIdx.x);
  const int q = order[s];
  const int64_t n = (block_off[q + 1] - block_off[q]) * nmax;
  const int64_t T = (n + kTile - 1) / kTile;
  const int64_t t = blockIdx.x - off[s];  // k + 1 tiles of L, then k + 1 of U
  const bool upper = t > k;
  const int64_t row = upper ? T - 1 - k : k;
  const int64_t col = upper ? T - 1 - (t - k - 1) : t;
  double2* X = inv + mat_off[q];
  const double2* Ti = tinv + tile_off[q] + row * 2048 + (upper ? 1024 : 0);
  const int r = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t i = row * kTile + r, j = col * kTile + 4 * g;
  if (row == col) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = 4 * g + u;
      if (i < n && j + u < n && (upper ? r <= c : r > c)) X[i + (j + u) * n] = Ti[c * 32 + r];
    }
    return;
  }
  extern __shared__ Tile3 tiles3[];
  Tile3& as = tiles3[0];
  Tile3& xs = tiles3[1];
  load_tinv(as, Ti);
  load_tile(xs, X, n, row, col);
  __syncthreads();
  double2 acc[4] = {};
  tile_product<-1>(as, xs, acc);
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (i < n && j + u < n) X[i + (j + u) * n] = acc[u];
}

__global__ void __launch_bounds__(kTileThreads)
    precond_inverse_update_kernel(int64_t k, int nact, const int* __restrict__ order, const int64_t* __restrict__ off,
                                  const int64_t* __restrict__ block_off, const int64_t* __restrict__ mat_off,
                                  const int64_t* __restrict__ tile_off, int nmax, const double2* __restrict__ lu,
                                  const double2* __restrict__ tinv, double2* __restrict__ inv) {
  const int s = tile_block(off, nact, blockIdx.x);
  const int q = order[s];
  const int64_t n = (block_off[q + 1] - block_off[q]) * nmax;
  const int64_t T = (n + kTile - 1) / kTile;
  const int64_t rem = T - 1 - k, half = rem * (k + 1);  // rem rows to come, k + 1 columns; L, then U
  int64_t t = blockIdx.x - off[s];
  const bool upper = t >= half;
  if (upper) t -= half;
  const int64_t mid = upper ? rem : k;
  const int64_t row = upper ? rem - 1 - t % rem : k + 1 + t % rem;
  const int64_t col = upper ? T - 1 - t / rem : t / rem;
  const double2* A = lu + mat_off[q];
  double2* X = inv + mat_off[q];
  extern __shared__ Tile3 tiles3[];
  Tile3& as = tiles3[0];
  Tile3& xs = tiles3[1];
  load_tile(as, A, n, row, mid);
  if (col == mid) load_tinv(xs, tinv + tile_off[q] + mid * 2048 + (upper ? 1024 : 0));
  else load_tile(xs, X, n, mid, col);
  const int r = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t i = row * kTile + r, j = col * kTile + 4 * g;
  double2 acc[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)  // the first term of S_ij is the one of k = j
    acc[u] = col != mid && i < n && j + u < n ? X[i + (j + u) * n] : make_double2(0.0, 0.0);
  __syncthreads();
  tile_product<1>(as, xs, acc);
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (i < n && j + u < n) X[i + (j + u) * n] = acc[u];
}
constexpr int kInvThreads = 256;

// one complex factor, read once per apply: past the caches' retention
__device__ __forceinline__ Pair2<float> load_stream(const Pair2<float>* p) {
  const float2 v = __ldcs(reinterpret_cast<const float2*>(p));
  return Pair2<float>{v.x, v.y};
}
__device__ __forceinline__ Pair2<double> load_stream(const Pair2<double>* p) {
  const double2 v = __ldcs(reinterpret_cast<const double2*>(p));
  return Pair2<double>{v.x, v.y};
}

// x = U^{-1} (L^{-1} (P y)) for one (block, RHS) per cluster of C CTAs.  Bound
// by HBM: every factor is read once.  The 32-row tiles are dealt round robin to
// the CTAs, one lane per row, so each column of a tile is one coalesced read of
// 256 (FP32) or 512 bytes.  A CTA's tiles are triangular, so their columns are
// laid end to end and cut into equal runs, one per warp, sixteen columns in
// flight each: with whole tiles per warp the longest row of a block set the time
// and half of the bandwidth was left (245 blocks of up to 810 unknowns, FP32:
// 237 -> 144 us).  A tile cut between warps is added up from their
// pieces in order, so results do not depend on timing.  Every CTA gathers the
// whole (pivot-permuted) block vector.
template <typename R, typename F>
__global__ void __launch_bounds__(kInvThreads, 3)
    precond_apply_inv_kernel(const int64_t* __restrict__ block_off, const int64_t* __restrict__ mat_off, int nmax,
                             const int* __restrict__ perm, const Pair2<F>* __restrict__ inv,
                             const int* __restrict__ pivperm, int64_t N, const Pair2<R>* __restrict__ x,
                             Pair2<R>* __restrict__ y) {
  using V = Pair2<F>;
  constexpr int NW = kInvThreads / 32;
  constexpr int U = sizeof(F) == 4 ? 16 : 8;  // columns in flight
  extern __shared__ __align__(16) unsigned char pi_smem[];
  __shared__ V head[NW][32];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = static_cast<int>(cluster.num_blocks());
  const int s = static_cast<int>(cluster.block_rank());
  const int64_t q = blockIdx.x / C;
  const int rhs = blockIdx.y;
  const int64_t s0 = block_off[q];
  const int n = static_cast<int>((block_off[q + 1] - s0) * nmax);
  const int T = (n + 31) / 32;
  const V* A = inv + mat_off[q];
  const int* pp = pivperm + s0 * nmax;
  const Pair2<R>* xr = x + (int64_t)rhs * N * nmax;
  Pair2<R>* yr = y + (int64_t)rhs * N * nmax;
  V* xv = reinterpret_cast<V*>(pi_smem);  // [n] P y
  V* tv = xv + n;                         // [n] t = L^{-1} P y
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int t = tid; t < n; t += blockDim.x) {
    const int src = pp[t];
    const int a = src / nmax;
    const int r = src - a * nmax;
    const Pair2<R> e = xr[(int64_t)perm[s0 + a] * nmax + r];
    xv[t] = V{static_cast<F>(e.re), static_cast<F>(e.im)};
  }
  // every CTA of the cluster has started (and gathered) before any writes
  // into another's shared memory
  cluster.sync();
  const int m = T > s ? (T - s + C - 1) / C : 0;  // own tiles: s + C k, k < m
  // one triangular product; emit(row, sum) by the lane of the row
  auto sweep = [&](auto lower_, const V* v, auto emit) {
    constexpr bool LOWER = decltype(lower_)::value;
    auto first = [&](int k) { return LOWER ? 0 : 32 * (s + C * k); };
    auto count = [&](int k) { return LOWER ? min(32 * (s + C * k + 1), n) : n - 32 * (s + C * k); };
    int64_t tot = 0;
    for (int k = 0; k < m; ++k) tot += count(k);
    const int64_t a0 = tot * w / NW, a1 = tot * (w + 1) / NW;
    int64_t base = 0, tail_end = -1;
    int tail_row = 0;
    V tail{0, 0};
    for (int k = 0; k < m && base < a1; ++k) {
      const int64_t end = base + count(k);
      const int64_t lo = a0 > base ? a0 : base, hi = a1 < end ? a1 : end;
      if (lo < hi) {
        const int i = 32 * (s + C * k) + lane;
        const int j0 = first(k) + static_cast<int>(lo - base), j1 = first(k) + static_cast<int>(hi - base);
        // columns of this row's triangle: j < i (unit diagonal implied) or j >= i
        const int b0 = i >= n ? j1 : (LOWER ? 0 : i), b1 = LOWER ? i : n;
        F re0 = 0, im0 = 0, re1 = 0, im1 = 0;
        for (int j = j0; j < j1; j += U) {
          V c[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            c[u] = j + u < j1 && j + u >= b0 && j + u < b1 ? load_stream(A + i + (int64_t)(j + u) * n) : V{0, 0};
#pragma unroll
          for (int u = 0; u < U; u += 2) {
            const V v0 = v[min(j + u, n - 1)], v1 = v[min(j + u + 1, n - 1)];
            re0 += c[u].re * v0.re - c[u].im * v0.im;
            im0 += c[u].re * v0.im + c[u].im * v0.re;
            re1 += c[u + 1].re * v1.re - c[u + 1].im * v1.im;
            im1 += c[u + 1].re * v1.im + c[u + 1].im * v1.re;
          }
        }
        const V sum{re0 + re1, im0 + im1};
        if (lo > base) {
          head[w][lane] = sum;  // a tile that an earlier warp began
        } else if (hi < end) {
          tail = sum;
          tail_end = end;
          tail_row = i;
        } else if (i < n) {
          emit(i, sum);
        }
      }
      base = end;
    }
    __syncthreads();
    if (tail_end >= 0) {
      for (int o = w + 1; o < NW && tot * o / NW < tail_end; ++o) {
        if (tot * o / NW == tot * (o + 1) / NW) continue;  // an empty run
        tail.re += head[o][lane].re;
        tail.im += head[o][lane].im;
      }
      if (tail_row < n) emit(tail_row, tail);
    }
  };
  // t = L^{-1} P y on own tiles, into every CTA's copy of t
  sweep(std::true_type{}, xv, [&](int i, V d) {
    const V t = V{xv[i].re + d.re, xv[i].im + d.im};
    for (int dst = 0; dst < C; ++dst) cluster.map_shared_rank(tv, dst)[i] = t;
  });
  cluster.sync();
  // x = U^{-1} t on own tiles
  sweep(std::false_type{}, tv, [&](int i, V o) {
    const int a = i / nmax;
    const int r = i - a * nmax;
    yr[(int64_t)perm[s0 + a] * nmax + r] = Pair2<R>{static_cast<R>(o.re), static_cast<R>(o.im)};
  });
}

// FP64 explicit inverses of L and U of every block (from the FP64 LU and
// FP64 tile inverses) into inv
cudaError_t launch_precond_tri_inverse(const PrecondPlan& plan, const int64_t* block_off, const int64_t* mat_off,
                                       const int64_t* tile_off, int nmax, const double* lu, const double* tinv,
                                       double* inv, cudaStream_t st) {
  const double2* T = reinterpret_cast<const double2*>(tinv);
  double2* X = reinterpret_cast<double2*>(inv);
  cudaError_t e = tile_smem(precond_inverse_row_kernel);
  if (e == cudaSuccess) e = tile_smem(precond_inverse_update_kernel);
  if (e != cudaSuccess) return e;
  for (size_t k = 0; k < plan.steps.size(); ++k) {
    const PrecondPlan::Step& p = plan.steps[k];
    precond_inverse_row_kernel<<<static_cast<unsigned>(p.rows), kTileThreads, 2 * sizeof(Tile3), st>>>(
        static_cast<int64_t>(k), p.active, plan.order, plan.off + p.rows_off, block_off, mat_off, tile_off, nmax, T, X);
    note_launch();
    if (p.inv_tiles > 0) {
      precond_inverse_update_kernel<<<static_cast<unsigned>(p.inv_tiles), kTileThreads, 2 * sizeof(Tile3), st>>>(
          static_cast<int64_t>(k), p.active, plan.order, plan.off + p.inv_tiles_off, block_off, mat_off, tile_off, nmax,
          reinterpret_cast<const double2*>(lu), T, X);
      note_launch();
    }
  }
  return cudaGetLastError();
}

// steps of the blocked factorisation and of the inverses for blocks of the
// given dimensions; `order` and `off` (host) go to the device
void precond_plan(const std::vector<int64_t>& dims, PrecondPlan& plan, std::vector<int>& order,
                  std::vector<int64_t>& off) {
  order.resize(dims.size());
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return dims[a] > dims[b]; });
  off.clear();
  plan.steps.clear();
  plan.dims.clear();
  for (int q : order) plan.dims.push_back(dims[q]);
  const int64_t steps = dims.empty() ? 0 : (plan.dims[0] + kTile - 1) / kTile;
  for (int64_t k = 0; k < steps; ++k) {
    PrecondPlan::Step p{};
    auto tiles = [&](int s) { return (plan.dims[s] + kTile - 1) / kTile; };
    while (p.active < static_cast<int>(order.size()) && tiles(p.active) > k) ++p.active;
    auto prefix = [&](int64_t& at, int64_t& total, auto count) {
      at = static_cast<int64_t>(off.size());
      total = 0;
      for (int s = 0; s < p.active; ++s) {
        off.push_back(total);
        total += count(tiles(s));
      }
    };
    prefix(p.columns_off, p.columns, [&](int64_t T) { return T - 1; });
    prefix(p.tiles_off, p.tiles, [&](int64_t T) { return (T - 1 - k) * (T - 1 - k); });
    prefix(p.rows_off, p.rows, [&](int64_t) { return 2 * (k + 1); });
    prefix(p.inv_tiles_off, p.inv_tiles, [&](int64_t T) { return 2 * (T - 1 - k) * (k + 1); });
    plan.steps.push_back(p);
  }
}

// position -> source index of the row interchanges of each block's LU
// (applied in order kk = 0..n-1, as the factorisation recorded them)
__global__ void pivot_perm_kernel(const int64_t* __restrict__ block_off, int nmax, const int* __restrict__ piv,
                                  int* __restrict__ pivperm) {
  const int64_t q = blockIdx.x;
  const int64_t s0 = block_off[q];
  const int64_t n = (block_off[q + 1] - s0) * nmax;
  const int* pv = piv + s0 * nmax;
  int* pp = pivperm + s0 * nmax;
  for (int64_t t = threadIdx.x; t < n; t += blockDim.x) pp[t] = static_cast<int>(t);
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int64_t kk = 0; kk < n; ++kk) {
      const int64_t p = pv[kk];
      if (p != kk) {
        const int t = pp[kk];
        pp[kk] = pp[p];
        pp[p] = t;
      }
    }
  }
}

cudaError_t launch_pivot_perm(int64_t nblocks, const int64_t* block_off, int nmax, const int* piv, int* pivperm,
                              cudaStream_t st) {
  if (nblocks <= 0) return cudaSuccess;
  pivot_perm_kernel<<<static_cast<unsigned>(nblocks), 256, 0, st>>>(block_off, nmax, piv, pivperm);
  note_launch();
  return cudaGetLastError();
}

template <typename R, typename F>
cudaError_t launch_apply_t(int64_t nblocks, const int64_t* block_off, const int64_t* mat_off, int nmax,
                           const int* perm, const void* mats, const int* piv, int64_t N, int nrhs, const void* x,
                           void* y, void* work, int max_block_dim, cudaStream_t st) {
  dim3 grid(static_cast<unsigned>(nblocks), static_cast<unsigned>(nrhs));
  const size_t smem = sizeof(Pair2<F>) * static_cast<size_t>(max_block_dim);
  if (smem <= 200 * 1024) {
    // the shared-memory opt-in, once on each device
    static PerDevice attr;
    cudaError_t se = cudaSuccess;
    if (attr.get(current_device, [&] {
          se = cudaFuncSetAttribute(precond_apply_kernel<R, F, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    200 * 1024);
          return se == cudaSuccess ? 1 : 0;
        }) == 0)
      return se != cudaSuccess ? se : cudaErrorInvalidConfiguration;
    precond_apply_kernel<R, F, true><<<grid, 256, smem, st>>>(
        block_off, mat_off, nmax, perm, static_cast<const Pair2<F>*>(mats), piv, N, static_cast<const Pair2<R>*>(x),
        static_cast<Pair2<R>*>(y), static_cast<Pair2<F>*>(work));
  } else {
    precond_apply_kernel<R, F, false><<<grid, 256, 0, st>>>(
        block_off, mat_off, nmax, perm, static_cast<const Pair2<F>*>(mats), piv, N, static_cast<const Pair2<R>*>(x),
        static_cast<Pair2<R>*>(y), static_cast<Pair2<F>*>(work));
  }
  note_launch();
  return cudaGetLastError();
}

template <typename R, typename F>
cudaError_t launch_apply_cluster_t(int64_t nblocks, const int64_t* block_off, const int64_t* mat_off,
                                   const int64_t* tile_off, int nmax, const int* perm, const void* mats,
                                   const void* tinv, const int* pivperm, int64_t N, int nrhs, const void* x, void* y,
                                   int max_block_dim, int csize, cudaStream_t st) {
  const size_t smem = sizeof(Pair2<F>) * static_cast<size_t>(max_block_dim);
  static PerDevice attr;
  cudaError_t se = cudaSuccess;
  if (attr.get(current_device, [&] {
        se = cudaFuncSetAttribute(precond_apply_cluster_kernel<R, F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kApplyClusterMaxSmem);
        return se == cudaSuccess ? 1 : 0;
      }) == 0)
    return se != cudaSuccess ? se : cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(nblocks * csize), static_cast<unsigned>(nrhs));
  cfg.blockDim = dim3(kApplyThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = static_cast<unsigned>(csize);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, precond_apply_cluster_kernel<R, F>, block_off, mat_off, tile_off, nmax,
                                           perm, static_cast<const Pair2<F>*>(mats), static_cast<const Pair2<F>*>(tinv),
                                           pivperm, N, static_cast<const Pair2<R>*>(x), static_cast<Pair2<R>*>(y));
  note_launch();
  return e;
}

// cluster size of the apply for blocks of about `mean_tiles` 32-row tiles
int precond_cluster_size(double mean_tiles) {
  if (mean_tiles >= 12.0) return 4;
  if (mean_tiles >= 4.0) return 2;
  return 1;
}

// the two-product form fits when both FP64 block vectors fit in shared memory
bool precond_inverse_fits(int max_block_dim) {
  return 2 * sizeof(Pair2<double>) * static_cast<size_t>(max_block_dim) <= kApplyClusterMaxSmem;
}

template <typename R>
cudaError_t launch_apply_inv(int64_t nblocks, const int64_t* block_off, const int64_t* mat_off, int nmax,
                             const int* perm, const R* inv, const int* pivperm, int64_t N, int nrhs, const void* x,
                             void* y, int max_block_dim, int csize, cudaStream_t st) {
  // three CTAs per SM keep enough loads in flight; more per block only where
  // there are fewer blocks, and for blocks with tiles to share out
  const int most = csize >= 4 ? 8 : (csize >= 2 ? 4 : 1);
  csize = 1;
  while (csize < most && nblocks * nrhs * csize < 3LL * device_sms()) csize *= 2;
  static PerDevice attr;
  cudaError_t se = cudaSuccess;
  if (attr.get(current_device, [&] {
        se = cudaFuncSetAttribute(precond_apply_inv_kernel<R, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kApplyClusterMaxSmem);
        return se == cudaSuccess ? 1 : 0;
      }) == 0)
    return se != cudaSuccess ? se : cudaErrorInvalidConfiguration;
  const size_t smem = 2 * sizeof(Pair2<R>) * static_cast<size_t>(max_block_dim);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(nblocks * csize), static_cast<unsigned>(nrhs));
  cfg.blockDim = dim3(kInvThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = static_cast<unsigned>(csize);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, precond_apply_inv_kernel<R, R>, block_off, mat_off, nmax, perm,
                                           reinterpret_cast<const Pair2<R>*>(inv), pivperm, N,
                                           static_cast<const Pair2<R>*>(x), static_cast<Pair2<R>*>(y));
  note_launch();
  return e;
}

// FP64 vectors use the FP64 factors (mats), FP32 vectors the FP32 copy
// (mats32).  With `inverse` set both hold the explicit inverses of L and U
// (the two-product form); otherwise the LU factors, solved by substitution:
// in the cluster form when tile inverses exist and the block vector fits in
// shared memory, else one CTA per block.
template <typename R>
cudaError_t launch_precond_apply(int64_t nblocks, const int64_t* block_off, const int64_t* mat_off, int nmax,
                                 const int* perm, const double* mats, const float* mats32, const int* piv, int64_t N,
                                 int nrhs, const void* x, void* y, double* work, int max_block_dim, cudaStream_t st,
                                 const int64_t* tile_off, const double* tinv, const float* tinv32, int csize,
                                 bool inverse) {
  if (nblocks <= 0) return cudaSuccess;
  constexpr size_t esz = sizeof(R) == 8 ? 16 : 8;
  if (inverse) {
    if constexpr (sizeof(R) == 8)
      return launch_apply_inv<double>(nblocks, block_off, mat_off, nmax, perm, mats, piv, N, nrhs, x, y,
                                      max_block_dim, csize >= 1 ? csize : 1, st);
    else
      return launch_apply_inv<float>(nblocks, block_off, mat_off, nmax, perm, mats32, piv, N, nrhs, x, y,
                                     max_block_dim, csize >= 1 ? csize : 1, st);
  }
  if (tinv && csize >= 1 && esz * static_cast<size_t>(max_block_dim) <= kApplyClusterMaxSmem) {
    if constexpr (sizeof(R) == 8)
      return launch_apply_cluster_t<double, double>(nblocks, block_off, mat_off, tile_off, nmax, perm, mats, tinv,
                                                    piv, N, nrhs, x, y, max_block_dim, csize, st);
    else
      return launch_apply_cluster_t<float, float>(nblocks, block_off, mat_off, tile_off, nmax, perm, mats32, tinv32,
                                                  piv, N, nrhs, x, y, max_block_dim, csize, st);
  }
  if constexpr (sizeof(R) == 8)
    return launch_apply_t<double, double>(nblocks, block_off, mat_off, nmax, perm, mats, piv, N, nrhs, x, y, work,
                                          max_block_dim, st);
  else
    return launch_apply_t<float, float>(nblocks, block_off, mat_off, nmax, perm, mats32, piv, N, nrhs, x, y, work,
                                        max_block_dim, st);
}
template cudaError_t launch_precond_apply<float>(int64_t, const int64_t*, const int64_t*, int, const int*,
                                                 const double*, const float*, const int*, int64_t, int, const void*,
                                                 void*, double*, int, cudaStream_t, const int64_t*, const double*,
                                                 const float*, int, bool);
template cudaError_t launch_precond_apply<double>(int64_t, const int64_t*, const int64_t*, int, const int*,
                                                  const double*, const float*, const int*, int64_t, int, const void*,
                                                  void*, double*, int, cudaStream_t, const int64_t*, const double*,
                                                  const float*, int, bool);

__global__ void f64_to_f32_kernel(int64_t n, const double* __restrict__ a, float* __restrict__ b) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    b[t] = static_cast<float>(a[t]);
}
cudaError_t launch_f64_to_f32(int64_t n, const double* a, float* b, cudaStream_t st) {
  const int64_t blocks = (n + 255) / 256;
  const int64_t cap = 16LL * device_sms();
  f64_to_f32_kernel<<<static_cast<unsigned>(blocks < cap ? (blocks > 0 ? blocks : 1) : cap), 256, 0, st>>>(
      n, a, b);
  note_launch();
  return cudaGetLastError();
}

}  // namespace celes
