// FP64 QR re-isometrisation on the GPU (Sec. 3.1, Fig. iso).
//
// A node tensor is viewed as the matrix A (M x k) whose column index is the
// link towards the next isometry centre; A = Q R with Q^T Q = 1 and
// R upper triangular, diag(R) >= 0. Columns are orthogonalised one after the
// other by classical Gram-Schmidt applied twice ("CGS2", numerically as
// orthogonal as Householder for full-rank A). A column whose remaining norm
// falls below 1e-13 of its original norm is rank-deficient: its R diagonal is
// set to 0 and, after the sweep over columns, it is replaced by a unit vector
// orthogonalised against all other columns (A = Q R still holds because every
// later column was orthogonalised against the zero column).
//
// One launch per QR (qr_slab_kernel) while the matrix fits the SMs' shared memory. Larger ones
// go column by column over At[j][row] = A[row][j] (each column contiguous):
// [dots] -> [update + dots] -> [update + norm] -> [finalise], every block reducing the
// partials itself.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "attn_internal.h"
#include "qr.h"

namespace attn {

namespace {

constexpr int QT = 256;   // threads per block
constexpr int QROWS = 256;   // rows per block (one per thread)

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// part[b][i] = sum_{rows of block b} At[i][row] * At[j][row], i < j
__device__ void partial_dots(const double* At, long M, int j, double* part, int nblk_stride) {
  const long r0 = (long)blockIdx.x * QROWS;
  const long r1 = min(M, r0 + QROWS);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* a = At + (long)j * M;
  for (int i = warp; i < j; i += QT / 32) {
    const double* q = At + (long)i * M;
    double s = 0.0;
    for (long r = r0 + lane; r < r1; r += 32) s = fma(q[r], a[r], s);
    s = warp_sum(s);
    if (lane == 0) part[(long)blockIdx.x * nblk_stride + i] = s;
  }
}

// h[i] = sum_b part[b][i] for i < j (into shared), R[i][j] += h[i] by block 0.
__device__ void reduce_h(const double* part, int nb, int j, int stride, double* h, double* R, int k, bool accum_R) {
  for (int i = threadIdx.x; i < j; i += QT) {
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += part[(long)b * stride + i];
    h[i] = s;
    if (accum_R && blockIdx.x == 0) R[(long)i * k + j] += s;
  }
  __syncthreads();
}

__global__ void qr_init_kernel(const double* At, long M, int k, double* nrm0, double* R) {
  // nrm0[j] = ||a_j|| (one block per column), R zeroed
  int j = blockIdx.x;
  __shared__ double sh[QT / 32];
  const double* a = At + (long)j * M;
  double s = 0.0;
  for (long r = threadIdx.x; r < M; r += QT) s = fma(a[r], a[r], s);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int w = 0; w < QT / 32; ++w) t += sh[w];
    nrm0[j] = sqrt(t);
  }
  for (int c = threadIdx.x; c < k; c += QT) R[(long)j * k + c] = 0.0;
}

__global__ void qr_dots_kernel(const double* At, long M, int j, double* part, int stride) {
  partial_dots(At, M, j, part, stride);
}

// a_j -= Q h (h from partials); then either the next dots or the norm partial.
__global__ void qr_update_kernel(double* At, long M, int j, int k, double* part, int nb, int stride, double* R,
                                 int next_is_norm, double* part2) {
  extern __shared__ double h[];
  reduce_h(part, nb, j, stride, h, R, k, true);
  const long r0 = (long)blockIdx.x * QROWS;
  const long r1 = min(M, r0 + QROWS);
  double* a = At + (long)j * M;
  for (long r = r0 + threadIdx.x; r < r1; r += QT) {
    double v = a[r];
    for (int i = 0; i < j; ++i) v = fma(-h[i], At[(long)i * M + r], v);
    a[r] = v;
  }
  __syncthreads();
  if (!next_is_norm) {
    partial_dots(At, M, j, part2, stride);
  } else {
    __shared__ double sh[QT / 32];
    double s = 0.0;
    for (long r = r0 + threadIdx.x; r < r1; r += QT) s = fma(a[r], a[r], s);
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0;
      for (int w = 0; w < QT / 32; ++w) t += sh[w];
      part2[blockIdx.x] = t;
    }
  }
}

__global__ void qr_norm_partial_kernel(const double* At, long M, int j, double* part) {
  __shared__ double sh[QT / 32];
  const long r0 = (long)blockIdx.x * QROWS;
  const long r1 = min(M, r0 + QROWS);
  const double* a = At + (long)j * M;
  double s = 0.0;
  for (long r = r0 + threadIdx.x; r < r1; r += QT) s = fma(a[r], a[r], s);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int w = 0; w < QT / 32; ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

__global__ void qr_finalise_kernel(double* At, long M, int j, int k, const double* part, int nb, const double* nrm0,
                                   double* R, int* deficient) {
  __shared__ double rj;
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += part[b];
    double r = sqrt(s);
    if (!(r > 1e-13 * nrm0[j]) || !(r > 1e-300)) {
      r = 0.0;
      if (blockIdx.x == 0) deficient[j] = 1;
    } else if (blockIdx.x == 0) {
      deficient[j] = 0;
    }
    rj = r;
    if (blockIdx.x == 0) R[(long)j * k + j] = r;
  }
  __syncthreads();
  const double inv = rj > 0.0 ? 1.0 / rj : 0.0;
  const long r0 = (long)blockIdx.x * QROWS;
  const long r1 = min(M, r0 + QROWS);
  double* a = At + (long)j * M;
  for (long r = r0 + threadIdx.x; r < r1; r += QT) a[r] *= inv;
}

// Replacement of deficient column j: a_j = e_t, then CGS2 against all other columns.
__global__ void qr_set_unit_kernel(double* At, long M, int j, long t) {
  double* a = At + (long)j * M;
  for (long r = blockIdx.x * (long)blockDim.x + threadIdx.x; r < M; r += (long)gridDim.x * blockDim.x)
    a[r] = (r == t) ? 1.0 : 0.0;
}

// single-block: a_j -= sum_{i != j} <q_i, a_j> q_i (all other columns), twice, then normalise; writes norm
__global__ void qr_fix_column_kernel(double* At, long M, int j, int k, double* out_norm) {
  extern __shared__ double h[];
  __shared__ double sh[QT / 32];
  double* a = At + (long)j * M;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = warp; i < k; i += QT / 32) {
      double s = 0.0;
      if (i != j) {
        const double* q = At + (long)i * M;
        for (long r = lane; r < M; r += 32) s = fma(q[r], a[r], s);
      }
      s = warp_sum(s);
      if (lane == 0) h[i] = s;
    }
    __syncthreads();
    for (long r = threadIdx.x; r < M; r += QT) {
      double v = a[r];
      for (int i = 0; i < k; ++i)
        if (i != j) v = fma(-h[i], At[(long)i * M + r], v);
      a[r] = v;
    }
    __syncthreads();
  }
  double s = 0.0;
  for (long r = threadIdx.x; r < M; r += QT) s = fma(a[r], a[r], s);
  s = warp_sum(s);
  if (lane == 0) sh[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int w = 0; w < QT / 32; ++w) t += sh[w];
    sh[0] = sqrt(t);
    *out_norm = sh[0];
  }
  __syncthreads();
  double inv = sh[0] > 0.5 ? 1.0 / sh[0] : 0.0;
  for (long r = threadIdx.x; r < M; r += QT) a[r] *= inv;
}

// Permute T[d0][d1][d2] into At[k = d_slot][M] (other two indices in order) and back.
__global__ void to_columns_kernel(const double* T, int d0, int d1, int d2, int slot, double* At) {
  long V = (long)d0 * d1 * d2;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < V; e += (long)gridDim.x * blockDim.x) {
    int c = e % d2;
    long t = e / d2;
    int b = t % d1;
    int a = t / d1;
    long col, row;
    if (slot == 0) { col = a; row = (long)b * d2 + c; }
    else if (slot == 1) { col = b; row = (long)a * d2 + c; }
    else { col = c; row = (long)a * d1 + b; }
    long M = V / (slot == 0 ? d0 : slot == 1 ? d1 : d2);
    At[col * M + row] = T[e];
  }
}

__global__ void from_columns_kernel(const double* At, int d0, int d1, int d2, int slot, double* T) {
  long V = (long)d0 * d1 * d2;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < V; e += (long)gridDim.x * blockDim.x) {
    int c = e % d2;
    long t = e / d2;
    int b = t % d1;
    int a = t / d1;
    long col, row;
    if (slot == 0) { col = a; row = (long)b * d2 + c; }
    else if (slot == 1) { col = b; row = (long)a * d2 + c; }
    else { col = c; row = (long)a * d1 + b; }
    long M = V / (slot == 0 ? d0 : slot == 1 ? d1 : d2);
    T[e] = At[col * M + row];
  }
}

// ---- the whole QR in one launch
//
// Every CTA keeps its rows of A (all columns) in shared memory from the first column to the
// last, reading and writing the tensor in place. What bounds a QR of this size is the chain of
// columns, each of which needs sums over all rows, so the two Gram-Schmidt passes share one
// reduction per column: the second pass of column j - 1 and the first of column j take their
// products with the same q_i together (delayed reorthogonalisation: D. Bielich, J. Langou,
// S. Thomas, K. Swirydowicz, I. Yamazaki, E. Boman, "Low-synch Gram-Schmidt with delayed
// reorthogonalization for Krylov solvers", Parallel Computing 112 (2022)). With c the second
// coefficients of w = a_{j-1} - Q s, its norm is |w|^2 - |c|^2, and its product with a_j follows
// from w . a_j. A column that the first pass cancelled to where |c| is no longer small beside
// |w| takes its second pass alone and repeats the reduction, so the result is as orthogonal as
// two full passes make it.
//
// Reduction: the CTAs of a cluster add their shares through distributed shared memory, each a
// slice of the values; several clusters meet through global partials and one grid barrier
// (cooperative launch; the wait is bounded). All sums run in a fixed order.
// [64, 64, 64] (4096 x 64): 1600 -> 585 us against four launches per column.
constexpr int kQrT = 256;    // threads
constexpr int kQrC = 8;      // CTAs per cluster
constexpr int kQrMaxK = 256;  // columns
constexpr long long kQrWait = 4000000000LL;  // cycles that the grid barrier waits at most

struct QrSlab {
  double* T;
  long rs_hi, rs_lo, cs;  // element (row, col) at (row / rlo) rs_hi + (row % rlo) rs_lo + col cs
  int rlo, M, k, rows, ld, nclus;
  double* R;
  int* defic;      // [k] rank-deficient columns, [k] = 1 when a wait gave up
  double* part;    // [2][clusters][2 kQrMaxK]
  unsigned* bar;   // arrivals, CTAs done
};

namespace cg = cooperative_groups;

struct QrShared {
  double loc[2][2 * kQrMaxK];  // this CTA's sums (two, so that one cluster barrier suffices)
  double tot[2 * kQrMaxK];     // sums over all rows
  double sum[2 * kQrT];        // partial sums of thread groups
  double nrm0[kQrMaxK], rprev[kQrMaxK];
  double rho, inv, sy;  // of the column being completed
  int again, dead;
};

// tot[0 .. nv) = sum of loc over all CTAs; `step` counts the reductions.
__device__ void qr_reduce(const QrSlab& q, QrShared& sh, int nv, unsigned step) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), cluster = blockIdx.x / kQrC, t = threadIdx.x, buf = step & 1;
  cl.sync();
  if (q.nclus == 1) {
    for (int v = t; v < nv; v += kQrT) {
      double s = 0.0;
#pragma unroll
      for (int r = 0; r < kQrC; ++r) s += *cl.map_shared_rank(&sh.loc[buf][v], r);
      sh.tot[v] = s;
    }
    __syncthreads();
    return;
  }
  const int v0 = nv * rank / kQrC, n = nv * (rank + 1) / kQrC - v0;  // this CTA's slice
  double* part = q.part + (long)buf * q.nclus * 2 * kQrMaxK;
  for (int v = t; v < n; v += kQrT) {
    double s = 0.0;
#pragma unroll
    for (int r = 0; r < kQrC; ++r) s += *cl.map_shared_rank(&sh.loc[buf][v0 + v], r);
    part[(long)cluster * 2 * kQrMaxK + v0 + v] = s;
  }
  __syncthreads();
  if (t == 0 && !sh.dead) {
    __threadfence();
    atomicAdd(q.bar, 1u);
    const unsigned target = (step + 1) * gridDim.x;
    const long long t0 = clock64();
    while (*(volatile unsigned*)q.bar < target) {
      if (clock64() - t0 > kQrWait) {
        sh.dead = 1;
        q.defic[q.k] = 1;
        break;
      }
    }
    __threadfence();
  }
  __syncthreads();
  // the slice over the clusters, four partial sums per value
  for (int e = t; e < 4 * n; e += kQrT) {
    const int v = e >> 2, h = e & 3;
    double s = 0.0;
    for (int c = h; c < q.nclus; c += 4) s += __ldcg(part + (long)c * 2 * kQrMaxK + v0 + v);
    sh.sum[e] = s;
  }
  __syncthreads();
  for (int e = t; e < n * kQrC; e += kQrT) {
    const int v = e / kQrC, r = e % kQrC;
    *cl.map_shared_rank(&sh.tot[v0 + v], r) = (sh.sum[4 * v] + sh.sum[4 * v + 1]) + (sh.sum[4 * v + 2] + sh.sum[4 * v + 3]);
  }
  cl.sync();
}

__global__ void __launch_bounds__(kQrT) qr_slab_kernel(const QrSlab q) {
  extern __shared__ double slab[];  // [rows][ld], ld odd: rows and columns both conflict-free
  __shared__ QrShared sh;
  const int t = threadIdx.x, k = q.k, ld = q.ld;
  const int r0 = blockIdx.x * q.rows, n = max(0, min(q.rows, q.M - r0));
  auto at = [&](int r, int c) {
    const int g = r0 + r;
    return (long)(g / q.rlo) * q.rs_hi + (long)(g % q.rlo) * q.rs_lo + (long)c * q.cs;
  };
  if (t == 0) sh.dead = 0;
  if (t == 0 && blockIdx.x == 0) q.defic[k] = 0;
  if (q.cs == 1) {
    for (int e = t; e < n * k; e += kQrT) slab[e / k * ld + e % k] = q.T[at(e / k, e % k)];
  } else {
    for (int e = t; e < n * k; e += kQrT) slab[e % n * ld + e / n] = q.T[at(e % n, e / n)];
  }
  __syncthreads();

  // loc = sums over this CTA's rows of columns 0 .. nc - 1 with column x (and, if y >= 0, y; with
  // themselves if x < 0): threads take a column and every G-th row
  auto dots = [&](int nc, int x, int y, double* loc) {
    int W = 16;
    while (W < nc) W *= 2;
    const int G = kQrT / W, i = t % W, g = t / W;
    double a0 = 0.0, a1 = 0.0, b0 = 0.0, b1 = 0.0;
    if (i < nc) {
      int r = g;
      for (; r + G < n; r += 2 * G) {
        const double *p = slab + r * ld, *p2 = p + G * ld;
        const double v = p[i], v2 = p2[i];
        a0 = fma(v, x < 0 ? v : p[x], a0);
        a1 = fma(v2, x < 0 ? v2 : p2[x], a1);
        if (y >= 0) {
          b0 = fma(v, p[y], b0);
          b1 = fma(v2, p2[y], b1);
        }
      }
      if (r < n) {
        const double* p = slab + r * ld;
        a0 = fma(p[i], x < 0 ? p[i] : p[x], a0);
        if (y >= 0) b0 = fma(p[i], p[y], b0);
      }
    }
    sh.sum[t] = a0 + a1;
    sh.sum[kQrT + t] = b0 + b1;
    __syncthreads();
    for (int v = t; v < (y >= 0 ? 2 * nc : nc); v += kQrT) {
      const double* p = sh.sum + (v >= nc ? kQrT + v - nc : v);
      double s = p[0];
      for (int h = 1; h < G; ++h) s += p[h * W];
      loc[v] = s;
    }
    __syncthreads();
  };
  // column x -= sum_{i < nc} Q_i cx_i, scaled by f; column y (if >= 0) -= sum Q_i cy_i + sy times the
  // new column x: threads take a row and every P-th column
  auto update = [&](int nc, int x, const double* cx, double f, int y, const double* cy, double sy) {
    int W = 16;
    while (W < n) W *= 2;
    const int P = kQrT / W, r = t % W, p = t / W;
    double a0 = 0.0, b0 = 0.0, a1 = 0.0, b1 = 0.0;
    if (r < n) {
      const double* row = slab + r * ld;
      int i = p;
      for (; i + P < nc; i += 2 * P) {
        const double v = row[i], v2 = row[i + P];
        a0 = fma(v, cx[i], a0);
        a1 = fma(v2, cx[i + P], a1);
        if (y >= 0) {
          b0 = fma(v, cy[i], b0);
          b1 = fma(v2, cy[i + P], b1);
        }
      }
      if (i < nc) {
        a0 = fma(row[i], cx[i], a0);
        if (y >= 0) b0 = fma(row[i], cy[i], b0);
      }
    }
    sh.sum[t] = a0 + a1;
    sh.sum[kQrT + t] = b0 + b1;
    __syncthreads();
    if (t < n) {
      double a = sh.sum[t], b = sh.sum[kQrT + t];
      for (int h = 1; h < P; ++h) {
        a += sh.sum[h * W + t];
        b += sh.sum[kQrT + h * W + t];
      }
      double* row = slab + t * ld;
      const double u = (row[x] - a) * f;
      row[x] = u;
      if (y >= 0) row[y] = fma(-sy, u, row[y] - b);
    }
    __syncthreads();
  };

  unsigned step = 0;
  dots(k, -1, -1, sh.loc[0]);
  qr_reduce(q, sh, k, step++);
  for (int i = t; i < k; i += kQrT) {
    sh.nrm0[i] = sqrt(sh.tot[i]);
    sh.rprev[i] = 0.0;
  }
  __syncthreads();
  for (int j = 1; j <= k; ++j) {  // column w = j - 1 is completed, column j takes its first pass
    const int w = j - 1, y = j < k ? j : -1;
    for (int again = 0;; ++again) {
      dots(j, w, y, sh.loc[step & 1]);
      qr_reduce(q, sh, y >= 0 ? 2 * j : j, step++);
      // tot: c_i (i < w), |w|^2; s_i, w . a_j. Every CTA has the same sums and takes the same
      // way; one warp works the scalars out (an FP64 instruction costs a warp 16 cycles of the SM)
      if (t < 32) {
        const double w2 = sh.tot[w];
        const float sc = rsqrtf((float)w2);
        float fc = 0.0f;  // |c|^2 / |w|^2
        for (int i = t; i < w; i += 32) {
          const double c = sh.tot[i];
          const float f = (float)c * sc;
          fc = fmaf(f, f, fc);
          sh.rprev[i] += c;
        }
        for (int o = 16; o > 0; o >>= 1) fc += __shfl_xor_sync(0xffffffffu, fc, o);
        // c below 1e-9 of w, the usual case: its square is nothing beside |w|^2, and FP32 is enough
        // for c . s, a correction of that size, while both columns' norms lie where no term of it that
        // matters leaves FP32's range
        const double ny = y >= 0 ? sh.nrm0[y] : 1.0;
        const bool mid = w2 > 1e-24 && w2 < 1e24 && ny > 1e-12 && ny < 1e12;
        double cc = 0.0, cs = 0.0;
        if (mid && fc <= 1e-18f) {
          float fs = 0.0f;
          for (int i = t; i < w && y >= 0; i += 32) fs = fmaf((float)sh.tot[i], (float)sh.tot[j + i], fs);
          for (int o = 16; o > 0; o >>= 1) fs += __shfl_xor_sync(0xffffffffu, fs, o);
          cs = (double)fs;
        } else {
          for (int i = t; i < w; i += 32) {
            const double c = sh.tot[i];
            cc = fma(c, c, cc);
            if (y >= 0) cs = fma(c, sh.tot[j + i], cs);
          }
          for (int o = 16; o > 0; o >>= 1) {
            cc += __shfl_xor_sync(0xffffffffu, cc, o);
            cs += __shfl_xor_sync(0xffffffffu, cs, o);
          }
        }
        if (t == 0) {
          const double d = w2 - cc, n0 = sh.nrm0[w];
          const double inv = rsqrt(d), rho = d > 0.0 ? d * inv : (d == d ? 0.0 : d);  // (a NaN stays one)
          const bool ok = rho > 1e-13 * n0 && rho > 1e-300;
          sh.again = cc > 0.25 * w2 && again < 3 && w2 > 1e-26 * n0 * n0;
          sh.rho = ok ? rho : 0.0;
          sh.inv = ok ? inv : 0.0;
          sh.sy = ok && y >= 0 ? (sh.tot[j + w] - cs) * inv : 0.0;
        }
      }
      __syncthreads();
      if (!sh.again) break;
      update(w, w, sh.tot, 1.0, -1, nullptr, 0.0);
    }
    const double rho = sh.rho, inv = sh.inv, sy = sh.sy;
    const bool ok = rho > 0.0;
    if (blockIdx.x == 0) {
      for (int i = t; i < k; i += kQrT)
        q.R[(long)i * k + w] = i < w ? sh.rprev[i] : (i == w ? rho : 0.0);
      if (t == 0) q.defic[w] = ok ? 0 : 1;
    }
    update(w, w, sh.tot, inv, y, sh.tot + j, sy);
    if (y >= 0)
      for (int i = t; i <= w; i += kQrT) sh.rprev[i] = i < w ? sh.tot[j + i] : sy;
    __syncthreads();
  }
  if (q.cs == 1) {
    for (int e = t; e < n * k; e += kQrT) q.T[at(e / k, e % k)] = slab[e / k * ld + e % k];
  } else {
    for (int e = t; e < n * k; e += kQrT) q.T[at(e % n, e / n)] = slab[e % n * ld + e / n];
  }
  if (t == 0 && q.nclus > 1) {  // the last CTA leaves the barrier as it found it
    __threadfence();
    if (atomicAdd(q.bar + 1, 1u) == gridDim.x - 1) {
      q.bar[0] = 0;
      q.bar[1] = 0;
    }
  }
  cg::this_cluster().sync();  // no CTA leaves while another may read its shared memory
}

int grid1(long n) { return (int)std::max<long>(1, std::min<long>((n + 255) / 256, 4096)); }

}  // namespace

static void qr_complete(attn_ctx* ctx, double* At, long M, int k, const std::vector<int>& hdef, double* part);

void qr_columns(attn_ctx* ctx, double* At, long M, int k, double* R, QRWork& w) {
  ATTN_REQUIRE(k >= 1 && M >= k, ATTN_EINVAL, "QR needs M >= k >= 1 (link wider than its other side)");
  const int nb = (int)((M + QROWS - 1) / QROWS);
  const int stride = k;
  w.part.reserve(sizeof(double) * ((size_t)nb * k + 16));
  w.part2.reserve(sizeof(double) * ((size_t)nb * k + 16));
  w.nrm0.reserve(sizeof(double) * k);
  w.defic.reserve(sizeof(int) * k);
  double* part = w.part.as<double>();
  double* part2 = w.part2.as<double>();
  double* nrm0 = w.nrm0.as<double>();
  int* def = w.defic.as<int>();
  cudaStream_t s = ctx->stream;
  qr_init_kernel<<<k, QT, 0, s>>>(At, M, k, nrm0, R);
  ctx->launches++;
  const size_t hsh = sizeof(double) * k;
  for (int j = 0; j < k; ++j) {
    if (j > 0) {
      qr_dots_kernel<<<nb, QT, 0, s>>>(At, M, j, part, stride);
      qr_update_kernel<<<nb, QT, hsh, s>>>(At, M, j, k, part, nb, stride, R, 0, part2);
      qr_update_kernel<<<nb, QT, hsh, s>>>(At, M, j, k, part2, nb, stride, R, 1, part);
      ctx->launches += 3;
    } else {
      qr_norm_partial_kernel<<<nb, QT, 0, s>>>(At, M, j, part);
      ctx->launches++;
    }
    qr_finalise_kernel<<<nb, QT, 0, s>>>(At, M, j, k, part, nb, nrm0, R, def);
    ctx->launches++;
  }
  ATTN_CHECK_CUDA(cudaGetLastError());
  // rank-deficient columns (rare): host check, one small sync
  std::vector<int> hdef(k);
  ATTN_CHECK_CUDA(cudaMemcpyAsync(hdef.data(), def, sizeof(int) * k, cudaMemcpyDeviceToHost, s));
  ATTN_CHECK_CUDA(cudaStreamSynchronize(s));
  qr_complete(ctx, At, M, k, hdef, part);
}

// Replaces the rank-deficient columns of At by unit vectors orthogonalised against the others.
static void qr_complete(attn_ctx* ctx, double* At, long M, int k, const std::vector<int>& hdef, double* part) {
  cudaStream_t s = ctx->stream;
  const size_t hsh = sizeof(double) * k;
  for (int j = 0; j < k; ++j) {
    if (!hdef[j]) continue;
    bool ok = false;
    for (long trial = 0; trial < std::min<long>(M, 64) && !ok; ++trial) {
      long t = ((long)j * 7919 + trial * 104729) % M;
      qr_set_unit_kernel<<<grid1(M), 256, 0, s>>>(At, M, j, t);
      qr_fix_column_kernel<<<1, QT, hsh, s>>>(At, M, j, k, part);
      ctx->launches += 2;
      double nrm = 0;
      ATTN_CHECK_CUDA(cudaMemcpyAsync(&nrm, part, sizeof(double), cudaMemcpyDeviceToHost, s));
      ATTN_CHECK_CUDA(cudaStreamSynchronize(s));
      ok = nrm > 0.5;
    }
    ATTN_REQUIRE(ok, ATTN_ENOTISOMETRIC, "QR could not complete a rank-deficient column");
  }
}

void qr_tensor(attn_ctx* ctx, double* T, const int d[3], int slot, double* R, QRWork& w) {
  const long V = (long)d[0] * d[1] * d[2];
  const int k = d[slot];
  const long M = V / std::max(k, 1);
  ATTN_REQUIRE(k >= 1 && M >= k, ATTN_EINVAL, "QR needs M >= k >= 1 (link wider than its other side)");
  QrSlab q;
  q.ld = k | 1;
  constexpr size_t kSmemMax = 200 * 1024;
  static PerDevice clusters;  // that are resident together with a full slab per SM
  const int most = clusters.get(current_device(), [] {
    ATTN_CHECK_CUDA(cudaFuncSetAttribute(qr_slab_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(kQrC);
    c.blockDim = dim3(kQrT);
    c.dynamicSmemBytes = kSmemMax;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kQrC;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    c.attrs = &attr;
    c.numAttrs = 1;
    int nc = 0;
    ATTN_CHECK_CUDA(cudaOccupancyMaxActiveClusters(&nc, qr_slab_kernel, &c));
    return std::max(nc, 1);
  });
  // Clusters by the cycles of a column: rows x k FP64 FMAs at two per cycle on the busiest SM
  // (both passes, both products), the cluster barriers and, with more than one cluster, the grid
  // barrier and the sums over the clusters (measured around 3 us).
  double best = 0.0;
  int nclus = 0;
  for (int c = 1; c <= most; ++c) {
    const long rows = (M + (long)c * kQrC - 1) / ((long)c * kQrC);
    if (rows > kQrT || sizeof(double) * rows * q.ld > kSmemMax || k > kQrMaxK) continue;
    const double cost = (double)rows * k + 1500.0 + (c > 1 ? 6000.0 + 20.0 * c : 0.0);
    if (!nclus || cost < best) {
      best = cost;
      nclus = c;
    }
  }
  if (!nclus) {
    w.cols.reserve(sizeof(double) * V);
    tensor_to_columns(ctx, T, d, slot, w.cols.as<double>());
    qr_columns(ctx, w.cols.as<double>(), M, k, R, w);
    columns_to_tensor(ctx, w.cols.as<double>(), d, slot, T);
    return;
  }
  q.T = T;
  q.M = (int)M;
  q.k = k;
  q.nclus = nclus;
  q.rows = (int)((M + (long)nclus * kQrC - 1) / ((long)nclus * kQrC));
  const long d1 = d[1], d2 = d[2];
  if (slot == 0) { q.rlo = d[2]; q.rs_hi = d2; q.rs_lo = 1; q.cs = d1 * d2; }
  else if (slot == 1) { q.rlo = d[2]; q.rs_hi = d1 * d2; q.rs_lo = 1; q.cs = d2; }
  else { q.rlo = d[1]; q.rs_hi = d1 * d2; q.rs_lo = d2; q.cs = 1; }
  q.R = R;
  w.defic.reserve(sizeof(int) * (kQrMaxK + 1));
  w.part.reserve(sizeof(double) * ((size_t)2 * most * 2 * kQrMaxK + 16));
  if (!w.bar_init) {
    w.bar.reserve(2 * sizeof(unsigned));
    ATTN_CHECK_CUDA(cudaMemsetAsync(w.bar.p, 0, 2 * sizeof(unsigned), ctx->stream));
    w.bar_init = true;
  }
  q.defic = w.defic.as<int>();
  q.part = w.part.as<double>();
  q.bar = w.bar.as<unsigned>();
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)(nclus * kQrC));
  c.blockDim = dim3(kQrT);
  c.dynamicSmemBytes = sizeof(double) * (size_t)q.rows * q.ld;
  c.stream = ctx->stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kQrC;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  c.attrs = attr;
  c.numAttrs = nclus > 1 ? 2 : 1;
  ATTN_CHECK_CUDA(cudaLaunchKernelEx(&c, qr_slab_kernel, q));
  ctx->launches++;
  // rank-deficient columns (rare) and a wait that gave up: host check, one small sync
  std::vector<int> hdef(k + 1);
  ATTN_CHECK_CUDA(cudaMemcpyAsync(hdef.data(), q.defic, sizeof(int) * (k + 1), cudaMemcpyDeviceToHost, ctx->stream));
  ATTN_CHECK_CUDA(cudaStreamSynchronize(ctx->stream));
  if (hdef[k]) {
    w.bar_init = false;
    throw Error{ATTN_ETIMEOUT, "a bounded wait in the QR kernel gave up"};
  }
  hdef.pop_back();
  if (std::any_of(hdef.begin(), hdef.end(), [](int v) { return v != 0; })) {
    w.cols.reserve(sizeof(double) * V);
    tensor_to_columns(ctx, T, d, slot, w.cols.as<double>());
    qr_complete(ctx, w.cols.as<double>(), M, k, hdef, w.part.as<double>());
    columns_to_tensor(ctx, w.cols.as<double>(), d, slot, T);
  }
}

void tensor_to_columns(attn_ctx* ctx, const double* T, const int d[3], int slot, double* At) {
  long V = (long)d[0] * d[1] * d[2];
  to_columns_kernel<<<grid1(V), 256, 0, ctx->stream>>>(T, d[0], d[1], d[2], slot, At);
  ctx->launches++;
  ATTN_CHECK_CUDA(cudaGetLastError());
}

void columns_to_tensor(attn_ctx* ctx, const double* At, const int d[3], int slot, double* T) {
  long V = (long)d[0] * d[1] * d[2];
  from_columns_kernel<<<grid1(V), 256, 0, ctx->stream>>>(At, d[0], d[1], d[2], slot, T);
  ctx->launches++;
  ATTN_CHECK_CUDA(cudaGetLastError());
}

}  // namespace attn
