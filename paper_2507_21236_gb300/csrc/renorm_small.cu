// Renormalisation O_r = T^T (A_r (x) B_r) T of all products of a link in one launch, for
// tensors that fit one SM's shared memory (Sec. 3.3.2, Fig. eff-op).
//
// The lower layers of a tree have most of its links, and tensors of 16 to 4096 entries whose
// three contractions take microseconds: as gathers, mode products and a contraction per kind of
// product they were about 25 launches a link, and the launches were the time. Here a CTA takes one
// product and a block of output columns j: the columns of W = (A_r (x) B_r) T are independent, so
//     W[x, y, j] = sum A_r[x, x'] B_r[y, y'] T[x', y', j],   O[i, j] = sum_{x, y} T[x, y, i] W[x, y, j]
// stays in shared memory from T to O. The operators are read in place through the product list
// (a kernel argument), so nothing is gathered or uploaded. Products that end behind the link are
// summed in groups of four before their contraction; a second kernel adds the groups.
// H_eff build with all links of a 16x16, m = 64 tree (192 of 253 links are this small): 124 -> 107 ms,
// a 4x4, m = 16 sweep 31.7 -> 27.3 ms.
#include <algorithm>

#include "state.h"

namespace attn {

namespace {

constexpr int kMaxProducts = 448;  // per launch (kernel arguments hold 4 KB)
constexpr int kRT = 256;           // threads
constexpr int kGroup = 4;          // products per group of the internal operator
constexpr size_t kMaxSmem = 96 * 1024;

struct RenormSmall {
  const double* T;
  const double *A, *B;    // operator stacks of slots x and y
  const double *ha, *hb;  // their internal operators
  double* out;            // [n][dt][dt]
  double* part;           // [groups][dt][dt]
  long sx, sy, st;        // T element (ix, iy, it) at ix sx + iy sy + it st
  int dx, dy, dt, n, nc;  // nc products after the first n form the internal operator
  int jb;                 // output columns per CTA
  // stack entry of the product on x and on y; -1: identity, -2: the internal operator
  short a[kMaxProducts], b[kMaxProducts];
};

__global__ void __launch_bounds__(kRT) renorm_small_kernel(const __grid_constant__ RenormSmall q) {
  extern __shared__ double sm[];
  const int dx = q.dx, dy = q.dy, dt = q.dt, dxy = dx * dy, t = threadIdx.x;
  const int j0 = blockIdx.y * q.jb, jb = min(q.jb, dt - j0), cols = dxy * jb;
  double* Ts = sm;                // [dxy][dt]
  double* W1 = Ts + dxy * dt;     // [dxy][jb]
  double* W2 = W1 + dxy * q.jb;   // the same
  double* As = W2 + dxy * q.jb;   // operators of the product
  double* Bs = As + dx * dx;
  double* red = Bs + dy * dy;     // [kRT]
  for (int e = t; e < dxy * dt; e += kRT) {
    // consecutive threads along the tensor's unit stride
    int ix, iy, it;
    if (q.st == 1) { it = e % dt; iy = e / dt % dy; ix = e / dt / dy; }
    else { iy = e % dy; it = e / dy % dt; ix = e / dy / dt; }
    Ts[(ix * dy + iy) * dt + it] = q.T[ix * q.sx + iy * q.sy + it * q.st];
  }
  const bool own = (int)blockIdx.x < q.n;
  const int r0 = own ? blockIdx.x : q.n + (blockIdx.x - q.n) * kGroup;
  const int r1 = own ? r0 + 1 : min(r0 + kGroup, q.n + q.nc);
  for (int r = r0; r < r1; ++r) {
    const int a = q.a[r], b = q.b[r];
    const double* ap = a >= 0 ? q.A + (long)a * dx * dx : q.ha;
    const double* bp = b >= 0 ? q.B + (long)b * dy * dy : q.hb;
    __syncthreads();
    if (a != -1)
      for (int e = t; e < dx * dx; e += kRT) As[e] = ap[e];
    if (b != -1)
      for (int e = t; e < dy * dy; e += kRT) Bs[e] = bp[e];
    __syncthreads();
    for (int e = t; e < cols; e += kRT) {  // B_r on y
      const int j = e % jb, xy = e / jb, iy = xy % dy;
      double s;
      if (b == -1) {
        s = Ts[xy * dt + j0 + j];
      } else {
        const double* col = Ts + (xy - iy) * dt + j0 + j;
        const double* row = Bs + iy * dy;
        double s0 = 0.0, s1 = 0.0;
        int y = 0;
        for (; y + 2 <= dy; y += 2) {
          s0 = fma(row[y], col[y * dt], s0);
          s1 = fma(row[y + 1], col[(y + 1) * dt], s1);
        }
        if (y < dy) s0 = fma(row[y], col[y * dt], s0);
        s = s0 + s1;
      }
      W1[e] = s;
    }
    __syncthreads();
    for (int e = t; e < cols; e += kRT) {  // A_r on x
      double s;
      if (a == -1) {
        s = W1[e];
      } else {
        const int ix = e / (dy * jb);
        const double* col = W1 + (e - ix * dy * jb);
        const double* row = As + ix * dx;
        double s0 = 0.0, s1 = 0.0;
        int x = 0;
        for (; x + 2 <= dx; x += 2) {
          s0 = fma(row[x], col[x * dy * jb], s0);
          s1 = fma(row[x + 1], col[(x + 1) * dy * jb], s1);
        }
        if (x < dx) s0 = fma(row[x], col[x * dy * jb], s0);
        s = s0 + s1;
      }
      W2[e] = r > r0 ? W2[e] + s : s;
    }
  }
  __syncthreads();
  // O[i][j] over (x, y): P threads per output where there are fewer outputs than threads
  double* out = (own ? q.out + (long)blockIdx.x * dt * dt : q.part + (long)(blockIdx.x - q.n) * dt * dt) + j0;
  const int outs = dt * jb;
  int P = 1;
  while (2 * P * outs <= kRT) P *= 2;
  for (int e0 = 0; e0 < outs; e0 += kRT / P) {
    const int e = e0 + t / P, p = t % P;
    double s0 = 0.0, s1 = 0.0;
    if (e < outs && t / P < kRT / P) {
      const int i = e / jb, j = e % jb;
      int xy = p;
      for (; xy + P < dxy; xy += 2 * P) {
        s0 = fma(Ts[xy * dt + i], W2[xy * jb + j], s0);
        s1 = fma(Ts[(xy + P) * dt + i], W2[(xy + P) * jb + j], s1);
      }
      if (xy < dxy) s0 = fma(Ts[xy * dt + i], W2[xy * jb + j], s0);
    }
    red[t] = s0 + s1;
    __syncthreads();
    if (p == 0 && e < outs) {
      double s = red[t];
      for (int h = 1; h < P; ++h) s += red[t + h];
      out[(long)(e / jb) * dt + e % jb] = s;
    }
    __syncthreads();
  }
}

__global__ void renorm_groups_kernel(const double* part, int groups, int len, double* hint) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < len; e += gridDim.x * blockDim.x) {
    double s = part[e];
    for (int g = 1; g < groups; ++g) s += part[(long)g * len + e];
    hint[e] = s;
  }
}

size_t smem_of(int dx, int dy, int dt, int jb) {
  return sizeof(double) * ((size_t)dx * dy * dt + 2 * (size_t)dx * dy * jb + (size_t)dx * dx + (size_t)dy * dy + kRT);
}

}  // namespace

bool renorm_small_fits(const int d[3], int x, int y, int t) {
  return (long)d[0] * d[1] * d[2] <= 4096 && d[x] <= 32 && d[y] <= 32 && smem_of(d[x], d[y], d[t], 1) <= kMaxSmem;
}

void renorm_small(attn_ctx* ctx, const double* T, const int d[3], int t, int x, int y, const double* A, const double* B,
                  const double* ha, const double* hb, const std::vector<std::pair<int, int>>& open, double* out,
                  const std::vector<std::pair<int, int>>& closed, double* hint, DevBuf& part) {
  RenormSmall q;
  q.T = T;
  q.A = A;
  q.B = B;
  q.ha = ha;
  q.hb = hb;
  const long stride[3] = {(long)d[1] * d[2], d[2], 1};
  q.sx = stride[x];
  q.sy = stride[y];
  q.st = stride[t];
  q.dx = d[x];
  q.dy = d[y];
  q.dt = d[t];
  const long osz = (long)d[t] * d[t];
  const int groups_all = ((int)closed.size() + kGroup - 1) / kGroup;
  if (groups_all) part.reserve(sizeof(double) * groups_all * osz);
  static PerDevice attr;
  attr.get(current_device(), [] {
    ATTN_CHECK_CUDA(cudaFuncSetAttribute(renorm_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
    return 1;
  });
  size_t io = 0, ic = 0;
  int groups_done = 0;
  while (io < open.size() || ic < closed.size()) {
    q.out = out + (long)io * osz;
    q.part = part.as<double>() + (long)groups_done * osz;
    q.n = (int)std::min<size_t>(open.size() - io, kMaxProducts);
    for (int r = 0; r < q.n; ++r) {
      q.a[r] = (short)open[io + r].first;
      q.b[r] = (short)open[io + r].second;
    }
    io += q.n;
    // whole groups only, so that the order of the sums does not depend on the launches
    q.nc = (int)std::min<size_t>(closed.size() - ic, (kMaxProducts - q.n) / kGroup * kGroup);
    for (int r = 0; r < q.nc; ++r) {
      q.a[q.n + r] = (short)closed[ic + r].first;
      q.b[q.n + r] = (short)closed[ic + r].second;
    }
    ic += q.nc;
    const int groups = (q.nc + kGroup - 1) / kGroup;
    groups_done += groups;
    const int blocks = q.n + groups;
    if (!blocks) continue;
    // columns per CTA: enough CTAs for two per SM, one column at least
    const long want = 2L * std::max(ctx->num_sms, 1);
    q.jb = (int)std::max<long>(1, std::min<long>(q.dt, (long)blocks * q.dt / want));
    while (q.jb > 1 && smem_of(q.dx, q.dy, q.dt, q.jb) > kMaxSmem) --q.jb;
    const dim3 grid(blocks, (q.dt + q.jb - 1) / q.jb);
    renorm_small_kernel<<<grid, kRT, smem_of(q.dx, q.dy, q.dt, q.jb), ctx->stream>>>(q);
    ctx->launches++;
  }
  if (groups_all) {
    renorm_groups_kernel<<<(int)std::min<long>((osz + 255) / 256, 64), 256, 0, ctx->stream>>>(part.as<double>(), groups_all,
                                                                                          (int)osz, hint);
    ctx->launches++;
  }
  ATTN_CHECK_CUDA(cudaGetLastError());
}

}  // namespace attn
