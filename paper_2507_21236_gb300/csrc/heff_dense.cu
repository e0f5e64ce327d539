// H_eff applied through one dense operator per link pair (Sec. 3.3.2: the products of a
// node summed before they meet the tensor).
//
// The pair products of kind (p, q) act on the joint index of two links only, so their sum
//     M[(i, j)][(i', j')] = sum_r A_r[i][i'] B_r[j][j']   (+ H_p[i][i'] delta_jj' + delta_ii' H_q[j][j'])
// is one PQ x PQ matrix, and an application to a tensor with S slices costs 2 (PQ)^2 S
// operations instead of 2 R (P + Q) PQ S: less as soon as R > PQ / (P + Q) products share the
// pair (64 at 128 x 128; the nodes of the 8x8 to 32x32 lattices have 50 to 300). Making M
// costs 2 R (PQ)^2, about half of one product-by-product application, once per H_eff.
//
// FP64 on the CUDA cores. This GPU executes two FP64 FMAs per SM and cycle, so the number of
// FMAs decides (M streams from L2 or HBM far below their rates), and a simple kernel saturates
// it: every CTA owns a block of y and adds the contributions of all three pair kinds to it,
// in a fixed order, with no workspace and no second launch.
//
// With f64_split, M is held as its six BF16 slices (12 bytes per entry, written once), and an
// application is one split GEMM per kind instead of two with a 1 GiB intermediate that has to be
// sliced in between. Measured (GB300, one
// application): [64]^3 with 140 products per pair 25.4 -> 5.5 ms; [16]^3 with 12
// 128 -> 12 us, where the product-by-product path spends its time on 17 launches; f64_split at
// [128]^3 with 288: 42.3 -> 3.4 ms (first application, which makes the slices: 42.7 -> 21.5 ms),
// error against 64 bits 1.1e-13 -> 7.7e-14.
#include <algorithm>
#include <cmath>

#include "heff.h"
#include "heff_dense.h"
#include "ozaki.h"

namespace attn {

namespace {

// ---------------------------------------------------------------- the operators
struct PairOp {
  const double* a;   // [R][P][P]
  const double* b;   // [R][Q][Q]
  const double* hp;  // internal operator on slot p, or null
  const double* hq;
  double* m;         // [P Q][P Q]
  int P, Q, R;
  int tiles_n, tile0;  // column tiles, first tile of this kind
};
struct PairOps {
  PairOp k[3];
  int n;
};

// M as a P^2 x Q^2 GEMM over the products (rows (i, i'), columns (j, j')); both operand
// stacks are contiguous along the output index, so no transpose is needed. 64 x 64 tiles,
// 4 x 4 per thread, 16 products per step.
constexpr int kBT = 64, kBK = 16;
__global__ void __launch_bounds__(256) pair_operator_kernel(const PairOps ops) {
  __shared__ double As[kBK][kBT], Bs[kBK][kBT];
  int ki = 0;
  if (ops.n > 1 && (int)blockIdx.x >= ops.k[1].tile0) ki = 1;
  if (ops.n > 2 && (int)blockIdx.x >= ops.k[2].tile0) ki = 2;
  const PairOp o = ki == 0 ? ops.k[0] : (ki == 1 ? ops.k[1] : ops.k[2]);
  const int t = blockIdx.x - o.tile0;
  const int P2 = o.P * o.P, Q2 = o.Q * o.Q;
  const int i0 = (t / o.tiles_n) * kBT, j0 = (t % o.tiles_n) * kBT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  for (int r0 = 0; r0 < o.R; r0 += kBK) {
#pragma unroll
    for (int q = 0; q < kBK * kBT / 256; ++q) {
      const int e = threadIdx.x + 256 * q, c = e & (kBT - 1), r = r0 + (e >> 6);
      As[e >> 6][c] = (r < o.R && i0 + c < P2) ? o.a[(long)r * P2 + i0 + c] : 0.0;
      Bs[e >> 6][c] = (r < o.R && j0 + c < Q2) ? o.b[(long)r * Q2 + j0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kBK; ++r) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[r][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[r][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  const long PQ = (long)o.P * o.Q;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int gi = i0 + ty + 16 * i;
    if (gi >= P2) continue;
    const int p = gi / o.P, pp = gi % o.P;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gj = j0 + tx + 16 * j;
      if (gj >= Q2) continue;
      const int q = gj / o.Q, qq = gj % o.Q;
      double v = acc[i][j];
      if (o.hp && q == qq) v += o.hp[gi];
      if (o.hq && p == pp) v += o.hq[gj];
      o.m[((long)p * o.Q + q) * PQ + (long)pp * o.Q + qq] = v;
    }
  }
}

// ---------------------------------------------------------------- the application
struct DenseApply {
  const double* m[3];  // dense operators per pair kind (null: none)
  const double* x;
  double* y;
  int d[3];
};

__device__ __forceinline__ void cp_async8(uint32_t dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

constexpr int kDT = 256;      // threads
constexpr int kDStages = 3;
constexpr int kDFoldK = 128;  // K entries summed before they join the total

// Shape of pair kind k in a TA x TB x TC block: rows (the block's extent along the pair,
// second link fastest) and columns (along the remaining link).
template <int TA, int TB, int TC, int k>
struct DenseKind {
  static constexpr int ROWS = k == 0 ? TA * TB : (k == 1 ? TA * TC : TB * TC);
  static constexpr int INNER = k == 0 ? TB : TC;
  static constexpr int COLS = k == 0 ? TC : (k == 1 ? TB : TA);
};

// One CTA: the TA x TB x TC block of y. Each kind is a small GEMM of the block's rows of M
// with x; blocks of fewer outputs than threads split every K step over G groups of threads,
// whose sums meet at the end in a fixed order. Each loading warp takes every eighth row, so a
// thread's rows are one pointer and one stride: with two warps per scheduler the integer work
// of a step, not its copies, was what a small block waited for (24.6 -> 16.4 us at [16]^3; with 128 K entries a step 12.3 us).
// HK: K entries per step and loading lane.
template <int TA, int TB, int TC, int HK>
struct DenseBlock {
  static constexpr int kDK = 32 * HK;     // K entries per step
  static constexpr int kDP = kDK + 1;     // padded row: the 32 rows a warp reads lie in different banks
  static constexpr int kDFold = kDFoldK / kDK;
  static constexpr int OUT = TA * TB * TC;
  static constexpr int G = OUT < kDT ? kDT / OUT : 1;    // thread groups over K
  static constexpr int PER = OUT < kDT ? 1 : OUT / kDT;  // outputs per thread
  static constexpr int R01 = TA * TB, R02 = TA * TC, R12 = TB * TC;
  static constexpr int RMAX = R01 > R02 ? (R01 > R12 ? R01 : R12) : (R02 > R12 ? R02 : R12);
  static constexpr int CMAX = TA > TB ? (TA > TC ? TA : TC) : (TB > TC ? TB : TC);
  static constexpr int STAGE = (RMAX + CMAX) * kDP;
  static_assert(R01 % 8 == 0 && R02 % 8 == 0 && R12 % 8 == 0 && 8 % TB == 0 && 8 % TC == 0 && CMAX <= 8,
                "eight loading warps share the rows and columns evenly");
  static_assert(OUT >= kDT ? OUT % kDT == 0 && kDT % R01 == 0 && kDT % R02 == 0 && kDT % R12 == 0 : kDT % OUT == 0,
                "outputs divide over the threads, with a thread's outputs in one row");

  const DenseApply& g;
  double* sm;
  int a0, b0, c0;  // block origin
  int K[3], n[3];  // reduction lengths and K steps of the kinds (0 steps: no operator)
  const double* mp[3];  // this thread's first row of M, at its K entry of step 0
  long mstride[3];      // to its next row (eight rows on)
  int live[3];          // how many of its rows are inside the tensor
  double acc[PER], tot[PER];

  __device__ DenseBlock(const DenseApply& g_, double* sm_) : g(g_), sm(sm_) {
    const int nb1 = (g.d[1] + TB - 1) / TB, nb2 = (g.d[2] + TC - 1) / TC;
    const int bid = blockIdx.x;
    a0 = bid / (nb1 * nb2) * TA;
    b0 = bid / nb2 % nb1 * TB;
    c0 = bid % nb2 * TC;
    setup<0>();
    setup<1>();
    setup<2>();
  }

  template <int k>
  __device__ void setup() {
    using D = DenseKind<TA, TB, TC, k>;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int outer0 = k == 2 ? b0 : a0, inner0 = k == 0 ? b0 : c0;
    const int no = k == 2 ? g.d[1] : g.d[0], ni = k == 0 ? g.d[1] : g.d[2];
    K[k] = no * ni;
    n[k] = g.m[k] ? (K[k] + kDK - 1) / kDK : 0;
    const int o = outer0 + w / D::INNER, i = inner0 + w % D::INNER;
    constexpr int step = 8 / D::INNER;  // links of the outer slot from one row to the next
    mp[k] = g.m[k] + ((long)o * ni + i) * K[k] + lane;
    mstride[k] = (long)step * ni * K[k];
    live[k] = i < ni && o < no ? min(D::ROWS / 8, (no - o + step - 1) / step) : 0;
  }

  static __device__ __forceinline__ void copy(double* dst, const double* src, bool in) {
    if (in) cp_async8((uint32_t)__cvta_generic_to_shared(dst), src);
    else *dst = 0.0;
  }

  // issue the copies of K step s of kind k into stage st
  template <int k>
  __device__ __forceinline__ void load(int s, int st) {
    using D = DenseKind<TA, TB, TC, k>;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = s * kDK;
    double* Ms = sm + st * STAGE + w * kDP + lane;
    double* Xs = sm + st * STAGE + RMAX * kDP;
    const double* src = mp[k] + k0;
    const int m1 = g.d[1], m2 = g.d[2];
#pragma unroll
    for (int h = 0; h < HK; ++h) {
      const int kg = k0 + 32 * h + lane;
      const bool kin = kg < K[k];
#pragma unroll
      for (int i = 0; i < D::ROWS / 8; ++i)
        copy(Ms + 8 * i * kDP + 32 * h, src + 32 * h + i * mstride[k], kin && i < live[k]);
      if (k > 0 && w < D::COLS) {
        if (k == 1) {
          const unsigned kp = (unsigned)kg / (unsigned)m2, kc = (unsigned)kg - kp * (unsigned)m2;
          copy(Xs + w * kDP + 32 * h + lane, g.x + ((long)kp * m1 + b0 + w) * m2 + kc, kin && b0 + w < m1);
        } else {
          copy(Xs + w * kDP + 32 * h + lane, g.x + (long)(a0 + w) * K[2] + kg, kin && a0 + w < g.d[0]);
        }
      }
    }
    if (k == 0) {  // x[k][c]: contiguous along the columns
#pragma unroll
      for (int e = threadIdx.x; e < D::COLS * kDK; e += kDT) {
        const int c = e % TC, kk = e / TC, ke = k0 + kk;
        copy(Xs + c * kDP + kk, g.x + (long)ke * m2 + c0 + c, ke < K[0] && c0 + c < m2);
      }
    }
  }
  // step `at` of the three kinds' steps in a row
  __device__ __forceinline__ void issue(int at, int st) {
    if (at < n[0]) load<0>(at, st);
    else if (at < n[0] + n[1]) load<1>(at - n[0], st);
    else if (at < n[0] + n[1] + n[2]) load<2>(at - n[0] - n[1], st);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }

  // all steps of kind k, the first being step `at` of the whole; adds its outputs to ysum
  template <int k>
  __device__ __forceinline__ void run(int& at, int& st, double* ysum) {
    using D = DenseKind<TA, TB, TC, k>;
    const int grp = G > 1 ? threadIdx.x / OUT : 0, o = G > 1 ? threadIdx.x % OUT : threadIdx.x;
    const int row = o % D::ROWS, col = o / D::ROWS;
    constexpr int CSTEP = PER > 1 ? kDT / D::ROWS : 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) acc[j] = tot[j] = 0.0;
    for (int s = 0; s < n[k]; ++s, ++at) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kDStages - 2) : "memory");
      __syncthreads();
      issue(at + kDStages - 1, st == 0 ? kDStages - 1 : st - 1);
      const double* mr = sm + st * STAGE + row * kDP + grp;
      const double* xc = sm + st * STAGE + RMAX * kDP + col * kDP + grp;
#pragma unroll
      for (int q = 0; q < kDK; q += G) {
        const double mv = mr[q];
#pragma unroll
        for (int j = 0; j < PER; ++j) acc[j] = fma(mv, xc[j * CSTEP * kDP + q], acc[j]);
      }
      // sums run over kDFoldK entries before they join the total, so that rounding grows with
      // the root of that many terms and not of the whole row of M
      if (s % kDFold == kDFold - 1) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
          tot[j] += acc[j];
          acc[j] = 0.0;
        }
      }
      st = st == kDStages - 1 ? 0 : st + 1;
    }
    if (n[k] == 0) return;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int cj = col + j * CSTEP, ro = row / D::INNER, ri = row % D::INNER;
      const int a = k == 2 ? cj : ro, b = k == 0 ? ri : (k == 1 ? cj : ro), c = k == 0 ? cj : ri;
      ysum[grp * OUT + (a * TB + b) * TC + c] += tot[j] + acc[j];
    }
    __syncthreads();  // the next kind's outputs belong to other threads
  }
};

template <int TA, int TB, int TC, int HK>
__global__ void __launch_bounds__(kDT) dense_apply_kernel(const __grid_constant__ DenseApply g) {
  using B = DenseBlock<TA, TB, TC, HK>;
  extern __shared__ double sm[];
  double* ysum = sm + kDStages * B::STAGE;  // [G][OUT]
  B blk(g, sm);
  for (int e = threadIdx.x; e < B::G * B::OUT; e += kDT) ysum[e] = 0.0;
#pragma unroll
  for (int i = 0; i < kDStages - 1; ++i) blk.issue(i, i);
  int at = 0, st = 0;
  blk.template run<0>(at, st, ysum);
  blk.template run<1>(at, st, ysum);
  blk.template run<2>(at, st, ysum);
  __syncthreads();
  for (int o = threadIdx.x; o < B::OUT; o += kDT) {
    double v = ysum[o];
#pragma unroll
    for (int q = 1; q < B::G; ++q) v += ysum[q * B::OUT + o];
    const int a = blk.a0 + o / (TB * TC), b = blk.b0 + o / TC % TB, c = blk.c0 + o % TC;
    if (a < g.d[0] && b < g.d[1] && c < g.d[2]) g.y[((long)a * g.d[1] + b) * g.d[2] + c] = v;
  }
}

template <int TA, int TB, int TC, int HK>
void launch_dense(cudaStream_t st, const DenseApply& g) {
  using B = DenseBlock<TA, TB, TC, HK>;
  constexpr size_t smem = sizeof(double) * (kDStages * B::STAGE + B::G * B::OUT);
  static PerDevice attr;
  attr.get(current_device(), [] {
    ATTN_CHECK_CUDA(cudaFuncSetAttribute(dense_apply_kernel<TA, TB, TC, HK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem));
    return 1;
  });
  const long blocks = (long)((g.d[0] + TA - 1) / TA) * ((g.d[1] + TB - 1) / TB) * ((g.d[2] + TC - 1) / TC);
  dense_apply_kernel<TA, TB, TC, HK><<<(unsigned)blocks, kDT, smem, st>>>(g);
}

// What the choices below weigh: the FP64 FMA rate that the kernels reach, a dependent launch
// and a device allocation (measured: 1.11 TFLOP/s at [64]^3, about 4 us and 50 us).
constexpr double kF64Rate = 1.1e12, kLaunch = 4e-6, kAlloc = 5e-5;

}  // namespace

// Device memory for dense operators: at most a sixteenth of the GPU per context and, for more
// than 64 MB at once, at most a quarter of what is free, so that programs with many handles or
// a pool of their own keep the product-by-product path instead of running out. False when
// there is no room: beyond these limits buf stays what it was, counted, for smaller operators of
// the same handle (a sweep's next node); where the allocation fails it is empty and not counted.
bool dense_reserve(attn_ctx* ctx, DevBuf& buf, size_t n, size_t& counted) {
  if (n <= buf.bytes) return true;
  bool ok = ctx->dense_bytes - counted + n <= ctx->total_mem / 16;
  if (ok && n > (64u << 20)) {
    size_t fr = 0, total = 0;
    ok = cudaMemGetInfo(&fr, &total) == cudaSuccess && n <= fr / 4 + buf.bytes;
    (void)cudaGetLastError();
  }
  if (!ok) return false;
  ctx->dense_bytes -= counted;
  counted = 0;
  try {
    buf.reserve(n);
  } catch (const Error& e) {
    if (e.status != ATTN_ENOMEM) throw;
    return false;
  }
  counted = buf.bytes;
  ctx->dense_bytes += counted;
  return true;
}

bool stream_capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
    (void)cudaGetLastError();
    return true;
  }
  return cs != cudaStreamCaptureStatusNone;
}

DenseF64::~DenseF64() {
  if (ctx) ctx->dense_bytes -= bytes;
}
DenseSplit::~DenseSplit() {
  if (ctx) ctx->dense_bytes -= bytes;
}

// Which pair kinds are worth a dense operator for `uses` applications, and whether making
// them pays. Per kind: (PQ)^2 S against R (P + Q) PQ S operations, and the launches of the
// product path (per kind a mode product, a sum over products and its split, and a share of
// the fill and the internal operators).
static bool plan_dense(const attn_heff* h, double uses, bool (&use)[3]) {
  // A handle's dense operators also cost an allocation; one that a state keeps for its local steps
  // counts none, not even the first time: its choice must not depend on what the state did before,
  // so that a resumed run repeats the original's bits.
  double gain = 0.0, build = kLaunch + (h->kept ? 0.0 : kAlloc);
  bool any = false;
  for (int k = 0; k < 3; ++k) {
    const double P = h->m[kPairP[k]], Q = h->m[kPairQ[k]], S = h->m[kPairS[k]], R = h->npair[k];
    use[k] = false;
    if (h->npair[k] == 0) continue;
    const double direct = 2.0 * R * (P + Q) * P * Q * S / kF64Rate + 5 * kLaunch;
    const double dense = 2.0 * P * Q * P * Q * S / kF64Rate;
    const double make = 2.0 * R * P * P * Q * Q / kF64Rate;
    if (dense >= direct) continue;
    use[k] = true;
    any = true;
    gain += direct - dense;
    build += make;
  }
  return any && uses * gain >= build;
}

void dense_invalidate(attn_heff* h) {
  if (h->dense) h->dense->ready = false;
  if (h->dense_s) h->dense_s->ready = false;
  h->f64_uses = h->split_uses = 0;
  h->expect = 1;
}

void dense_release(attn_heff* h) {
  delete h->dense;
  delete h->dense_s;
  h->dense = nullptr;
  h->dense_s = nullptr;
}

// The dense FP64 operators of h, made when they pay for the applications so far plus the
// ones announced (h->expect); null when the product-by-product path is the cheaper one.
DenseF64* dense_f64(attn_heff* h) {
  attn_ctx* ctx = h->ctx;
  if (h->dense && h->dense->ready) return h->dense;
  // an application counts for itself and for those already made: a caller who comes back
  // will come back again
  const double uses = std::max<double>(h->expect, h->f64_uses > 0 ? 1 + 4.0 * h->f64_uses : 1.0);
  ++h->f64_uses;
  bool use[3];
  if (!plan_dense(h, uses, use) || stream_capturing(ctx->stream) || !h->f64_retry.due()) return nullptr;
  if (!h->dense) h->dense = new DenseF64();
  DenseF64* d = h->dense;
  d->ctx = ctx;
  size_t need = 0;
  for (int k = 0; k < 3; ++k) {
    const size_t pq = (size_t)h->m[kPairP[k]] * h->m[kPairQ[k]];
    d->at[k] = need;
    if (use[k]) need += pq * pq;
  }
  if (!dense_reserve(ctx, d->buf, sizeof(double) * need, d->bytes)) {
    h->f64_retry.failed();
    return nullptr;
  }
  h->f64_retry = DenseRetry();
  PairOps ops;
  ops.n = 0;
  int tiles = 0;
  bool hint_done[3] = {false, false, false};
  for (int k = 0; k < 3; ++k) {
    d->use[k] = use[k];
    if (!use[k]) continue;
    const int p = kPairP[k], q = kPairQ[k];
    PairOp& o = ops.k[ops.n++];
    o.P = h->m[p];
    o.Q = h->m[q];
    o.R = h->npair[k];
    o.a = h->pa[k].as<double>();
    o.b = h->pb[k].as<double>();
    o.m = d->m(k);
    // an internal operator joins the first dense kind that acts on its link
    o.hp = h->has_hint[p] && !hint_done[p] ? h->hint[p].as<double>() : nullptr;
    o.hq = h->has_hint[q] && !hint_done[q] ? h->hint[q].as<double>() : nullptr;
    hint_done[p] = hint_done[q] = true;
    o.tiles_n = (o.Q * o.Q + kBT - 1) / kBT;
    o.tile0 = tiles;
    tiles += o.tiles_n * ((o.P * o.P + kBT - 1) / kBT);
  }
  for (int s = 0; s < 3; ++s) d->hint[s] = hint_done[s];
  ctx->prof_begin(1);
  pair_operator_kernel<<<tiles, 256, 0, ctx->stream>>>(ops);
  ctx->prof_end(1, 0.0);
  ctx->launches++;
  ATTN_CHECK_CUDA(cudaGetLastError());
  d->ready = true;
  return d;
}

// Algorithmic FLOPs that one application through the sum of kind k stands for: its products one by one
// (2 m_l V per operator), and with the first such kind the internal operators in the sums.
static double products_flops(const attn_heff* h, int k, const bool (&use)[3], const bool (&hint)[3]) {
  double fl = 2.0 * h->npair[k] * (h->m[kPairP[k]] + h->m[kPairQ[k]]) * h->V;
  for (int q = 0; q < k; ++q)
    if (use[q]) return fl;
  for (int s = 0; s < 3; ++s)
    if (hint[s] && h->has_hint[s]) fl += 2.0 * h->m[s] * h->V;
  return fl;
}

// y = (dense kinds) x; every entry of y is written.
void dense_apply_f64(attn_heff* h, const DenseF64* d, const double* x, double* y) {
  attn_ctx* ctx = h->ctx;
  DenseApply g;
  double fl = 0.0;
  for (int k = 0; k < 3; ++k) {
    g.m[k] = d->use[k] ? d->m(k) : nullptr;
    if (d->use[k]) fl += products_flops(h, k, d->use, d->hint);
    g.d[k] = h->m[k];
  }
  g.x = x;
  g.y = y;
  // Block of y by the outputs that the busiest SM computes (FP64 FMAs bound the kernel), weighted by
  // what a block shape loses to its loads, and K steps of 128 where they are not much padding, 64
  // otherwise; measured at 8 to 96 on all links, where the rule takes the fastest or one within 5 %
  // (16: 12.4 us against 16.5 with steps of 32; 32: 200 against 232; 64: 5.46 ms against 5.67).
  const long sms = std::max(ctx->num_sms, 1);
  const int* m = h->m;
  auto cost = [&](int ta, int tb, int tc, double weight) {
    const long blocks = (long)((m[0] + ta - 1) / ta) * ((m[1] + tb - 1) / tb) * ((m[2] + tc - 1) / tc);
    return weight * (double)((blocks + sms - 1) / sms * (ta * tb * tc));
  };
  const double c[3] = {cost(4, 4, 8, 1.0), cost(4, 4, 4, 1.01), cost(4, 4, 2, 1.06)};
  const int best = (int)(std::min_element(c, c + 3) - c);
  long K = 0, padded = 0;
  for (int k = 0; k < 3; ++k)
    if (g.m[k]) {
      const long pq = (long)m[kPairP[k]] * m[kPairQ[k]];
      K += pq;
      padded += (pq + 127) / 128 * 128;
    }
  const bool wide = 10 * padded <= 11 * K;
  ctx->prof_begin(1);
  if (best == 0) launch_dense<4, 4, 8, 2>(ctx->stream, g);
  else if (best == 1 && wide) launch_dense<4, 4, 4, 4>(ctx->stream, g);
  else if (best == 1) launch_dense<4, 4, 4, 2>(ctx->stream, g);
  else if (wide) launch_dense<4, 4, 2, 4>(ctx->stream, g);
  else launch_dense<4, 4, 2, 2>(ctx->stream, g);
  ctx->prof_end(1, fl);
  ctx->launches++;
  ATTN_CHECK_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------- as BF16 slices
namespace {

// M += H_p (x) 1 and 1 (x) H_q (either may be null) on the rows r0 <= i Q + j < r1 that m
// holds; one thread per row, since both add to the row's diagonal entry.
__global__ void add_internal_kernel(double* m, int P, int Q, long r0, long r1, const double* hp, const double* hq) {
  const long PQ = (long)P * Q;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < r1 - r0; e += (long)gridDim.x * blockDim.x) {
    const int i = (int)((r0 + e) / Q), j = (int)((r0 + e) % Q);
    double* row = m + e * PQ;
    if (hp)
      for (int ii = 0; ii < P; ++ii) row[(long)ii * Q + j] += hp[(long)i * P + ii];
    if (hq)
      for (int jj = 0; jj < Q; ++jj) row[(long)i * Q + jj] += hq[(long)j * Q + jj];
  }
}

// y[a][b][c] = sum over the K parts of the kinds' outputs P01[c][(a, b)], P02[b][(a, c)],
// P12[a][(b, c)], in that order; 32 x 32 tiles of the (b, c) plane, the first through shared memory.
struct SplitParts {
  const double* p[3];
  int n[3];
};
__global__ void split_combine_kernel(double* __restrict__ y, int m0, int m1, int m2, const SplitParts s) {
  __shared__ double t[32][33];
  const long V = (long)m0 * m1 * m2;
  const int a = blockIdx.z, b0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  auto sum = [&](const double* p, int n, long at) {
    double v = p[at];
    int i = 1;
    for (; i + 4 <= n; i += 4) {  // four loads in flight
      const double a = p[at + i * V], b = p[at + (i + 1) * V], c = p[at + (i + 2) * V], d = p[at + (i + 3) * V];
      v = (((v + a) + b) + c) + d;
    }
    for (; i < n; ++i) v += p[at + i * V];
    return v;
  };
  if (s.n[0]) {
    for (int cc = threadIdx.y; cc < 32; cc += blockDim.y) {
      const int c = c0 + cc, b = b0 + threadIdx.x;
      if (b < m1 && c < m2) t[threadIdx.x][cc] = sum(s.p[0], s.n[0], ((long)c * m0 + a) * m1 + b);
    }
    __syncthreads();
  }
  for (int bb = threadIdx.y; bb < 32; bb += blockDim.y) {
    const int b = b0 + bb, c = c0 + threadIdx.x;
    if (b < m1 && c < m2) {
      double v = s.n[0] ? t[bb][threadIdx.x] : 0.0;
      if (s.n[1]) v += sum(s.p[1], s.n[1], ((long)b * m0 + a) * m2 + c);
      if (s.n[2]) v += sum(s.p[2], s.n[2], ((long)a * m1 + b) * m2 + c);
      y[((long)a * m1 + b) * m2 + c] = v;
    }
  }
}

// Times of the split path on this GPU (measured at 64 and 128 on all links): product by product
// 25 ps per intermediate entry and product (both GEMM stages, exponents and slicing of the
// intermediate), slices of M 20 ps per entry to make, 1.4 ps per entry and 64 slices to apply,
// and the launches of a kind; FP64 FMAs as above.
constexpr double kSplitProd = 25e-12, kSplitMake = 20e-12, kSplitUse = 1.4e-12, kSplitKind = 5e-5;
constexpr long kStage = 1L << 27;  // doubles of M made at a time (1 GiB)

// Rows of M made at a time: whole 128-row tiles within the stage, and where that goes whole values of the
// first link as well (one GEMM per stage). Where it does not (a second link with few factors of two:
// 113 x 113 would take all of M, 1.3 GB, 191 x 191 7 GB) tiles alone.
long stage_rows(int P, int Q) {
  const long PQ = (long)P * Q;
  int unit = 1;
  while (unit < 128 && (unit * Q) % 128) ++unit;
  const long step = std::max<long>(1, std::min<long>(P, kStage / (PQ * Q)) / unit) * unit;
  if (std::min<long>(step, P) * Q * PQ <= kStage) return step * Q;
  return std::max<long>(1, kStage / PQ / 128) * 128;
}

}  // namespace

DenseSplit* dense_split(attn_heff* h) {
  attn_ctx* ctx = h->ctx;
  if (h->dense_s && h->dense_s->ready) return h->dense_s;
  const double uses = std::max<double>(h->expect, h->split_uses > 0 ? 1 + 4.0 * h->split_uses : 1.0);
  ++h->split_uses;
  bool use[3], any = false;
  double gain = 0.0, build = 2e-4;  // and two allocations
  size_t need = 0, ne = 0, at[3], eat[3];
  int kpart[3] = {0, 0, 0};
  for (int k = 0; k < 3; ++k) {
    const double P = h->m[kPairP[k]], Q = h->m[kPairQ[k]], S = h->m[kPairS[k]], R = h->npair[k];
    const double direct = R * h->V * kSplitProd + kSplitKind;
    const double dense = P * Q * P * Q * std::ceil(S / 64.0) * kSplitUse + kSplitKind;
    at[k] = need;
    eat[k] = ne;
    // (a slice row has at most 65536 entries: the int64 sums of the split GEMM)
    use[k] = h->npair[k] > 0 && 2.0 * dense < direct && P * Q <= 65536.0 && P >= 16 && Q >= 16;
    if (!use[k]) continue;
    any = true;
    gain += direct - dense;
    build += P * Q * P * Q * kSplitMake * (1.0 + R / 600.0);
    const long pq = (long)P * (long)Q;
    kpart[k] = oz_kparts((int)pq, (int)S, pq, std::max(ctx->num_sms, 1));
    const long parts = (pq + kpart[k] - 1) / kpart[k];
    need += ozaki_slice_bytes(parts, pq, kpart[k], 128);
    ne += (size_t)(parts * pq);
  }
  if (!any || uses * gain < build || stream_capturing(ctx->stream) || !h->split_retry.due()) return nullptr;
  if (!h->dense_s) h->dense_s = new DenseSplit();
  DenseSplit* d = h->dense_s;
  d->ctx = ctx;
  if (!dense_reserve(ctx, d->slices, need, d->bytes)) {
    h->split_retry.failed();
    return nullptr;
  }
  bool hint_done[3] = {false, false, false};
  try {
    // all memory before any work
    d->exps.reserve(sizeof(int) * ne);
    size_t most = 0;
    for (int k = 0; k < 3; ++k) {
      const long P = h->m[kPairP[k]], Q = h->m[kPairQ[k]];
      if (use[k]) most = std::max(most, (size_t)(std::min(stage_rows((int)P, (int)Q), P * Q) * P * Q));
    }
    ctx->ws[0].reserve(sizeof(double) * most);
    double* stage = ctx->ws[0].as<double>();
    for (int k = 0; k < 3; ++k) {
      d->use[k] = use[k];
      d->at[k] = at[k];
      d->eat[k] = eat[k];
      d->kpart[k] = kpart[k];
      if (!use[k]) continue;
      const int p = kPairP[k], q = kPairQ[k], P = h->m[p], Q = h->m[q], R = h->npair[k];
      const long PQ = (long)P * Q, parts = (PQ + kpart[k] - 1) / kpart[k], tiles = (PQ + 127) / 128;
      const long part_slices = tiles * (kpart[k] / 64) * 6 * 128 * 64;
      const double* hp = h->has_hint[p] && !hint_done[p] ? h->hint[p].as<double>() : nullptr;
      const double* hq = h->has_hint[q] && !hint_done[q] ? h->hint[q].as<double>() : nullptr;
      hint_done[p] = hint_done[q] = true;
      const long rows = stage_rows(P, Q);
      for (long r0 = 0; r0 < PQ; r0 += rows) {
        const long r1 = std::min(PQ, r0 + rows);
        // M[(i, j)][(i', j')] = sum_r A_r[i][i'] B_r[j][j'], a batch entry per (i, j): all whole i at once,
        // the part of one at either end
        for (long r = r0; r < r1;) {
          const int i = (int)(r / Q), j = (int)(r % Q);
          const bool whole = j == 0 && r1 - r >= Q;
          GemmF64 g;
          g.split_ok = true;
          g.counted = false;
          g.M = P; g.N = Q; g.K = R;
          g.Bhi = whole ? (int)((r1 - r) / Q) : 1;
          g.Blo = whole ? Q : (int)std::min<long>(Q - j, r1 - r);
          g.A = h->pa[k].as<double>() + (long)i * P; g.aM = 1; g.aK = (long)P * P; g.aBhi = P;
          g.B = h->pb[k].as<double>() + (long)j * Q; g.bN = 1; g.bK = (long)Q * Q; g.bBlo = Q;
          g.C = stage + (r - r0) * PQ; g.cM = Q; g.cN = 1; g.cBhi = Q * PQ; g.cBlo = PQ;
          gemm_f64(ctx, g);
          r += (long)g.Bhi * g.Blo;
        }
        if (hp || hq) {
          add_internal_kernel<<<(int)std::min<long>((r1 - r0 + 127) / 128, 4096), 128, 0, ctx->stream>>>(stage, P, Q, r0, r1,
                                                                                                     hp, hq);
          ctx->launches++;
        }
        OzView v;
        v.p = stage;
        v.sR = PQ; v.sK = 1;
        v.rows = (int)(r1 - r0);
        v.K = (int)PQ;
        v.kpart = kpart[k];
        auto* s = reinterpret_cast<__nv_bfloat16*>(d->slices.as<uint8_t>() + at[k]) +
                  r0 / 128 * (kpart[k] / 64) * 6 * 128 * 64;
        v.nblo = (int)parts;
        ozaki_slice_to(ctx, v, kpart[k], 128, s, d->exps.as<int>() + eat[k] + r0, part_slices, PQ);
      }
    }
  } catch (const Error& e) {  // no memory for the exponents or the stage: product by product, as without M
    if (e.status != ATTN_ENOMEM) throw;
    d->slices.release();
    ctx->dense_bytes -= d->bytes;
    d->bytes = 0;
    h->split_retry.failed();
    return nullptr;
  }
  h->split_retry = DenseRetry();
  for (int s = 0; s < 3; ++s) d->hint[s] = hint_done[s];
  ATTN_CHECK_CUDA(cudaGetLastError());
  d->ready = true;
  return d;
}

void dense_apply_split(attn_heff* h, const DenseSplit* d, const double* x, double* y) {
  attn_ctx* ctx = h->ctx;
  const int m0 = h->m[0], m1 = h->m[1], m2 = h->m[2];
  SplitParts parts;
  size_t total = 0, off[3];
  for (int k = 0; k < 3; ++k) {
    const long pq = (long)h->m[kPairP[k]] * h->m[kPairQ[k]];
    parts.n[k] = d->use[k] ? (int)((pq + d->kpart[k] - 1) / d->kpart[k]) : 0;
    off[k] = total;
    total += (size_t)parts.n[k] * h->V;
  }
  ctx->ws[0].reserve(sizeof(double) * total);
  for (int k = 0; k < 3; ++k) {
    parts.p[k] = ctx->ws[0].as<double>() + off[k];
    if (!d->use[k]) continue;
    OzView q;  // x as [slice][K]: the slices of kind k along its third link
    q.p = x;
    q.rows = h->m[kPairS[k]];
    if (k == 0) { q.sR = 1; q.sK = m2; q.K = m0 * m1; }
    else if (k == 1) { q.sR = m2; q.sK = 1; q.K = m2; q.G = m0; q.sG = (long)m1 * m2; }
    else { q.sR = (long)m1 * m2; q.sK = 1; q.K = m1 * m2; }
    q.kpart = d->kpart[k];
    q.nblo = parts.n[k];
    const long pq = (long)h->m[kPairP[k]] * h->m[kPairQ[k]];
    gemm_f64_presliced(ctx, reinterpret_cast<const __nv_bfloat16*>(d->slices.as<uint8_t>() + d->at[k]),
                       d->exps.as<int>() + d->eat[k], (int)pq, q, ctx->ws[0].as<double>() + off[k],
                       products_flops(h, k, d->use, d->hint));
  }
  dim3 grid((m2 + 31) / 32, (m1 + 31) / 32, m0);
  split_combine_kernel<<<grid, dim3(32, 8), 0, ctx->stream>>>(y, m0, m1, m2, parts);
  ctx->launches++;
  ATTN_CHECK_CUDA(cudaGetLastError());
}

}  // namespace attn
