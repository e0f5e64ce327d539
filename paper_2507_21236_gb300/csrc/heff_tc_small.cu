// Pair products of an H_eff whose links are all at most 64, on the tcgen05 tensor cores: the
// same arithmetic as sandwich_tc_kernel (heff_tc.cu),
//     stage 1   D1 = B_r X_s^T,   Z = D1 rounded to the operand type,   stage 2   D2 += Z^T A_r^T,
// arranged for narrow matrices.
//
// What bounds products of this size is the chain stage 1 -> conversion -> stage 2, some thousand
// cycles a product whatever its width, and an MMA has 128 lanes whether 64 or 32 rows fill them. So
// a CTA takes several slices through the chain at once and fills the lanes with them:
//   * lanes are blocks of 64 (Q > 32) or 32 rows, one per slice: the operand of stage 1 is B_r
//     repeated down the 128 rows, its other operand the X of all slices side by side (N = up to 256),
//     so one group of MMAs computes every (lane block, slice) pair;
//   * the conversion takes from each lane block the columns of its own slice and packs them into
//     the same columns of Z, which leaves a full 128-lane operand;
//   * stage 2 multiplies that by A_r: one group of MMAs for two (or four) slices.
// Two such groups of slices share a stage 1 while N allows (four slices at 64, eight at 32). D1 is
// free again once the conversion has read it, so stage 1 of the next product overlaps stage 2 of this
// one; Z has two buffers in BF16 (FP32 Z of TF32 operands takes one).
// Tensor memory: D1 columns 0-255, Z 256-383, D2 384-511.
//
// A unit of work is a product and a set of slices; the units of all kinds are cut into equal runs, one
// per SM (persistent), outputs that two runs share meet by FP32 atomics. kPP: three-link products,
// where each product brings its own X. [64]^3 with 60 to 95 products per pair, TF32: 125 -> 41 us,
// [32]^3 with 45 to 70, BF16: 41 -> 11 us.
//
// Warp roles (384 threads): 0 = TMA producer, 1 = TMEM allocation and stage 1, 2 = stage 2, 4-11 =
// conversion and epilogue (four warps per group of slices). All waits are bounded; on a timeout
// the CTA records an error code, stops issuing, drains its copies and MMAs and frees TMEM.
#include <algorithm>

#include "heff.h"
#include "heff_tc_small.h"
#include "tc_ptx.h"

namespace attn {

namespace {

using namespace tc;

constexpr int kThreads = 384;
constexpr int kMaxStages = 7;
constexpr int kRowBytes = 128;  // one row of a K block
constexpr uint32_t kZ = 256, kD2 = 384;

struct SmMaps {
  CUtensorMap x[3], a[3], b[3];
};

template <bool kPP, bool kTF>
__global__ void __launch_bounds__(kThreads, 1) small_tc_kernel(const __grid_constant__ SmMaps maps,
                                                               const __grid_constant__ SmParams prm) {
  constexpr int KB = kTF ? 32 : 64;  // entries per 128-byte K block
  constexpr int KS = kTF ? 8 : 16;   // entries per MMA K step
  constexpr int NKB = kTF ? 2 : 1;   // K blocks of a 64-wide operand
  constexpr int kB = 128 * kRowBytes * NKB, kA = 64 * kRowBytes * NKB, kX = 256 * kRowBytes * NKB;
  constexpr int kStage = kB + kA + (kPP ? kX : 0);
  constexpr int NS = kPP ? (kTF ? 2 : 3) : (kTF ? 3 : 7);
  constexpr int NZ = kTF ? 1 : 2;    // Z buffers per group
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t sX = base, sRing = kPP ? base : base + kX, sBar = sRing + NS * kStage;
  enum {
    XFULL = 0,
    XEMPTY = 1,
    FULL = 2,
    EMPTY = FULL + kMaxStages,   // both issuers are done with a stage
    D1FULL = EMPTY + kMaxStages,
    D1EMPTY = D1FULL + 1,        // the conversion has read D1
    ZFULL = D1EMPTY + 1,         // [group][buffer]
    ZEMPTY = ZFULL + 4,          // [group][buffer]: stage 2 has read it
    D2FULL = ZEMPTY + 4,
    D2EMPTY = D2FULL + 1,
    DONE = D2EMPTY + 1,          // [issuer]: every MMA has completed
    NBAR = DONE + 2
  };
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + (sBar - base));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NBAR);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto bar = [&](int i) { return sBar + 8u * (uint32_t)i; };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the CTA's runs; static indices into the parameter struct keep it out of local memory
  const int s0 = prm.seg_start[blockIdx.x], nseg = prm.seg_start[blockIdx.x + 1] - s0;
  auto seg_at = [&](int j) { return prm.segs[s0 + j]; };  // {kind, slice set, first product, products | atomic << 30}
  auto kind_of = [&](int k) -> SmKind { return k == 0 ? prm.kind[0] : (k == 1 ? prm.kind[1] : prm.kind[2]); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < NBAR; ++i) {
      int count = 1;
      if (i >= EMPTY && i < EMPTY + kMaxStages) count = 2;
      if (i == D1EMPTY || i == D2EMPTY) count = 8;
      if (i >= ZFULL && i < ZFULL + 4) count = 4;
      mbar_init(bar(i), count);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---- producer: per run the X of its slices, per product B_r (once per lane block) and A_r
    int st = 0, issued = 0, xissued = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int j = 0; ok && j < nseg; ++j) {
      const int4 g = seg_at(j);
      const SmKind k = kind_of(g.x);
      const CUtensorMap *mX = &maps.x[g.x], *mA = &maps.a[g.x], *mB = &maps.b[g.x];
      const int n = g.w & 0x3FFFFFFF, nsl = k.nsl, first = g.y * nsl, rows = k.lb;
      const int nkbQ = (k.Q + KB - 1) / KB, nkbP = (k.P + KB - 1) / KB;
      const uint32_t xbytes = (uint32_t)(nsl * nkbQ * k.P * kRowBytes);
      const uint32_t bytes = (uint32_t)((128 * nkbQ + k.P * nkbP) * kRowBytes) + (kPP ? xbytes : 0u);
      if (!kPP) {
        if (j > 0 && !mbar_wait(bar(XEMPTY), (j - 1) & 1, prm.err, 81, abort_flag)) break;
        mbar_expect_tx(bar(XFULL), xbytes);
        for (int kb = 0; kb < nkbQ; ++kb)
          for (int u = 0; u < nsl; ++u)
            tma_load_3d(sX + (kb * nsl + u) * k.P * kRowBytes, mX, KB * kb, 0, first + u, bar(XFULL));
        ++xissued;
      }
      for (int r = g.z; r < g.z + n; ++r) {
        if (issued >= NS && !mbar_wait(bar(EMPTY + st), ph ^ 1u, prm.err, 82, abort_flag)) {
          ok = false;
          break;
        }
        mbar_expect_tx(bar(FULL + st), bytes);
        const uint32_t dst = sRing + st * kStage;
        for (int kb = 0; kb < nkbQ; ++kb)
          for (int b = 0; b < 128; b += rows)
            tma_load_3d(dst + (kb * 128 + b) * kRowBytes, mB, KB * kb, 0, r, bar(FULL + st));
        for (int kb = 0; kb < nkbP; ++kb) tma_load_3d(dst + kB + kb * k.P * kRowBytes, mA, KB * kb, 0, r, bar(FULL + st));
        if (kPP)
          for (int kb = 0; kb < nkbQ; ++kb)
            for (int u = 0; u < nsl; ++u)
              tma_load_3d(dst + kB + kA + (kb * nsl + u) * k.P * kRowBytes, mX, KB * kb, 0, r * k.S + first + u,
                          bar(FULL + st));
        ++issued;
        if (++st == NS) { st = 0; ph ^= 1u; }
      }
    }
    // drain: every issued copy must land before the CTA exits
    if (xissued > 0) {
      long long t0 = clock64();
      while (!mbar_try_wait(bar(XFULL), (xissued - 1) & 1) && clock64() - t0 < kWaitCycles) {}
    }
    for (int q = (issued > NS ? issued - NS : 0); q < issued; ++q) {
      long long t0 = clock64();
      while (!mbar_try_wait(bar(FULL + q % NS), (q / NS) & 1) && clock64() - t0 < kWaitCycles) {}
    }
  } else if (warp == 1 && lane == 0) {
    // ---- stage 1: D1[(lane block, j)][(slice, i')] = sum_j' B_r[j][j'] X_slice[i'][j']
    int st = 0, cnt = 0;
    uint32_t ph = 0;
    bool ok = true;
    const uint64_t dR0 = sw128_desc(sRing), dX0 = sw128_desc(sX);
    for (int j = 0; ok && j < nseg; ++j) {
      const int4 g = seg_at(j);
      const SmKind k = kind_of(g.x);
      const int n = g.w & 0x3FFFFFFF, steps = k.Q / KS;
      const uint32_t id = idesc_of<kTF>(128, k.nsl * k.P);
      const uint32_t xkb = (uint32_t)(k.nsl * k.P * kRowBytes) >> 4;  // to the next K block of X
      if (!kPP && !mbar_wait_limit(bar(XFULL), j & 1, prm.err, 83, abort_flag, prm.wait)) break;
      for (int r = 0; r < n; ++r, ++cnt) {
        if (!mbar_wait_limit(bar(FULL + st), ph, prm.err, 84, abort_flag, prm.wait) ||
            (cnt > 0 && !mbar_wait_limit(bar(D1EMPTY), (cnt - 1) & 1, prm.err, 85, abort_flag, prm.wait))) {
          ok = false;
          break;
        }
        fence_after();
        const uint64_t dB = dR0 + (uint64_t)((st * kStage) >> 4);
        const uint64_t dX = kPP ? dB + (uint64_t)((kB + kA) >> 4) : dX0;
        for (int s = 0; s < steps; ++s)
          mma_ss<kTF>(tmem, dB + (uint64_t)((s >> 2) * (128 * kRowBytes >> 4) + 2 * (s & 3)),
                      dX + (uint64_t)((s >> 2) * xkb + 2 * (s & 3)), id, s > 0 ? 1u : 0u);
        mma_commit(bar(D1FULL));
        mma_commit(bar(EMPTY + st));
        if (++st == NS) { st = 0; ph ^= 1u; }
      }
      if (ok && !kPP) mma_commit(bar(XEMPTY));
    }
    mma_commit(bar(DONE));
    long long t0 = clock64();
    while (!mbar_try_wait(bar(DONE), 0) && clock64() - t0 < kWaitCycles) {}
  } else if (warp == 2 && lane == 0) {
    // ---- stage 2: D2[group][(lane block, j)][i] += sum_i' Z[(lane block, j)][i'] A_r[i][i']
    int st = 0, zc[2] = {0, 0};  // products of each group so far
    uint32_t ph = 0;
    bool ok = true;
    const uint64_t dR0 = sw128_desc(sRing);
    for (int j = 0; ok && j < nseg; ++j) {
      const int4 g = seg_at(j);
      const SmKind k = kind_of(g.x);
      const int n = g.w & 0x3FFFFFFF, steps = k.P / KS;
      const uint32_t id = idesc_of<kTF>(128, k.P);
      const uint32_t akb = (uint32_t)(k.P * kRowBytes) >> 4;
      // the run's first MMAs restart D2: the epilogue must have read the last run's
      if (j > 0 && !mbar_wait_limit(bar(D2EMPTY), (j - 1) & 1, prm.err, 86, abort_flag, prm.wait)) break;
      for (int r = 0; ok && r < n; ++r) {
        if (!mbar_wait_limit(bar(FULL + st), ph, prm.err, 87, abort_flag, prm.wait)) {
          ok = false;
          break;
        }
        const uint64_t dA = dR0 + (uint64_t)((st * kStage + kB) >> 4);
        for (int gr = 0; gr < k.ngrp; ++gr) {
          const int zb = zc[gr] % NZ, zi = 2 * gr + zb;
          if (!mbar_wait_limit(bar(ZFULL + zi), (zc[gr] / NZ) & 1, prm.err, 88, abort_flag, prm.wait)) {
            ok = false;
            break;
          }
          fence_after();  // Z was written by tcgen05.st in other threads
          const uint32_t z = tmem + kZ + (kTF ? 64u * (uint32_t)gr : 32u * (uint32_t)zi);
          for (int s = 0; s < steps; ++s)
            mma_ts<kTF>(tmem + kD2 + 64u * (uint32_t)gr, z + 8u * (uint32_t)s,
                        dA + (uint64_t)((s >> 2) * akb + 2 * (s & 3)), id, (r > 0 || s > 0) ? 1u : 0u);
          mma_commit(bar(ZEMPTY + zi));
          ++zc[gr];
        }
        if (!ok) break;
        mma_commit(bar(EMPTY + st));
        if (++st == NS) { st = 0; ph ^= 1u; }
      }
      if (!ok) break;
      mma_commit(bar(D2FULL));
    }
    mma_commit(bar(DONE + 1));
    long long t0 = clock64();
    while (!mbar_try_wait(bar(DONE + 1), 0) && clock64() - t0 < kWaitCycles) {}
  } else if (warp >= 4) {
    // ---- conversion of group gr: warp q4 holds lanes 32 q4 .. + 31, whose lane block's slice it takes
    const int gr = (warp - 4) >> 2, q4 = warp & 3;
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    int cnt = 0, zc = 0;
    bool ok = true;
    for (int j = 0; ok && j < nseg; ++j) {
      const int4 g = seg_at(j);
      const SmKind k = kind_of(g.x);
      const int n = g.w & 0x3FFFFFFF, nblk = 128 / k.lb, blk = q4 * 32 / k.lb;
      const bool mine = gr < k.ngrp;
      const uint32_t src = tmem + lane_off + (uint32_t)((gr * nblk + blk) * k.P);
      for (int r = 0; r < n; ++r, ++cnt) {
        // warp-uniform: the TMEM accesses below are .sync.aligned
        if (!__all_sync(0xffffffffu, mbar_wait_limit(bar(D1FULL), cnt & 1, prm.err, 89, abort_flag, prm.wait))) {
          ok = false;
          break;
        }
        fence_after();
        if (!mine) {
          if (lane == 0) mbar_arrive(bar(D1EMPTY));
          continue;
        }
        const int zb = zc % NZ, zi = 2 * gr + zb;
        const uint32_t z = tmem + lane_off + kZ + (kTF ? 64u * (uint32_t)gr : 32u * (uint32_t)zi);
        uint32_t w[64];
        if (kTF) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float v[16];
            if (16 * c < k.P) tmem_ld16(src + 16 * c, v);
#pragma unroll
            for (int h = 0; h < 16; ++h) w[16 * c + h] = __float_as_uint(v[h]);
          }
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float v[16];
            if (16 * c < k.P) tmem_ld16(src + 16 * c, v);
#pragma unroll
            for (int h = 0; h < 8; ++h) {
              const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * h], v[2 * h + 1]);
              w[8 * c + h] = *reinterpret_cast<const uint32_t*>(&p);
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(D1EMPTY));
        if (zc >= NZ && !__all_sync(0xffffffffu, mbar_wait_limit(bar(ZEMPTY + zi), (zc / NZ - 1) & 1, prm.err, 90, abort_flag,
                                                                 prm.wait))) {
          ok = false;
          break;
        }
        fence_after();
        {
          uint32_t lo[32];
#pragma unroll
          for (int h = 0; h < 32; ++h) lo[h] = w[h];
          tmem_st32(z, lo);
        }
        if (kTF && k.P > 32) {
          uint32_t hi[32];
#pragma unroll
          for (int h = 0; h < 32; ++h) hi[h] = w[32 + h];
          tmem_st32(z + 32, hi);
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(ZFULL + zi));
        ++zc;
      }
      if (!ok) break;
      // the run's result; every warp takes part in the phases, whether it has columns or not
      if (!__all_sync(0xffffffffu, mbar_wait_limit(bar(D2FULL), j & 1, prm.err, 91, abort_flag, prm.wait))) break;
      fence_after();
      const int jl = (q4 * 32 + lane) % k.lb, s = g.y * k.nsl + gr * nblk + blk;
      if (mine) {
        const bool atomic = (g.w >> 30) & 1, in = jl < k.Q && s < k.S;
        float* yp = k.Y + (long)s * k.P * k.Q + jl;  // walks down column jl of Y_s
        for (int c0 = 0; c0 < k.P; c0 += 16) {
          float v[16];
          tmem_ld16(tmem + lane_off + kD2 + 64u * (uint32_t)gr + (uint32_t)c0, v);
          if (in) {
#pragma unroll
            for (int c = 0; c < 16; ++c) {
              if (atomic) atomicAdd(yp + (long)(c0 + c) * k.Q, v[c]);
              else yp[(long)(c0 + c) * k.Q] = v[c];
            }
          }
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(D2EMPTY));
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// 3-D map over [d2][d1][d0] operands with a {128 bytes, rows, 1} box (rows past d1 read zero).
void encode(CUtensorMap* map, const void* ptr, bool tf, int d0, int d1, int d2, int rows) {
  const int es = tf ? 4 : 2;
  cuuint64_t dims[3] = {(cuuint64_t)d0, (cuuint64_t)d1, (cuuint64_t)d2};
  cuuint64_t strides[2] = {(cuuint64_t)d0 * es, (cuuint64_t)d0 * d1 * es};
  cuuint32_t box[3] = {(cuuint32_t)(128 / es), (cuuint32_t)rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = tensor_map_encoder()(map, tf ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                                    const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  ATTN_REQUIRE(r == CUDA_SUCCESS, ATTN_ECUDA, "cuTensorMapEncodeTiled failed for a small H_eff operand");
}

size_t smem_of(bool pp, bool tf) {
  const size_t nkb = tf ? 2 : 1, kB = 128 * 128 * nkb, kA = 64 * 128 * nkb, kX = 256 * 128 * nkb;
  const size_t ns = pp ? (tf ? 2 : 3) : (tf ? 3 : 7);
  return 1024 + (pp ? 0 : kX) + ns * (kB + kA + (pp ? kX : 0)) + 512;
}

}  // namespace

struct SmallTc::Maps {
  SmMaps m;
};
SmallTc::SmallTc() : maps(new Maps) {}
SmallTc::~SmallTc() { delete maps; }

bool small_tc_fits(const attn_heff* h) { return h->m[0] <= 64 && h->m[1] <= 64 && h->m[2] <= 64; }

void SmallTc::add_kind(bool tf, int P, int Q, int S, int R, int nx, const void* x, const void* a, const void* b, float* y,
                       bool accumulate) {
  const int i = prm.nkinds++;
  SmKind& k = prm.kind[i];
  k.P = P;
  k.Q = Q;
  k.S = S;
  k.R = R;
  k.lb = Q <= 32 ? 32 : 64;
  const int blocks = 128 / k.lb;
  k.ngrp = 2 * blocks * P <= 256 ? 2 : 1;
  k.nsl = blocks * k.ngrp;
  k.Y = y;
  k.accumulate = accumulate ? 1 : 0;
  encode(&maps->m.x[i], x, tf, Q, P, nx, P);
  encode(&maps->m.a[i], a, tf, P, P, R, P);
  encode(&maps->m.b[i], b, tf, Q, Q, R, k.lb);
}

// Cuts the units (kind, slice set, product) into one run per SM of equal MMA work.
void SmallTc::cut(int sms, cudaStream_t st) {
  double total = 0.0;
  auto cost = [](const SmKind& k) { return 600.0 + k.Q * 8.0 + k.P * 4.0; };  // cycles of a product (chain and MMAs)
  for (int k = 0; k < prm.nkinds; ++k)
    total += (double)((prm.kind[k].S + prm.kind[k].nsl - 1) / prm.kind[k].nsl) * prm.kind[k].R * cost(prm.kind[k]);
  // a run of fewer than two products spends more on its X and its output than on them
  grid = (int)std::max(1.0, std::min<double>(sms, total / 2000.0));
  hsegs.clear();
  hstart.assign(grid + 1, 0);
  const double per = total / grid;
  double pos = 0.0;
  int cur = -1;
  shared = false;
  for (int k = 0; k < prm.nkinds; ++k) {
    const SmKind& kp = prm.kind[k];
    const double w = cost(kp);
    for (int set = 0; set < (kp.S + kp.nsl - 1) / kp.nsl; ++set) {
      const size_t first = hsegs.size();
      for (int r = 0; r < kp.R; ++r, pos += w) {
        const int c = std::min(grid - 1, (int)(pos / per));
        if (hsegs.size() > first && c == cur) {
          ++hsegs.back().w;
        } else {
          for (int cc = cur + 1; cc <= c; ++cc) hstart[cc] = (int)hsegs.size();
          hsegs.push_back(make_int4(k, set, r, 1));
          cur = c;
        }
      }
      if (hsegs.size() - first > 1 || kp.accumulate)
        for (size_t i = first; i < hsegs.size(); ++i) {
          hsegs[i].w |= 1 << 30;
          shared = true;
        }
    }
  }
  for (int cc = cur + 1; cc <= grid; ++cc) hstart[cc] = (int)hsegs.size();
  segs.reserve(sizeof(int4) * std::max<size_t>(hsegs.size(), 1));
  seg_start.reserve(sizeof(int) * hstart.size());
  ATTN_CHECK_CUDA(cudaMemcpyAsync(segs.p, hsegs.data(), sizeof(int4) * hsegs.size(), cudaMemcpyHostToDevice, st));
  ATTN_CHECK_CUDA(cudaMemcpyAsync(seg_start.p, hstart.data(), sizeof(int) * hstart.size(), cudaMemcpyHostToDevice, st));
  prm.segs = segs.as<int4>();
  prm.seg_start = seg_start.as<int>();
}

void SmallTc::launch(bool pp, bool tf, int* err, long long wait, cudaStream_t st) {
  prm.err = err;
  prm.wait = wait;
  static PerDevice attr;
  attr.get(current_device(), [] {
    ATTN_CHECK_CUDA(cudaFuncSetAttribute(small_tc_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(false, false)));
    ATTN_CHECK_CUDA(cudaFuncSetAttribute(small_tc_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(false, true)));
    ATTN_CHECK_CUDA(cudaFuncSetAttribute(small_tc_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(true, false)));
    ATTN_CHECK_CUDA(cudaFuncSetAttribute(small_tc_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(true, true)));
    return 1;
  });
  const size_t smem = smem_of(pp, tf);
  if (tf) {
    if (pp) small_tc_kernel<true, true><<<grid, kThreads, smem, st>>>(maps->m, prm);
    else small_tc_kernel<false, true><<<grid, kThreads, smem, st>>>(maps->m, prm);
  } else {
    if (pp) small_tc_kernel<true, false><<<grid, kThreads, smem, st>>>(maps->m, prm);
    else small_tc_kernel<false, false><<<grid, kThreads, smem, st>>>(maps->m, prm);
  }
}

}  // namespace attn
