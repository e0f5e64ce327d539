// FP64-accurate GEMM from exact BF16 slice products on the tensor cores (internal).
#pragma once

#include <cuda_bf16.h>

#include "attn_internal.h"

namespace attn {

// A strided FP64 operand seen as [batches][rows][K'] with K' = G K: entry
// (bh, bl, r, g K + k) at p + bh sBhi + bl sBlo + r sR + g sG + k sK.
struct OzView {
  const double* p = nullptr;
  long sR = 0, sK = 0, sG = 0, sBhi = 0, sBlo = 0;
  int rows = 0, K = 0, G = 1;
  int nbhi = 1, nblo = 1;  // distinct batch entries of this operand
  // K' in parts of kpart (a multiple of 64), each a batch entry bl with row exponents of its
  // own; 0: undivided. The last part may be shorter.
  long kpart = 0;
};

// Row exponents E (|entry| < 2^E per row; -2000 for a zero row) and six BF16 slices
// of 2^-E times each row (Kpad >= K G, a multiple of 64), stored tiled: per batch entry,
// tile of tile_rows rows and 64-wide K block, the six [tile_rows][64] slice blocks.
void ozaki_slice(attn_ctx* ctx, const OzView& v, long Kpad, int tile_rows, DevBuf& slices, DevBuf& exps);

// The same into memory of at least ozaki_slice_bytes and one int per row and batch
// (batch entries slice_stride slices' entries and exp_stride exponents apart).
void ozaki_slice_to(attn_ctx* ctx, const OzView& v, long Kpad, int tile_rows, __nv_bfloat16* slices, int* exps,
                    long slice_stride, long exp_stride);
size_t ozaki_slice_bytes(long batches, long rows, long Kpad, int tile_rows);

// C[s][j][i] = sum over K part s of P[i][k] Q[j][k] for an operand P of M rows sliced beforehand
// (ozaki_slice of a view in K parts, 128-row tiles) and a view Q in the same parts: one dense
// [Q.rows][M] matrix per part, to be added up; flops: what the profile records for it.
void gemm_f64_presliced(attn_ctx* ctx, const __nv_bfloat16* ps, const int* pe, int M, const OzView& q, double* C,
                        double flops);
// Part length for an M x N product over K: 4 to 16 K blocks, the fewest on the busiest SM. Short
// parts also keep the error down: what the scheme drops goes with the product of the row
// scales, and the largest of 1024 entries exceeds the typical one by less than that of 16384
// (error of an application at 128 on all links: 1.5e-13 with one part, see heff_dense.cu).
int oz_kparts(int M, int N, long K, int sms);

// The GemmF64 contraction C = alpha sum_g A_g B_g + beta C, computed from the
// slices' exact BF16 products (normwise error about (K + 2) 2^-46 of the row scales).
void gemm_f64_ozaki(attn_ctx* ctx, const GemmF64& g);

// Read and clear the split GEMM's device error word (0 = ok).
int ozaki_error(attn_ctx* ctx);

}  // namespace attn
