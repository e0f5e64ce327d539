// One dense operator per link pair of an effective Hamiltonian (internal).
#pragma once

#include "attn_internal.h"

struct attn_heff;

namespace attn {

// FP64 operators M_k [P Q][P Q] of the pair kinds whose products are summed (use[k]), one
// after another in one buffer; hint[s]: the internal operator of slot s is part of one of them.
struct DenseF64 {
  attn_ctx* ctx = nullptr;
  DevBuf buf;
  size_t at[3] = {0, 0, 0};
  double* m(int k) const { return buf.as<double>() + at[k]; }
  bool use[3] = {false, false, false}, hint[3] = {false, false, false};
  bool ready = false;
  size_t bytes = 0;  // counted in ctx->dense_bytes
  ~DenseF64();
};

// The same operators as BF16 slices (ozaki.h) for applications with f64_split: six slices of each
// M_k in 128-row tiles and the row exponents, one kind after another.
struct DenseSplit {
  attn_ctx* ctx = nullptr;
  DevBuf slices, exps;
  size_t at[3] = {0, 0, 0}, eat[3] = {0, 0, 0};  // first slice byte and exponent of each kind
  int kpart[3] = {0, 0, 0};                      // entries of a row that share an exponent
  bool use[3] = {false, false, false}, hint[3] = {false, false, false};
  bool ready = false;
  size_t bytes = 0;
  ~DenseSplit();
};

// When to ask again for memory that was refused: at the next application the first three times, then
// after ever more of them (1, 2, 4 .. 64), since every attempt may allocate and free gigabytes.
struct DenseRetry {
  int refused = 0, wait = 0;
  bool due() {
    if (wait == 0) return true;
    --wait;
    return false;
  }
  void failed() {
    if (refused < 10) ++refused;
    wait = (1 << refused) / 16;
  }
};

// buf of at least n bytes within the context's share of device memory for dense operators;
// `counted` is what buf has in that count.
bool dense_reserve(attn_ctx* ctx, DevBuf& buf, size_t n, size_t& counted);
bool stream_capturing(cudaStream_t st);

DenseF64* dense_f64(attn_heff* h);
void dense_apply_f64(attn_heff* h, const DenseF64* d, const double* x, double* y);
// The slices, made when they pay; null when products (or FP64 FMAs) are the faster way.
DenseSplit* dense_split(attn_heff* h);
void dense_apply_split(attn_heff* h, const DenseSplit* d, const double* x, double* y);
void dense_invalidate(attn_heff* h);
void dense_release(attn_heff* h);

}  // namespace attn
