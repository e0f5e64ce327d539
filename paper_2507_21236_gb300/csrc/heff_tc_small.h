// Tensor-core pair products for links of at most 64 (internal).
#pragma once

#include <vector>

#include "attn_internal.h"

struct attn_heff;

namespace attn {

struct SmKind {
  int P, Q, S, R;  // slice rows and columns, slices, products
  int lb;          // lanes per slice (32 or 64)
  int ngrp, nsl;   // groups of slices sharing a stage 1, slices per unit
  float* Y;        // [S][P][Q] FP32 output
  int accumulate;  // add to Y instead of writing it
};
struct SmParams {
  SmKind kind[3];
  int nkinds = 0;
  int* err;
  long long wait;  // wait limit (cycles) of the MMA-issue, conversion and epilogue threads
  const int4* segs;  // {kind, slice set, first product, products | 1 << 30 when added atomically}
  const int* seg_start;
};

// One launch: kinds are added, the work is cut into runs, then it can be launched any number of times.
struct SmallTc {
  SmParams prm;
  struct Maps;
  Maps* maps;
  int grid = 0;
  bool shared = false;  // some output is added to atomically: zero the outputs first
  std::vector<int4> hsegs;
  std::vector<int> hstart;
  DevBuf segs, seg_start;
  SmallTc();
  SmallTc(const SmallTc&) = delete;
  SmallTc& operator=(const SmallTc&) = delete;
  ~SmallTc();
  // nx: slices of x (S, or products x S where each product has its own)
  void add_kind(bool tf, int P, int Q, int S, int R, int nx, const void* x, const void* a, const void* b, float* y,
                bool accumulate);
  void cut(int sms, cudaStream_t st);
  void launch(bool pp, bool tf, int* err, long long wait, cudaStream_t st);
};

bool small_tc_fits(const attn_heff* h);

}  // namespace attn
