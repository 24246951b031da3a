// Interface between the direct path's host side (direct.cu) and its kernel
// instances (direct_inst.cu, compiled once per family).
#pragma once

#include "internal.h"

namespace gbg {

// How an operand's elements are read (direct_kernel.cuh, Operand).
enum LoadMode { kRows = 0, kVec = 1, kScalar = 2 };

struct DirectArgs {
  const float* A; const float* B;
  int64_t lda, ldb, sa, sb;
  int64_t m, n, k;
  float alpha, beta;
  float* C; int64_t ldc, sc;
  int tiles_m, tiles_n;     // tiles of 128 rows (PAIR: 256) x BN columns
  int nkc, slices, slice_chunks;
  int cluster_slices;       // slices that reduce in the cluster (slices, or 1)
  float* partial;           // slices beyond a cluster: raw 128 x BN tiles ...
  int* partial_exp;         // ... and their exponents (kDirectExpInts)
  int* status;
};

// CTAs of a plan's clusters.
inline int direct_cluster_ctas(const DirectPlan& plan) {
  return (plan.in_cluster ? plan.slices : 1) * (plan.pair ? 2 : 1);
}

template <int PARTS, int MA>
cudaError_t launch_direct_mode(const DirectPlan& plan, int mb, const DirectArgs& S, int64_t items, cudaStream_t s);
// Whether the device can hold a cluster of the plan's instance.
template <int PARTS, int MA>
bool direct_mode_fits(const DirectPlan& plan, int mb);

}  // namespace gbg
