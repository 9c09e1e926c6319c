// Neighbour lists whose entries carry their matrix element: the step kernel for
// models with many coupling values and for spins above 1/2, where an
// amplitude per bond and state would otherwise be recomputed by every lane of
// every state at every step.
//
// Entry 0 of a state's list is (count, diagonal of 2(H - b)/a, 2M), the others
// (first chunk of the neighbour's row, matrix element of 2H/a): a matrix
// element is two words, high and low limb in fixed point (FxCoef) or the
// float pair hi + lo.  The first step (A = 1/a) halves the row's sum, which is exact
// for floats.  Lists are padded to whole batches with an all-zero row.
#pragma once

#include <algorithm>

#include "kpm_fixed.cuh"
#include "kpm_internal.h"

namespace kpm {

#ifndef KPM_WEIGHTED_BATCH
#define KPM_WEIGHTED_BATCH 4
#endif
constexpr int kWeightedBatch = KPM_WEIGHTED_BATCH;  // padding of the lists

// Above this size of the lists the matrix-free kernels are used.
constexpr uint64_t kWeightedMaxBytes = (uint64_t)32 << 30;

// Words of 16 bytes per state for at most `entries` neighbours.
inline int weighted_stride(int entries) {
  return 1 + (entries + kWeightedBatch - 1) / kWeightedBatch * kWeightedBatch;
}

struct WeightedRun {
  const uint4 *lists = nullptr;
  int stride = 0;
  const Tile *tiles = nullptr;
  const int32_t *tile_begin = nullptr, *tile_end = nullptr;
  int n_tiles = 0, n_sectors = 0;
  const double *scale = nullptr;  // fixed point: [n_sectors] 1 / (U^2 dim)
  int64_t unit = 0;               // fixed point: U
  int *flag = nullptr;
  RowLayout lay;
  bool full = false;              // M-weighted sums too
  bool exact_dots = false;        // FP32: dot products as if summed in FP64
};

// U for rows of at most `entries` neighbours: (entries + 1) 8 U <= 2^62 keeps the
// middle limbs of a row's sum, that and kFxMaxRow 2^59, below 2^63 (kpm_fixed.cuh).
inline int64_t weighted_unit(int entries) {
  return std::min<int64_t>((int64_t)1 << 54,
                           ((int64_t)1 << 62) / (kFxRange * ((int64_t)entries + 1))) - 1;
}

// Step kernel of a run (fixed point for KPM_FP64; at most two chunks per lane).
size_t weighted_smem(const WeightedRun &r);
void *weighted_kernel_ptr(const WeightedRun &r, int precision);
int launch_weighted_step(const WeightedRun &r, int precision, int grid, const void *x, void *zy,
                         int first, double *partials, const double *prev_partials,
                         double *prev_sums, int sum_parts, int *queue, int *next_queue, cudaStream_t s);

}  // namespace kpm
