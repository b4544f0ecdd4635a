// The cooperative solve kernel's interface (resident.cu).
#pragma once

#include "passes.cuh"

namespace pc {

constexpr int kResidentThreads = 512;         // one CTA per SM, up to 128 registers per thread
constexpr int kResidentSmem = 220 * 1024;   // dynamic shared memory (the arguments take 3 KB beside it)

struct ResidentArgs {
  PassArgs<float> pass[5];   // the passes of a solve (2 dim - 1), in order
  GridDev g;
  const void *s;             // the source the residuals read: (hi, lo) pairs or FP64
  float2 *p2;                // the iterate
  double *f64;               // p in FP64
  DevStats *st;
  unsigned *bar;             // arrivals and exits, zero at the start and at the end
  int tables_at;             // slots of shared memory before the tables
  int sweeps, adaptive, singular;
  int grid;                  // CTAs
  int cluster;               // the grid is one cluster (small grids), else a cooperative launch
  int row_tiles;             // row tiles per CTA (consecutive)
  int own_at;                // slots of shared memory before the own rows' planes
  float tol;
};

pc_status launch_resident(const ResidentArgs &R, int dim, bool pairs, size_t smem, cudaStream_t st);
pc_status prepare_resident();
// CTAs of the largest cluster the kernel runs as (16, else 8; 0: none).
int resident_cluster_size();

}  // namespace pc
