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
  unsigned polls;            // of one grid barrier at most
  unsigned *gave_up;         // host word: set where a barrier ran out of them
};

// The plain FP64 solve of a small grid: its passes, the gauge and p in one launch (resident64.cu).
struct Resident64Args {
  PassArgs<double> pass[5];
  const double *s;
  double *p;
  DevStats *st;
  double *partials;          // one sum of p per CTA
  unsigned *bar;
  int grid, cluster, row_tiles, tables_at, own_at;
  int gauge;                 // 0 none, 1 zero mean, 2 zero first cell
  double inv_cells;
  unsigned polls;
  unsigned *gave_up;
};
cudaError_t launch_resident64(const Resident64Args &R, int dim, size_t smem, cudaStream_t st);
pc_status prepare_resident64();

cudaError_t launch_resident(const ResidentArgs &R, int dim, bool pairs, size_t smem, cudaStream_t st);
pc_status prepare_resident();
// CTAs of the largest cluster the kernel runs as on the device, which is current (16, else 8; 0: none).
int resident_cluster_size(int device);

#ifdef __CUDACC__
// Barrier of the whole grid (a cooperative launch: every CTA is resident). bar counts arrivals;
// phase is the number of barriers passed. Bounded: after `polls` looks at the count it gives up and
// returns false, and the caller leaves the kernel. A CTA that left does not arrive at the next barrier,
// so every other CTA gives up there at the latest.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned &phase, unsigned polls) {
  __shared__ int ok;
  __syncthreads();
  ++phase;
  if (threadIdx.x == 0) {
    const unsigned want = phase * gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned seen = 0;
    int good = 0;
    for (unsigned it = 0; it < polls; ++it) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      if (seen >= want) {
        good = 1;
        break;
      }
    }
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}
// End of a kernel with grid barriers, by one thread of each CTA: the host learns of a barrier that gave up
// (its CTA has filled its rows of the result with NaN), and the last CTA leaves the counters at zero.
__device__ __forceinline__ void leave_grid(unsigned *bar, bool good, unsigned *gave_up) {
  if (!good) {
    *reinterpret_cast<volatile unsigned *>(gave_up) = 1u;
    __threadfence_system();
  }
  if (atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
    bar[0] = 0u;
    bar[1] = 0u;
  }
}

// Barrier of a grid that is one cluster: the hardware's (0.2 us against 1.2 for the grid barrier).
__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();   // .aligned: the warp arrives as one
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
#endif

}  // namespace pc
