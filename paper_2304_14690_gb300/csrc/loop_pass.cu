// Looped transform passes (loop_pass.cuh) as kernels of their own: single-problem launches (items
// == nullptr: the pass A1, CTA b transforming tiles b * chunk, ...) and batched ones (CTA b
// transforming tiles items[b].y .. items[b].y + items[b].z - 1 of args[items[b].x]).
#include "loop_pass.cuh"

namespace pc {

// IEEE: for solves that divide to nearest (PassArgs::ieee_div), in all their passes: with the dividing pass
// alone, each change of kernel cost a batch of five requests about 1 us (222 us against 216).
// FP32: 64 registers for four CTAs per SM, at which 24 bytes per thread spill (108 read back per tile,
// in L1): 64 2D problems 830 us, with three CTAs and no spill 840.
template <typename Real, bool IEEE>
__global__ void __launch_bounds__(loop::kThreads, sizeof(Real) == 4 ? 4 : 2)
    loop_kernel(PassArgs<Real> A1, const PassArgs<Real> *__restrict__ args, const int4 *__restrict__ items) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  typename Cplx<Real>::T *buf = reinterpret_cast<typename Cplx<Real>::T *>(smem_raw);
  __shared__ __align__(16) PassArgs<Real> A;
  __shared__ __align__(16) typename Cplx<Real>::T w16tab[10];
  loop::fill_w16(w16tab);
  int t0, t1;
  {
    const unsigned *src;
    if (items) {
      const int4 it = items[blockIdx.x];
      src = reinterpret_cast<const unsigned *>(args + it.x);
      t0 = it.y;
      t1 = it.y + it.z;
    } else {
      src = reinterpret_cast<const unsigned *>(&A1);
      t0 = blockIdx.x * A1.chunk;
      t1 = min(t0 + A1.chunk, A1.ntiles);
    }
    unsigned *dst = reinterpret_cast<unsigned *>(&A);
    for (int w = threadIdx.x; w < (int)(sizeof(PassArgs<Real>) / 4); w += blockDim.x) dst[w] = src[w];
  }
  __syncthreads();
  if (A.gate.st && refine_stopped_before(A.gate.st, A.gate.j, A.gate.tol)) return;   // refinement already ended
  for (int t = t0; t < t1; ++t) {
    if (t > t0) __syncthreads();   // the previous tile no longer reads the buffers
    loop::pass_tile<Real, IEEE>(A, t, buf, w16tab);
  }
}

pc_status launch_loop(const PassArgs<float> &A, const PassArgs<float> *dargs, const int4 *ditems, unsigned grid,
                      size_t smem, bool ieee, cudaStream_t st) {
  if (grid == 0) return PC_OK;
  launch_pdl(ieee ? loop_kernel<float, true> : loop_kernel<float, false>, grid, loop::kThreads, smem, st, A, dargs, ditems);
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}
pc_status launch_loop(const PassArgs<double> &A, unsigned grid, size_t smem, cudaStream_t st) {
  if (grid == 0) return PC_OK;
  launch_pdl(loop_kernel<double, false>, grid, loop::kThreads, smem, st, A, (const PassArgs<double> *)nullptr, (const int4 *)nullptr);
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

pc_status prepare_loop(int lim) {
  PC_CUDA_TRY(cudaFuncSetAttribute(loop_kernel<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
  PC_CUDA_TRY(cudaFuncSetAttribute(loop_kernel<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
  PC_CUDA_TRY(cudaFuncSetAttribute(loop_kernel<double, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
  return PC_OK;
}

}  // namespace pc
