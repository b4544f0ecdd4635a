// The plain FP64 solve of a grid up to a million cells as one launch: the passes of resident.cu in
// FP64 (the same looped body, tables in shared memory, a barrier of the grid or of the cluster
// between passes), then the gauge on the rows each CTA still holds. The three or five passes and
// the two gauge kernels of small grids are bound by their launches (64^2 projection with a zero
// mode 50 -> 44 us); on large ones the FP64 pipe bounds (two lanes per SM and clock: about 60 us of
// a 1024 x 512 solve) and one launch still saves the passes' ramps and tails.
#include "loop_pass.cuh"
#include "resident.cuh"

namespace pc {

using loop::Quad;

// Sum over the CTA, fixed order (shuffle tree, then the warps' sums in order); valid in thread 0.
__device__ __forceinline__ double cta_sum(double v) {
  __shared__ double sh[kResidentThreads / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = threadIdx.x < kResidentThreads / 32 ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  return t;
}

template <int DIM, bool CLUSTER>
__global__ void __launch_bounds__(kResidentThreads, 1) resident64_kernel(const __grid_constant__ Resident64Args R) {
  constexpr int NP = 2 * DIM - 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2 *buf = reinterpret_cast<double2 *>(smem_raw);
  __shared__ __align__(16) PassArgs<double> As[NP];
  __shared__ __align__(16) double2 w16tab[10];
  __shared__ double shift_s;
  const double2 *tabs = buf + R.tables_at;
  {
    const unsigned *src = reinterpret_cast<const unsigned *>(R.pass);
    unsigned *dst = reinterpret_cast<unsigned *>(As);
    for (int w = threadIdx.x; w < (int)(sizeof(As) / 4); w += blockDim.x) dst[w] = src[w];
    loop::fill_w16(w16tab);
    double2 *to = buf + R.tables_at;
    for (int k = 0; k < DIM; ++k) {
      const PassArgs<double> &A = R.pass[k];
      for (int i = A.tw_first + threadIdx.x; i < A.tw_last; i += blockDim.x) to[A.tw_at + i] = __ldg(A.tw + i);
      for (int i = threadIdx.x; i < A.st_count; i += blockDim.x) to[A.st_at + i] = __ldg(A.stw + i);
      if (A.do_div)
        for (int i = threadIdx.x; i < A.n; i += blockDim.x) reinterpret_cast<double *>(to)[A.lam_at + i] = __ldg(A.lam[A.axis] + i);
    }
  }
  if (CLUSTER) pdl_enter();
  double *own = reinterpret_cast<double *>(buf + R.own_at);
  const int nl = R.pass[0].n, line0 = blockIdx.x * R.row_tiles * R.pass[0].L;
  const int lines = max(0, min(R.row_tiles * R.pass[0].L, R.pass[0].lines - line0));
  unsigned phase = 0;
  bool good = true;
  __syncthreads();
#pragma unroll 1
  for (int ps = 0; ps < NP && good; ++ps) {
    const PassArgs<double> &A = As[ps];
    const bool first = ps == 0, final_pass = ps == NP - 1, row = first || final_pass;
    const void *src = first ? (const void *)R.s : A.src;
    const loop::Store<double> out = loop::store_of(A);
    const SharedTables<double> tb{tabs + A.tw_at, tabs + A.st_at, reinterpret_cast<const double *>(tabs) + A.lam_at};
    const int t0 = row ? (int)blockIdx.x * R.row_tiles : (int)blockIdx.x, step = row ? 1 : (int)gridDim.x;
    const int t1 = row ? min(t0 + R.row_tiles, A.ntiles) : A.ntiles;
#pragma unroll 1
    for (int tile = t0; tile < t1; tile += step) {
      if (tile != t0) __syncthreads();
      const int d0 = (tile - t0) * A.L;
      loop::pass_tile<double, false>(
          A, tile, buf, tb, w16tab,
          [&](int, int base, int qd, int stride) { return loop::load_src4<double>(src, SRC_WORK, base + 4 * qd * stride, stride); },
          [&](int l, int base, int qd, int stride, const Quad<double> &x) {
            if (!final_pass) {
              loop::store_dst4(out, base + 4 * qd * stride, stride, x);
              return;
            }
            double2 *o = reinterpret_cast<double2 *>(own + (d0 + l) * nl + 4 * qd);
            o[0] = make_double2(x.x, x.y);
            o[1] = make_double2(x.z, x.w);
          });
    }
    if (final_pass) break;
    if constexpr (CLUSTER) cluster_barrier();
    else good = grid_barrier(R.bar, phase, R.polls);
  }
  __syncthreads();
  const int cells = lines * nl, c0 = line0 * nl;
  double shift = 0.0;
  if (R.gauge && good) {
    // the gauge constant: each CTA's sum of its rows, added up in the order of the CTAs by every CTA
    double v = 0.0;
    if (R.gauge == 1)
      for (int i = threadIdx.x; i < cells; i += blockDim.x) v += own[i];
    v = cta_sum(v);
    if (threadIdx.x == 0) {
      R.partials[blockIdx.x] = v;
      if (c0 == 0 && cells > 0) R.st->corner_p = own[0];
    }
    if constexpr (CLUSTER) cluster_barrier();
    else good = grid_barrier(R.bar, phase, R.polls);
    double t = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) t += __ldcg(R.partials + b);
    t = cta_sum(t);
    if (threadIdx.x == 0) {
      shift_s = R.gauge == 1 ? t * R.inv_cells : __ldcg(&R.st->corner_p);
      if (blockIdx.x == 0) {
        R.st->sum_p = t;
        R.st->shift = shift_s;
      }
    }
    __syncthreads();
    shift = shift_s;
  }
  if (good)
    for (int i = 2 * threadIdx.x; i < cells; i += 2 * blockDim.x) {
      const double2 v = *reinterpret_cast<const double2 *>(own + i);
      *reinterpret_cast<double2 *>(R.p + c0 + i) = make_double2(v.x - shift, v.y - shift);
    }
  if constexpr (!CLUSTER) {
    if (!good)   // a barrier gave up: these rows have no result
      for (int i = threadIdx.x; i < cells; i += blockDim.x) R.p[c0 + i] = __longlong_as_double(0x7ff8000000000000LL);
    __syncthreads();
    if (threadIdx.x == 0) leave_grid(R.bar, good, R.gave_up);
  }
}

template <int DIM>
static cudaError_t launch64(const Resident64Args &R, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)R.grid);
  cfg.blockDim = dim3(kResidentThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  cfg.attrs = at;
  if (R.cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)R.grid;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = tl_plain_launch ? 1 : 2;
    return cudaLaunchKernelEx(&cfg, resident64_kernel<DIM, true>, R);
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, resident64_kernel<DIM, false>, R);
  }
}

cudaError_t launch_resident64(const Resident64Args &R, int dim, size_t smem, cudaStream_t st) {
  return dim == 2 ? launch64<2>(R, smem, st) : launch64<3>(R, smem, st);
}

template <int DIM>
static pc_status prepare64() {
  PC_CUDA_TRY(cudaFuncSetAttribute(resident64_kernel<DIM, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmem));
  PC_CUDA_TRY(cudaFuncSetAttribute(resident64_kernel<DIM, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmem));
  PC_CUDA_TRY(cudaFuncSetAttribute(resident64_kernel<DIM, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  return PC_OK;
}
pc_status prepare_resident64() {
  PC_TRY(prepare64<2>());
  return prepare64<3>();
}

}  // namespace pc
