// The whole refined solve of one problem as one cooperative kernel (§2.3 three-step solve and its
// FP32 refinement): every transform pass of every sweep, the residuals between them and the
// stopping rule.
//
// On grids of a few hundred cells per axis a pass is bound by latency: a launch of its own takes
// 8-9 us on a 1024 x 512 grid (launch and code fetch, one round of loads, the stages of one or two
// tiles per SM, the stores), at a few percent of any throughput. Here the CTAs stay resident (one per
// SM, 512 threads) and meet at a barrier of the grid between passes instead (1.4 us each):
//   - the passes share one body for all lengths (loop_pass.cuh), whose code stays in the SMs'
//     instruction caches, and their tables stay in shared memory;
//   - a CTA owns consecutive rows of the grid, whose source and iterate stay in its shared memory
//     as planes of high and low parts; a row tile forms the residual of its own cells as the input
//     of its forward transform, two cells per instruction, and only the rows next to other CTAs'
//     go through global memory (in 3D all);
//   - a sweep that the rule ended costs nothing.
// One call of the solve with walls on every side (two sweeps run; the sum of the source and the gauge with
// it) on a GB300, before (one launch per pass and residual) and now: 128^2 104 -> 55 us, 512^2 156 -> 75,
// 1024 x 512 217 -> 96, 1024^2 274 -> 159, 96^3 268 -> 193; with an outlet 128^2 43, 512^2 59, 1024 x 512 78.
// A phase of the 1024 x 512 grid takes about 7 us: five half-stages per transform at
// 0.35 us each (latency and issue alike: 38% of the issue slots), 1 us to load, 1 to store, the
// barrier.
#include <atomic>
#include <type_traits>

#include "loop_pass.cuh"
#include "dfloat.cuh"
#include "resident.cuh"

namespace pc {

using loop::Quad;

// Four consecutive values as two packed pairs: from global memory past L1 (other CTAs write it), or
// from the planes of high and low parts in shared memory.
struct Four { DF2 a, b; };
__device__ __forceinline__ Four load_four(const float2 *p) {
  const float4 u = __ldcg(reinterpret_cast<const float4 *>(p)), v = __ldcg(reinterpret_cast<const float4 *>(p + 2));
  return Four{DF2{f2_pack(u.x, u.z), f2_pack(u.y, u.w)}, DF2{f2_pack(v.x, v.z), f2_pack(v.y, v.w)}};
}
__device__ __forceinline__ Four load_four(const double *p) {
  const double2 u = __ldcg(reinterpret_cast<const double2 *>(p)), v = __ldcg(reinterpret_cast<const double2 *>(p + 2));
  return Four{df2_of(df_of(u.x), df_of(u.y)), df2_of(df_of(v.x), df_of(v.y))};
}
__device__ __forceinline__ Four load_planes(const float *hi, const float *lo) {
  const ulonglong2 h = *reinterpret_cast<const ulonglong2 *>(hi), l = *reinterpret_cast<const ulonglong2 *>(lo);
  return Four{DF2{F2{h.x}, F2{l.x}}, DF2{F2{h.y}, F2{l.y}}};
}
__device__ __forceinline__ void store_planes(float *hi, float *lo, const Four &v) {
  *reinterpret_cast<ulonglong2 *>(hi) = make_ulonglong2(v.a.hi.v, v.b.hi.v);
  *reinterpret_cast<ulonglong2 *>(lo) = make_ulonglong2(v.a.lo.v, v.b.lo.v);
}
__device__ __forceinline__ void store_pairs(float2 *p, const Four &v) {
  float4 u, w;
  f2_unpack(v.a.hi, u.x, u.z);
  f2_unpack(v.a.lo, u.y, u.w);
  f2_unpack(v.b.hi, w.x, w.z);
  f2_unpack(v.b.lo, w.y, w.w);
  *reinterpret_cast<float4 *>(p) = u;
  *reinterpret_cast<float4 *>(p + 2) = w;
}
// pair_add (loop_pass.cuh) on two pairs.
__device__ __forceinline__ DF2 pair_add2(DF2 old, F2 x) {
  const F2 s = f2_add(old.hi, x), z = f2_sub(s, old.hi);
  const F2 e = f2_add(f2_add(f2_sub(old.hi, f2_sub(s, z)), f2_sub(x, z)), old.lo);
  const F2 hi = f2_add(s, e);
  return DF2{hi, f2_sub(e, f2_sub(hi, s))};
}

// The rows a CTA owns (consecutive lines of the last axis): their source and iterate stay in its
// shared memory as planes of high and low parts.
struct Own {
  float *ph, *pl, *sh, *sl;
  int line0, lines;
};

// Residual of the cells 4 qd .. + 3 of own line d (residual_body of project.cu, two cells per
// operation: the same operations in the same order), and its max norms. Rows of other CTAs are read
// from p.
template <int DIM>
__device__ __forceinline__ Quad<float> residual_quad(const GridDev &g, const Own &o, const float2 *p, DF mean, bool singular,
                                                     int d, int qd, float &rmx, float &smx) {
  const int x = 4 * qd, nl = g.n[DIM - 1], at = d * nl + x, row = o.line0 + d;
  int i[3] = {0, 0, 0};
  if (DIM == 2) {
    i[0] = row;
  } else {
    i[0] = row / g.n[1];
    i[1] = row - i[0] * g.n[1];
  }
  const Four pc = load_planes(o.ph + at, o.pl + at);
  Four lo[DIM], hi[DIM];
#pragma unroll
  for (int a = 0; a < DIM - 1; ++a) {
    const int st = a == DIM - 2 ? 1 : g.n[1];   // in rows
    const bool l_in = i[a] > 0, h_in = i[a] < g.n[a] - 1, per = g.periodic[a];
    const int rl = l_in ? row - st : (per ? row + (g.n[a] - 1) * st : row);
    const int rh = h_in ? row + st : (per ? row - (g.n[a] - 1) * st : row);
    const int dl = rl - o.line0, dh = rh - o.line0;
    if ((unsigned)dl < (unsigned)o.lines) lo[a] = load_planes(o.ph + dl * nl + x, o.pl + dl * nl + x);
    else lo[a] = load_four(p + rl * nl + x);
    if ((unsigned)dh < (unsigned)o.lines) hi[a] = load_planes(o.ph + dh * nl + x, o.pl + dh * nl + x);
    else hi[a] = load_four(p + rh * nl + x);
    if (!l_in && !per) { lo[a].a = ghost(g.lo_kind[a], pc.a); lo[a].b = ghost(g.lo_kind[a], pc.b); }
    if (!h_in && !per) { hi[a].a = ghost(g.hi_kind[a], pc.a); hi[a].b = ghost(g.hi_kind[a], pc.b); }
  }
  {
    // neighbours along the row
    constexpr int a = DIM - 1;
    const int al = x > 0 ? at - 1 : at + nl - 1, ar = x + 4 < nl ? at + 4 : at + 4 - nl;
    DF2 l = DF2{f2_pack(0.0f, o.ph[al]), f2_pack(0.0f, o.pl[al])}, r = DF2{f2_pack(o.ph[ar], 0.0f), f2_pack(o.pl[ar], 0.0f)};
    if (x == 0 && !g.periodic[a]) {
      const DF2 e = ghost(g.lo_kind[a], pc.a);
      l = DF2{F2{e.hi.v << 32}, F2{e.lo.v << 32}};   // the first cell's in the upper half
    }
    if (x + 4 >= nl && !g.periodic[a]) {
      const DF2 e = ghost(g.hi_kind[a], pc.b);
      r = DF2{F2{e.hi.v >> 32}, F2{e.lo.v >> 32}};   // the last cell's in the lower half
    }
    lo[a].a = df2_mid(l, pc.a);
    lo[a].b = df2_mid(pc.a, pc.b);
    hi[a].a = lo[a].b;
    hi[a].b = df2_mid(pc.b, r);
  }
  DF2 u, v;
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    const DF ih2{g.ih2_hi[a], g.ih2_lo[a]};
    const DF2 tu = second_difference2(lo[a].a, pc.a, hi[a].a, ih2), tv = second_difference2(lo[a].b, pc.b, hi[a].b, ih2);
    u = a == 0 ? tu : df2_sum(u, tu);
    v = a == 0 ? tv : df2_sum(v, tv);
  }
  const Four sc = load_planes(o.sh + at, o.sl + at);
  DF2 su = sc.a, sv = sc.b;
  smx = max_abs(max_abs(smx, su.hi), sv.hi);
  if (singular) {
    const DF2 m = df2_of(mean, mean);
    su = df2_diff(su, m);
    sv = df2_diff(sv, m);
  }
  const DF2 ru = df2_diff(su, u), rv = df2_diff(sv, v);
  const F2 r0 = f2_add(ru.hi, ru.lo), r1 = f2_add(rv.hi, rv.lo);
  rmx = max_abs(max_abs(rmx, r0), r1);
  Quad<float> q;
  f2_unpack(r0, q.x, q.y);
  f2_unpack(r1, q.z, q.w);
  return q;
}

// Maximum over the CTA of non-negative v, merged into *dst by one atomic maximum of its bits.
__device__ __forceinline__ void cta_max(float v, float *dst) {
  __shared__ float sh[kResidentThreads / 32];
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < kResidentThreads / 32 ? sh[threadIdx.x] : 0.0f;
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned *>(dst), __float_as_uint(v));
  }
}

// IEEE: the pass of axis 0 divides to nearest (PassArgs::ieee_div).
template <int DIM, typename SV, bool CLUSTER, bool IEEE>
__global__ void __launch_bounds__(kResidentThreads, 1) resident_kernel(const __grid_constant__ ResidentArgs R) {
  constexpr int NP = 2 * DIM - 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *buf = reinterpret_cast<float2 *>(smem_raw);
  __shared__ __align__(16) PassArgs<float> As[NP];
  __shared__ float2 w16tab[10];
  __shared__ int stop;
  const float2 *tabs = buf + R.tables_at;
  {
    const unsigned *src = reinterpret_cast<const unsigned *>(R.pass);
    unsigned *dst = reinterpret_cast<unsigned *>(As);
    for (int w = threadIdx.x; w < (int)(sizeof(As) / 4); w += blockDim.x) dst[w] = src[w];
    loop::fill_w16(w16tab);
    // the tables of every axis, once: a barrier of the grid empties L1 (a stage that read them from
    // L2 took 800 cycles however small the tile)
    float2 *to = buf + R.tables_at;
    for (int k = 0; k < DIM; ++k) {   // passes 0 .. DIM - 1 cover the axes
      const PassArgs<float> &A = R.pass[k];
      for (int i = A.tw_first + threadIdx.x; i < A.tw_last; i += blockDim.x) to[A.tw_at + i] = __ldg(A.tw + i);
      for (int i = threadIdx.x; i < A.st_count; i += blockDim.x) to[A.st_at + i] = __ldg(A.stw + i);
      if (A.do_div)
        for (int i = threadIdx.x; i < A.n; i += blockDim.x) reinterpret_cast<float *>(to)[A.lam_at + i] = __ldg(A.lam[A.axis] + i);
    }
  }
  if (CLUSTER) pdl_enter();   // a plain launch in the stream's chain: what is above does not depend on it
  const SV *s = static_cast<const SV *>(R.s);
  const int nl = R.g.n[DIM - 1], own = R.row_tiles * R.pass[0].L * nl;   // cells
  Own o;
  o.ph = reinterpret_cast<float *>(buf + R.own_at);
  o.pl = o.ph + own;
  o.sh = o.pl + own;
  o.sl = o.sh + own;
  o.line0 = blockIdx.x * R.row_tiles * R.pass[0].L;
  o.lines = max(0, min(R.row_tiles * R.pass[0].L, R.pass[0].lines - o.line0));
  unsigned phase = 0;
  bool good = true, ended = false;
  __syncthreads();
#pragma unroll 1
  for (int j = 0; j <= R.sweeps && good && !ended; ++j) {
    DF mean{0.0f, 0.0f};
    if (j > 0 && R.singular) mean = df_of(__ldcg(&R.st->mean_s));
#pragma unroll 1
    for (int ps = 0; ps < NP && good && !ended; ++ps) {
      const PassArgs<float> &A = As[ps];
      const bool first = ps == 0, final_pass = ps == NP - 1, row = first || final_pass;
      const void *src = A.src;
      const loop::Store<float> out = loop::store_of(A);
      float rmx = 0.0f, smx = 0.0f;
      const SharedTables<float> tb{tabs + A.tw_at, tabs + A.st_at, reinterpret_cast<const float *>(tabs) + A.lam_at};
      // row passes: the CTA's own consecutive tiles; column passes: every gridDim.x-th tile
      const int t0 = row ? (int)blockIdx.x * R.row_tiles : (int)blockIdx.x, step = row ? 1 : (int)gridDim.x;
      const int t1 = row ? min(t0 + R.row_tiles, A.ntiles) : A.ntiles;
#pragma unroll 1
      for (int tile = t0; tile < t1; tile += step) {
        if (tile != t0) __syncthreads();   // the previous tile's outputs have left the buffers
        const int d0 = (tile - t0) * A.L;
        loop::pass_tile<float, IEEE>(
            A, tile, buf, tb, w16tab,
            [&](int l, int base, int qd, int stride) -> Quad<float> {
              if (!first) return loop::load_src4<float>(src, SRC_WORK, base + 4 * qd * stride, stride);
              if (j > 0) return residual_quad<DIM>(R.g, o, R.p2, mean, R.singular, d0 + l, qd, rmx, smx);
              const int c = base + 4 * qd, at = (d0 + l) * nl + 4 * qd;
              const Four v = load_four(s + c);
              store_planes(o.sh + at, o.sl + at, v);
              Quad<float> q;
              if constexpr (sizeof(SV) == 8 && !std::is_same<SV, float2>::value) {
                q = loop::load_src4<float>(s, SRC_F64, c, 1);   // as an FP32 pass takes an FP64 source
              } else {
                f2_unpack(v.a.hi, q.x, q.y);
                f2_unpack(v.b.hi, q.z, q.w);
              }
              return q;
            },
            [&](int l, int base, int qd, int stride, const Quad<float> &x) {
              if (!final_pass) {
                loop::store_dst4(out, base + 4 * qd * stride, stride, x);
                return;
              }
              const int d = d0 + l, at = d * nl + 4 * qd;
              const F2 xa = f2_pack(x.x, x.y), xb = f2_pack(x.z, x.w), zero = f2_pack(0.0f, 0.0f);
              Four v;
              if (j == 0) {
                v = Four{DF2{xa, zero}, DF2{xb, zero}};
              } else {
                const Four old = load_planes(o.ph + at, o.pl + at);
                v = Four{pair_add2(old.a, xa), pair_add2(old.b, xb)};
              }
              store_planes(o.ph + at, o.pl + at, v);
              // the rows that other CTAs read: the first and the last own one, in 3D any
              if (DIM == 3 || d == 0 || d == o.lines - 1) store_pairs(R.p2 + base + 4 * qd, v);
            });
      }
      if (first && j > 0 && R.adaptive) {
        cta_max(rmx, &R.st->rmax[j - 1]);
        if (j == 1) cta_max(smx, &R.st->smax);
      }
      if (j == R.sweeps && final_pass) break;
      if constexpr (CLUSTER) cluster_barrier();
      else good = grid_barrier(R.bar, phase, R.polls);
      if (first && j > 0 && R.adaptive && good) {
        if (threadIdx.x == 0) stop = refine_stopped_before(R.st, j, R.tol) ? 1 : 0;
        __syncthreads();
        ended = stop != 0;
      }
    }
  }
  __syncthreads();
  if (good) {
    // the iterate in pairs (the gradient reads it) and in FP64
    const int nq = o.lines * nl / 4, c0 = o.line0 * nl;
    for (int i = threadIdx.x; i < nq; i += blockDim.x) {
      const Four v = load_planes(o.ph + 4 * i, o.pl + 4 * i);
      store_pairs(R.p2 + c0 + 4 * i, v);
      float h[4], l[4];
      f2_unpack(v.a.hi, h[0], h[1]);
      f2_unpack(v.b.hi, h[2], h[3]);
      f2_unpack(v.a.lo, l[0], l[1]);
      f2_unpack(v.b.lo, l[2], l[3]);
      double2 *f = reinterpret_cast<double2 *>(R.f64 + c0 + 4 * i);
      f[0] = make_double2(f2d_bits(h[0]) + f2d_bits(l[0]), f2d_bits(h[1]) + f2d_bits(l[1]));
      f[1] = make_double2(f2d_bits(h[2]) + f2d_bits(l[2]), f2d_bits(h[3]) + f2d_bits(l[3]));
    }
  }
  if constexpr (!CLUSTER) {
    if (!good)   // a barrier gave up: these rows have no result
      for (int i = threadIdx.x; i < o.lines * nl; i += blockDim.x) {
        R.p2[o.line0 * nl + i] = make_float2(__int_as_float(0x7fc00000), 0.0f);
        R.f64[o.line0 * nl + i] = __longlong_as_double(0x7ff8000000000000LL);
      }
    __syncthreads();
    if (threadIdx.x == 0) leave_grid(R.bar, good, R.gave_up);
  }
}

template <int DIM, typename SV, bool IEEE>
static cudaError_t launch(const ResidentArgs &R, size_t smem, cudaStream_t st) {
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
    return cudaLaunchKernelEx(&cfg, resident_kernel<DIM, SV, true, IEEE>, R);
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, resident_kernel<DIM, SV, false, IEEE>, R);
  }
}

cudaError_t launch_resident(const ResidentArgs &R, int dim, bool pairs, size_t smem, cudaStream_t st) {
  auto of = [&](auto ieee) {
    constexpr bool I = decltype(ieee)::value;
    if (dim == 2) return pairs ? launch<2, float2, I>(R, smem, st) : launch<2, double, I>(R, smem, st);
    return pairs ? launch<3, float2, I>(R, smem, st) : launch<3, double, I>(R, smem, st);
  };
  return R.pass[dim - 1].ieee_div ? of(std::true_type{}) : of(std::false_type{});
}

template <int DIM, typename SV, bool IEEE>
static pc_status prepare_one() {
  PC_CUDA_TRY(cudaFuncSetAttribute(resident_kernel<DIM, SV, false, IEEE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmem));
  PC_CUDA_TRY(cudaFuncSetAttribute(resident_kernel<DIM, SV, true, IEEE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmem));
  PC_CUDA_TRY(cudaFuncSetAttribute(resident_kernel<DIM, SV, true, IEEE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  return PC_OK;
}
pc_status prepare_resident() {
  PC_TRY((prepare_one<2, float2, false>()));
  PC_TRY((prepare_one<2, float2, true>()));
  PC_TRY((prepare_one<2, double, false>()));
  PC_TRY((prepare_one<2, double, true>()));
  PC_TRY((prepare_one<3, float2, false>()));
  PC_TRY((prepare_one<3, float2, true>()));
  PC_TRY((prepare_one<3, double, false>()));
  return prepare_one<3, double, true>();
}

int resident_cluster_size(int device) {
  static std::atomic<int> known[kMaxDevices];   // 1 + the size
  if (device < 0 || device >= kMaxDevices) return 0;
  const int have = known[device].load(std::memory_order_relaxed);
  if (have) return have - 1;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  cfg.blockDim = dim3(kResidentThreads);
  cfg.dynamicSmemBytes = kResidentSmem;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  int size = 0;
  for (int n : {16, 8}) {
    at[0].val.clusterDim.x = (unsigned)n;
    cfg.gridDim = dim3((unsigned)n);
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, resident_kernel<3, double, true, true>, &cfg) == cudaSuccess && fit > 0) {
      size = n;
      break;
    }
    cudaGetLastError();
  }
  known[device].store(1 + size, std::memory_order_relaxed);
  return size;
}

}  // namespace pc
