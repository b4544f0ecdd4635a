// Transform passes whose FFT loops over identical butterflies (cell-grid families 0-2, even M =
// n/2 = 2^a 3^b 5^c). The line length is a run-time value and only the radix of a stage is compiled
// in, so one small body serves every length: the code of a pass stays in the instruction cache
// while the CTAs of a persistent kernel (resident.cu) run pass after pass, and any number of
// lines can share a CTA, down to the one or two per SM that a small grid leaves.
//   - A tile is L lines of M complex slots, line-major in shared memory, one slot of padding every
//     W (W slots fill the 32 banks): slot q of line l at l * LS + q + q / W, LS = W / L mod W. The
//     lanes of a stage read consecutive slots and write slots R apart (first stage) or
//     consecutive ones; either way, and for the column tiles' scatter across lines, they fall into
//     different banks.
//   - A stage takes butterfly j of line l per thread and iteration, reads its R slots from one
//     buffer, twiddles, transforms them in registers and writes the other: one barrier per stage.
//     Its twiddles come from a table per stage ([r - 1][k], k fast), so that a warp's loads are
//     consecutive.
//   - Wrappers and radices are those of pairs.cuh; the schedule of a length with a compile-time
//     pass is that pass's variant 0 (lean_pass.cuh), so both give a line the same bits.
#pragma once

#include "pairs.cuh"

namespace pc {
namespace loop {

constexpr int kThreads = 256;   // CTA size of a looped pass on its own (resident.cu: 512)

template <typename Real> struct Slots;
template <> struct Slots<float> { static constexpr int kShift = 4; };    // 16 float2 fill the banks
template <> struct Slots<double> { static constexpr int kShift = 3; };   // 8 double2

// Slots between the lines of a tile of L lines.
template <typename Real>
__host__ __device__ inline int line_slots(int M, int L) {
  constexpr int W = 1 << Slots<Real>::kShift;
  const int base = M + (M >> Slots<Real>::kShift);
  const int want = L <= W ? W / L : 1;
  const int off = (want - base) & (W - 1);
  return base + off;
}
template <typename Real>
inline size_t tile_smem(int M, int L) {   // two buffers, and the lines' eigenvalue sums
  return 2 * (size_t)L * line_slots<Real>(M, L) * 2 * sizeof(Real) + (size_t)L * sizeof(Real);
}

template <typename Real>
__device__ __forceinline__ int at(int q) { return q + (q >> Slots<Real>::kShift); }

// i / d for i < 2^16 (magic = ceil(2^32 / d)).
__device__ __forceinline__ int fdiv(int i, unsigned magic) { return (int)__umulhi((unsigned)i, magic); }

// Reads and writes of a stage. Slots that lie a multiple of W apart are a constant number of padded
// slots apart, which is so for all but short or odd lengths; the radix consecutive slots that the
// first stage writes share a padding block.
template <typename Real, int R>
__device__ __forceinline__ void read_slots(const typename Cplx<Real>::T *line, int q0, int step, typename Cplx<Real>::T *v) {
  constexpr int S = Slots<Real>::kShift, W = 1 << S;
  if ((step & (W - 1)) == 0) {
    const typename Cplx<Real>::T *p = line + at<Real>(q0);
    const int d = step + (step >> S);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = p[r * d];
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = line[at<Real>(q0 + r * step)];
  }
}
template <typename Real, int R>
__device__ __forceinline__ void write_slots(typename Cplx<Real>::T *line, int q0, int step, const typename Cplx<Real>::T *v) {
  constexpr int S = Slots<Real>::kShift, W = 1 << S;
  typename Cplx<Real>::T *p = line + at<Real>(q0);
  if ((step & (W - 1)) == 0) {
    const int d = step + (step >> S);
#pragma unroll
    for (int r = 0; r < R; ++r) p[r * d] = v[r];
  } else if (W % R == 0 && step == 1) {
#pragma unroll
    for (int r = 0; r < R; ++r) p[r] = v[r];
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) line[at<Real>(q0 + r * step)] = v[r];
  }
}

// One Stockham stage of radix R over the L lines of a tile: butterfly j reads slots j + r M/R,
// twiddles them by w_{Ns R}^{r (j mod Ns)} and writes slots (j / Ns) Ns R + (j mod Ns) + r Ns.
// pre >= 0: a factor per input slot from there in the tables (the DCT-IV pre-twiddle, first stage).
template <typename Real, int R, typename Tables>
__device__ __forceinline__ void stage(const typename Cplx<Real>::T *in, typename Cplx<Real>::T *out, int L, int LS,
                                      const StageInfo &s, const Tables &tb, int pre) {
  using T = typename Cplx<Real>::T;
  const int MR = s.mr, Ns = s.Ns, total = L * MR;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    const int l = fdiv(i, s.mr_magic), j = i - l * MR;
    const int q = s.shift >= 0 ? (j >> s.shift) : fdiv(j, s.magic);
    const int k = j - q * Ns;
    T v[R];
    read_slots<Real, R>(in + l * LS, j, MR, v);
    if (pre >= 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = cmul(v[r], tb.tw(pre + j + r * MR));
    }
    if (Ns > 1) {
      const int w = s.stride_m + k;
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tb.st(w + (r - 1) * Ns));
    }
    dft_small<R>(v);
    write_slots<Real, R>(out + l * LS, q * Ns * R + k, Ns, v);
  }
}

// A radix-16 stage as its two halves of radix-4 butterflies, with the operations of small_dft<16> in
// the same order (input k1 + 4 k2, output j2 + 4 j1): four times the threads, for tiles that leave
// most of a CTA idle at one butterfly of 16 per thread (a radix-16 stage of 2048 slots: four
// warps per SM, 1300 cycles). The intermediate values go through `out`; the result is back in `in`.
template <typename Real, typename Tables>
__device__ __forceinline__ void stage16_split(typename Cplx<Real>::T *in, typename Cplx<Real>::T *out, int L, int LS,
                                              const StageInfo &s, const Tables &tb, int pre,
                                              const typename Cplx<Real>::T *w16tab) {
  using T = typename Cplx<Real>::T;
  const int MR = s.mr, Ns = s.Ns, quarter = 4 * MR, total = L * quarter;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    const int lk = fdiv(i, s.mr_magic), j = i - lk * MR, k1 = lk & 3, l = lk >> 2;
    const int q = s.shift >= 0 ? (j >> s.shift) : fdiv(j, s.magic);
    const int k = j - q * Ns;
    T v[4];
    read_slots<Real, 4>(in + l * LS, j + k1 * MR, quarter, v);
    if (pre >= 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = cmul(v[r], tb.tw(pre + j + (k1 + 4 * r) * MR));
    }
    if (Ns > 1) {
      const int w = s.stride_m + k;
      if (k1) v[0] = cmul(v[0], tb.st(w + (k1 - 1) * Ns));
#pragma unroll
      for (int r = 1; r < 4; ++r) v[r] = cmul(v[r], tb.st(w + (k1 + 4 * r - 1) * Ns));
    }
    dft4<T, false>(v[0], v[1], v[2], v[3]);
#pragma unroll
    for (int r = 1; r < 4; ++r) v[r] = cmul_w16<T, false>(v[r], w16tab[k1 * r], k1 * r == 6);   // (1, 0) and (0, -1) are exact
    write_slots<Real, 4>(out + l * LS, 4 * k1 * MR + j, MR, v);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    const int lk = fdiv(i, s.mr_magic), j = i - lk * MR, j2 = lk & 3, l = lk >> 2;
    const int q = s.shift >= 0 ? (j >> s.shift) : fdiv(j, s.magic);
    const int k = j - q * Ns;
    T v[4];
    read_slots<Real, 4>(out + l * LS, j2 * MR + j, quarter, v);
    dft4<T, false>(v[0], v[1], v[2], v[3]);
    if (Ns == 1) {   // outputs 16 q + j2 + 4 j1: one padding block
      T *p = in + l * LS + at<Real>(16 * q + j2);
      if constexpr (Slots<Real>::kShift == 4) {
#pragma unroll
        for (int r = 0; r < 4; ++r) p[4 * r] = v[r];
      } else {
#pragma unroll
        for (int r = 0; r < 4; ++r) (in + l * LS)[at<Real>(16 * q + j2 + 4 * r)] = v[r];
      }
    } else {
      write_slots<Real, 4>(in + l * LS, q * Ns * 16 + k + j2 * Ns, 4 * Ns, v);
    }
  }
}

// Forward FFT of every line of the tile, ping-ponging between a and b; the result is left in a.
// Called by every thread of the CTA, after a barrier; ends with one. Radix-16 stages run as their halves.
template <typename Real, typename Tables>
__device__ __forceinline__ void fft(const PassArgs<Real> &A, int L, int LS, typename Cplx<Real>::T *&a,
                                    typename Cplx<Real>::T *&b, const Tables &tb, int pre,
                                    const typename Cplx<Real>::T *w16tab) {
  using T = typename Cplx<Real>::T;
  const int nst = A.nst;
#pragma unroll 1
  for (int s = 0; s < nst; ++s) {
    const StageInfo si = A.st[s];
    const int p0 = s == 0 ? pre : -1;
    if (si.R == 16) {
      stage16_split<Real>(a, b, L, LS, si, tb, p0, w16tab);
      __syncthreads();
      continue;
    }
    // Not a switch: with one, and an IEEE division elsewhere in the kernel, nvcc 13.0 let warps whose lanes
    // end their loops at different iterations into the barrier in parts (a 60 x 720 solve off by 5e4,
    // differently in each run). The warp barrier below is there for the same reason.
    const int radix = si.R;
    if (radix == 8) stage<Real, 8>(a, b, L, LS, si, tb, p0);
    else if (radix == 4) stage<Real, 4>(a, b, L, LS, si, tb, p0);
    else if (radix == 2) stage<Real, 2>(a, b, L, LS, si, tb, p0);
    else if (radix == 3) stage<Real, 3>(a, b, L, LS, si, tb, p0);
    else stage<Real, 5>(a, b, L, LS, si, tb, p0);
    __syncthreads();
    T *t = a;
    a = b;
    b = t;
  }
}
// e^{-2 pi i e/16} for the products k1 j2 of the split stage (e <= 9), for a CTA's shared memory.
template <typename T>
__device__ __forceinline__ void fill_w16(T *tab) {
  if (threadIdx.x == 0) {
    tab[0] = w16<T, false>(0); tab[1] = w16<T, false>(1); tab[2] = w16<T, false>(2); tab[3] = w16<T, false>(3);
    tab[4] = w16<T, false>(4); tab[5] = w16<T, false>(0); tab[6] = w16<T, false>(6); tab[7] = w16<T, false>(0);
    tab[8] = w16<T, false>(0); tab[9] = w16<T, false>(9);
  }
}

template <typename Real> struct Quad { Real x, y, z, w; };

// Forward scatter of the values at positions 4 qd .. 4 qd + 3 of a line: in order (real DFT), by
// Makhoul's reordering (times (-1)^j for DST-II), or as DCT-IV's z_q = (x_2q, x_{n-1-2q}).
template <typename Real>
__device__ __forceinline__ void scatter_quad(typename Cplx<Real>::T *line, int M, int fam, int kind, int qd,
                                             const Quad<Real> &x) {
  using T = typename Cplx<Real>::T;
  if (fam == 0) {
    line[at<Real>(2 * qd)] = cmk<T>(x.x, x.y);
    line[at<Real>(2 * qd + 1)] = cmk<T>(x.z, x.w);
  } else if (fam == 1) {
    const bool dd = kind == KIND_DD;
    line[at<Real>(qd)] = cmk<T>(x.x, x.z);
    line[at<Real>(M - 1 - qd)] = dd ? cmk<T>(-x.w, -x.y) : cmk<T>(x.w, x.y);
  } else {
    Real *re = reinterpret_cast<Real *>(line);
    const int c = kind == KIND_ND ? 0 : 1;
    re[2 * at<Real>(2 * qd) + c] = x.x;
    re[2 * at<Real>(2 * qd + 1) + c] = x.z;
    re[2 * at<Real>(M - 1 - 2 * qd) + (c ^ 1)] = x.y;
    re[2 * at<Real>(M - 2 - 2 * qd) + (c ^ 1)] = x.w;
  }
}

// Outputs 4 qd .. 4 qd + 3 of a line after the final FFT (before the 1/M normalisation).
template <typename Real, typename Tables>
__device__ __forceinline__ Quad<Real> gather_quad(const typename Cplx<Real>::T *line, int M, int fam, int kind, int qd,
                                                  const Tables &tb) {
  using T = typename Cplx<Real>::T;
  if (fam == 0) {
    const T a = line[at<Real>(2 * qd)], b = line[at<Real>(2 * qd + 1)];
    return Quad<Real>{a.x, -a.y, b.x, -b.y};
  }
  if (fam == 1) {
    const T zq = line[at<Real>(qd)], zm = line[at<Real>(M - 1 - qd)];
    if (kind == KIND_DD) return Quad<Real>{zq.x, zm.y, -zq.y, -zm.x};
    return Quad<Real>{zq.x, -zm.y, -zq.y, zm.x};
  }
  const int tp = tw_dct4post(M);
  const int qa = 2 * qd, qb = M - 1 - 2 * qd, qc = 2 * qd + 1, qe = M - 2 - 2 * qd;
  const T ya = cmul(line[at<Real>(qa)], tb.tw(tp + qa)), yb = cmul(line[at<Real>(qb)], tb.tw(tp + qb));
  const T yc = cmul(line[at<Real>(qc)], tb.tw(tp + qc)), ye = cmul(line[at<Real>(qe)], tb.tw(tp + qe));
  if (kind == KIND_ND) return Quad<Real>{ya.x, -yb.y, yc.x, -ye.y};
  return Quad<Real>{ya.x, yb.y, yc.x, ye.y};
}

// Global loads past L1 (the arrays a persistent kernel's other CTAs wrote).
__device__ __forceinline__ Quad<float> load4(const float *s, int stride) {
  if (stride == 1) {
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(s));
    return Quad<float>{v.x, v.y, v.z, v.w};
  }
  return Quad<float>{__ldcg(s), __ldcg(s + stride), __ldcg(s + 2 * stride), __ldcg(s + 3 * stride)};
}
__device__ __forceinline__ Quad<double> load4(const double *s, int stride) {
  if (stride == 1) {
    const double2 a = __ldcg(reinterpret_cast<const double2 *>(s)), b = __ldcg(reinterpret_cast<const double2 *>(s + 2));
    return Quad<double>{a.x, a.y, b.x, b.y};
  }
  return Quad<double>{__ldcg(s), __ldcg(s + stride), __ldcg(s + 2 * stride), __ldcg(s + 3 * stride)};
}
template <typename Real>
__device__ __forceinline__ Quad<Real> load_src4(const void *src, int mode, int g, int stride) {
  if constexpr (sizeof(Real) == 4) {
    if (mode == SRC_F64) {   // truncated to FP32, as every FP32 pass takes an FP64 source
      const Quad<double> v = load4(static_cast<const double *>(src) + g, stride);
      return Quad<float>{d2f_rz_bits(v.x), d2f_rz_bits(v.y), d2f_rz_bits(v.z), d2f_rz_bits(v.w)};
    }
  }
  return load4(static_cast<const Real *>(src) + g, stride);
}

// The pair (hi, lo) of the refinement iterate += x (Knuth's TwoSum), renormalised.
__device__ __forceinline__ float2 pair_add(float2 old, float x) {
  const float s1 = __fadd_rn(old.x, x), z = __fsub_rn(s1, old.x);
  const float e = __fadd_rn(__fadd_rn(__fsub_rn(old.x, __fsub_rn(s1, z)), __fsub_rn(x, z)), old.y);
  const float hi = __fadd_rn(s1, e);
  return make_float2(hi, __fsub_rn(e, __fsub_rn(hi, s1)));
}

// A pass's destination in registers.
template <typename Real>
struct Store {
  int dst_mode;
  void *dst;
  double *f64;
};
template <typename Real>
__device__ __forceinline__ Store<Real> store_of(const PassArgs<Real> &A) { return Store<Real>{A.dst_mode, A.dst, A.f64}; }

// Store of the outputs 4 qd .. 4 qd + 3 of a line by the destination's mode.
__device__ __forceinline__ void store_dst4(const Store<float> &A, int g, int stride, const Quad<float> &x) {
  if (A.dst_mode == DST_WORK) {
    float *d = static_cast<float *>(A.dst) + g;
    if (stride == 1) {
      *reinterpret_cast<float4 *>(d) = make_float4(x.x, x.y, x.z, x.w);
    } else {
      d[0] = x.x; d[stride] = x.y; d[2 * stride] = x.z; d[3 * stride] = x.w;
    }
    return;
  }
  const float v[4] = {x.x, x.y, x.z, x.w};
  if (A.dst_mode == DST_PAIR_SET || A.dst_mode == DST_PAIR_ADD) {
    float2 *d = static_cast<float2 *>(A.dst) + g;
    float2 r[4];
    if (A.dst_mode == DST_PAIR_ADD) {
      if (stride == 1) {
        const float4 a = __ldcg(reinterpret_cast<const float4 *>(d)), b = __ldcg(reinterpret_cast<const float4 *>(d + 2));
        r[0] = make_float2(a.x, a.y); r[1] = make_float2(a.z, a.w);
        r[2] = make_float2(b.x, b.y); r[3] = make_float2(b.z, b.w);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) r[c] = __ldcg(d + c * stride);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) r[c] = pair_add(r[c], v[c]);
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) r[c] = make_float2(v[c], 0.0f);
    }
    if (stride == 1) {
      *reinterpret_cast<float4 *>(d) = make_float4(r[0].x, r[0].y, r[1].x, r[1].y);
      *reinterpret_cast<float4 *>(d + 2) = make_float4(r[2].x, r[2].y, r[3].x, r[3].y);
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) d[c * stride] = r[c];
    }
    if (A.f64) {
      double w[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) w[c] = f2d_bits(r[c].x) + f2d_bits(r[c].y);
      double *f = A.f64 + g;
      if (stride == 1) {
        *reinterpret_cast<double2 *>(f) = make_double2(w[0], w[1]);
        *reinterpret_cast<double2 *>(f + 2) = make_double2(w[2], w[3]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) f[c * stride] = w[c];
      }
    }
    return;
  }
  double *d = static_cast<double *>(A.dst) + g;   // FP64 set or accumulate
#pragma unroll 1
  for (int c = 0; c < 4; ++c)
    d[c * stride] = A.dst_mode == DST_F64_SET ? f2d_bits(v[c]) : d[c * stride] + f2d_bits(v[c]);
}
__device__ __forceinline__ void store_dst4(const Store<double> &A, int g, int stride, const Quad<double> &x) {
  double *d = static_cast<double *>(A.dst) + g;   // FP64 passes: DST_WORK and DST_F64_SET alike
  if (stride == 1) {
    *reinterpret_cast<double2 *>(d) = make_double2(x.x, x.y);
    *reinterpret_cast<double2 *>(d + 2) = make_double2(x.z, x.w);
  } else {
    d[0] = x.x; d[stride] = x.y; d[2 * stride] = x.z; d[3 * stride] = x.w;
  }
}

// Division by an eigenvalue sum. FP32: to nearest where the axis's general pass rounds to nearest
// (A.ieee_div), else the approximate one of the compile-time pass (2 ulp, and zero for divisors beyond 2^126),
// whose bits this pass shares. To nearest: the quotient of an approximate reciprocal, corrected once by
// its exact remainder (Markstein, IBM J. Res. Dev. 34, 1990), for divisors that A.div_scale brings into
// the middle of the range. Of 2^30 random quotients one differs from the IEEE one, by an ulp (errors up to
// 0.50000003 ulp; fdividef 2.1); the IEEE operator itself cost the 400^2 solve 2 us (59.4 against 57.5).
// IEEE: the kernel holds both; those without keep the registers of the approximate one.
template <bool IEEE>
__device__ __forceinline__ float divide(float a, float b, bool ieee) {
  if constexpr (IEEE) {
    if (ieee) {
      float y;
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(b));
      const float q = __fmul_rn(a, y);
      return __fmaf_rn(__fmaf_rn(-q, b, a), y, q);
    }
  }
  return __fdividef(a, b);
}
template <bool IEEE>
__device__ __forceinline__ double divide(double a, double b, bool) { return a / b; }

// A tile in registers: line l (l < valid) starts at cell b0 + l * bstep and runs at `stride`.
struct Tile {
  int L, lbits, M, LS, kind, stride, b0, bstep, valid;
  unsigned half_magic;
  bool col;
};
template <typename Real>
__device__ __forceinline__ Tile tile_of(const PassArgs<Real> &A, int tile) {
  Tile t;
  t.L = A.L;
  t.lbits = A.lbits;
  t.M = A.M;
  t.LS = A.ls;
  t.kind = A.kind;
  t.half_magic = A.half_magic;
  t.col = A.col;
  if (t.col) {
    const int per = A.tiles_per_outer, o = tile / per, f0 = (tile - o * per) * t.L;
    t.stride = A.stride;
    t.b0 = o * A.n * A.stride + f0;
    t.bstep = 1;
    t.valid = A.inner - f0;
  } else {
    t.stride = 1;
    t.b0 = tile * t.L * A.n;
    t.bstep = A.n;
    t.valid = A.lines - tile * t.L;
  }
  return t;
}
// Line and quad (or pair) of item i of a tile: across the lines on column tiles (coalesced over
// adjacent lines), along the line on row tiles.
__device__ __forceinline__ void item_of(const Tile &t, bool across, int i, int &l, int &q) {
  if (across) {
    l = i & (t.L - 1);
    q = i >> t.lbits;
  } else {
    l = fdiv(i, t.half_magic);
    q = i - l * (t.M >> 1);
  }
}

// Eigenvalue sum of the other axes on the lines of a dividing tile (axis 0: a line's first cell is
// the flat index of its other axes).
template <typename Real>
__device__ __forceinline__ void fill_lambda(const PassArgs<Real> &A, const Tile &t, Real *lam) {
  if ((int)threadIdx.x < t.L) {
    const int f = t.b0 + (int)threadIdx.x;
    Real lo = 1;
    if ((int)threadIdx.x < t.valid) {
      if (A.dim == 2) {
        lo = __ldg(A.lam[1] + f);
      } else {
        const int n2 = A.shape[2], i1 = f / n2;
        lo = (Real)0 + __ldg(A.lam[1] + i1);
        lo += __ldg(A.lam[2] + (f - i1 * n2));
      }
    }
    lam[threadIdx.x] = lo;
  }
}

// Post-processing, division (the zero mode of a singular problem: coefficient 0 of the line at
// cell 0) and pre-processing between the two halves of a dividing pass, pair by pair in registers,
// in place.
template <typename Real, int FAM, bool IEEE, typename Tables>
__device__ __forceinline__ void divide_tile(const PassArgs<Real> &A, const Tile &t, typename Cplx<Real>::T *z,
                                            const Real *lam, const Tables &tb) {
  using T = typename Cplx<Real>::T;
  const int M = t.M, total = t.L * (M >> 1);
  const bool dv = A.do_div, ieee = A.ieee_div, singular = A.singular && t.b0 == 0;
  const Real sc = IEEE ? A.div_scale : (Real)1;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    int l, k, qa, qb, pos[4];
    item_of(t, false, i, l, k);
    T *line = z + l * t.LS;
    Real val[4];
    pair_positions<FAM>(M, k, t.kind, pos);
    pair_slots<FAM>(M, k, qa, qb);
    T *pa = line + at<Real>(qa), *pb = line + at<Real>(qb);
    fwd_values<FAM>(*pa, *pb, M, k, t.kind, tb, val);
    if (dv) {
      const Real lo = lam[l] * sc;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        val[c] = (singular && l == 0 && pos[c] == 0) ? (Real)0 : divide<IEEE>(val[c], fma_rn(tb.lam(pos[c]), sc, lo), ieee);
    }
    T za, zb;
    inv_values<FAM>(val, M, k, t.kind, tb, za, zb);
    *pa = za;
    *pb = zb;
  }
}
// Coefficients of a forward-only pass to global memory.
template <typename Real, int FAM, typename Tables>
__device__ __forceinline__ void store_coefs(const PassArgs<Real> &A, const Tile &t, const typename Cplx<Real>::T *z,
                                            const Tables &tb) {
  using T = typename Cplx<Real>::T;
  const int M = t.M, total = t.L * (M >> 1);
  Real *d = static_cast<Real *>(A.dst) + t.b0;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    int l, k, qa, qb, pos[4];
    item_of(t, t.col, i, l, k);
    if (l >= t.valid) continue;
    const T *line = z + l * t.LS;
    Real val[4];
    pair_positions<FAM>(M, k, t.kind, pos);
    pair_slots<FAM>(M, k, qa, qb);
    fwd_values<FAM>(line[at<Real>(qa)], line[at<Real>(qb)], M, k, t.kind, tb, val);
    Real *dl = d + l * t.bstep;
#pragma unroll
    for (int c = 0; c < 4; ++c) dl[pos[c] * t.stride] = val[c];
  }
}
// Coefficients of an inverse-only pass from global memory into the slots.
template <typename Real, int FAM, typename Tables>
__device__ __forceinline__ void load_coefs(const PassArgs<Real> &A, const Tile &t, typename Cplx<Real>::T *z,
                                           const Tables &tb) {
  using T = typename Cplx<Real>::T;
  const int M = t.M, total = t.L * (M >> 1);
  const Real *s = static_cast<const Real *>(A.src) + t.b0;
#pragma unroll 2
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    int l, k, qa, qb, pos[4];
    item_of(t, t.col, i, l, k);
    Real val[4] = {0, 0, 0, 0};
    pair_positions<FAM>(M, k, t.kind, pos);
    if (l < t.valid) {
      const Real *sl = s + l * t.bstep;
#pragma unroll
      for (int c = 0; c < 4; ++c) val[c] = __ldcg(sl + pos[c] * t.stride);
    }
    pair_slots<FAM>(M, k, qa, qb);
    T za, zb, *line = z + l * t.LS;
    inv_values<FAM>(val, M, k, t.kind, tb, za, zb);
    line[at<Real>(qa)] = za;
    line[at<Real>(qb)] = zb;
  }
}

// One pass over a tile: [forward transform] [division] [inverse transform] as A asks. quad(l, base,
// qd, stride) yields the input values at positions 4 qd .. 4 qd + 3 of line l (first cell base), and
// put(l, base, qd, stride, x) takes the outputs of a final inverse. buf: two buffers of L lines, then the
// lines' eigenvalue sums. The two halves share one copy of the FFT (a loop that is not unrolled). The
// caller puts a barrier before it; it ends without.
template <typename Real, bool IEEE, typename Tables, typename QuadFn, typename PutFn>
__device__ __forceinline__ void pass_tile(const PassArgs<Real> &A, int tile, typename Cplx<Real>::T *buf,
                                          const Tables &tb, const typename Cplx<Real>::T *w16tab, QuadFn quad, PutFn put) {
  using T = typename Cplx<Real>::T;
  const Tile t = tile_of(A, tile);
  const int M = t.M, fam = A.fam, total = t.L * (M >> 1);
  T *a = buf, *b = buf + t.L * t.LS;
  Real *lam = reinterpret_cast<Real *>(b + t.L * t.LS);
  const bool fwd = A.do_fwd, inv = A.do_inv;
  if (A.do_div) fill_lambda(A, t, lam);
  if (fwd) {
#pragma unroll 2
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
      int l, qd;
      item_of(t, t.col, i, l, qd);
      Quad<Real> x{0, 0, 0, 0};
      if (l < t.valid) x = quad(l, t.b0 + l * t.bstep, qd, t.stride);
      scatter_quad<Real>(a + l * t.LS, M, fam, t.kind, qd, x);
    }
  } else {
    if (fam == 0) load_coefs<Real, 0>(A, t, a, tb);
    else if (fam == 1) load_coefs<Real, 1>(A, t, a, tb);
    else load_coefs<Real, 2>(A, t, a, tb);
  }
  __syncthreads();
#pragma unroll 1
  for (int half = fwd ? 0 : 1; half < (inv ? 2 : 1); ++half) {
    fft<Real>(A, t.L, t.LS, a, b, tb, fam == 2 && half == 0 ? tw_dct4pre(M) : -1, w16tab);
    if (half == 0 && inv) {
      if (fam == 0) divide_tile<Real, 0, IEEE>(A, t, a, lam, tb);
      else if (fam == 1) divide_tile<Real, 1, IEEE>(A, t, a, lam, tb);
      else divide_tile<Real, 2, IEEE>(A, t, a, lam, tb);
      __syncwarp();
      __syncthreads();
    }
  }
  if (!inv) {
    if (fam == 0) store_coefs<Real, 0>(A, t, a, tb);
    else if (fam == 1) store_coefs<Real, 1>(A, t, a, tb);
    else store_coefs<Real, 2>(A, t, a, tb);
    return;
  }
  const Real scale = A.out_scale;
#pragma unroll 2
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    int l, qd;
    item_of(t, t.col, i, l, qd);
    if (l >= t.valid) continue;
    Quad<Real> x = gather_quad<Real>(a + l * t.LS, M, fam, t.kind, qd, tb);
    x.x = mul_rn(x.x, scale);
    x.y = mul_rn(x.y, scale);
    x.z = mul_rn(x.z, scale);
    x.w = mul_rn(x.w, scale);
    put(l, t.b0 + l * t.bstep, qd, t.stride, x);
  }
}

// The pass on its plain source.
template <typename Real, bool IEEE>
__device__ __forceinline__ void pass_tile(const PassArgs<Real> &A, int tile, typename Cplx<Real>::T *buf,
                                          const typename Cplx<Real>::T *w16tab) {
  const void *src = A.src;
  const int mode = A.src_mode;
  const GlobalTables<Real> tb{A.tw, A.stw, A.lam[A.axis]};
  const Store<Real> out = store_of(A);
  pass_tile<Real, IEEE>(
      A, tile, buf, tb, w16tab,
      [&](int, int base, int qd, int stride) { return load_src4<Real>(src, mode, base + 4 * qd * stride, stride); },
      [&](int, int base, int qd, int stride, const Quad<Real> &x) { store_dst4(out, base + 4 * qd * stride, stride, x); });
}

}  // namespace loop
}  // namespace pc
