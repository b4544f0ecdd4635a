// Transform-based Poisson solve on the pressure grid (§2.3, three-step algorithm):
//   1. forward 1D transforms along each axis in turn,
//   2. division by the sum of the 1D eigenvalues of the central-difference Laplacian,
//   3. backward 1D transforms.
// One kernel launch per axis pass; grids up to about a million cells take all the passes of a solve in
// one launch (resident.cu, resident64.cu). The contiguous (last) axis is processed in row tiles, the
// other axes in column tiles of adjacent lines so that every global access is coalesced without a
// transpose. The division is fused into the pass of axis 0, which does its forward
// transform, the division and its inverse transform on the tile while it sits in shared memory.
// 2D: [fwd ax1] -> [fwd ax0, divide, inv ax0] -> [inv ax1]; 3D adds ax1 passes around the middle.
//
// Mixed precision: the transforms run in FP32; the iterate p is kept as FP32 (hi, lo) pairs and corrected
// by sweeps p += solve32(s - L_h p) whose residual is formed on such pairs (iterative refinement).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "lean_pass.cuh"
#include "loop_pass.cuh"
#include "resident.cuh"

namespace pc {

// ----------------------------------------------------------------------------- host side

// Radix schedule of a length-M FFT with at most E slots per thread: the largest power-of-two
// radices up to min(E, 16) first, then the factors 3 and 5.
static void radix_plan(int M, int E, int *radix, int &nr) {
  nr = 0;
  int m = M;
  int rmax = E < 16 ? E : 16;
  if (rmax < 2) rmax = 2;
  for (int r = rmax; r >= 2; r >>= 1)
    while (m % r == 0) { radix[nr++] = r; m /= r; }
  while (m % 3 == 0) { radix[nr++] = 3; m /= 3; }
  while (m % 5 == 0) { radix[nr++] = 5; m /= 5; }
}

static int ilog2(int v) {
  int b = 0;
  while ((1 << b) < v) ++b;
  return b;
}

// A complex FFT length the passes take: 2^a 3^b 5^c, at most 2048.
static bool fft_length_supported(int M) {
  if (M < 2 || M > 2048) return false;
  int m = M;
  for (int r : {2, 3, 5}) while (m % r == 0) m /= r;
  return m == 1;
}

bool axis_length_supported(int n) { return n >= 2 && (n & 1) == 0 && fft_length_supported(n / 2); }

int fft_length_of(int kind, int n) {
  if (kind == KIND_VNN) return n - 1;   // DCT-I of m + 1 unknowns: real DFT of length 2m
  if (kind == KIND_VDD) return n + 1;   // DST-I of m - 1 unknowns: real DFT of length 2m
  return n / 2;
}

bool vertex_axis_supported(int kind, int m) {
  if (kind == KIND_VNN || kind == KIND_VDD) return fft_length_supported(m);
  return axis_length_supported(m);   // P-P and the quarter-wave pairs: length m, m even
}

// Schedule of the looped passes of a cell-grid axis: variant 0 of the length's compile-time pass
// where it has one; else the power of two in radices of 16 and 8, then 3 and 5. Every stage has at
// least two butterflies per line. Returns false where the axis has no looped pass.
static bool loop_schedule(AxisInfo &ax) {
  const int M = ax.M;
  ax.loop_nst = 0;
  if (pass_family(ax.kind) > 2 || (M & 1) || M < 6) return false;
  int radix[kMaxRadices], nr = 0;
  if (lean::length_ok(M)) {
    for (int s = 0; lean::radix_of(M, 0, s) > 0; ++s) radix[nr++] = lean::radix_of(M, 0, s);
  } else {
    int m = M, two = 0;
    while (m % 2 == 0) { m /= 2; ++two; }
    if (m == 1 && two == 3) { radix[nr++] = 4; radix[nr++] = 2; two = 0; }   // M = 8
    while (two >= 6 || two == 4) { radix[nr++] = 16; two -= 4; }
    if (two == 5) { radix[nr++] = 8; two = 2; }
    if (two) radix[nr++] = 1 << two;
    while (m % 3 == 0) { radix[nr++] = 3; m /= 3; }
    while (m % 5 == 0) { radix[nr++] = 5; m /= 5; }
  }
  int Ns = 1, off = 0;
  for (int s = 0; s < nr; ++s) {
    StageInfo &si = ax.loop_st[s];
    si.R = radix[s];
    si.Ns = Ns;
    si.stride_m = off;
    si.shift = ((Ns & (Ns - 1)) == 0) ? ilog2(Ns) : -1;
    si.magic = (unsigned)(((1ULL << 32) + Ns - 1) / Ns);
    si.mr = M / si.R;
    if (si.mr < 2) return false;
    si.mr_magic = (unsigned)(((1ULL << 32) + si.mr - 1) / si.mr);
    if (Ns > 1) off += (si.R - 1) * Ns;
    Ns *= si.R;
  }
  if (Ns != M) return false;
  ax.loop_nst = nr;
  return true;
}
static int loop_twiddles(const AxisInfo &ax) {
  int n = 0;
  for (int s = 0; s < ax.loop_nst; ++s)
    if (ax.loop_st[s].Ns > 1) n += (ax.loop_st[s].R - 1) * ax.loop_st[s].Ns;
  return n;
}

pc_status build_axis_tables(Plan *p) {
  for (int a = 0; a < p->dim; ++a) {
    AxisInfo &ax = p->ax[a];
    const int n = ax.n, M = fft_length_of(ax.kind, n);
    const int nt = 2 * M;   // length of the real transform the FFT serves (n for cell kinds)
    ax.M = M;
    std::vector<double2> tw(tw_total(M));
    auto put = [&](int off, int k, double ang) { tw[off + k] = make_double2(std::cos(ang), std::sin(ang)); };
    const double pi = 3.14159265358979323846;
    for (int k = 0; k < M; ++k) put(0, k, -2.0 * pi * k / M);
    for (int k = 0; k <= M; ++k) put(tw_rdft(M), k, -2.0 * pi * k / nt);
    for (int k = 0; k <= M; ++k) put(tw_quarter(M), k, -pi * k / (2.0 * nt));
    for (int k = 0; k < M; ++k) put(tw_dct4pre(M), k, -pi * (4.0 * k + 1.0) / (4.0 * nt));
    for (int k = 0; k < M; ++k) put(tw_dct4post(M), k, -pi * k / (double)nt);
    // stage twiddles of the looped passes, w_{Ns R}^{r k} = w_M^{r k M/(Ns R)} with k fast
    loop_schedule(ax);
    tw.resize(tw_total(M) + loop_twiddles(ax));
    for (int s = 0; s < ax.loop_nst; ++s) {
      const StageInfo &si = ax.loop_st[s];
      if (si.Ns == 1) continue;
      const int step = M / (si.Ns * si.R);
      for (int r = 1; r < si.R; ++r)
        for (int k = 0; k < si.Ns; ++k) tw[tw_total(M) + si.stride_m + (r - 1) * si.Ns + k] = tw[r * k * step];
    }
    std::vector<float2> tw32(tw.size());
    for (size_t i = 0; i < tw.size(); ++i) tw32[i] = make_float2((float)tw[i].x, (float)tw[i].y);
    // eigenvalues per spectral index with the angle theta of each basis vector (th = theta/2):
    // central finite differences -(4/h^2) sin^2(theta/2), pseudo-spectral -(theta/h)^2
    std::vector<double> lam(n);
    std::vector<float> lam32(n);
    const double c = -4.0 / (ax.h * ax.h);
    for (int m = 0; m < n; ++m) {
      double th;  // sin argument
      switch (ax.kind) {
        case KIND_PP: {
          int w = (m == 0) ? 0 : (m == 1 ? n / 2 : m / 2);
          th = pi * w / n;
          break;
        }
        case KIND_NN: th = pi * m / (2.0 * n); break;
        case KIND_DD: th = pi * (m + 1.0) / (2.0 * n); break;
        // vertex grids: M cells on DCT-I / DST-I axes, basis cos(pi k j/M) and sin(pi (k+1) j/M)
        // for coefficient k; n cells on quarter-wave axes, theta = pi (k + 1/2)/n
        case KIND_VNN: th = pi * m / (2.0 * M); break;
        case KIND_VDD: th = pi * (m + 1.0) / (2.0 * M); break;
        default: th = pi * (2.0 * m + 1.0) / (4.0 * n); break;   // ND, DN, VND, VDN
      }
      double s = std::sin(th);
      lam[m] = p->eigen == PC_EIG_SPECTRAL ? -(2.0 * th / ax.h) * (2.0 * th / ax.h) : c * s * s;
      lam32[m] = (float)lam[m];
    }
    PC_TRY(plan_alloc(p, (void **)&ax.tw64, tw.size() * sizeof(double2)));
    PC_TRY(plan_alloc(p, (void **)&ax.tw32, tw32.size() * sizeof(float2)));
    PC_TRY(plan_alloc(p, (void **)&ax.lam64, n * sizeof(double)));
    PC_TRY(plan_alloc(p, (void **)&ax.lam32, n * sizeof(float)));
    PC_CUDA_TRY(cudaMemcpy(ax.tw64, tw.data(), tw.size() * sizeof(double2), cudaMemcpyHostToDevice));
    PC_CUDA_TRY(cudaMemcpy(ax.tw32, tw32.data(), tw32.size() * sizeof(float2), cudaMemcpyHostToDevice));
    PC_CUDA_TRY(cudaMemcpy(ax.lam64, lam.data(), n * sizeof(double), cudaMemcpyHostToDevice));
    PC_CUDA_TRY(cudaMemcpy(ax.lam32, lam32.data(), n * sizeof(float), cudaMemcpyHostToDevice));
  }
  return PC_OK;
}

// The common part of a pass's arguments: axis, geometry, tables, source and destination.
template <typename Real>
static void fill_pass(const Plan *p, const PassSpec &ps, PassArgs<Real> &A) {
  using T = typename Cplx<Real>::T;
  const AxisInfo &ax = p->ax[ps.axis];
  memset(&A, 0, sizeof(A));
  A.axis = ps.axis;
  A.kind = ax.kind;
  A.n = ax.n;
  A.M = ax.M;
  A.tw = (const T *)(sizeof(Real) == 8 ? (const void *)ax.tw64 : (const void *)ax.tw32);
  A.dim = p->dim;
  int stride = 1;
  for (int b = 0; b < p->dim; ++b) A.shape[b] = (int)p->n[b];
  for (int b = ps.axis + 1; b < p->dim; ++b) stride *= (int)p->n[b];
  A.stride = stride;
  A.col = ps.axis != p->dim - 1;
  A.do_fwd = ps.fwd;
  A.do_div = ps.div;
  A.do_inv = ps.inv;
  for (int b = 0; b < p->dim; ++b)
    A.lam[b] = (const Real *)(sizeof(Real) == 8 ? (const void *)p->ax[b].lam64 : (const void *)p->ax[b].lam32);
  A.singular = p->singular;
  A.src_mode = ps.src_mode;
  A.src = ps.src;
  A.dst_mode = ps.dst_mode;
  A.dst = ps.dst;
  A.out_scale = (Real)inv_scale(ax.M);
  A.f64 = ps.f64;
  A.gate = ps.gate;
  A.chunk = ps.chunk > 1 ? ps.chunk : 1;
}

// Tiles of L lines of a pass.
template <typename Real>
static long long fill_tiles(const Plan *p, PassArgs<Real> &A, int L) {
  long long tiles;
  if (A.col) {
    const long long outer = p->ncells / ((long long)A.stride * A.n);
    A.inner = A.stride;
    A.tiles_per_outer = (A.stride + L - 1) / L;
    tiles = outer * A.tiles_per_outer;
  } else {
    const long long lines = p->ncells / A.n;
    A.lines = (int)lines;
    tiles = (lines + L - 1) / L;
  }
  A.L = L;
  A.lbits = ilog2(L);
  A.ntiles = (int)tiles;
  return tiles;
}

// A looped pass with tiles of L lines (L a power of two).
template <typename Real>
static long long fill_loop(const Plan *p, const PassSpec &ps, PassArgs<Real> &A, int L) {
  using T = typename Cplx<Real>::T;
  const AxisInfo &ax = p->ax[ps.axis];
  fill_pass<Real>(p, ps, A);
  A.loop = 1;
  A.fam = pass_family(ax.kind);
  A.ieee_div = !lean::length_ok(ax.M);   // lengths with a compile-time pass keep its division, and its bits
  A.div_scale = 1;
  if (sizeof(Real) == 4 && ps.div && A.ieee_div) {
    double top = 0.0;   // of the eigenvalue sums, FD or spectral
    for (int a = 0; a < p->dim; ++a) top += 9.87 / (p->h[a] * p->h[a]);
    A.div_scale = (Real)(top > 0x1p100 ? 0x1p-64 : (top < 0x1p-60 ? 0x1p64 : 1.0));
    A.out_scale *= A.div_scale;
  }
  A.nst = ax.loop_nst;
  for (int s = 0; s < ax.loop_nst; ++s) A.st[s] = ax.loop_st[s];
  A.stw = A.tw + tw_total(ax.M);
  A.half_magic = (unsigned)(((1ULL << 32) + ax.M / 2 - 1) / (ax.M / 2));
  A.ls = loop::line_slots<Real>(ax.M, L);
  return fill_tiles<Real>(p, A, L);
}

// Slots of a looped pass's tile: 2048 in FP32 (35 KB: six CTAs of 256 threads per SM) and 1024 in
// FP64 in a launch of its own (4096: 64 2D problems 868 us against 823), up to 4096 on the resident CTAs.
constexpr int kLoopSlots = 2048;

static bool aligned16(const void *q) { return ((uintptr_t)q & 15) == 0; }

// Whether the compile-time and the looped passes can run a pass: they move row tiles in 16-byte
// accesses (16-byte aligned arrays), store forward coefficients as work and read inverse-only
// coefficients in the pass precision.
static bool quad_io(const Plan *p, const PassSpec &ps, bool fp32) {
  const bool row = ps.axis == p->dim - 1;
  return (!ps.fwd || ps.inv || ps.dst_mode == DST_WORK) && (!fp32 || ps.fwd || ps.src_mode != SRC_F64) &&
         (!row || (aligned16(ps.src) && aligned16(ps.dst) && aligned16(ps.f64)));
}

// SMs of a device (of the part of it that the process may use), asked for once.
static int sm_count(int device) {
  static std::atomic<int> known[kMaxDevices];
  if (device < 0 || device >= kMaxDevices) return 1;
  int n = known[device].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || n < 1) n = 1;
    known[device].store(n, std::memory_order_relaxed);
  }
  return n;
}

template <typename Real>
pc_status build_pass(const Plan *p, const PassSpec &ps, PassArgs<Real> &A, long long &tiles, int &threads,
                     size_t &smem, int batch_threads) {
  const int axis = ps.axis;
  const AxisInfo &ax = p->ax[axis];
  const int M = ax.M;
  // slots per thread; 0 and 1 (FP32 only): variant 0 or 1 of the lean pass of the length
  // (lean_pass.cuh) where it has one, else the looped pass (loop_pass.cuh) where it has one, else 4;
  // FP64: 2, the default, the looped pass where the axis has one
  const bool fp32 = sizeof(Real) == 4;
  int E = fp32 ? ax.slots32 : ax.slots64;
  const bool deflt = fp32 ? E <= 1 : E == 2;
  const bool quad = quad_io(p, ps, fp32);
  bool all = true;   // an axis without a looped pass (odd M, vertex kinds): none on the others either
  for (int a = 0; a < p->dim; ++a) all = all && p->ax[a].loop_nst > 0;
  // variant 0 on grids beyond the cooperative solve (192^3: 871 us against 982 with looped passes);
  // below, where many problems share a launch, one kernel for all their lengths and families is the
  // better one (64 2D problems 845 us with up to six lean kernels side by side, 823 looped; 12
  // requests 1572 and 1459). The bits are the same.
  const bool lean = fp32 && deflt && pass_family(ax.kind) <= 2 && lean::length_ok(M) && quad &&
                    (E == 1 || !all || p->ncells > kResidentCells);
  const int lv = E == 1 ? 1 : 0;
  // unrefined solves return the transforms' own rounding (1e-7): their bits stay those of the
  // general pass at the lengths without a compile-time one
  const bool general = fp32 && unrefined(p) && !lean::length_ok(M);
  // FP64 lines of 4096 values leave one CTA per SM its shared memory for (4096 x 128: 229 us against
  // the general pass's 206; 2048 x 256: 160 against 238)
  const bool too_long = !fp32 && M > 1024;
  if (deflt && !lean && quad && all && !general && !too_long) {
    // lines per tile: as many as the slots allow; a problem alone takes fewer where the GPU would
    // not be full (the lines do not depend on it)
    const int slots = fp32 ? kLoopSlots : kLoopSlots / 2;
    int L = axis == p->dim - 1 ? 1 : 4;   // column tiles: four lines fill half a sector in FP32, one in FP64
    while (L < 32 && 2 * L * M <= slots) L *= 2;
    if (batch_threads <= 0) {
      const long long lines = p->ncells / ax.n, sms = sm_count(p->device);
      while (L > 4 && lines / L < 2 * sms) L /= 2;
      while (L > 1 && lines / L < sms) L /= 2;   // few long lines (1024 x 96 in FP64: 152 us at four lines, 57 at one)
    }
    while (L > 1 && loop::tile_smem<Real>(M, L) > 160 * 1024) L /= 2;
    tiles = fill_loop<Real>(p, ps, A, L);
    threads = loop::kThreads;
    smem = loop::tile_smem<Real>(M, L);
    return PC_OK;
  }
  fill_pass<Real>(p, ps, A);
  if (E <= 1) E = 4;
  // threads per line: a power of two with at most E slots per thread; the kernel instance is
  // the smallest power of two >= M / tpl. A line must fit one CTA: longer lines take more
  // slots per thread (up to 16)
  while (E < 16 && (M + E - 1) / E > kMaxPassThreads) E *= 2;
  const int tpl = 1 << ilog2((M + E - 1) / E);
  const int emax = 1 << ilog2((M + tpl - 1) / tpl);
  A.emax = emax;
  if (!lean) {
    int radix[kMaxRadices], nr;
    radix_plan(M, emax, radix, nr);
    A.nst = nr;
    int Ns = 1;
    for (int i = 0; i < nr; ++i) {
      StageInfo &si = A.st[i];
      si.R = radix[i];
      si.Ns = Ns;
      si.stride_m = M / (Ns * si.R);
      si.shift = ((Ns & (Ns - 1)) == 0) ? ilog2(Ns) : -1;
      si.magic = (unsigned)(((1ULL << 32) + Ns - 1) / Ns);
      Ns *= si.R;
    }
  }
  if (lean) {
    // compile-time tile: L lines of T = M / E threads each, 256 threads
    tiles = fill_tiles<Real>(p, A, lean::lines_of(M, lv));
    A.lean = lean::lean_id(M, pass_family(ax.kind));
    threads = lean::kThreads;
    smem = lean::smem_of(M, lv);
    return PC_OK;
  }
  const int stride = A.stride;
  const int max_threads = batch_threads > 0 ? batch_threads : 256;
  const int max_lines = max_threads / tpl > 0 ? max_threads / tpl : 1;
  const int budget = 8192;          // complex slots per tile (two buffers: 2 x 64 KB in FP32)
  // CTAs per SM the tile size aims for (part of the plan's schedule; 152 SMs on both dies)
  const int want_ctas = ((sizeof(Real) == 8) ? ax.ctas64 : ax.ctas32) * 152;
  int L;
  if (A.col) {
    // 32-byte row segments when the grid allows it, fewer lines when CTAs would be too few
    L = 32;
    while (L > 1 && (L * M > budget || L > max_lines)) L /= 2;
    long long outer = p->ncells / ((long long)stride * ax.n);
    const int Lmin = (sizeof(Real) == 8) ? 4 : 8;
    while (L > Lmin && batch_threads <= 0 && outer * ((stride + L - 1) / L) < want_ctas) L /= 2;
    if (L > stride) L = 1 << (ilog2(stride + 1) - 1);
    A.inner = stride;
    A.tiles_per_outer = (stride + L - 1) / L;
    tiles = outer * A.tiles_per_outer;
  } else {
    long long lines = p->ncells / ax.n;
    L = budget / M;
    if (L < 1) L = 1;
    L = 1 << (ilog2(L + 1) - 1);
    while (L > max_lines) L /= 2;
    while (L > 1 && batch_threads <= 0 && (lines + L - 1) / L < want_ctas) L /= 2;
    A.lines = (int)lines;
    tiles = (lines + L - 1) / L;
  }
  A.L = L;
  A.lbits = ilog2(L);
  A.tpl_bits = ilog2(tpl);
  threads = L * tpl;
  A.ntiles = (int)tiles;
  if (threads > kMaxPassThreads || L * M > budget)
    return fail(PC_ERR_UNSUPPORTED, "axis %d: tile of %d x %d too large", axis, L, M);
  if (batch_threads > 0 && emax > kBatchPassEmax)
    return fail(PC_ERR_UNSUPPORTED, "axis %d: %d slots per thread exceed the batched kernel", axis, emax);
  smem = 2 * (size_t)L * M * sizeof(typename Cplx<Real>::T) + (size_t)L * (sizeof(Real) + 2 * sizeof(int));
  return PC_OK;
}

template pc_status build_pass<float>(const Plan *, const PassSpec &, PassArgs<float> &, long long &, int &, size_t &, int);
template pc_status build_pass<double>(const Plan *, const PassSpec &, PassArgs<double> &, long long &, int &, size_t &, int);

template <typename Real>
static pc_status launch_pass(Plan *p, const PassSpec &ps, cudaStream_t st) {
  PassArgs<Real> A;
  long long tiles;
  int threads;
  size_t smem;
  PC_TRY(build_pass<Real>(p, ps, A, tiles, threads, smem, 0));
  tiles = (tiles + A.chunk - 1) / A.chunk;   // CTAs
  if (A.loop) {
    // one instance for all passes of a solve: its code stays in the instruction caches
    if constexpr (sizeof(Real) == 4) PC_TRY(launch_loop(A, nullptr, nullptr, (unsigned)tiles, smem, !lean::length_ok(p->ax[0].M), st));
    else PC_TRY(launch_loop(A, (unsigned)tiles, smem, st));
    count_launch(p);
    return PC_OK;
  }
  if constexpr (sizeof(Real) == 4) {
    if (A.lean) {
      PC_TRY(launch_lean(A.lean, A, nullptr, nullptr, (unsigned)tiles, threads, smem, st));
      count_launch(p);
      return PC_OK;
    }
    // FP32 passes: the instance of the axis's transform family (one translation unit each)
    switch (pass_family(A.kind)) {
      case 0: PC_TRY(launch_pass_f32_family0(A, tiles, threads, smem, st)); break;
      case 1: PC_TRY(launch_pass_f32_family1(A, tiles, threads, smem, st)); break;
      case 2: PC_TRY(launch_pass_f32_family2(A, tiles, threads, smem, st)); break;
      default: PC_TRY(launch_pass_vertex_f32(A, tiles, threads, smem, st)); break;
    }
  } else {
    if (pass_family(A.kind) >= 3) PC_TRY(launch_pass_vertex_f64(A, tiles, threads, smem, st));
    else PC_TRY((launch_axis_pass_spec<Real, -1, false>(A, tiles, threads, smem, st)));
  }
  count_launch(p);
  return PC_OK;
}

// Kernel attributes set once per device, before any stream capture.
constexpr int kPassSmem = 200 * 1024;   // dynamic shared memory of any pass
pc_status prepare_kernels() {
  const int lim = kPassSmem;
  PC_TRY(prepare_pass_f32_family0(lim));
  PC_TRY(prepare_pass_f32_family1(lim));
  PC_TRY(prepare_pass_f32_family2(lim));
  PC_TRY(prepare_pass_vertex(lim));
  PC_TRY(prepare_batched_f32(lim));
  PC_TRY(prepare_lean(lim));
  PC_TRY(prepare_loop(lim));
  PC_TRY(prepare_resident());
  PC_TRY(prepare_resident64());
  PC_TRY((prepare_axis_pass_spec<double, -1, false>(lim)));
  return PC_OK;
}

std::vector<PassSpec> solve_pass_specs(const Plan *p, bool fp32, int src_mode, const void *src,
                                       int dst_mode, void *dst, double *f64, RefineGate gate, int chunk) {
  std::vector<PassSpec> v;
  void *work = fp32 ? (void *)p->work32 : (void *)p->work64;
  const int d = p->dim;
  int cur_mode = src_mode;
  const void *cur = src;
  for (int a = d - 1; a >= 1; --a) {     // forward passes: last axis down to axis 1
    v.push_back(PassSpec{a, true, false, false, cur_mode, cur, DST_WORK, work, nullptr, gate, chunk});
    cur_mode = SRC_WORK;
    cur = work;
  }
  v.push_back(PassSpec{0, true, true, true, cur_mode, cur, DST_WORK, work, nullptr, gate, chunk});   // axis 0, division
  for (int a = 1; a < d; ++a) {         // inverse passes: axis 1 up to the last axis
    const bool final_pass = (a == d - 1);
    v.push_back(PassSpec{a, false, false, true, SRC_WORK, work, final_pass ? dst_mode : DST_WORK,
                         final_pass ? dst : work, final_pass ? f64 : nullptr, gate, chunk});
  }
  return v;
}

// Full solve with Real precision: src (cells, src_mode) -> dst (dst_mode).
template <typename Real>
static pc_status solve_real(Plan *p, int src_mode, const void *src, int dst_mode, void *dst,
                            cudaStream_t st, double *f64 = nullptr, RefineGate gate = RefineGate{nullptr, 0, 0.0f},
                            int chunk = 1) {
  if (p->dim < 2) return fail(PC_ERR_UNSUPPORTED, "dim 1");
  for (const PassSpec &ps : solve_pass_specs(p, sizeof(Real) == 4, src_mode, src, dst_mode, dst, f64, gate, chunk))
    PC_TRY(launch_pass<Real>(p, ps, st));
  return PC_OK;
}

// Slots [first, end) of an axis's table that the wrappers of its family read.
static void tables_of(const AxisInfo &ax, int &first, int &end) {
  const int fam = pass_family(ax.kind), M = ax.M;
  first = fam == 2 ? tw_dct4pre(M) : tw_rdft(M);
  end = fam == 0 ? tw_quarter(M) : fam == 1 ? tw_dct4pre(M) : tw_total(M);
}

// Grids that run as one cluster of 16 CTAs: the hardware barrier saves about 1 us at each of ten
// barriers, the work of more cells per SM costs it again (2D: 128^2 43 us against 49 as a grid of
// all SMs, 160 x 200 62 against 52; 3D: 20^3 80 against 84, 24^3 74 against 72).
constexpr long long kClusterCells2D = 20000, kClusterCells3D = 8192;
static bool cluster_grid(const Plan *p) {
  return p->ncells <= (p->dim == 2 ? kClusterCells2D : kClusterCells3D) && resident_cluster_size(p->device) > 0;
}

// Slots up to which a tile of the cooperative solve takes more lines where more CTAs would not be faster
// (FP64: half of them): the grid leaves SMs to solves on other streams. Projections in us, one after the
// other / on 8 streams: 256^2 mixed 64 CTAs 75.9 / 26.4, 128 CTAs 75.5 / 48.7, 32 CTAs 78.6 / 15.7; 192^2
// 48 CTAs 69.4 / 18.8, 96 CTAs 68.0 / 49.9, 24 CTAs 75.3 / 11.4; 32^3 32 CTAs 115.5 / 21.8, 128 CTAs 113.7 /
// 66.1; FP64 128^2 32 CTAs 54.4 / 10.2, 128 CTAs 54.3 / 35.1; 256^2 64 CTAs 70.9 / 25.4, 128 CTAs 65.8 / 40.7.
constexpr int kSpreadSlots = 512;

// Tiles, tables and own rows of a cooperative solve's passes: lines per tile as few as give every SM
// at most one tile, more while the tile has no more than `spread` slots, and fewer again where the
// buffers would not leave room for the own rows (own_bytes per cell). Behind the tiles: per axis the
// wrappers' factors its family reads, the stage twiddles and, on the dividing pass, the eigenvalues.
template <typename Real>
static bool resident_layout(const Plan *p, const std::vector<PassSpec> &specs, PassArgs<Real> *pass, int sms, int spread,
                            int cap0, int own_bytes, int &grid, int &row_tiles, int &tables_at, int &own_at, size_t &smem) {
  constexpr int kSlot = 2 * (int)sizeof(Real);
  const int np = (int)specs.size(), last = p->dim - 1;
  int slots = 0, at[3][3];
  for (int k = 0; k < p->dim; ++k) {
    const AxisInfo &ax = p->ax[specs[k].axis];
    int *t = at[specs[k].axis], first, end;
    tables_of(ax, first, end);
    t[0] = slots - first;
    slots += end - first;
    t[1] = slots;
    slots += loop_twiddles(ax);
    t[2] = 2 * slots;
    if (specs[k].div) slots += (ax.n + 1) / 2;
  }
  slots = (slots + 1) & ~1;
  bool fits = false;
  for (int cap = cap0; cap >= cap0 / 4 && !fits; cap /= 2) {
    long long most = 0;
    size_t tiles_smem = 0;
    for (int k = 0; k < np; ++k) {
      const int M = p->ax[specs[k].axis].M;
      const long long lines = p->ncells / p->ax[specs[k].axis].n;
      long long run = 1;   // lines side by side: a column tile's do not go beyond
      for (int b = specs[k].axis + 1; b < p->dim; ++b) run *= p->n[b];
      if (specs[k].axis == last) run = lines;
      int L = 1;
      while ((lines + L - 1) / L > sms && 2 * L * M <= cap) L *= 2;
      while (L < run && 2 * L * M <= spread) L *= 2;
      const long long tiles = fill_loop<Real>(p, specs[k], pass[k], L);
      most = tiles > most ? tiles : most;
      const size_t b = loop::tile_smem<Real>(M, L);
      tiles_smem = b > tiles_smem ? b : tiles_smem;
    }
    grid = (int)(most < sms ? most : sms);
    row_tiles = (pass[0].ntiles + grid - 1) / grid;
    tables_at = (int)((tiles_smem + 15) / 16 * 16 / kSlot) + (kSlot == 8 ? 0 : 1);
    own_at = tables_at + slots;
    smem = (size_t)own_at * kSlot + (size_t)row_tiles * pass[0].L * p->ax[last].n * own_bytes;
    fits = smem <= (size_t)kResidentSmem;
  }
  for (int k = 0; k < np; ++k) {
    PassArgs<Real> &A = pass[k];
    const AxisInfo &ax = p->ax[specs[k].axis];
    const int *t = at[specs[k].axis];
    tables_of(ax, A.tw_first, A.tw_last);
    A.tw_at = t[0];
    A.st_at = t[1];
    A.st_count = loop_twiddles(ax);
    A.lam_at = t[2];
  }
  return fits;
}

// A grid that does not fit at once (a context held to fewer SMs than the device reports) is not launched:
// the solve takes one launch per pass.
static pc_status resident_taken(Plan *p, cudaError_t e, bool &taken) {
  if (e == cudaErrorCooperativeLaunchTooLarge) {
    cudaGetLastError();
    return PC_OK;
  }
  PC_CUDA_TRY(e);
  count_launch(p);
  taken = true;
  return PC_OK;
}

pc_status solve_resident(Plan *p, const double *s64, const float2 *s2, double *pout, int sweeps, bool adaptive,
                         float tol, const GridDev &g, cudaStream_t st, bool &taken) {
  taken = false;
  if (p->wait_polls == 0 || p->ncells > kResidentCells || sweeps > kMaxRefine) return PC_OK;
  for (int a = 0; a < p->dim; ++a) {
    if (p->ax[a].slots32 != 0 || p->ax[a].loop_nst == 0) return PC_OK;
    if (unrefined(p) && !lean::length_ok(p->ax[a].M)) return PC_OK;   // see build_pass
  }
  const void *rs = s2 ? (const void *)s2 : (const void *)s64;
  if (!aligned16(rs) || !aligned16(pout)) return PC_OK;
  ResidentArgs R;
  memset(&R, 0, sizeof(R));
  R.cluster = cluster_grid(p);
  size_t smem = 0;
  if (!resident_layout<float>(p, solve_pass_specs(p, true, SRC_F32, rs, DST_PAIR_SET, p->p2), R.pass,
                              R.cluster ? resident_cluster_size(p->device) : sm_count(p->device),
                              R.cluster ? 0 : kSpreadSlots, 2 * kLoopSlots, 16, R.grid, R.row_tiles,
                              R.tables_at, R.own_at, smem))
    return PC_OK;
  R.g = g;
  R.s = rs;
  R.p2 = p->p2;
  R.f64 = pout;
  R.st = p->dstats;
  R.bar = p->dstats->bar;
  R.sweeps = sweeps;
  R.adaptive = adaptive;
  R.singular = p->singular;
  R.tol = tol;
  R.polls = p->wait_polls;
  R.gave_up = p->gave_up;
  return resident_taken(p, launch_resident(R, p->dim, s2 != nullptr, smem, st), taken);
}

// Largest grid of the FP64 solve in one launch (96^3 236 us against 275 by launches, 512^2 76 against
// 80, 1024 x 96 41 against 57), and as one cluster (64^2 with a zero mode 31 against 33; beyond, the
// FP64 pipes of 16 SMs are too few).
constexpr long long kResident64Cells = 1LL << 20, kCluster64Cells = 4096;

pc_status solve_resident64(Plan *p, const double *s, double *pout, int gauge, cudaStream_t st, bool &taken) {
  taken = false;
  if (p->wait_polls == 0 || p->ncells > kResident64Cells || !aligned16(s) || !aligned16(pout)) return PC_OK;
  for (int a = 0; a < p->dim; ++a)
    if (p->ax[a].slots64 != 2 || p->ax[a].loop_nst == 0 || p->ax[a].M > 1024) return PC_OK;
  Resident64Args R;
  memset(&R, 0, sizeof(R));
  R.cluster = p->ncells <= kCluster64Cells && resident_cluster_size(p->device) > 0;
  size_t smem = 0;
  if (!resident_layout<double>(p, solve_pass_specs(p, false, SRC_F64, s, DST_F64_SET, pout), R.pass,
                               R.cluster ? resident_cluster_size(p->device) : sm_count(p->device),
                               R.cluster ? 0 : kSpreadSlots / 2, kLoopSlots, 8, R.grid, R.row_tiles,
                               R.tables_at, R.own_at, smem))
    return PC_OK;
  if (R.grid > 2 * (p->ncells / 256) + 64) return PC_OK;   // the partial sums' array (partial_slots)
  R.s = s;
  R.p = pout;
  R.st = p->dstats;
  R.partials = p->partials;
  R.bar = p->dstats->bar;
  R.gauge = gauge;
  R.inv_cells = 1.0 / (double)p->ncells;
  R.polls = p->wait_polls;
  R.gave_up = p->gave_up;
  return resident_taken(p, launch_resident64(R, p->dim, smem, st), taken);
}

pc_status solve_fp64_grid(Plan *p, const double *s, double *pout, cudaStream_t st) {
  return solve_real<double>(p, SRC_F64, s, DST_F64_SET, pout, st);
}

pc_status solve_fp32_grid(Plan *p, int src_mode, const void *s, int dst_mode, void *dst,
                          cudaStream_t st, double *f64, RefineGate gate, int chunk) {
  return solve_real<float>(p, src_mode, s, dst_mode, dst, st, f64, gate, chunk);
}

}  // namespace pc
