// The real-to-real wrappers of the transform passes around their half-length complex FFT (M slots
// for n = 2M real values), one pair of slots at a time, and the radix-3 and radix-5 butterflies.
// Every kernel that transforms cell-grid lines by pairs (lean_pass.cuh, loop_pass.cuh) takes its
// arithmetic from here, with the order of operations and the fused multiply-adds written out, so
// that a line has the same bits whichever kernel transforms it.
#pragma once

#include "axis_pass.cuh"

namespace pc {

// A pass's tables: the wrappers' factors (tw, layout of fft.cuh's table offsets), the stage twiddles of
// a looped pass and the eigenvalues of its axis, read from global memory through L1, or from a
// CTA's shared memory (a barrier of the grid empties L1, so the resident kernel keeps them there).
template <typename Real>
struct GlobalTables {
  using T = typename Cplx<Real>::T;
  const T *w, *s;
  const Real *l;
  __device__ __forceinline__ T tw(int i) const { return __ldg(w + i); }
  __device__ __forceinline__ T st(int i) const { return __ldg(s + i); }
  __device__ __forceinline__ Real lam(int i) const { return __ldg(l + i); }
};
template <typename Real>
struct SharedTables {
  using T = typename Cplx<Real>::T;
  const T *w, *s;
  const Real *l;
  __device__ __forceinline__ T tw(int i) const { return w[i]; }
  __device__ __forceinline__ T st(int i) const { return s[i]; }
  __device__ __forceinline__ Real lam(int i) const { return l[i]; }
};

// e^{-2 pi i/3}: cos = -1/2, sin = -sqrt(3)/2
template <typename T>
__device__ __forceinline__ void dft3(T &a0, T &a1, T &a2) {
  using R = decltype(T::x);
  const R c = (R)0.86602540378443864676;
  const T s = cadd(a1, a2), d = csub(a1, a2);
  const T t = cmk<T>(fma_rn((R)-0.5, s.x, a0.x), fma_rn((R)-0.5, s.y, a0.y));
  a0 = cadd(a0, s);
  // y1 = t - i c d, y2 = t + i c d
  a1 = cmk<T>(fma_rn(c, d.y, t.x), fma_rn(-c, d.x, t.y));
  a2 = cmk<T>(fma_rn(-c, d.y, t.x), fma_rn(c, d.x, t.y));
}

// Radix 5 by the sums and differences of the mirrored inputs: cos and sin of 2 pi/5 and 4 pi/5.
template <typename T>
__device__ __forceinline__ void dft5(T *v) {
  using R = decltype(T::x);
  const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;
  const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;
  const T p = cadd(v[1], v[4]), m = csub(v[1], v[4]), q = cadd(v[2], v[3]), k = csub(v[2], v[3]);
  const T a = cmk<T>(fma_rn(c1, p.x, fma_rn(c2, q.x, v[0].x)), fma_rn(c1, p.y, fma_rn(c2, q.y, v[0].y)));
  const T b = cmk<T>(fma_rn(c2, p.x, fma_rn(c1, q.x, v[0].x)), fma_rn(c2, p.y, fma_rn(c1, q.y, v[0].y)));
  // -i times these is added to outputs 1, 2 and subtracted from 4, 3
  const T g = cmk<T>(fma_rn(s1, m.x, mul_rn(s2, k.x)), fma_rn(s1, m.y, mul_rn(s2, k.y)));
  const T h = cmk<T>(fma_rn(s2, m.x, -mul_rn(s1, k.x)), fma_rn(s2, m.y, -mul_rn(s1, k.y)));
  v[0] = cadd(v[0], cadd(p, q));
  v[1] = cmk<T>(a.x + g.y, a.y - g.x);
  v[4] = cmk<T>(a.x - g.y, a.y + g.x);
  v[2] = cmk<T>(b.x + h.y, b.y - h.x);
  v[3] = cmk<T>(b.x - h.y, b.y + h.x);
}

// Forward DFT of radix R in registers (2, 3, 4, 5, 8, 16), natural order.
template <int R, typename T>
__device__ __forceinline__ void dft_small(T *v) {
  if constexpr (R == 3) dft3(v[0], v[1], v[2]);
  else if constexpr (R == 5) dft5(v);
  else small_dft<T, R, false>(v, nullptr, 0);
}

// Natural coefficient index -> position in the pass's coefficient layout (DST-II reversed).
template <int FAM>
__device__ __forceinline__ int coef_pos(int kind, int n, int i) {
  return (FAM == 1 && kind == KIND_DD) ? n - 1 - i : i;
}

// The four coefficient positions of pair k (k in [0, M/2)) in the order fwd_values and inv_values
// use: family 0 the packed real DFT [X0, X_{n/2}, Re X1, Im X1, ...] (k = 0: X0, X_{n/2} and
// the self-paired V_{M/2}); family 1 X_k, X_{n-k}, X_{M-k}, X_{M+k} (k = 0: X_0, X_M, X_{M/2},
// X_{n-M/2}), DST-II reversed; family 2 X_2q, X_{n-1-2q} for q = k and q = M - 1 - k.
template <int FAM>
__device__ __forceinline__ void pair_positions(int M, int k, int kind, int (&pos)[4]) {
  const int n = 2 * M;
  if constexpr (FAM == 2) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = h == 0 ? k : M - 1 - k;
      pos[2 * h] = 2 * q;
      pos[2 * h + 1] = n - 1 - 2 * q;
    }
  } else if constexpr (FAM == 0) {
    if (k == 0) { pos[0] = 0; pos[1] = 1; pos[2] = M; pos[3] = M + 1; }
    else { pos[0] = 2 * k; pos[1] = 2 * k + 1; pos[2] = 2 * (M - k); pos[3] = 2 * (M - k) + 1; }
  } else {
    const int i0 = (k == 0) ? 0 : k, i1 = (k == 0) ? M : n - k, i2 = (k == 0) ? M / 2 : M - k,
              i3 = (k == 0) ? n - M / 2 : M + k;
    pos[0] = coef_pos<FAM>(kind, n, i0);
    pos[1] = coef_pos<FAM>(kind, n, i1);
    pos[2] = coef_pos<FAM>(kind, n, i2);
    pos[3] = coef_pos<FAM>(kind, n, i3);
  }
}

// The slots of pair k: families 0 and 1 slots k and M - k (k = 0: slots 0 and M/2), family 2 slots
// k and M - 1 - k.
template <int FAM>
__device__ __forceinline__ void pair_slots(int M, int k, int &qa, int &qb) {
  qa = k;
  if constexpr (FAM == 2) qb = M - 1 - k;
  else qb = k == 0 ? M / 2 : M - k;
}

// Forward post-processing of pair k from its two slots za, zb of the FFT: the four coefficients at
// pair_positions. Family 0: real DFT in packed order; family 1: DCT-II (DST-II reversed); family
// 2: DCT-IV / DST-IV.
template <int FAM, typename T, typename Tables>
__device__ __forceinline__ void fwd_values(T za, T zb, int M, int k, int kind, const Tables &tb,
                                           decltype(T::x) (&val)[4]) {
  using R = decltype(T::x);
  if constexpr (FAM == 2) {
    const int tp = tw_dct4post(M);
    const T ya = cmul(za, tb.tw(tp + k)), yb = cmul(zb, tb.tw(tp + M - 1 - k));
    val[0] = ya.x;
    val[1] = (kind == KIND_ND) ? -ya.y : ya.y;
    val[2] = yb.x;
    val[3] = (kind == KIND_ND) ? -yb.y : yb.y;
  } else {
    const int wq = tw_quarter(M);
    if (k == 0) {
      const R V0 = za.x + za.y, VM = za.x - za.y;
      const T Vh = cmk<T>(zb.x, -zb.y);   // V_{M/2} = conj Z_{M/2}
      if constexpr (FAM == 0) {
        val[0] = V0;
        val[1] = VM;
        val[2] = Vh.x;
        val[3] = Vh.y;
      } else {
        const T th = cmul(Vh, tb.tw(wq + M / 2));
        val[0] = V0;
        val[1] = mul_rn(tb.tw(wq + M).x, VM);
        val[2] = th.x;
        val[3] = -th.y;
      }
      return;
    }
    // V_k = E + w^k O, V_{M-k} = conj(E - w^k O); E = (Z_k + conj Z_{M-k})/2, O = -i (Z_k - conj Z_{M-k})/2
    const T Eh = cmk<T>((R)0.5 * (za.x + zb.x), (R)0.5 * (za.y - zb.y));
    const T O = cmk<T>((R)0.5 * (za.y + zb.y), (R)-0.5 * (za.x - zb.x));
    const T Ow = cmul(O, tb.tw(tw_rdft(M) + k));
    const T Vk = cmk<T>(Eh.x + Ow.x, Eh.y + Ow.y);
    const T Vm = cmk<T>(Eh.x - Ow.x, Ow.y - Eh.y);
    if constexpr (FAM == 0) {
      val[0] = Vk.x;
      val[1] = Vk.y;
      val[2] = Vm.x;
      val[3] = Vm.y;
    } else {
      // t = e^{-i pi k/(2n)} V_k: X_k = Re t, X_{n-k} = -Im t
      const T tk = cmul(Vk, tb.tw(wq + k)), tm = cmul(Vm, tb.tw(wq + M - k));
      val[0] = tk.x;
      val[1] = -tk.y;
      val[2] = tm.x;
      val[3] = -tm.y;
    }
  }
}

// Inverse pre-processing of pair k from its four coefficients: the conjugated slots the forward FFT
// then inverts (family 2: the slots themselves, DCT-IV being its own inverse up to 2/n).
template <int FAM, typename T, typename Tables>
__device__ __forceinline__ void inv_values(const decltype(T::x) (&val)[4], int M, int k, int kind,
                                           const Tables &tb, T &za, T &zb) {
  using R = decltype(T::x);
  if constexpr (FAM == 2) {
    const int t4 = tw_dct4pre(M);
    const T a = (kind == KIND_ND) ? cmk<T>(val[0], val[1]) : cmk<T>(val[1], val[0]);   // X_2q, X_{n-1-2q}
    const T b = (kind == KIND_ND) ? cmk<T>(val[2], val[3]) : cmk<T>(val[3], val[2]);
    za = cmul(a, tb.tw(t4 + k));
    zb = cmul(b, tb.tw(t4 + M - 1 - k));
  } else {
    const int wq = tw_quarter(M);
    if (k == 0) {
      R a, b;
      T xh;   // the self-paired coefficient V_{M/2}
      if constexpr (FAM == 0) {
        a = val[0];
        b = val[1];
        xh = cmk<T>(val[2], val[3]);
      } else {
        const T wM = tb.tw(wq + M);
        a = val[0];
        b = fma_rn(val[1], wM.x, -mul_rn(val[1], wM.y));   // Re V_M, V_M = (X_M - i X_M) conj(wq_M)
        xh = cmulc(cmk<T>(val[2], -val[3]), tb.tw(wq + M / 2));
      }
      za = cmk<T>((R)0.5 * (a + b), (R)-0.5 * (a - b));   // conj Z_0
      zb = xh;                                            // conj Z_{M/2} = V_{M/2}
      return;
    }
    T xk, xm;   // V_k, V_{M-k}
    if constexpr (FAM == 0) {
      xk = cmk<T>(val[0], val[1]);
      xm = cmk<T>(val[2], val[3]);
    } else {
      // V_i = (X_i - i X_{n-i}) e^{+i pi i/(2n)}
      xk = cmulc(cmk<T>(val[0], -val[1]), tb.tw(wq + k));
      xm = cmulc(cmk<T>(val[2], -val[3]), tb.tw(wq + M - k));
    }
    // Z_k = E + i O, Z_{M-k} = conj(E - i O); E = (V_k + conj V_{M-k})/2, O = (V_k - conj V_{M-k}) conj(w^k)/2
    const T Eh = cmk<T>((R)0.5 * (xk.x + xm.x), (R)0.5 * (xk.y - xm.y));
    const T D = cmk<T>((R)0.5 * (xk.x - xm.x), (R)0.5 * (xk.y + xm.y));
    const T O = cmulc(D, tb.tw(tw_rdft(M) + k));
    za = cmk<T>(Eh.x - O.y, -(Eh.y + O.x));   // conj(E + i O)
    zb = cmk<T>(Eh.x + O.y, Eh.y - O.x);      // E - i O
  }
}

}  // namespace pc
