// Accessors of the compressed (HODLR) storage: block factors, leaf triangles,
// the near-diagonal band, projection slots, and Sigma^R from whichever
// storage holds an element.
#pragma once
#include "dev_util.cuh"

namespace hk {

template <int NO, typename S>
__device__ __forceinline__ S* Up(const Dev& d, int X, int n, int b, int p) {
  const long long rows = d.b_r1[b] - d.b_r0[b];
  return static_cast<S*>(d.hod[X].U) + ((long long)n * d.utot + d.b_uoff[b] + p * rows) * d.rmax;
}
template <int NO, typename S>
__device__ __forceinline__ S* Vp(const Dev& d, int X, int n, int b, int p) {
  const long long cols = d.b_c1[b] - d.b_c0[b];
  return static_cast<S*>(d.hod[X].V) + ((long long)n * d.vtot + d.b_voff[b] + p * cols) * d.rmax;
}
template <int NO>
__device__ __forceinline__ double* Sp(const Dev& d, int X, int n, int b, int p) {
  return d.hod[X].S + (((long long)n * d.nblk + b) * (NO * NO) + p) * d.rmax;
}
template <int NO>
__device__ __forceinline__ int* Rk(const Dev& d, int X, int n, int b, int p) {
  return d.hod[X].rank + ((long long)n * d.nblk + b) * (NO * NO) + p;
}
// element (t, l) of leaf j of component X (t, l inside the leaf, l <= t)
template <int NO, typename S>
__device__ __forceinline__ S* Lf(const Dev& d, int X, int n, int j, int t, int l) {
  const int A = j * d.L;
  return static_cast<S*>(d.hod[X].leaf) + ((long long)n * d.leaftot + d.leafoff[j] + tri(t - A) + (l - A)) * (NO * NO);
}
template <int NO, typename S>
__device__ __forceinline__ S* Bd(const Dev& d, int n, int t, int dd) {
  return static_cast<S*>(d.band) + (((long long)n * d.nt + t) * d.k + (dd - 1)) * (NO * NO);
}
// sweep projection slots: [n][row/col][maxl][no2][rmax]
template <int NO>
__device__ __forceinline__ double2* Pj(const Dev& d, int n, int which, int lv, int p) {
  return d.proj + ((((long long)n * NO + which) * d.maxl + lv) * (NO * NO) + p) * d.rmax;
}

// Sigma^R(t, l), l <= t, from whichever storage holds it.
template <int NO, typename S>
__device__ __forceinline__ zd sr_any(const Dev& d, int n, int t, int l, int x, int y) {
  if (t >= d.cdir) return ld(el<NO, S>(d.SR, d, n, t, l) + x * NO + y);
  const int jt = t / d.L, jl = l / d.L;
  if (jt == jl) return ld(Lf<NO, S>(d, 2, n, jt, t, l) + x * NO + y);
  for (int lv = 0; lv < d.maxl; ++lv) {
    const int b = d.rowblk[jt * d.maxl + lv];
    if (b < 0 || l < d.b_c0[b] || l >= d.b_c1[b]) continue;
    const int p = x * NO + y, rk = *Rk<NO>(d, 2, n, b, p);
    const S* U = Up<NO, S>(d, 2, n, b, p) + (long long)(t - d.b_r0[b]) * d.rmax;
    const S* V = Vp<NO, S>(d, 2, n, b, p) + (long long)(l - d.b_c0[b]) * d.rmax;
    const double* S = Sp<NO>(d, 2, n, b, p);
    zd s = zd();
    for (int q = 0; q < rk; ++q) s += ld(U + q) * ld(V + q).conj() * S[q];
    return s;
  }
  return zd();
}
template <int NO, typename S>
__device__ __forceinline__ zd srx_any(const Dev& d, int n, int a, int b, int x, int y) {
  if (a >= b) return sr_any<NO, S>(d, n, a, b, x, y);
  return -sr_any<NO, S>(d, n, b, a, y, x).conj();
}

// A solved value: FP64, or float-float in the complex64 form (about 48 bits
// on the FP32 pipes; an FP64 instruction holds a warp's pipe for 64 cycles,
// and the epilogue of a sweep's chunk in FP64 took most of the chunk's time).
template <typename S> struct Val { using t = zd; };
template <> struct Val<float2> { using t = cff; };
__device__ __forceinline__ void vset(zd& v, const zd& x) { v = x; }
__device__ __forceinline__ void vset(cff& v, const zd& x) { v = cff_of(x); }
__device__ __forceinline__ zd v64(const zd& v) { return v; }
__device__ __forceinline__ zd v64(const cff& v) { return cff_val(v); }
__device__ __forceinline__ zd vadd(const zd& a, const zd& b) { return a + b; }
__device__ __forceinline__ cff vadd(const cff& a, const cff& b) { return cff_add(a, b); }
__device__ __forceinline__ zd vbulk(const zd& v) { return v; }                      // in the bulk arithmetic
__device__ __forceinline__ zf vbulk(const cff& v) { return zf(v.re.hi, v.im.hi); }
__device__ __forceinline__ zd vreal(const zd& a, double s, float2) { return a * s; }
__device__ __forceinline__ cff vreal(const cff& a, double, float2 s) {
  return {ff_mul(a.re, {s.x, s.y}), ff_mul(a.im, {s.x, s.y})};
}
// acc + (-i a_j / h) y
__device__ __forceinline__ zd vbdf(const zd& acc, const zd& y, const DevW& W, int j) {
  return zd(fma(W.ah[j], y.im, acc.re), fma(-W.ah[j], y.re, acc.im));
}
__device__ __forceinline__ cff vbdf(const cff& acc, const cff& y, const DevW& W, int j) {
  const ffl a{W.ahf[j].x, W.ahf[j].y};
  return {ff_add(acc.re, ff_mul(a, y.im)), ff_add(acc.im, ff_neg(ff_mul(a, y.re)))};
}
__device__ __forceinline__ zd vshfl_xor(const zd& a, int off) { return wshfl(a, off); }
__device__ __forceinline__ cff vshfl_xor(const cff& a, int off) { return cff_shfl_xor(a, off); }
template <typename T, int N>
__device__ __forceinline__ T pick(const T (&v)[N], int i) {   // v[i] without indexed registers
  T r = v[0];
#pragma unroll
  for (int j = 1; j < N; ++j)
    if (i == j) r = v[j];
  return r;
}

// Element of the lesser source as a solved value.
__device__ __forceinline__ void stV(double2* p, const zd& v) { st(p, v); }
__device__ __forceinline__ void stV(double2* p, const cff& v) {
  *reinterpret_cast<float4*>(p) = make_float4(v.re.hi, v.re.lo, v.im.hi, v.im.lo);
}

}  // namespace hk
