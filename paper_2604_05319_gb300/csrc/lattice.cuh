// Lattice helpers of the 2D Hubbard model (Sec. 4.2) shared by the
// real-time self-energy (kernels_hodlr.cu) and the equilibrium solve
// (matsubara_dev.cu): the k-point of a thread, the reflection-reduced k-set,
// and 2D Fourier transforms over L x L grids held in shared memory.
#pragma once
#include "common.cuh"

namespace hk {

constexpr int kLatMaxK = 256;
// instance holding grid point q = m_x L + m_y (ys: reflection-reduced k-set)
__device__ __forceinline__ int lat_inst(int q, int L, int ys) {
  if (!ys) return q;
  const int y = q % L;
  return (q / L) * (L / 2 + 1) + min(y, L - y);
}
// grid point q is the instance's own k-point (not a reflected copy)
__device__ __forceinline__ bool lat_owner(int q, int L, int ys) { return !ys || q % L <= L / 2; }
// ---- one-dimensional transforms of L points held by one thread ----------
__device__ __forceinline__ zd mul_i(const zd& a, int sg) { return sg > 0 ? zd(-a.im, a.re) : zd(a.im, -a.re); }
__device__ __forceinline__ zd tw_mul(const zd& a, double c, double s, int sg) {   // a e^{i sg phi}, (c, s) = e^{i phi}
  const double t = sg > 0 ? s : -s;
  return zd(fma(a.re, c, -a.im * t), fma(a.re, t, a.im * c));
}
__device__ __forceinline__ void fft4(zd& a, zd& b, zd& c, zd& d, int sg) {
  const zd t0 = a + c, t1 = a - c, t2 = b + d, t3 = mul_i(b - d, sg);
  a = t0 + t2; b = t1 + t3; c = t0 - t2; d = t1 - t3;
}
constexpr double kC8 = 0.70710678118654752440, kC16 = 0.92387953251128675613, kS16 = 0.38268343236508977173;
// v (strided by st) -> its transform with e^{sg 2 pi i / L}, in place
__device__ __forceinline__ void fft16(zd* v, int st, int sg) {
  zd x[16];
#pragma unroll
  for (int n = 0; n < 16; ++n) x[n] = v[n * st];
#pragma unroll
  for (int n = 0; n < 4; ++n) fft4(x[n], x[n + 4], x[n + 8], x[n + 12], sg);   // x[n + 4 k1] = A[n][k1]
  x[5] = tw_mul(x[5], kC16, kS16, sg);     // times w16^{n k1}
  x[9] = tw_mul(x[9], kC8, kC8, sg);
  x[13] = tw_mul(x[13], kS16, kC16, sg);
  x[6] = tw_mul(x[6], kC8, kC8, sg);
  x[10] = mul_i(x[10], sg);
  x[14] = tw_mul(x[14], -kC8, kC8, sg);
  x[7] = tw_mul(x[7], kS16, kC16, sg);
  x[11] = tw_mul(x[11], -kC8, kC8, sg);
  x[15] = tw_mul(x[15], -kC16, -kS16, sg);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    fft4(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3], sg);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[(k1 + 4 * k2) * st] = x[4 * k1 + k2];
  }
}
__device__ __forceinline__ void fft8(zd* v, int st, int sg) {
  zd x[8];
#pragma unroll
  for (int n = 0; n < 8; ++n) x[n] = v[n * st];
  fft4(x[0], x[2], x[4], x[6], sg);
  fft4(x[1], x[3], x[5], x[7], sg);
  x[3] = tw_mul(x[3], kC8, kC8, sg);
  x[5] = mul_i(x[5], sg);
  x[7] = tw_mul(x[7], -kC8, kC8, sg);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k * st] = x[2 * k] + x[2 * k + 1];
    v[(k + 4) * st] = x[2 * k] - x[2 * k + 1];
  }
}
// any L <= 16, from the points and the twiddles tw[m] = e^{2 pi i m / L} in shared memory
__device__ __forceinline__ void dft_any(zd* v, int st, const zd* tw, int L, int sg) {
  zd out[16];
#pragma unroll
  for (int y = 0; y < 16; ++y) {
    if (y >= L) break;
    zd s = v[0];
    int e = 0;
    for (int m = 1; m < L; ++m) {
      e += y;
      if (e >= L) e -= L;
      const zd w = tw[e];
      s = cfma(v[m * st], sg > 0 ? w : w.conj(), s);
    }
    out[y] = s;
  }
#pragma unroll
  for (int y = 0; y < 16; ++y)
    if (y < L) v[y * st] = out[y];
}
// In-place 2D transforms with sign sg of ng grids (index m_x, m_y; rows of
// L + 1 elements, so that the threads of a warp hit different banks), one
// thread per row, then per column.  The CTA synchronises before the call; it
// is synchronised after it.  A thread's 16-point transform is 0.17 thousand
// FP64 operations; the direct sums, two thousand per thread and grid of 256
// points, made Sigma of 256 k-points at T = 360 take 262 us.
__device__ __forceinline__ void lat_fft2(zd* g, int ng, const zd* tw, int L, int sg) {
  const int gsz = L * (L + 1);
  for (int pass = 0; pass < 2; ++pass) {
    for (int e = threadIdx.x; e < ng * L; e += blockDim.x) {
      zd* v = g + (e / L) * gsz + (pass == 0 ? (e % L) * (L + 1) : e % L);
      const int st = pass == 0 ? 1 : L + 1;
      if (L == 16) fft16(v, st, sg);
      else if (L == 8) fft8(v, st, sg);
      else dft_any(v, st, tw, L, sg);
    }
    __syncthreads();
  }
}
constexpr int kLatT = 4;   // times or nodes per CTA (64-byte pieces of a k-point's row)
constexpr size_t lat_smem(int L) { return sizeof(zd) * 2 * kLatT * L * (L + 1); }

// tw[m] = e^{2 pi i m / L}, m < L, written by the first L threads (the
// caller synchronises before use)
__device__ __forceinline__ void lat_twiddles(zd* tw, int L) {
  const int q = threadIdx.x;
  if (q < L) {
    double sn, cs;
    sincospi(2.0 * q / L, &sn, &cs);
    tw[q] = zd(cs, sn);
  }
}

}  // namespace hk
