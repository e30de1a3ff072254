// Device helpers shared by the dense and the compressed (HODLR) kernels:
// indexing, Appendix A integration rule, warp reductions, small solves.
#pragma once
#include "common.cuh"
#include "state.h"

namespace hk {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kSMs = 152;   // of a GB300: batches below a CTA for each of them leave SMs idle

// The kernels of a time step run one after the other on one stream, and each
// begins with pdl_start.  Where the sweeps have at most kEarlyCtas CTAs the
// others are launched with programmatic stream serialization (launch_k): the
// next kernel's CTAs are set up while this one runs, and wait there until every
// earlier kernel has finished and its writes are visible.  That takes the launch
// latency out of the gaps (1 x 64, FP64: 11.9 -> 10.6 ms; 5 x 150, complex64:
// 15.8 -> 14.9; 8 x 300, N_o = 2, FP64: 73.5 -> 71.9).  Larger batches place
// their CTAs worse when they come early, next to those still running (12 x 300,
// N_o = 2, FP64: 76.6 -> 81.7; 40 x 150, FP64: 43.8 -> 44.8; lattice of 256,
// T = 360: 90.7 -> 97.6); for the sweeps themselves see early_sweep.
constexpr int kEarlyCtas = 16;
__device__ __forceinline__ void pdl_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch_on(bool early, void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_k(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, const Dev& d, A... args) {
  return launch_on(d.no * d.n_inst <= kEarlyCtas, kern, grid, threads, smem, s, d, args...);
}

// Let a kernel ask for all the dynamic shared memory that its static arrays leave
// of a CTA's opt-in limit; *room is lowered to that size.  The setting belongs to
// the kernel and the device, not to a handle: it is made when a handle is created,
// always to this same value, and a launch never touches it.  Set to a launch's own
// size before each launch, one thread's handle could lower it between another
// thread's setting and launch, which was then refused.
template <typename K>
inline cudaError_t open_smem(K kern, int* room) {
  int dev = 0, cap = 0;
  cudaFuncAttributes a;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, kern);
  if (e != cudaSuccess) return e;
  const int left = cap - (int)a.sharedSizeBytes;
  *room = left < *room ? left : *room;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, left);
}

__device__ __forceinline__ long long tri(int T) { return (long long)T * (T + 1) / 2; }

// First uncompressed row of instance n.  An instance whose last step comes
// before N_t - 1 stops taking part in the compression once its rows end: its
// front freezes at the last whole leaf of rows older than k + 1 steps, and
// the rows after it stay in their ring slots, which no later kernel writes.
__device__ __forceinline__ int front_of(const Dev& d, int n) {
  const int lk = d.last[n] - d.k;
  const int fz = lk >= d.L ? (lk / d.L) * d.L : 0;
  return d.cdir < fz ? d.cdir : fz;
}

__device__ __forceinline__ void* ringX(const Dev& d, int X) {
  return X == 0 ? d.GR : X == 1 ? d.GL : X == 2 ? d.SR : d.SL;
}

// Row T of a two-time component: the dense lower triangle, or (compressed
// storage) the ring of uncompressed rows, slot T mod ring.
// S is the storage element type (double2 or float2).
template <int NO, typename S>
__device__ __forceinline__ S* el(void* base, const Dev& d, int n, int T, int t) {
  S* b = static_cast<S*>(base);
  if (d.ring) return b + (((long long)n * d.ring + (T % d.ring)) * d.nt + t) * (NO * NO);
  return b + ((long long)n * d.ntri + tri(T) + t) * (NO * NO);
}
// FP64 copy of element (T, t) of component X (complex64 compressed form).
template <int NO>
__device__ __forceinline__ double2* el64(const Dev& d, int X, int n, int T, int t) {
  return d.ring64[X] + (((long long)n * d.ring + (T % d.ring)) * d.nt + t) * (NO * NO);
}
// Entry q of element (T, t) of component X in FP64: from the FP64 copy when
// there is one (and it is seeded), else from the storage.
template <int NO, typename S>
__device__ __forceinline__ zd ldx(const Dev& d, int X, int n, int T, int t, int q) {
  if (d.ring64[X] && d.use64) return ld(el64<NO>(d, X, n, T, t) + q);
  return ld(el<NO, S>(ringX(d, X), d, n, T, t) + q);
}
// Write entry q of element (T, t) of component X: the storage (rounded in the
// complex64 form) and the FP64 copy.
template <int NO, typename S>
__device__ __forceinline__ void stx(const Dev& d, int X, int n, int T, int t, int q, const zd& v) {
  st(el<NO, S>(ringX(d, X), d, n, T, t) + q, v);
  if (d.ring64[X]) st(el64<NO>(d, X, n, T, t) + q, v);
}

// Mixed components G^tv, Sigma^tv: complex128 in both precision forms (their
// DLR convolution is ill-conditioned; they are r/T times smaller than a row set).
template <int NO>
__device__ __forceinline__ double2* tv(void* base, const Dev& d, int n, int T, int i) {
  return static_cast<double2*>(base) + (((long long)n * d.nt + T) * d.r + i) * (NO * NO);
}
template <int NO>
__device__ __forceinline__ double2* epsp(const Dev& d, int n, int t) {  // eps(t), t >= -1
  return d.eps + ((long long)n * (d.nt + 1) + (t + 1)) * (NO * NO);
}

__device__ __forceinline__ double rule_w(const DevW& w, int n, int l) {
  const int k = w.k;
  if (n <= 0) return 0.0;
  if (n <= k) return (l >= 0 && l <= k) ? w.I0[n][l] : 0.0;
  if (n < 2 * k + 1) {
    double s = 0.0;
    if (l >= 0 && l <= k) s += w.I0[n - k][l];
    if (l >= n - k && l <= n) s += w.I0[k][l - (n - k)];
    return s;
  }
  if (l < 0 || l > n) return 0.0;
  if (l <= k) return w.omega[l];
  if (l >= n - k) return w.omega[n - l];
  return 1.0;
}

// The same rule in the arithmetic R of the bulk sums (float tables for float).
template <typename R>
__device__ __forceinline__ R rule_wr(const DevW& w, int n, int l) {
  if constexpr (sizeof(R) == sizeof(double)) {
    return rule_w(w, n, l);
  } else {
    const int k = w.k;
    if (n <= 0) return 0.0f;
    if (n <= k) return (l >= 0 && l <= k) ? w.I0f[n][l] : 0.0f;
    if (n < 2 * k + 1) {
      float s = 0.0f;
      if (l >= 0 && l <= k) s += w.I0f[n - k][l];
      if (l >= n - k && l <= n) s += w.I0f[k][l - (n - k)];
      return s;
    }
    if (l < 0 || l > n) return 0.0f;
    if (l <= k) return w.omegaf[l];
    if (l >= n - k) return w.omegaf[n - l];
    return 1.0f;
  }
}

// Element of the lesser source q(t): FP64, or in the complex64 form a
// float-float pair of the same 16 bytes, so that the lesser sweep takes it
// without FP64 conversions.
template <typename S>
__device__ __forceinline__ auto ldv(const double2* p) {
  if constexpr (sizeof(S) == sizeof(double2)) {
    return ld(p);
  } else {
    const float4 v = *reinterpret_cast<const float4*>(p);
    return cff{{v.x, v.y}, {v.z, v.w}};
  }
}
template <typename S>
__device__ __forceinline__ zd ldv64(const double2* p) {
  if constexpr (sizeof(S) == sizeof(double2)) return ld(p);
  else return cff_val(ldv<S>(p));
}
template <typename S>
__device__ __forceinline__ void stv(double2* p, const zd& v) {
  if constexpr (sizeof(S) == sizeof(double2)) {
    st(p, v);
  } else {
    const cff f = cff_of(v);
    *reinterpret_cast<float4*>(p) = make_float4(f.re.hi, f.re.lo, f.im.hi, f.im.lo);
  }
}

constexpr int FOLD = 8;  // terms summed in R before they enter the compensated accumulator

__device__ __forceinline__ zd wshfl(zd v, int off) {
  return zd(__shfl_xor_sync(FULL, v.re, off), __shfl_xor_sync(FULL, v.im, off));
}
template <int L>
__device__ __forceinline__ void warp_sum(zd (&v)[L]) {
#pragma unroll
  for (int off = 16; off; off >>= 1)
#pragma unroll
    for (int i = 0; i < L; ++i) v[i] += wshfl(v[i], off);
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int off = 16; off; off >>= 1) v = fmax(v, __shfl_xor_sync(FULL, v, off));
  return v;
}

// Sigma^R(a, b) continued above the diagonal: -[Sigma^R(b, a)]^dagger for a < b.
template <int NO, typename S>
__device__ __forceinline__ zd srx(const Dev& d, int n, int a, int b, int x, int y) {
  if (a >= b) return ld(el<NO, S>(d.SR, d, n, a, b) + x * NO + y);
  return -ld(el<NO, S>(d.SR, d, n, b, a) + y * NO + x).conj();
}
// Sigma^<(t, l) anywhere (Eq. GLantiHerm)
template <int NO, typename S>
__device__ __forceinline__ zd sless(const Dev& d, int n, int t, int l, int x, int y) {
  if (t <= l) return ld(el<NO, S>(d.SL, d, n, l, t) + x * NO + y);
  return -ld(el<NO, S>(d.SL, d, n, t, l) + y * NO + x).conj();
}

// ---------------------------------------------------------------------------
// Warp-parallel dense solve A X = B (n <= 32, nrhs <= 32), A and B in shared
// memory, LU with partial pivoting; lane r owns row r during elimination.
// With nrhs = 0 it only factors (L below the diagonal, row swaps in piv).
// ---------------------------------------------------------------------------
static __device__ __noinline__ void warp_lu_solve(int n, zd* A, zd* B, int nrhs, int* piv) {
  const int lane = threadIdx.x & 31;
  for (int c = 0; c < n; ++c) {
    double v = (lane >= c && lane < n) ? A[lane * n + c].abs2() : -1.0;
    int p = lane;
#pragma unroll
    for (int off = 16; off; off >>= 1) {
      double v2 = __shfl_xor_sync(FULL, v, off);
      int p2 = __shfl_xor_sync(FULL, p, off);
      if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
    }
    if (piv && lane == 0) piv[c] = p;
    if (p != c) {
      for (int j = lane; j < n; j += 32) { zd t = A[c * n + j]; A[c * n + j] = A[p * n + j]; A[p * n + j] = t; }
      for (int j = lane; j < nrhs; j += 32) { zd t = B[c * nrhs + j]; B[c * nrhs + j] = B[p * nrhs + j]; B[p * nrhs + j] = t; }
    }
    __syncwarp();
    if (lane > c && lane < n) {
      zd f = cdiv(A[lane * n + c], A[c * n + c]);
      A[lane * n + c] = f;
      for (int j = c + 1; j < n; ++j) A[lane * n + j] -= f * A[c * n + j];
      for (int j = 0; j < nrhs; ++j) B[lane * nrhs + j] -= f * B[c * nrhs + j];
    }
    __syncwarp();
  }
  for (int j = lane; j < nrhs; j += 32)
    for (int c = n - 1; c >= 0; --c) {
      zd s = B[c * nrhs + j];
      for (int m = c + 1; m < n; ++m) s -= A[c * n + m] * B[m * nrhs + j];
      B[c * nrhs + j] = cdiv(s, A[c * n + c]);
    }
  __syncwarp();
}
// Solve with a factor from warp_lu_solve(nrhs = 0) for one right-hand side b.
__device__ __forceinline__ void lu_apply(int n, const zd* A, const int* piv, zd* b) {
  for (int c = 0; c < n; ++c)
    if (piv[c] != c) { zd t = b[c]; b[c] = b[piv[c]]; b[piv[c]] = t; }
  for (int c = 0; c < n; ++c)
    for (int r = c + 1; r < n; ++r) b[r] -= A[r * n + c] * b[c];
  for (int c = n - 1; c >= 0; --c) {
    zd s = b[c];
    for (int m = c + 1; m < n; ++m) s -= A[c * n + m] * b[m];
    b[c] = cdiv(s, A[c * n + c]);
  }
}

// 1 / a: the real reciprocal from an FP32 estimate by two Newton steps (an FP64
// division is a sequence of some ten dependent FP64 instructions, each holding
// the pipe for 64 cycles of the warp).  The exponent of |a|^2 is set aside
// meanwhile, so the estimate covers the range of FP64.
__device__ __forceinline__ zd crecip(const zd& a) {
  const double d = a.abs2();
  const int hi = __double2hiint(d), e = (hi >> 20) - 1023;
  if (e < -1021 || e > 1020) return cdiv(zd(1.0), a);   // zero, subnormal, about to overflow, not finite
  const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(d));   // d = m 2^e
  double y = (double)(1.0f / (float)m);
  y = y * fma(-m, y, 2.0);
  y = y * fma(-m, y, 2.0);
  y = __hiloint2double(__double2hiint(y) - (e << 20), __double2loint(y));
  return zd(a.re * y, -a.im * y);
}
// A key to choose pivots by: the upper words of max(|re|, |im|), which order like
// the values over the range of FP64 (squares in FP32 order nothing outside 1e-22
// to 1.8e19) and take no FP64 instruction.
__device__ __forceinline__ int pivot_key(const zd& a) {
  return max(__double2hiint(a.re) & 0x7fffffff, __double2hiint(a.im) & 0x7fffffff);
}
// Inverse of the NO x NO matrix A (shared memory, row-major) into out by one
// warp, Gauss-Jordan with partial pivoting; lane e < NO^2 owns element e of A
// and of out.  Every lane of the warp calls it.
template <int NO>
__device__ __forceinline__ void warp_inv(const zd* A, zd* tmp, zd* out) {
  constexpr int NO2 = NO * NO;
  const int lane = threadIdx.x & 31, r = lane / NO, c = lane % NO;
  if constexpr (NO == 1) {
    if (lane == 0) out[0] = crecip(A[0]);
    __syncwarp();
    return;
  }
  if (lane < NO2) {
    tmp[lane] = A[lane];
    out[lane] = zd(r == c ? 1.0 : 0.0);
  }
  __syncwarp();
  for (int p = 0; p < NO; ++p) {
    int pr = p;
    int best = pivot_key(tmp[p * NO + p]);
    for (int q = p + 1; q < NO; ++q) {
      const int v = pivot_key(tmp[q * NO + p]);
      if (v > best) { best = v; pr = q; }
    }
    zd a = zd(), o = zd(), f = zd(), ap = zd(), op = zd(), piv = tmp[pr * NO + p];
    if (lane < NO2) {   // rows p and pr change places
      const int src = r == p ? pr : r == pr ? p : r;
      a = tmp[src * NO + c];
      o = out[src * NO + c];
      f = tmp[src * NO + p];
      ap = tmp[pr * NO + c];
      op = out[pr * NO + c];
    }
    __syncwarp();
    const zd ip = crecip(piv);
    if (lane < NO2) {
      ap = ap * ip;
      op = op * ip;
      tmp[lane] = r == p ? ap : a - f * ap;
      out[lane] = r == p ? op : o - f * op;
    }
    __syncwarp();
  }
}

// In-place Gauss-Jordan inverse with partial pivoting of the n x n matrix A
// (leading dimension ld, shared memory, n <= 20); every thread calls it.
static __device__ __noinline__ void gj_inverse(int n, zd* A, int ld) {
  __shared__ zd col[20];
  __shared__ int prow[20];
  const int tid = threadIdx.x;
  for (int c = 0; c < n; ++c) {
    if (tid < 32) {
      int v = (tid >= c && tid < n) ? pivot_key(A[tid * ld + c]) : -1;
      int p = tid;
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        const int v2 = __shfl_xor_sync(FULL, v, off);
        const int p2 = __shfl_xor_sync(FULL, p, off);
        if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
      }
      if (p != c && tid < n) { const zd t = A[c * ld + tid]; A[c * ld + tid] = A[p * ld + tid]; A[p * ld + tid] = t; }
      if (tid == 0) prow[c] = p;
      __syncwarp();
      if (tid < n) col[tid] = tid == c ? crecip(A[c * ld + c]) : A[tid * ld + c];
      __syncwarp();
      if (tid < n) A[c * ld + tid] = tid == c ? col[c] : A[c * ld + tid] * col[c];   // the scaled pivot row
    }
    __syncthreads();
    for (int e = tid; e < n * n; e += blockDim.x) {
      const int r = e / n, j = e % n;
      if (r == c) continue;
      const zd f = col[r];
      A[r * ld + j] = j == c ? -(f * col[c]) : A[r * ld + j] - f * A[c * ld + j];
    }
    __syncthreads();
  }
  if (tid < n)   // undo the row exchanges on the columns, last first
    for (int c = n - 1; c >= 0; --c)
      if (prow[c] != c) { const zd t = A[tid * ld + c]; A[tid * ld + c] = A[tid * ld + prow[c]]; A[tid * ld + prow[c]] = t; }
  __syncthreads();
}

// small vector solve M x = r (column vector)
template <int NO>
__device__ void solve_col(const M<NO>& Mm, const zd* r, zd* x) {
  M<NO> B = M<NO>::zero();
#pragma unroll
  for (int j = 0; j < NO; ++j) B.a[j][0] = r[j];
  M<NO> X = solve_left<NO>(Mm, B);
#pragma unroll
  for (int j = 0; j < NO; ++j) x[j] = X.a[j][0];
}

__device__ __forceinline__ double fermi(double e, double beta) { return 0.5 * (1.0 - tanh(0.5 * beta * e)); }

}  // namespace hk
