// Mixed component of a time step: its own kernel (k_mixed) for large batches,
// extra CTAs of the retarded sweep's launch for small ones (neither needs the
// other's result).
#pragma once
#include "dev_util.cuh"

namespace hk {

// ---------------------------------------------------------------------------
// Mixed component at step T, Eq. KBET.  One CTA per instance and group of NI
// nodes: a lane owns element (i, z, y) of the group's rows of G^tv (adjacent
// elements, 16-byte loads) and all N_o products with column z of Sigma^R; the
// warps, and the lanes left over by a small group, split the history l and the
// convolution sum a.  Groups fill a warp (32 elements) where that gives a CTA to
// every SM (256 lattice points: 38 us an iteration, 76 us with small groups);
// with fewer, groups of 64 bytes or one node spread the FP64 products over more
// SMs (3 instances, FP64, N_o = 1, T = 256: 19 us with groups of 32, 16 with 4).  (One
// warp per node over all l read 16 bytes of every row and node apart, and its
// lane 0 solved an N_o x N_o system per node: 158 us for 128 instances at
// N_o = 2, T = 600; 110 us for 16 at N_o = 4, T = 290.)  Bound by latency at two
// CTAs per SM, so a thread's addresses advance by constants and the BDF rows are
// loaded before their sum (128 x 600: 16.7 -> 14.7 ms of a pass).
// ---------------------------------------------------------------------------
template <int NO> constexpr int kNodes = 32 / (NO * NO);                      // nodes per CTA
template <int NO> constexpr int kNodesFew = NO == 1 ? 4 : NO == 2 ? 2 : 1;    // with few instances
template <int NO, typename S, int NI>
__device__ __forceinline__ void mixed_nodes(const Dev& d, int T, int group, int n) {
  constexpr int NO2 = NO * NO, E = NI * NO2, LS = 32 / E, NS = 8 * LS;   // elements, slices per warp and CTA
  constexpr bool kLanes = LS > 1 && E * LS == 32;   // a warp's slices are combined by shuffles
  constexpr int NR = kLanes ? 8 : NS;               // partial sums per element
  constexpr bool MX = sizeof(S) == sizeof(float2);
  using R = typename Bulk<S>::R;
  const int i0 = group * NI;
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = d.k, ni = min(NI, d.r - i0);
  const double h = d.h;
  const DevW& W = d.w;
  __shared__ zd red[NR][NO][E];
  __shared__ zd Mi[NO2];       // inverse of the point's matrix
  __shared__ double serr[8];
  if (tid < NO2) {
    const int x = tid / NO, y = tid % NO;
    Mi[tid] = (x == y ? zd(0, W.a[0] / h) : zd()) - ld(epsp<NO>(d, n, T) + tid) -
              ld(el<NO, S>(d.SR, d, n, T, T) + tid) * (h * rule_w(W, T, T));
  }
  const int el_ = lane % E, slice = warp * LS + lane / E;
  const bool act = lane < LS * E && el_ < ni * NO2;
  const int z = (el_ % NO2) / NO;
  const double2* G = tv<NO>(d.GTV, d, n, 0, i0) + (act ? el_ : 0);
  const long long gs = (long long)d.r * NO2;   // from row l to row l + 1
  const S* Sr = el<NO, S>(d.SR, d, n, T, 0) + z;
  constexpr int UB = 8;        // rows in flight
  KAcc<R> ka[NO];              // h sum_l w_l Sigma^R(T,l) G^tv(l, tau_i): FP32 products, compensated, in the complex64 form
  const bool start = T < 2 * k + 1;   // the rule of the first steps has weights everywhere
  const double2* Gl = G + slice * gs;
  const S* Sl = Sr + (long long)slice * NO2;
  const long long gst = NS * gs;      // between a slice's rows
  for (int l0 = slice; l0 < T; l0 += NS * UB, Gl += UB * gst, Sl += UB * NS * NO2) {
    double2 g[UB];
#pragma unroll
    for (int u = 0; u < UB; ++u) g[u] = l0 + NS * u < T ? Gl[u * gst] : make_double2(0, 0);
#pragma unroll
    for (int u0 = 0; u0 < UB; u0 += 4) {
      cx<R> pa[NO];
#pragma unroll
      for (int x = 0; x < NO; ++x) pa[x] = cx<R>(0);
#pragma unroll
      for (int u = u0; u < u0 + 4; ++u) {
        const int l = l0 + NS * u;
        if (l < T) {
          cx<R> gv;
          if constexpr (MX) gv = zf(f32_of(g[u].x), f32_of(g[u].y));
          else gv = zd(g[u].x, g[u].y);
          if (start || l <= k || T - l <= k) gv = gv * rule_wr<R>(W, T, l);
#pragma unroll
          for (int x = 0; x < NO; ++x) pa[x] = cfma(ldr<R>(Sl + u * NS * NO2 + x * NO), gv, pa[x]);
        }
      }
#pragma unroll
      for (int x = 0; x < NO; ++x) ka[x].add(pa[x]);
    }
  }
  zd acc[NO];
#pragma unroll
  for (int x = 0; x < NO; ++x) acc[x] = ka[x].get() * h;
  const double2* C = d.wconv + ((long long)n * d.r * d.r + i0) * NO2 + (act ? el_ : 0);
  const double2* St = tv<NO>(d.STV, d, n, T, 0) + z;
#pragma unroll 4
  for (int a = slice; a < d.r; a += NS) {   // sum_a Sigma^tv(T, tau_a) W[a][i]
    const zd c = ld(C + (long long)a * gs);
#pragma unroll
    for (int x = 0; x < NO; ++x) acc[x] = cfma(ld(St + (long long)a * NO2 + x * NO), c, acc[x]);
  }
#pragma unroll
  for (int x = 0; x < NO; ++x) {
    if constexpr (kLanes) {
#pragma unroll
      for (int off = 16; off >= E; off >>= 1) acc[x] += wshfl(acc[x], off);
      if (lane < E) red[warp][x][el_] = acc[x];
    } else {
      if (lane < LS * E) red[slice][x][el_] = acc[x];
    }
  }
  __syncthreads();
  if constexpr (NO == 1) {
    if (tid == 0) Mi[0] = cdiv(zd(1.0), Mi[0]);
    __syncthreads();
  } else {
    gj_inverse(NO, Mi, NO);
  }
  zd rhs = zd();
  double e = 0.0;
  const int i = tid / NO2, x = (tid % NO2) / NO, y = tid % NO;
  if (tid < ni * NO2) {
    for (int w2 = 0; w2 < NR; ++w2)
#pragma unroll
      for (int zz = 0; zz < NO; ++zz) rhs += red[w2][x][i * NO2 + zz * NO + y];
    const double2* gp = tv<NO>(d.GTV, d, n, T, i0) + tid;
    zd g[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) g[j] = j < k ? ld(gp - (j + 1) * gs) : zd();
#pragma unroll
    for (int j = 0; j < 5; ++j) rhs += zd(W.ah[j + 1] * g[j].im, -W.ah[j + 1] * g[j].re);
  }
  __syncthreads();
  zd* rs = &red[0][0][0];
  if (tid < ni * NO2) rs[tid] = rhs;
  __syncthreads();
  if (tid < ni * NO2) {
    zd v = zd();
#pragma unroll
    for (int m = 0; m < NO; ++m) v = cfma(Mi[x * NO + m], rs[i * NO2 + m * NO + y], v);
    double2* p = tv<NO>(d.GTV, d, n, T, i0) + tid;
    e = max_change(0.0, sqrt((v - ld(p)).abs2()));
    st(p, v);
  }
  e = warp_max(e);
  if (lane == 0) serr[warp] = e;
  __syncthreads();
  if (tid == 0) {
    for (int w2 = 1; w2 < 8; ++w2) e = fmax(e, serr[w2]);
    atomic_max_nonneg(d.err + n, e);
  }
}

}  // namespace hk
