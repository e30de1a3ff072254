// Compressed (HODLR) form of the time step (Sec. 2.2, Fig. 2): the two-time
// components are stored as dense leaf triangles on the diagonal, U S V^dagger
// blocks below them (one scalar TSVD per orbital pair, Sec. 2.3), and a ring
// of the most recent uncompressed rows (the red and green regions: the
// current row and the rows not yet old enough to compress).
//
// History integrals over compressed rows use block projections:
//   retarded row (columns t' of Sigma^R):  pi_B = sum_s y(s) U_B(s,:) S_B,
//     contribution to t' = pi_B . conj(V_B(t',:))
//   lesser column (rows t of Sigma^R):     rho_B = S_B sum_l w_l conj(V_B(l,:)) x(l),
//     contribution to t = U_B(t,:) . rho_B
//   lesser source (Sigma^<, both triangles): each block is used as B and -B^dagger.
// Gregory weights differ from 1 only near the ends (App. A): lower-end weights
// omega_l, l <= k, are folded into the projections; near-diagonal block entries
// (|t - t'| <= k) get an explicit (w - 1) correction from a dense band copy.
//
// update_blocks (Sec. 3.1): whenever a whole leaf of rows is older than k+1
// steps, its rows are appended to every block containing them by a batched
// Brand update: P = R V, E = R - P V^dagger (projected twice in the complex64
// form), an orthonormal basis Q of E's rows by Gram-Schmidt (a second pass for
// the rows that add a direction), the core K = [[S, 0], [P, C]] (C = E Q^dagger),
// its SVD by a column-pivoted QR and one-sided Jacobi on R^dagger, truncation of
// singular values below the SVD tolerance (Sec. 2.2), and rotation of U, V.
#include "hodlr_util.cuh"
#include "lattice.cuh"

namespace hk {

// ---------------------------------------------------------------------------
// Lesser source with compressed Sigma^< (two-sided HODLR matvec).
// Stored S[r][c] = Sigma^<(c, r), c <= r.  q(t) = h sum_l w_l Sigma^<(t,l) g_l,
// g_l = [G^R(T,l)]^dagger:  l >= t uses S[l][t] (column t), l < t uses
// -S[t][l]^dagger (row t).
// Projections per (block, pair (x,z), y):
//   P1 = S o sum_{rows l} w_l g_l[z][y] U(l,:),  q(t in cols) += P1 . conj(V(t,:))
//   P2 = - S o sum_{cols l} w_l g_l[z][y] V(l,:),  q(t in rows) += conj(U(t,:)) . P2
// ---------------------------------------------------------------------------
// P1 (which = 0) or P2 (which = 1) of (block, pair), entry q, all y < N_o, in
// the bulk arithmetic R of the form, inside complex128-sized slots.
template <int NO, typename R>
__device__ __forceinline__ cx<R>* Psrc(const Dev& d, int n, int b, int p, int which) {
  return reinterpret_cast<cx<R>*>(d.proj + (long long)d.n_inst * NO * d.maxl * NO * NO * d.rmax +
                                  ((((long long)n * d.nblk + b) * (NO * NO) + p) * 2 + which) * d.rmax * NO);
}

// The projections: one CTA per instance, block side and 256 rows of it (or
// columns), so that a block of a thousand rows is not one warp's loop over
// all of them.  A warp takes one pair (N_o = 1, 2: 8 or 2 warps share a pair's
// rows), all y, lanes packed by the pair's rank (8, 16 or 32 per factor row,
// 64 entries of the rank per pass).  Sides longer than 256 leave one partial
// sum per CTA in spart; the CTA that finds itself the last of its side (a
// counter that it sets back) adds them in their order, so the sum does not
// depend on which one that is.
// In sides longer than that the chunks are of 128 rows: the chain per CTA halves,
// and the sums over chunks are there anyway (1 instance, N_o = 2, T = 1089: 10.4 ->
// 7.6 ms of a pass; 128 instances, T = 600: 36.4 -> 35.6).  128 rows everywhere
// would split sides that need no partial sums (16 instances, N_o = 4, T = 290:
// 17.6 -> 19.3).
// s_tab: (block, side, chunk, first slot of the side's partial sums).
template <int NO, typename S>
__global__ void __launch_bounds__(256) k_src_proj(Dev d, int T) {
  pdl_start();
  constexpr int NO2 = NO * NO;
  using R = typename Bulk<S>::R;
  using V = typename Val<S>::t;
  const int4 job = d.s_tab[blockIdx.x];
  const int b = job.x, which = job.y, ch = job.z, n = blockIdx.y;
  const int c = d.cdir;
  if (!d.active[n] || d.b_r0[b] >= c) return;
  const int lo = which == 0 ? d.b_r0[b] : d.b_c0[b], hi = which == 0 ? min(d.b_r1[b], c) : d.b_c1[b];
  const int rows = src_chunk(which == 0 ? d.b_r1[b] - d.b_r0[b] : d.b_c1[b] - d.b_c0[b]);
  const int l0 = lo + ch * rows, l1 = min(l0 + rows, hi), nch = (hi - lo + rows - 1) / rows;
  if (l0 >= hi) return;
  const DevW& W = d.w;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int WPJ = NO == 1 ? 8 : NO == 2 ? 2 : 1, NGRP = 8 / WPJ;   // warps per pair
  __shared__ V red[WPJ > 1 ? 8 : 1][NO * 64];
  __shared__ int s_last;
  const int grp = warp / WPJ, wig = warp % WPJ;
  V* part = reinterpret_cast<V*>(d.spart) + ((long long)n * d.s_parts + job.w) * (NO2 * NO) * d.rmax;   // [chunk][p][q][y]
  auto finish = [&](int p, int q, int y, const V& v) {   // the whole side's sum
    const double s = Sp<NO>(d, 3, n, b, p)[q];
    const zd r = v64(v) * (which == 0 ? s : -s);
    Psrc<NO, R>(d, n, b, p, which)[q * NO + y] = cx<R>((R)r.re, (R)r.im);
  };
  for (int p0 = 0; p0 < NO2; p0 += NGRP) {
    const int p = p0 + grp;
    const bool act = p < NO2;
    const int z = which == 0 ? p % NO : p / NO;
    const int rk = act ? *Rk<NO>(d, 3, n, b, p) : 0;
    const S* F = which == 0 ? Up<NO, S>(d, 3, n, b, act ? p : 0) : Vp<NO, S>(d, 3, n, b, act ? p : 0);
    int rkall = rk;   // of the pairs taken together (the groups meet at barriers)
    if (WPJ > 1) {
      for (int g = 0; g < NGRP; ++g) rkall = max(rkall, *Rk<NO>(d, 3, n, b, p0 + g));
    }
    for (int qb = 0; qb < rkall; qb += 64) {
      const int rem = max(0, min(rk - qb, 64)), lpr = rem <= 8 ? 8 : rem <= 16 ? 16 : 32;
      const int rps = 32 / lpr, sub = lane / lpr, q0 = qb + lane % lpr;
      const int stride = WPJ * rps;
      KAcc<R> acc[NO][2];
      if (rem > 0)
        for (int lb = l0 + wig * rps + sub; lb < l1; lb += stride * FOLD) {
          cx<R> pp[NO][2];
#pragma unroll
          for (int y = 0; y < NO; ++y) pp[y][0] = pp[y][1] = cx<R>(0);
#pragma unroll
          for (int jj = 0; jj < FOLD; ++jj) {
            const int l = lb + stride * jj;
            if (l < l1) {
              const R wl = rule_wr<R>(W, T, l);
              const S* gp = el<NO, S>(d.GR, d, n, T, l);
              cx<R> g[NO];   // w_l g_l[z][y] = w_l conj(G^R(T,l)[y][z])
#pragma unroll
              for (int y = 0; y < NO; ++y) g[y] = ldr<R>(gp + y * NO + z).conj() * wl;
              const S* fr = F + (long long)(l - lo) * d.rmax;
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int q = q0 + lpr * u;
                if (q < rk) {
                  const cx<R> f = ldr<R>(fr + q);
#pragma unroll
                  for (int y = 0; y < NO; ++y) pp[y][u] = cfma(g[y], f, pp[y][u]);
                }
              }
            }
          }
#pragma unroll
          for (int y = 0; y < NO; ++y) {
            acc[y][0].add(pp[y][0]);
            acc[y][1].add(pp[y][1]);
          }
        }
#pragma unroll
      for (int y = 0; y < NO; ++y)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int q = q0 + lpr * u;
          if (lpr * u < rem) {   // (warp-uniform)
            const V r = kacc_lanes(acc[y][u], lpr, 32);
            if (sub == 0 && q < rk && q < qb + 64) {
              if (WPJ > 1) red[warp][y * 64 + q - qb] = r;
              else if (nch == 1) finish(p, q, y, r);
              else part[((long long)(ch * NO2 + p) * d.rmax + q) * NO + y] = r;
            }
          }
        }
      if (WPJ > 1) {
        __syncthreads();
        if (act)
          for (int e = wig * 32 + lane; e < NO * rem; e += WPJ * 32) {
            const int y = e / rem, qq = e % rem;
            V r = red[grp * WPJ][y * 64 + qq];
#pragma unroll
            for (int w2 = 1; w2 < WPJ; ++w2) r = vadd(r, red[grp * WPJ + w2][y * 64 + qq]);
            if (nch == 1) finish(p, qb + qq, y, r);
            else part[((long long)(ch * NO2 + p) * d.rmax + qb + qq) * NO + y] = r;
          }
        __syncthreads();
      }
    }
  }
  if (nch == 1) return;
  __threadfence();
  __syncthreads();
  int* cnt = d.s_cnt + ((long long)n * d.nblk + b) * 2 + which;
  if (tid == 0) {
    s_last = atomicAdd(cnt, 1) == nch - 1;
    if (s_last) *cnt = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int p = 0; p < NO2; ++p) {
    const int rk = *Rk<NO>(d, 3, n, b, p);
    for (int e = tid; e < rk * NO; e += blockDim.x) {
      V r;
      vset(r, zd());
      for (int i = 0; i < nch; ++i) r = vadd(r, part[(long long)(i * NO2 + p) * d.rmax * NO + e]);
      finish(p, e / NO, e % NO, r);
    }
  }
}

// Sum of products of FP64 data.  Complex64 form: both factors as float-float
// pairs, every product's rounding error kept by a fused multiply-add and every
// sum's by TwoSum, both collected in a second float (the compensated dot
// product of Ogita, Rump and Oishi): about 48 bits on the FP32 pipes, 12
// instructions per real product where an FP64 one holds the pipe for 64 cycles.
struct Dot2 {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(const ffl& a, const ffl& b) {
    const float p = a.hi * b.hi;
    const float e = fmaf(a.hi, b.hi, -p);
    const ffl t = ff_two_sum(s, p);
    s = t.hi;
    c = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, c + (t.lo + e)));
  }
};
template <typename S> struct DotC;
template <> struct DotC<double2> {
  zd a{};
  __device__ __forceinline__ DotC() : a(0.0) {}
  __device__ __forceinline__ void add(const zd& x, const zd& y) { a = cfma(x, y, a); }
  __device__ __forceinline__ zd get() const { return a; }
};
template <> struct DotC<float2> {
  Dot2 re, im;
  __device__ __forceinline__ void add(const cff& x, const cff& y) {
    re.add(x.re, y.re);
    re.add(ff_neg(x.im), y.im);
    im.add(x.re, y.im);
    im.add(x.im, y.re);
  }
  __device__ __forceinline__ cff get() const { return {ff_two_sum(re.s, re.c), ff_two_sum(im.s, im.c)}; }
};
template <typename S>
__device__ __forceinline__ auto ld_split(const double2* p) {   // complex128 data as a Val<S>
  if constexpr (sizeof(S) == sizeof(double2)) {
    return ld(p);
  } else {
    const double2 v = *p;
    return cff{ff_of_bits(v.x), ff_of_bits(v.y)};
  }
}
__device__ __forceinline__ zd vmul_mi(const zd& a) { return zd(a.im, -a.re); }   // -i a
__device__ __forceinline__ cff vmul_mi(const cff& a) { return {a.im, ff_neg(a.re)}; }

// q(t).  CTAs x < c / 32: 32 compressed columns t < c; lanes along t (adjacent
// elements of every uncompressed row), the terms of the sum split over the 8
// warps: uncompressed rows l in [c, T] (at most a leaf plus k + 1, staged
// weighted G^A), the leaf, the packed entries of all blocks over the leaf
// (both sides) with kEB loads in flight, and the mixed part - i sum_a
// Sigma^tv(t, tau_a) v_a.  The other CTAs: 8 uncompressed rows t >= c, one warp
// each, lanes along the row.  One thread per t over all terms (the earlier form)
// was a chain of some thousand loads and FP64 products, on T / 128 CTAs; projections
// and source together took 554 us at N_o = 2, complex64, 128 instances, T = 600
// (now 360), 400 us in FP64 at 16 instances, T = 300 (123), 970 us at N_o = 4,
// complex64, 16 instances, T = 290 (152).
// With the rows' g staged in shared memory and each entry's pointers kept there:
// 25.1 -> 18.8 ms of a pass at N_o = 1, complex64, 304 instances, T = 384, and
// 46.3 -> 37.0 at N_o = 2, 128 instances, T = 600.
constexpr int kEB = 4;
template <int NO, typename S>
__global__ void __launch_bounds__(256) k_src_q(Dev d, int T, int uselist) {
  pdl_start();
  constexpr int NO2 = NO * NO;
  using R = typename Bulk<S>::R;
  using V = typename Val<S>::t;
  const int n = blockIdx.y;
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = d.cdir, L = d.L, ntile = c / 32;
  const DevW& W = d.w;
  extern __shared__ __align__(16) char dyn[];
  V* vs = reinterpret_cast<V*>(dyn);              // [r][NO2] v_a
  V* red = vs + d.r * NO2;                        // [8][NO2][32] partial sums of the warps
  for (int e = tid; e < d.r * NO2; e += blockDim.x) vset(vs[e], ld(d.vvec + (long long)n * d.r * NO2 + e));
  KAcc<R> ka[NO2];   // the history sums: compensated FP32 in the complex64 form
  DotC<S> mx[NO2];   // the mixed part
  cx<R> pa[NO2];
  auto fold = [&]() {
#pragma unroll
    for (int q = 0; q < NO2; ++q) {
      ka[q].add(pa[q]);
      pa[q] = cx<R>(0);
    }
  };
#pragma unroll
  for (int q = 0; q < NO2; ++q) pa[q] = cx<R>(0);
  auto gw = [&](int l, int z, int y) {   // w_l g_l[z][y]
    return ldr<R>(el<NO, S>(d.GR, d, n, T, l) + y * NO + z).conj() * rule_wr<R>(W, T, l);
  };
  // pa[x][y] += sum_z Sx[x][z] g[z][y], Sx = S or -S^dagger
  auto mac = [&](const cx<R>* s, bool low, const cx<R>* g) {
#pragma unroll
    for (int x = 0; x < NO; ++x)
#pragma unroll
      for (int z = 0; z < NO; ++z) {
        const cx<R> sxz = low ? -s[z * NO + x].conj() : s[x * NO + z];
#pragma unroll
        for (int y = 0; y < NO; ++y) pa[x * NO + y] = cfma(sxz, g[z * NO + y], pa[x * NO + y]);
      }
  };
  auto mixed = [&](int t, int a0, int da) {
    const double2* sv = tv<NO>(d.STV, d, n, t, 0);
#pragma unroll(NO <= 2 ? 2 : 1)
    for (int a = a0; a < d.r; a += da)
#pragma unroll
      for (int x = 0; x < NO; ++x)
#pragma unroll
        for (int z = 0; z < NO; ++z) {
          const V s = ld_split<S>(sv + (long long)a * NO2 + x * NO + z);
#pragma unroll
          for (int y = 0; y < NO; ++y) mx[x * NO + y].add(s, vs[a * NO2 + z * NO + y]);
        }
  };
  if ((int)blockIdx.x >= ntile) {   // uncompressed rows, one warp each, lanes along the row
    const int t = c + ((int)blockIdx.x - ntile) * 8 + warp;
    const bool row = t <= T;
    const S* srow = el<NO, S>(d.SL, d, n, row ? t : T, 0);
    cx<R>* gt = reinterpret_cast<cx<R>*>(red);   // [256][NO2] w_l g_l, shared by the CTA's rows
    cx<R> s[NO2];
    for (int lt = 0; lt <= T; lt += 256) {
      const int ln = min(256, T + 1 - lt);
      __syncthreads();
      for (int e = tid; e < ln * NO2; e += blockDim.x) gt[e] = gw(lt + e / NO2, (e % NO2) / NO, e % NO);
      __syncthreads();
      if (row) {
#pragma unroll
        for (int jj = 0; jj < FOLD; ++jj) {
          const int li = lane + 32 * jj, l = lt + li;
          if (li < ln) {
            const S* sp = l >= t ? el<NO, S>(d.SL, d, n, l, t) : srow + (long long)l * NO2;
#pragma unroll
            for (int q = 0; q < NO2; ++q) s[q] = ldr<R>(sp + q);
            mac(s, l < t, gt + li * NO2);
          }
        }
        fold();
      }
    }
    if (!row) return;
    V hist[NO2];
#pragma unroll
    for (int q = 0; q < NO2; ++q) hist[q] = vreal(kacc_lanes(ka[q], 1, 32), d.h, W.hf);
    mixed(t, lane, 32);
#pragma unroll
    for (int q = 0; q < NO2; ++q) {
      V v = vmul_mi(mx[q].get());
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) v = vadd(v, vshfl_xor(v, off));
      if (lane == 0) stV(d.qsrc + ((long long)n * d.nt + t) * NO2 + q, vadd(hist[q], v));
    }
    return;
  }
  // 32 compressed columns
  const int t = blockIdx.x * 32 + lane, jt = blockIdx.x * 32 / L, A = jt * L;
  cx<R>* gr = reinterpret_cast<cx<R>*>(red + 8 * NO2 * 32);   // [kRingRows][NO2] w_l g_l of the uncompressed rows
  cx<R>* gl = gr + kRingRows * NO2;                            // [L][NO2] of the leaf
  int* rk = reinterpret_cast<int*>(gl + 64 * NO2);            // per slot (target x, side, level, other index): rank,
  const int nslot = 2 * d.maxl * NO2;
  int* start = rk + nslot;                                    // first packed entry,
  const S** fp = reinterpret_cast<const S**>(((unsigned long long)(start + nslot + 1) + 7) & ~7ull);   // factor row of the first t,
  const cx<R>** pp = reinterpret_cast<const cx<R>**>(fp + nslot);           // and projections [q][y]
  unsigned short* list = reinterpret_cast<unsigned short*>(pp + nslot);     // entries: slot * 128 + q
  const int nr = T + 1 - c;
  for (int e = tid; e < nr * NO2; e += blockDim.x) gr[e] = gw(c + e / NO2, (e % NO2) / NO, e % NO);
  for (int e = tid; e < L * NO2; e += blockDim.x) gl[e] = gw(A + e / NO2, (e % NO2) / NO, e % NO);
  for (int s = tid; s < nslot; s += blockDim.x) {
    const int x = s / (2 * d.maxl * NO), which = (s / (d.maxl * NO)) & 1, lv = (s / NO) % d.maxl, z = s % NO;
    const int p = which == 0 ? x * NO + z : z * NO + x;
    int b = (which == 0 ? d.colblk : d.rowblk)[jt * d.maxl + lv];
    if (b >= 0 && d.b_r0[b] >= c) b = -1;
    rk[s] = b >= 0 ? *Rk<NO>(d, 3, n, b, p) : 0;
    if (b >= 0) {
      fp[s] = which == 0 ? Vp<NO, S>(d, 3, n, b, p) + (long long)(blockIdx.x * 32 - d.b_c0[b]) * d.rmax
                         : Up<NO, S>(d, 3, n, b, p) + (long long)(blockIdx.x * 32 - d.b_r0[b]) * d.rmax;
      pp[s] = Psrc<NO, R>(d, n, b, p, which);
    }
  }
  __syncthreads();
  if (warp == 0) {
    int carry = 0;
    for (int s0 = 0; s0 < nslot; s0 += 32) {
      const int r = s0 + lane < nslot ? rk[s0 + lane] : 0;
      int x = r;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
      }
      if (s0 + lane < nslot) start[s0 + lane] = carry + x - r;
      carry += __shfl_sync(FULL, x, 31);
    }
    if (lane == 0) start[nslot] = carry;
  }
  __syncthreads();
  if (uselist) {
    for (int s = warp; s < nslot; s += 8)
      for (int q = lane; q < rk[s]; q += 32) list[start[s] + q] = (unsigned short)(s * 128 + q);
    __syncthreads();
  }
  cx<R> s[NO2];
  const int ring0 = c % d.ring;
  const S* sring = static_cast<const S*>(d.SL) + ((long long)n * d.ring * d.nt + t) * NO2;
  for (int l0 = warp; l0 < nr; l0 += 8 * FOLD) {   // the uncompressed rows
#pragma unroll
    for (int jj = 0; jj < FOLD; ++jj) {
      const int l = l0 + 8 * jj;
      if (l < nr) {
        int slot = ring0 + l;
        if (slot >= d.ring) slot -= d.ring;
        const S* sp = sring + (long long)slot * d.nt * NO2;
#pragma unroll
        for (int q = 0; q < NO2; ++q) s[q] = ldr<R>(sp + q);
        mac(s, false, gr + l * NO2);
      }
    }
    fold();
  }
  const S* leaf = static_cast<const S*>(d.hod[3].leaf) + ((long long)n * d.leaftot + (long long)jt * (L * (L + 1) / 2)) * NO2;
  for (int l0 = warp; l0 < L; l0 += 8 * FOLD) {   // the leaf, both triangles
#pragma unroll
    for (int jj = 0; jj < FOLD; ++jj) {
      const int l = A + l0 + 8 * jj;
      if (l < A + L) {
        const int hi = max(l, t) - A, lo = min(l, t) - A;
        const S* sp = leaf + (hi * (hi + 1) / 2 + lo) * NO2;
#pragma unroll
        for (int q = 0; q < NO2; ++q) s[q] = ldr<R>(sp + q);
        mac(s, l < t, gl + (l - A) * NO2);
      }
    }
    fold();
  }
  const int tstr = lane * d.rmax;
#pragma unroll
  for (int x = 0; x < NO; ++x) {   // the blocks
    auto entries = [&](auto at, int e0, int e1, int stride) {   // kEB entries from e0, at(e) = slot * 128 + q
      cx<R> f[kEB], P[kEB][NO];
#pragma unroll
      for (int u = 0; u < kEB; ++u) {
        const int e = e0 + stride * u, le = at(min(e, e1 - 1)), sl = le >> 7, q = le & 127;
        f[u] = e < e1 ? ldr<R>(fp[sl] + tstr + q).conj() : cx<R>(0);
#pragma unroll
        for (int y = 0; y < NO; ++y) P[u][y] = pp[sl][q * NO + y];
      }
#pragma unroll
      for (int y = 0; y < NO; ++y) {
        cx<R> sum = cx<R>(0);
#pragma unroll
        for (int u = 0; u < kEB; ++u) sum = cfma(P[u][y], f[u], sum);
        ka[x * NO + y].add(sum);
      }
    };
    if (uselist) {
      const int e1 = start[(x + 1) * 2 * d.maxl * NO];
      for (int e0 = start[x * 2 * d.maxl * NO] + warp; e0 < e1; e0 += 8 * kEB)
        entries([&](int e) { return (int)list[e]; }, e0, e1, 8);
    } else {
      for (int sl = x * 2 * d.maxl * NO; sl < (x + 1) * 2 * d.maxl * NO; ++sl)
        for (int q0 = warp; q0 < rk[sl]; q0 += 8 * kEB) entries([&](int q) { return sl * 128 + q; }, q0, rk[sl], 8);
    }
  }
#pragma unroll
  for (int q = 0; q < NO2; ++q) red[(warp * NO2 + q) * 32 + lane] = vreal(kacc_lanes(ka[q], 32, 32), d.h, W.hf);
  mixed(t, warp, 8);
#pragma unroll
  for (int q = 0; q < NO2; ++q) {
    V& v = red[(warp * NO2 + q) * 32 + lane];
    v = vadd(v, vmul_mi(mx[q].get()));
  }
  __syncthreads();
  for (int e = tid; e < 32 * NO2; e += blockDim.x) {
    const int tt = e / NO2, q = e % NO2;
    V a[8];
#pragma unroll
    for (int w2 = 0; w2 < 8; ++w2) a[w2] = red[(w2 * NO2 + q) * 32 + tt];
#pragma unroll
    for (int s2 = 4; s2; s2 >>= 1)
#pragma unroll
      for (int w2 = 0; w2 < s2; ++w2) a[w2] = vadd(a[w2], a[w2 + s2]);
    stV(d.qsrc + ((long long)n * d.nt + blockIdx.x * 32) * NO2 + e, a[0]);
  }
}

// ---------------------------------------------------------------------------
// update_blocks: compress the rows [A, A+nb) of every component
// ---------------------------------------------------------------------------
template <int NO, typename S>
__global__ void k_comp_copy(Dev d, int A, int nb) {
  constexpr int NO2 = NO * NO;
  const int n = blockIdx.y;
  if (A + nb + d.k > d.last[n]) return;   // the instance's rows end before this leaf is final
  const int j = A / d.L;
  const long long ntr = (long long)nb * (nb + 1) / 2;
  const long long total = 4 * ntr + (long long)nb * d.k;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    if (idx < 4 * ntr) {
      const int X = (int)(idx / ntr);
      long long e = idx % ntr;
      int i = (int)((sqrt(8.0 * e + 1.0) - 1.0) * 0.5);
      while ((long long)i * (i + 1) / 2 > e) --i;
      while ((long long)(i + 1) * (i + 2) / 2 <= e) ++i;
      const int l = (int)(e - (long long)i * (i + 1) / 2);
      const int t = A + i, col = A + l;
      const S* src = el<NO, S>(ringX(d, X), d, n, t, col);
      S* dst = Lf<NO, S>(d, X, n, j, t, col);
#pragma unroll
      for (int q = 0; q < NO2; ++q) dst[q] = src[q];
    } else {
      const long long e = idx - 4 * ntr;
      const int t = A + (int)(e / d.k), dd = (int)(e % d.k) + 1;
      S* dst = Bd<NO, S>(d, n, t, dd);
      if (t - dd >= 0) {
        const S* src = el<NO, S>(d.SR, d, n, t, t - dd);
#pragma unroll
        for (int q = 0; q < NO2; ++q) dst[q] = src[q];
      } else {
#pragma unroll
        for (int q = 0; q < NO2; ++q) st(dst + q, zd());
      }
    }
  }
}

// ---------------------------------------------------------------------------
// update_blocks, the TSVD.  One CTA per (component X, level slot, pair p) x
// instance.  With E the new rows of the block, V the block's right factor:
//   P = E V, E -= P V^dagger (twice in the complex64 form);
//   Gram-Schmidt of the residual rows, E = C Q: row by row, a row whose residual
//     is below a quarter of the threshold adds no basis direction;
//   the core K = [[S, 0], [P, C]]: R of a column-pivoted QR, then one-sided
//     Jacobi (round-robin pairs) on the columns of R^dagger, whose normalised
//     columns are the right singular vectors W of K;
//   truncation, U' = [[U, 0], [0, I]] K W / sigma, V' = [V, Q^dagger] W.
// It is bound by the arithmetic of one SM and the latency of its phases, so:
// tiles of E and V in shared memory; the Gram-Schmidt's second pass (against V
// and Q) for accepted rows only, which then update every later row at once
// (two passes over all 64 rows one after the other, five barriers each, were
// the largest part); the pivoted QR makes the Jacobi matrix n x n and graded (4
// to 6 sweeps instead of up to 12 on 64 + r rows), and needs no accumulation of
// the rotations; a rotation's angle is found in FP32 and only its
// normalisation in full precision.
// Precision: FP64, and in the complex64 form float-float throughout (about 48
// bits, on the FP32 pipes).  That form truncates at the rounding floor of its
// stored rows (below), so every step must round well below that floor;
// measured on the C4 batch, FP32 variants of the projections (even with FP64
// folds), of the residual rows, of the rotation of V, or of the core Jacobi
// each put rounding directions above it and the ranks grew to r_max within a
// few hundred steps.
// ---------------------------------------------------------------------------
constexpr double kF32Unit = 5.9604644775390625e-8;  // 2^-24, complex64 unit roundoff
constexpr size_t kTsvdSmem = 100 * 1024;            // dynamic shared memory: two CTAs per SM

// real numbers of the same precision as Val<S>
__device__ __forceinline__ double rmul(double a, double b) { return a * b; }
__device__ __forceinline__ ffl rmul(const ffl& a, const ffl& b) { return ff_mul(a, b); }
__device__ __forceinline__ zd vscl(const zd& a, double s) { return a * s; }
__device__ __forceinline__ cff vscl(const cff& a, const ffl& s) { return {ff_mul(a.re, s), ff_mul(a.im, s)}; }
__device__ __forceinline__ zd vmul(const zd& a, const zd& b) { return a * b; }
__device__ __forceinline__ cff vmul(const cff& a, const cff& b) { return cff_mul(a, b); }
__device__ __forceinline__ zd vneg(const zd& a) { return -a; }
__device__ __forceinline__ cff vneg(const cff& a) { return {ff_neg(a.re), ff_neg(a.im)}; }
__device__ __forceinline__ zd vconj(const zd& a) { return a.conj(); }
__device__ __forceinline__ cff vconj(const cff& a) { return {a.re, ff_neg(a.im)}; }
__device__ __forceinline__ zd vof(const double2& a) { return zd(a.x, a.y); }
__device__ __forceinline__ cff vof(const float2& a) { return {{a.x, 0.f}, {a.y, 0.f}}; }
__device__ __forceinline__ double vnorm2(const zd& a) { return a.abs2(); }
__device__ __forceinline__ float vtop(const zd&) { return 0.f; }
__device__ __forceinline__ float vtop(const cff& a) { return fmaxf(fabsf(a.re.hi), fabsf(a.im.hi)); }
__device__ __forceinline__ float vnorm2(const cff& a) { return a.re.hi * a.re.hi + a.im.hi * a.im.hi; }
// 1 / sqrt(x) from an FP32 estimate by two Newton steps
__device__ __forceinline__ double rsq(double x) {
  const int e = ((__double2hiint(x) >> 20) & 0x7ff) - 1023;   // scale by an even power of two into the FP32 range
  const int e2 = e & ~1;
  const double xs = x * __hiloint2double((1023 - e2) << 20, 0);
  double y = (double)rsqrtf((float)xs);
  y = y * fma(-0.5 * xs * y, y, 1.5);
  y = y * fma(-0.5 * xs * y, y, 1.5);
  return y * __hiloint2double((1023 - e2 / 2) << 20, 0);
}
__device__ __forceinline__ ffl rsq(const ffl& x) {
  const float y0 = rsqrtf(x.hi);
  ffl y{y0, 0.f};
  const ffl xh{-0.5f * x.hi, -0.5f * x.lo};
#pragma unroll
  for (int i = 0; i < 2; ++i) y = ff_mul(y, ff_add(ff_mul(ff_mul(xh, y), y), {1.5f, 0.f}));
  return y;
}
// x >= 0 as m 4^e, m in [1, 4), of FP32 precision (zero: m = 0), on the integer
// pipes: the decisions on a rotation are taken in FP32 without its range
struct Quad {
  float m;
  int e;
};
__device__ __forceinline__ Quad quad_of(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), f = hi >> 20 & 0x7ffu, e = f - 1023u;
  const unsigned m = (127u + (e & 1u)) << 23 | (hi & 0xfffffu) << 3 | (unsigned)__double2loint(x) >> 29;
  return {f ? __uint_as_float(m) : 0.f, (int)e >> 1};
}
__device__ __forceinline__ Quad quad_of(const ffl& x) {
  const unsigned b = __float_as_uint(x.hi), f = b >> 23 & 0xffu, e = f - 127u;
  return {f ? __uint_as_float((127u + (e & 1u)) << 23 | (b & 0x7fffffu)) : 0.f, (int)e >> 1};
}
// a 2^e (e kept within the exponents of normal numbers)
__device__ __forceinline__ zd vldexp(const zd& a, int e) {
  return a * __hiloint2double((1023 + min(max(e, -1022), 1022)) << 20, 0);
}
__device__ __forceinline__ cff vldexp(const cff& a, int e) {
  const float s = __int_as_float((127 + min(max(e, -126), 126)) << 23);
  return {{a.re.hi * s, a.re.lo * s}, {a.im.hi * s, a.im.lo * s}};
}
__device__ __forceinline__ double rtop(double x) { return x; }
__device__ __forceinline__ float rtop(const ffl& x) { return x.hi; }
__device__ __forceinline__ double r64(double x) { return x; }
__device__ __forceinline__ double r64(const ffl& x) { return ff_val(x); }
template <typename S> struct Re { using t = double; };
template <> struct Re<float2> { using t = ffl; };
__device__ __forceinline__ float vnorm32(const zd& a) { return (float)a.abs2(); }
__device__ __forceinline__ float vnorm32(const cff& a) { return vnorm2(a); }
__device__ __forceinline__ double rof(double x, double2*) { return x; }
__device__ __forceinline__ ffl rof(double x, float2*) { return ff_of(x); }
// sum of |a|^2
template <typename S> struct Nrm2;
template <> struct Nrm2<double2> {
  double s = 0.0;
  __device__ __forceinline__ void add(const zd& a) { s = fma(a.re, a.re, fma(a.im, a.im, s)); }
  __device__ __forceinline__ double get() const { return s; }
};
template <> struct Nrm2<float2> {
  Dot2 s;
  __device__ __forceinline__ void add(const cff& a) { s.add(a.re, a.re); s.add(a.im, a.im); }
  __device__ __forceinline__ ffl get() const { return ff_two_sum(s.s, s.c); }
};
__device__ __forceinline__ double rshfl(double a, int off) { return __shfl_xor_sync(FULL, a, off); }
__device__ __forceinline__ ffl rshfl(const ffl& a, int off) {
  return {__shfl_xor_sync(FULL, a.hi, off), __shfl_xor_sync(FULL, a.lo, off)};
}
__device__ __forceinline__ double radd(double a, double b) { return a + b; }
__device__ __forceinline__ ffl radd(const ffl& a, const ffl& b) { return ff_add(a, b); }
// sums over the lanes reached by xor offsets from n / 2 down (all lanes call)
template <typename T> __device__ __forceinline__ T vsum(T v, int n) {
  for (int off = n >> 1; off; off >>= 1) v = vadd(v, vshfl_xor(v, off));
  return v;
}
template <typename T> __device__ __forceinline__ T rsum(T v, int n) {
  for (int off = n >> 1; off; off >>= 1) v = radd(v, rshfl(v, off));
  return v;
}
// a - sum of products, the sum started from a
__device__ __forceinline__ void dot_from(DotC<double2>& s, const zd& a) { s.a = a; }
__device__ __forceinline__ void dot_from(DotC<float2>& s, const cff& a) {
  s.re.s = a.re.hi; s.re.c = a.re.lo;
  s.im.s = a.im.hi; s.im.c = a.im.lo;
}

template <int NO, typename S>
__global__ void __launch_bounds__(256, 2) k_tsvd(Dev d, int A, int nb, int n0) {
  constexpr int NO2 = NO * NO;
  using V = typename Val<S>::t;
  using R = typename Re<S>::t;
  const int n = n0 + blockIdx.y;   // instances n0 .. n0 + gridDim.y - 1 share the workspace
  const int X = blockIdx.x / (d.maxl * NO2);
  const int lv = (blockIdx.x / NO2) % d.maxl;
  const int p = blockIdx.x % NO2;
  const int b = d.rowblk[(A / d.L) * d.maxl + lv];
  if (b < 0 || A + nb + d.k > d.last[n]) return;   // the instance's rows end before this leaf is final
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = d.b_r0[b], c0 = d.b_c0[b];
  const int ncol = d.b_c1[b] - c0, rmax = d.rmax, L = d.L;
  const int ld_k = rmax + L;
  double2* ws = d.tsvd_ws + (((long long)blockIdx.y * 4 + X) * NO2 + p) * d.tsvd_ws_per + d.ws_lvoff[lv];
  V* Em = reinterpret_cast<V*>(ws);                   // [nb][ncol]
  V* Qm = Em + (long long)L * ncol;                   // [nb][ncol]
  V* Pm = Qm + (long long)L * ncol;                   // [nb][rmax]
  V* Cm = Pm + (long long)L * rmax;                   // [nb][nb]
  V* g1 = Cm + (long long)L * L;                      // [ld_k][ld_k] R^dagger, where it does not fit in shared memory
  V* g2 = g1 + (long long)ld_k * ld_k;                // [ld_k][ld_k] the core while it is factorised, then K W / sigma
  extern __shared__ __align__(16) char dyn[];
  V* sm = reinterpret_cast<V*>(dyn);
  constexpr int kSm = kTsvdSmem / sizeof(V);
  __shared__ double s_w[8], s_norm[64], s_sig[256];
  __shared__ int s_ord[256], s_flag, s_piv;
  __shared__ V s_coef[256];
  int* rkp = Rk<NO>(d, X, n, b, p);
  const int r = *rkp;
  S* U = Up<NO, S>(d, X, n, b, p);
  S* Vf = Vp<NO, S>(d, X, n, b, p);
  double* Sv = Sp<NO>(d, X, n, b, p);
  // E <- new rows (and max |E| for the complex64 rounding floor below).  The
  // complex64 form reads them from its FP64 copies: rows free of storage
  // rounding, whose residuals against V hold real directions only.
  float top = 0.f;
  {
    void* ring = ringX(d, X);
    double emax = 0.0;
    for (int i = warp; i < nb; i += 8)
      for (int l = lane; l < ncol; l += 32) {
        V v;
        if (d.ring64[X]) v = ld_split<S>(el64<NO>(d, X, n, A + i, c0 + l) + p);
        else vset(v, ld(el<NO, S>(ring, d, n, A + i, c0 + l) + p));
        emax = fmax(emax, (double)vnorm2(v));
        top = fmaxf(top, vtop(v));
        Em[(long long)i * ncol + l] = v;
      }
    emax = warp_max(emax);
    top = (float)warp_max((double)top);
    if (lane == 0) { s_w[warp] = emax; s_norm[warp] = top; }
  }
  __syncthreads();
  // The complex64 form's squares have the range of FP32: rows and singular values
  // far from 1 are brought there by a power of two, which changes no digit, and the
  // new singular values taken back.
  double up = 1.0, down = 1.0;
  if constexpr (sizeof(S) == sizeof(float2)) {
    double big = r > 0 ? Sv[0] : 0.0;
    for (int w2 = 0; w2 < 8; ++w2) big = fmax(big, s_norm[w2]);
    if (big > 0.0 && (big < 0x1p-20 || big > 0x1p50)) {   // (the same for every thread)
      const int e = min(max((__double2hiint(big) >> 20) - 1023, -126), 126);
      up = __hiloint2double((1023 - e) << 20, 0);
      down = __hiloint2double((1023 + e) << 20, 0);
      __syncthreads();
      double emax = 0.0;
      for (int i = warp; i < nb; i += 8)
        for (int l = lane; l < ncol; l += 32) {
          const V v = vldexp(Em[(long long)i * ncol + l], -e);
          emax = fmax(emax, (double)vnorm2(v));
          Em[(long long)i * ncol + l] = v;
        }
      emax = warp_max(emax);
      if (lane == 0) s_w[warp] = emax;
      __syncthreads();
    }
  }
  // Truncation threshold: eps_SVD, raised in the complex64 storage form to
  // the rounding floor of the appended rows.  Their rounding is a matrix of
  // independent entries below 2^-24 max|E|, whose largest singular value
  // stays below 2^-24 max|E| (sqrt(nb) + sqrt(ncol)); directions under that
  // level are storage noise, and keeping them would let the rank grow by the
  // leaf size at every append.
  double tol = d.svd_tol * up;
  if (sizeof(S) == sizeof(float2)) {
    double emax = 0.0;
    for (int w2 = 0; w2 < 8; ++w2) emax = fmax(emax, s_w[w2]);
    tol = fmax(tol, kF32Unit * sqrt(emax) * (sqrt((double)nb) + sqrt((double)ncol)));
  }
  constexpr int TC = 32;   // columns of a tile
  // P = E V, E -= P V^dagger: once in the FP64 form, whose V is orthonormal to
  // rounding; twice in the complex64 form, whose stored V is so to 2^-24 only (one
  // pass leaves parts of that size along V in every row, about the threshold, and
  // the ranks of the C2 run reached r_max).  The residual of a pass goes through
  // its own coefficients, kept in Q's storage (r <= ncol), free until the
  // Gram-Schmidt below.
  constexpr int kPasses = sizeof(S) == sizeof(double2) ? 1 : 2;
  for (int pass = 0; pass < (r > 0 ? kPasses : 1); ++pass) {
  for (int qb = 0; qb < r; qb += 64) {   // the coefficients E V
    const int rq = min(r - qb, 64), lg = rq <= 4 ? 2 : rq <= 8 ? 3 : rq <= 16 ? 4 : rq <= 32 ? 5 : 6;
    const int q = tid & ((1 << lg) - 1), i0 = tid >> lg, di = blockDim.x >> lg;   // rows i0 + di o
    V* Et = sm;                       // [64][TC + 1]
    V* Vt = sm + 64 * (TC + 1);       // [TC][64]
    DotC<S> acc[16];
    for (int l0 = 0; l0 < ncol; l0 += TC) {
      for (int e = tid; e < nb * TC; e += blockDim.x)
        if (l0 + e % TC < ncol) Et[(e / TC) * (TC + 1) + e % TC] = Em[(long long)(e / TC) * ncol + l0 + e % TC];
      for (int e = tid; e < TC * rq; e += blockDim.x)
        if (l0 + e / rq < ncol) Vt[(e / rq) * 64 + e % rq] = vof(Vf[(long long)(l0 + e / rq) * rmax + qb + e % rq]);
      __syncthreads();
      const int lc = min(TC, ncol - l0);
      if (q < rq)
        for (int l = 0; l < lc; ++l) {
          const V v = Vt[l * 64 + q];
#pragma unroll
          for (int o = 0; o < 16; ++o) {
            const int i = i0 + di * o;
            if (i >= nb) break;
            acc[o].add(Et[i * (TC + 1) + l], v);
          }
        }
      __syncthreads();
    }
    if (q < rq)
#pragma unroll
      for (int o = 0; o < 16; ++o) {
        const int i = i0 + di * o;
        if (i < nb) {
          const V c = acc[o].get();
          V* pp = Pm + (long long)i * rmax + qb + q;
          *pp = pass == 0 ? c : vadd(*pp, c);
          Qm[(long long)i * ncol + qb + q] = c;
        }
      }
    __syncthreads();
  }
  // the residual, and the norms of its rows (rows w, w + 8, ... to warp w)
  {
    Nrm2<S> nr[8];
    const int rows = (nb + 7) / 8;
    for (int qb = 0; qb == 0 || qb < r; qb += 64) {
      const int rq = max(0, min(r - qb, 64));
      const bool lastq = qb + 64 >= r;
      V* Pt = sm;                     // [64][64]
      V* Vt = sm + 64 * 64;           // [TC][65]
      for (int e = tid; e < nb * rq; e += blockDim.x) Pt[(e / rq) * 64 + e % rq] = vneg(Qm[(long long)(e / rq) * ncol + qb + e % rq]);
      for (int l0 = 0; l0 < ncol; l0 += TC) {
        for (int e = tid; e < TC * rq; e += blockDim.x)
          if (l0 + e / rq < ncol) Vt[(e / rq) * 65 + e % rq] = vconj(vof(Vf[(long long)(l0 + e / rq) * rmax + qb + e % rq]));
        __syncthreads();
        if (l0 + lane < ncol) {
#pragma unroll
          for (int o = 0; o < 8; ++o) {
            const int i = warp + 8 * o;
            if (o >= rows || i >= nb) break;
            V* ep = Em + (long long)i * ncol + l0 + lane;
            V v = *ep;
            if (rq) {
              DotC<S> acc;
              dot_from(acc, v);
              for (int q = 0; q < rq; ++q) acc.add(Pt[i * 64 + q], Vt[lane * 65 + q]);
              v = acc.get();
              *ep = v;
            }
            if (lastq) nr[o].add(v);
          }
        }
        __syncthreads();
      }
    }
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const R s = rsum(nr[o].get(), 32);
      if (lane == 0 && warp + 8 * o < nb) s_norm[warp + 8 * o] = r64(s);
    }
  }
  __syncthreads();
  }
  for (int e = tid; e < L * L; e += blockDim.x) vset(Cm[e], zd());
  __syncthreads();
  // ---- Gram-Schmidt on the rows of E: E = C Q, rows of Q orthonormal.
  // Residual rows below a quarter of the threshold add no basis direction
  // (a higher floor, the rounding level of one stored row, rejects rows that
  // are each at noise level but together carry a direction above the
  // threshold: measured on the C4 batch, the ranks then grew about threefold).
  // Every thread takes the same decisions from the same sums.
  const double delta = 0.25 * tol, delta2 = delta * delta;
  int ke = 0;
  for (int j = 0; j < nb && r + ke < ncol; ++j) {
    {   // the next row above the floor
      const bool a = lane < nb && lane >= j && s_norm[lane] > delta2;
      const bool c = lane + 32 < nb && lane + 32 >= j && s_norm[lane + 32] > delta2;
      const unsigned lo = __ballot_sync(FULL, a), hi = __ballot_sync(FULL, c);
      if (lo) j = __ffs(lo) - 1;
      else if (hi) j = 31 + __ffs(hi);
      else break;
    }
    V* v = Em + (long long)j * ncol;
    // second pass of the accepted row: against V, then against the rows of Q
    for (int e = warp; e < r + ke; e += 8) {
      DotC<S> s;
      if (e < r)
        for (int l = lane; l < ncol; l += 32) s.add(vof(Vf[(long long)l * rmax + e]), v[l]);
      else
        for (int l = lane; l < ncol; l += 32) s.add(vconj(Qm[(long long)(e - r) * ncol + l]), v[l]);
      const V c = vsum(s.get(), 32);
      if (lane == 0) s_coef[e] = c;
    }
    __syncthreads();
    Nrm2<S> ns;
    for (int l = tid; l < ncol; l += blockDim.x) {
      DotC<S> s;
      dot_from(s, v[l]);
      for (int e = 0; e < r; ++e) s.add(vneg(s_coef[e]), vconj(vof(Vf[(long long)l * rmax + e])));
      for (int e = 0; e < ke; ++e) s.add(vneg(s_coef[r + e]), Qm[(long long)e * ncol + l]);
      const V x = s.get();
      v[l] = x;
      ns.add(x);
    }
    {
      const R s = rsum(ns.get(), 32);
      if (lane == 0) s_w[warp] = r64(s);
    }
    for (int e = tid; e < r + ke; e += blockDim.x) {
      V* c = e < r ? Pm + (long long)j * rmax + e : Cm + (long long)j * L + e - r;
      *c = vadd(*c, s_coef[e]);
    }
    __syncthreads();
    double n2 = 0.0;
    for (int w2 = 0; w2 < 8; ++w2) n2 += s_w[w2];
    if (!(n2 > delta2)) continue;
    const double nrm = sqrt(n2);
    const R inv = rof(1.0 / nrm, (S*)nullptr);
    V* q = Qm + (long long)ke * ncol;
    for (int l = tid; l < ncol; l += blockDim.x) q[l] = vscl(v[l], inv);
    if (tid == 0) vset(Cm[(long long)j * L + ke], zd(nrm));
    __syncthreads();
    // every later row loses its part along q; four rows at a time per warp
    for (int ib = j + 1 + warp * 4; ib < nb; ib += 32) {
      DotC<S> s[4];
      for (int l = lane; l < ncol; l += 32) {
        const V qc = vconj(q[l]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (ib + u < nb) s[u].add(qc, Em[(long long)(ib + u) * ncol + l]);
      }
      V c[4];
      Nrm2<S> m2[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) c[u] = vsum(s[u].get(), 32);
      for (int l = lane; l < ncol; l += 32) {
        const V ql = q[l];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (ib + u < nb) {
            V* ep = Em + (long long)(ib + u) * ncol + l;
            const V x = vadd(*ep, vneg(vmul(c[u], ql)));
            *ep = x;
            m2[u].add(x);
          }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const R t = rsum(m2[u].get(), 32);
        if (lane == 0 && ib + u < nb) {
          s_norm[ib + u] = r64(t);
          Cm[(long long)(ib + u) * L + ke] = c[u];
        }
      }
    }
    ++ke;
    __syncthreads();
  }
  __syncthreads();
  const int m = r + nb, nk = r + ke;  // core rows, columns
  // ---- the core K = [[diag(S), 0], [P, C]], column by column, and its column-pivoted QR ----
  V* Xr = nk * nk <= kSm ? sm : g1;                                       // [col][nk] R^dagger
  V* Kw = Xr == sm && nk * nk + m * nk <= kSm ? sm + nk * nk : g2;        // [col][m]
  for (int e = tid; e < nk * m; e += blockDim.x) {
    const int col = e / m, row = e % m;
    V v;
    if (row < r) vset(v, col == row ? zd(Sv[row] * up) : zd());
    else if (col < r) v = Pm[(long long)(row - r) * rmax + col];
    else v = Cm[(long long)(row - r) * L + (col - r)];
    Kw[e] = v;
  }
  for (int e = tid; e < nk * nk; e += blockDim.x) vset(Xr[e], zd());
  __syncthreads();
  for (int col = warp; col < nk; col += 8) {
    Nrm2<S> s;
    for (int i = lane; i < m; i += 32) s.add(Kw[col * m + i]);
    const R t = rsum(s.get(), 32);
    if (lane == 0) s_sig[col] = r64(t);
  }
  __syncthreads();
  const double drop2 = 1e-14 * tol * tol;   // columns this far below the threshold add nothing
  int nr = 0;                               // columns of R^dagger
  for (; nr < nk; ++nr) {
    if (warp == 0) {   // the largest remaining column (taken ones have norm -1)
      double best = -1.0;
      int arg = 0;
      for (int col = lane; col < nk; col += 32)
        if (s_sig[col] > best) { best = s_sig[col]; arg = col; }
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        const double b2 = __shfl_xor_sync(FULL, best, off);
        const int a2 = __shfl_xor_sync(FULL, arg, off);
        if (b2 > best || (b2 == best && a2 < arg)) { best = b2; arg = a2; }
      }
      if (lane == 0) { s_piv = best > drop2 ? arg : -1; s_w[0] = best; }
    }
    __syncthreads();
    const int pv = s_piv;
    if (pv < 0) break;
    const double nrm = sqrt(s_w[0]);
    const R inv = rof(1.0 / nrm, (S*)nullptr);
    for (int i = tid; i < m; i += blockDim.x) Kw[pv * m + i] = vscl(Kw[pv * m + i], inv);
    if (tid == 0) {
      vset(Xr[nr * nk + pv], zd(nrm));
      s_sig[pv] = -1.0;
    }
    __syncthreads();
    for (int col = warp; col < nk; col += 8) {
      if (s_sig[col] < 0.0) continue;
      DotC<S> s;
      for (int i = lane; i < m; i += 32) s.add(vconj(Kw[pv * m + i]), Kw[col * m + i]);
      const V c = vsum(s.get(), 32);
      Nrm2<S> t;
      for (int i = lane; i < m; i += 32) {
        const V x = vadd(Kw[col * m + i], vneg(vmul(c, Kw[pv * m + i])));
        Kw[col * m + i] = x;
        t.add(x);
      }
      const R t2 = rsum(t.get(), 32);
      if (lane == 0) {
        Xr[nr * nk + col] = vconj(c);
        s_sig[col] = r64(t2);
      }
    }
    __syncthreads();
  }
  __syncthreads();
  // ---- one-sided Jacobi (Hestenes) on the columns of R^dagger, round-robin pairing, a half-warp per pair ----
  const auto small2 = (decltype(rtop(R())))(1e-6 * tol * tol);   // two columns both this small are truncated: left as they are
  const int npad = nr + (nr & 1);
  for (int sweep = 0; sweep < 40; ++sweep) {
    if (tid == 0) s_flag = 0;
    __syncthreads();
    for (int round = 0; round < npad - 1; ++round) {
      // round-robin tournament: position 0 fixed, positions 1..npad-1 rotate
      auto at = [&](int i) { return i == 0 ? 0 : ((i - 1 + round) % (npad - 1)) + 1; };
      for (int pr0 = warp * 2; pr0 < npad / 2; pr0 += 16) {
        const int pr = pr0 + (lane >> 4), hl = lane & 15;
        int ia = 0, ib = 0;
        bool act = pr < npad / 2;
        if (act) {
          ia = at(pr);
          ib = at(npad - 1 - pr);
          act = ia < nr && ib < nr;
        }
        V *xa = Xr + ia * nk, *xb = Xr + ib * nk;
        Nrm2<S> na, nbm;
        DotC<S> ng;
        if (act)
          for (int i = hl; i < nk; i += 16) {
            const V x = xa[i], y = xb[i];
            na.add(x);
            nbm.add(y);
            ng.add(vconj(x), y);
          }
        const R al = rsum(na.get(), 16), be = rsum(nbm.get(), 16);
        const V ga = vsum(ng.get(), 16);
        const Quad qa = quad_of(al), qb = quad_of(be);   // |a|^2 = fa 4^ea, |b|^2 = fb 4^eb, <a, b> = gs 2^(ea + eb)
        const V gs = vldexp(ga, -(qa.e + qb.e));
        const float fa = qa.m, fb = qb.m, fg = sqrtf(vnorm32(gs));
        const int de = qb.e - qa.e;
        const float eps = sizeof(S) == sizeof(double2) ? 1e-14f : 1e-13f;
        act = act && fa * fb > 0.f && fg > eps * sqrtf(fa * fb) && (rtop(al) >= small2 || rtop(be) >= small2) && abs(de) <= 100;
        if (act) {
          Nrm2<S> g2;
          g2.add(gs);
          V ph = vscl(vconj(gs), rsq(g2.get()));           // e^{-i phi}
          float tf;   // tan of the angle: 1 / (zeta + sign sqrt(1 + zeta^2)), zeta = (|b|^2 - |a|^2) / (2 |<a, b>|)
          if (abs(de) > 20) {   // 1 / (2 zeta)
            tf = (de > 0 ? fg / fb : -fg / fa) * __int_as_float((127 - abs(de)) << 23);
          } else {
            const float u = __int_as_float((127 + de) << 23), v = __int_as_float((127 - de) << 23);
            const float zeta = (fb * u - fa * v) / (2.f * fg);
            tf = fabsf(zeta) < 1e18f ? (zeta >= 0.f ? 1.f : -1.f) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta)) : 0.5f / zeta;
          }
          R cs, sn;
          if constexpr (sizeof(S) == sizeof(double2)) {
            cs = rsq(fma((double)tf, (double)tf, 1.0));
            sn = cs * (double)tf;
          } else {
            cs = rsq(ff_add(ff_mul({tf, 0.f}, {tf, 0.f}), {1.f, 0.f}));
            sn = ff_mul(cs, {tf, 0.f});
          }
          if (hl == 0) s_flag = 1;
          for (int i = hl; i < nk; i += 16) {
            const V x = xa[i], y = vmul(xb[i], ph);
            xa[i] = vadd(vscl(x, cs), vneg(vscl(y, sn)));
            xb[i] = vadd(vscl(x, sn), vscl(y, cs));
          }
        }
      }
      __syncthreads();
    }
    if (!s_flag) break;
    if (sweep == 39 && tid == 0) atomicAdd(d.status + 1, 1);
    __syncthreads();
  }
  // ---- singular values, sorted, truncated; W = the normalised columns ----
  for (int col = warp; col < nr; col += 8) {
    Nrm2<S> s;
    for (int i = lane; i < nk; i += 32) s.add(Xr[col * nk + i]);
    const R t = rsum(s.get(), 32);
    if (lane == 0) s_sig[col] = sqrt(r64(t));
  }
  __syncthreads();
  if (tid < nr) {   // position in descending order (ties by index)
    const double s = s_sig[tid];
    int pos = 0;
    for (int i = 0; i < nr; ++i) pos += s_sig[i] > s || (s_sig[i] == s && i < tid);
    s_ord[pos] = tid;
  }
  if (tid == 0) s_flag = 0;
  __syncthreads();
  if (tid < nr && s_sig[tid] > tol) atomicAdd(&s_flag, 1);
  __syncthreads();
  int rn = s_flag;
  if (rn > rmax) {
    if (tid == 0) atomicAdd(d.status, 1);
    rn = rmax;
  }
  for (int e = tid; e < rn * nk; e += blockDim.x) {
    V* x = Xr + s_ord[e / nk] * nk + e % nk;
    *x = vscl(*x, rof(1.0 / s_sig[s_ord[e / nk]], (S*)nullptr));
  }
  __syncthreads();
  // K W / sigma, [rn][m]: the first r rows S W / sigma, the others (P W + C W) / sigma
  V* Kt = Xr == sm && nk * nk + rn * m <= kSm ? sm + nk * nk : g2;
  for (int e = tid; e < rn * m; e += blockDim.x) {
    const int jj = e / m, row = e % m;
    const V* w = Xr + s_ord[jj] * nk;
    const R inv = rof(1.0 / s_sig[s_ord[jj]], (S*)nullptr);
    V v;
    if (row < r) {
      v = vscl(w[row], rof(Sv[row] * up, (S*)nullptr));
    } else {
      DotC<S> s;
      for (int q = 0; q < r; ++q) s.add(Pm[(long long)(row - r) * rmax + q], w[q]);
      for (int q = 0; q < ke; ++q) s.add(Cm[(long long)(row - r) * L + q], w[r + q]);
      v = s.get();
    }
    Kt[e] = vscl(v, inv);
  }
  __syncthreads();
  // U' and V': lp lanes per row, up to four entries each; a row is read by its lanes before they write it
  const int lp = rn <= 4 ? 4 : rn <= 8 ? 8 : rn <= 16 ? 16 : 32, sub = tid / lp, j0 = tid % lp, rstep = blockDim.x / lp;
  auto rotate = [&](int rows, auto entry, S* out) {
    for (int row0 = 0; row0 < rows; row0 += rstep) {
      const int row = row0 + sub;
      V res[4];
#pragma unroll
      for (int t2 = 0; t2 < 4; ++t2) {
        const int jj = j0 + lp * t2;
        vset(res[t2], zd());
        if (jj < rn && row < rows) res[t2] = entry(row, jj);
      }
      __syncwarp();
      if (row < rows)
        for (int t2 = 0; t2 * lp < rmax; ++t2) {
          const int jj = j0 + lp * t2;
          if (jj < rmax) {
            V v = res[0];
            if (t2 == 1) v = res[1];
            if (t2 == 2) v = res[2];
            if (t2 == 3) v = res[3];
            if (jj >= rn) vset(v, zd());
            if constexpr (sizeof(S) == sizeof(double2)) st(out + (long long)row * rmax + jj, v);
            else out[(long long)row * rmax + jj] = make_float2(v.re.hi, v.im.hi);
          }
        }
      __syncwarp();
    }
  };
  const int nold = A - r0;   // old rows r0..A-1, new rows A..A+nb-1
  rotate(nold + nb, [&](int row, int jj) {
    if (row >= nold) return Kt[jj * m + r + row - nold];
    DotC<S> s;
    for (int q = 0; q < r; ++q) s.add(vof(U[(long long)row * rmax + q]), Kt[jj * m + q]);
    return s.get();
  }, U);
  rotate(ncol, [&](int l, int jj) {
    const V* w = Xr + s_ord[jj] * nk;
    DotC<S> s;
    for (int q = 0; q < r; ++q) s.add(vof(Vf[(long long)l * rmax + q]), w[q]);
    for (int e = 0; e < ke; ++e) s.add(vconj(Qm[(long long)e * ncol + l]), w[r + e]);
    return s.get();
  }, Vf);
  for (int q = tid; q < rmax; q += blockDim.x) Sv[q] = (q < rn) ? s_sig[s_ord[q]] * down : 0.0;
  if (tid == 0) *rkp = rn;
}

// Row T of G^R and G^< (any T <= current) in complex128 into out_r, out_l
// ([T+1][no2] each, pinned host memory), from the dense triangle, the ring, the
// leaves or the blocks.  One launch and one synchronisation per row: a copy of
// each component through pageable memory, each waited for, and a conversion on
// the host took some 45 us, half of them gaps (304 instances, T = 384, a row of
// each at the end: 106.9 -> 98.7 ms a pass).
template <int NO, typename S>
__global__ void k_row_out(Dev d, int n, int T, double2* out_r, double2* out_l) {
  constexpr int NO2 = NO * NO;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t > T) return;
  for (int X = 0; X < 2; ++X) {
    double2* out = (X == 0) ? out_r : out_l;
    if (!out) continue;
    for (int p = 0; p < NO2; ++p) {
      zd v;
      if (!d.ring || T >= front_of(d, n)) {
        v = ld(el<NO, S>(ringX(d, X), d, n, T, t) + p);
      } else {
        const int jT = T / d.L, jt = t / d.L;
        if (jT == jt) {
          v = ld(Lf<NO, S>(d, X, n, jT, T, t) + p);
        } else {
          v = zd();
          for (int lv = 0; lv < d.maxl; ++lv) {
            const int b = d.rowblk[jT * d.maxl + lv];
            if (b < 0 || t < d.b_c0[b] || t >= d.b_c1[b]) continue;
            const int rk = *Rk<NO>(d, X, n, b, p);
            const S* U = Up<NO, S>(d, X, n, b, p) + (long long)(T - d.b_r0[b]) * d.rmax;
            const S* V = Vp<NO, S>(d, X, n, b, p) + (long long)(t - d.b_c0[b]) * d.rmax;
            const double* Sv = Sp<NO>(d, X, n, b, p);
            for (int q = 0; q < rk; ++q) v += ld(U + q) * ld(V + q).conj() * Sv[q];
          }
        }
      }
      st(out + (long long)t * NO2 + p, v);
    }
  }
}

// rho(t) = xi i G^<(t, t) of every instance, from a row (dense or ring) or a leaf.
template <int NO, typename S>
__global__ void k_density_at(Dev d, int t, double2* out) {
  constexpr int NO2 = NO * NO;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= d.n_inst * NO2) return;
  const int n = e / NO2, q = e % NO2;
  if (t > d.last[n]) {   // past the instance's last step
    st(out + e, zd());
    return;
  }
  const S* p = (!d.ring || t >= front_of(d, n)) ? el<NO, S>(d.GL, d, n, t, t) : Lf<NO, S>(d, 1, n, t / d.L, t, t);
  st(out + e, ld(p + q) * zd(0, (double)d.xi));
}


// ---------------------------------------------------------------------------
// 2D Hubbard lattice, second Born (Sec. 4.2), N_o = 1, one instance per
// k = 2 pi (m_x, m_y)/L (instance m_x L + m_y), or, with the reflection
// k_y -> -k_y of a drive along x (Sec. 4.2, the L(L/2+1) k-set), one
// instance per m_y <= L/2 (instance m_x (L/2+1) + m_y; k-point (m_x, L - m_y)
// reads instance (m_x, m_y)):
//   X_r = (1/N_k) sum_k e^{+i k.r} X_k,
//   Sigma^>_r = U(T)U(t) G^>_r(T,t)^2 G^<_{-r}(t,T),
//   Sigma^<_r = U(T)U(t) G^<_r(T,t)^2 G^>_{-r}(t,T),
//   Sigma_k = sum_r e^{-i k.r} Sigma_r,  Sigma^R = Sigma^> - Sigma^<,
// where Y_{-r} = (1/N_k) sum_k e^{-i k.r} Y_k of Y_k = -[X_k]^* is -[X_r]^*, so
// G^<_{-r}(t,T) and G^>_{-r}(t,T) come from the transforms of G^<(T,t) and
// G^>(T,t).  Mixed: Sigma^tv_r = U(T)U(0_|) G^tv_r(T,tau)^2 G^vt_{-r}(tau,T).
// One CTA per kLatT times of the current row (or DLR nodes of the mixed row):
// two grids each, FP64-bound.
// ---------------------------------------------------------------------------
template <typename S>
__global__ void __launch_bounds__(128) k_sigma_lattice(Dev d, int T) {
  pdl_start();
  extern __shared__ __align__(16) zd grid[];   // [2][kLatT] grids of L rows of L + 1
  __shared__ zd tw[16];
  if (!d.active[0]) return;   // (the k-points iterate together)
  const int L = (int)d.mpar[0], ys = (int)d.mpar[1], N = L * L, gsz = L * (L + 1);
  const int ntb = (T + kLatT) / kLatT, tid = threadIdx.x;
  lat_twiddles(tw, L);
  const double* U = d.drU;   // U(t) of instance 0 (the same for every k)
  const double invN = 1.0 / N;
  zd *X1 = grid, *X2 = grid + kLatT * gsz;
  auto at = [&](int e, int* q) {   // element e: time (fastest) and grid point
    *q = e / kLatT;
    return (e % kLatT) * gsz + (*q / L) * (L + 1) + *q % L;
  };
  if ((int)blockIdx.x < ntb) {
    const int t0 = blockIdx.x * kLatT;
    for (int e = tid; e < kLatT * N; e += blockDim.x) {
      int q;
      const int o = at(e, &q), t = t0 + e % kLatT, nq = lat_inst(q, L, ys);
      zd gg = zd(), gl = zd();
      if (t <= T) {
        gl = -ldx<1, S>(d, 1, nq, T, t, 0).conj();   // G^<(T, t)
        gg = ldx<1, S>(d, 0, nq, T, t, 0) + gl;      // G^>(T, t)
      }
      X1[o] = gg;
      X2[o] = gl;
    }
    __syncthreads();
    lat_fft2(grid, 2 * kLatT, tw, L, +1);
    for (int e = tid; e < kLatT * N; e += blockDim.x) {
      int q;
      const int o = at(e, &q), t = t0 + e % kLatT;
      const double uu = t <= T ? U[T + 1] * U[t + 1] : 0.0;
      const zd g = X1[o] * invN, l = X2[o] * invN;
      X1[o] = g * g * -l.conj() * uu;    // Sigma^>_r
      X2[o] = l * l * -g.conj() * uu;    // Sigma^<_r
    }
    __syncthreads();
    lat_fft2(grid, 2 * kLatT, tw, L, -1);
    for (int e = tid; e < kLatT * N; e += blockDim.x) {
      int q;
      const int o = at(e, &q), t = t0 + e % kLatT;
      if (t > T || !lat_owner(q, L, ys)) continue;
      const int nq = lat_inst(q, L, ys);
      stx<1, S>(d, 2, nq, T, t, 0, X1[o] - X2[o]);
      stx<1, S>(d, 3, nq, T, t, 0, -X2[o].conj());
    }
  } else {
    const int i0 = (blockIdx.x - ntb) * kLatT, r = d.r, ni = min(kLatT, r - i0);
    for (int q = tid; q < N; q += blockDim.x) {
      const int nq = lat_inst(q, L, ys), o = (q / L) * (L + 1) + q % L;
      const double2* G = tv<1>(d.GTV, d, nq, T, 0);
      zd gb[kLatT];                                          // G^tv(T, beta - tau_i)
#pragma unroll
      for (int i = 0; i < kLatT; ++i) gb[i] = zd();
      for (int c = 0; c < r; ++c) {
        const zd g = ld(G + c);
#pragma unroll
        for (int i = 0; i < kLatT; ++i) {
          const double rv = i < ni ? d.rev[(i0 + i) * r + c] : 0.0;
          gb[i] = zd(fma(g.re, rv, gb[i].re), fma(g.im, rv, gb[i].im));
        }
      }
#pragma unroll
      for (int i = 0; i < kLatT; ++i) {
        X1[i * gsz + o] = i < ni ? ld(G + i0 + i) : zd();
        X2[i * gsz + o] = gb[i];
      }
    }
    __syncthreads();
    lat_fft2(grid, 2 * kLatT, tw, L, +1);
    const double uu = U[T + 1] * U[0] * -(double)d.xi;       // G^vt_{-r}(tau_i, T) = -xi [G^tv_r(T, beta - tau_i)]^*
    for (int e = tid; e < kLatT * N; e += blockDim.x) {
      int q;
      const int o = at(e, &q);
      const zd x = X1[o] * invN, y = X2[o] * invN;
      X1[o] = x * x * y.conj() * uu;
    }
    __syncthreads();
    lat_fft2(grid, kLatT, tw, L, -1);
    for (int e = tid; e < kLatT * N; e += blockDim.x) {
      int q;
      const int o = at(e, &q), i = i0 + e % kLatT;
      if (i < r && lat_owner(q, L, ys)) st(tv<1>(d.STV, d, lat_inst(q, L, ys), T, i), X1[o]);
    }
  }
}

// Lattice observables at time t (Sec. 4.2): n = -(i/N) sum_k G^<_k(t,t),
// E_kin = -(2i/N) sum_k eps_k G^<_k(t,t), eps_k = -2(cos k_x + cos k_y),
// j = -(2i/N) sum_k 2 sin(k_x - A(t)) G^<_k(t,t); out = (n, E_kin, j).  The
// sums run over the whole L x L grid (a reflected k-point reads its mirror).
template <typename S>
__global__ void __launch_bounds__(kLatMaxK) k_lattice_obs(Dev d, int t, double* out) {
  __shared__ double red[3][kLatMaxK];
  const int L = (int)d.mpar[0], ys = (int)d.mpar[1], N = L * L, q = threadIdx.x;
  double v[3] = {0, 0, 0};
  if (q < N) {
    const int nq = lat_inst(q, L, ys);
    const S* p = (!d.ring || t >= d.cdir) ? el<1, S>(d.GL, d, nq, t, t) : Lf<1, S>(d, 1, nq, t / d.L, t, t);
    const double mi = (-ld(p) * zd(0, 1)).re;            // Re(-i G^<(t,t))
    const double kx = 2.0 * M_PI * (q / L) / L, ky = 2.0 * M_PI * (q % L) / L;
    const double A = d.drA[t + 1];
    v[0] = mi / N;
    v[1] = 2.0 * (-2.0 * (cos(kx) + cos(ky))) * mi / N;
    v[2] = 2.0 * 2.0 * sin(kx - A) * mi / N;
  }
  for (int c = 0; c < 3; ++c) red[c][q] = v[c];
  __syncthreads();
  if (q == 0) {
    for (int c = 0; c < 3; ++c) {
      double s = 0.0;
      for (int e = 0; e < N; ++e) s += red[c][e];   // fixed order
      out[c] = s;
    }
  }
}

#define HK_DISPATCH(NOV, ...)                                                   \
  switch ((NOV) * 2 + d.prec) {                                                 \
    case 2: { constexpr int NO = 1; using S = double2; __VA_ARGS__; break; }           \
    case 3: { constexpr int NO = 1; using S = float2; __VA_ARGS__; break; }            \
    case 4: { constexpr int NO = 2; using S = double2; __VA_ARGS__; break; }           \
    case 5: { constexpr int NO = 2; using S = float2; __VA_ARGS__; break; }            \
    case 6: { constexpr int NO = 3; using S = double2; __VA_ARGS__; break; }           \
    case 7: { constexpr int NO = 3; using S = float2; __VA_ARGS__; break; }            \
    case 8: { constexpr int NO = 4; using S = double2; __VA_ARGS__; break; }           \
    case 9: { constexpr int NO = 4; using S = float2; __VA_ARGS__; break; }            \
    default: return cudaErrorInvalidValue;                                      \
  }

// Dynamic shared memory of k_src_q; the list of packed entries is left out
// where ranks, levels and orbitals would make it too large.
template <int NO, typename S>
static cudaError_t src_q(const Dev& d, int T, cudaStream_t s) {
  const size_t n2 = NO * NO, es = sizeof(S), ns = 2 * (size_t)d.maxl * n2;
  size_t bytes = ((size_t)d.r * n2 + 8 * n2 * 32) * 16 + (kRingRows + 64) * n2 * es + (2 * ns + 1) * 4 + 8 + ns * 16;
  const size_t list = ns * d.rmax * 2;
  const int uselist = ns * 128 <= 65536 && bytes + list <= 200 * 1024;
  if (uselist) bytes += list;
  const int nrow = T + 1 - d.cdir;
  return launch_k(k_src_q<NO, S>, dim3(d.cdir / 32 + (nrow + 7) / 8, d.n_inst), 256, bytes, s, d, T, uselist);
}
cudaError_t open_history(const Dev& d) {
  cudaError_t e = cudaErrorInvalidValue;
  int room = 1 << 30;
  HK_DISPATCH(d.no, {
    if ((e = open_smem(k_src_q<NO, S>, &room)) == cudaSuccess) e = open_smem(k_tsvd<NO, S>, &room);
  })
  return e;
}
cudaError_t launch_src_h(const Dev& d, int T, int njob, cudaStream_t s) {
  if (d.cdir > 0 && T + 1 - d.cdir > kRingRows) return cudaErrorInvalidValue;
  if (njob > 0) {
    cudaError_t e = cudaErrorInvalidValue;
    HK_DISPATCH(d.no, e = launch_k(k_src_proj<NO, S>, dim3(njob, d.n_inst), 256, 0, s, d, T));
    if (e != cudaSuccess) return e;
  }
  HK_DISPATCH(d.no, return (src_q<NO, S>(d, T, s)));
  return cudaSuccess;
}
cudaError_t launch_compress(const Dev& d, int A, int nb, cudaStream_t s) {
  {
    dim3 g(64, d.n_inst);
    HK_DISPATCH(d.no, (k_comp_copy<NO, S><<<g, 256, 0, s>>>(d, A, nb)));
  }
  HK_DISPATCH(d.no, {
    for (int n0 = 0; n0 < d.n_inst; n0 += d.tsvd_group) {
      dim3 g(4 * d.maxl * d.no * d.no, min(d.tsvd_group, d.n_inst - n0));
      k_tsvd<NO, S><<<g, 256, kTsvdSmem, s>>>(d, A, nb, n0);
    }
  })
  return cudaGetLastError();
}
cudaError_t launch_density_at(const Dev& d, int t, double2* out, cudaStream_t s) {
  HK_DISPATCH(d.no, (k_density_at<NO, S><<<(d.n_inst * d.no * d.no + 127) / 128, 128, 0, s>>>(d, t, out)));
  return cudaGetLastError();
}
cudaError_t launch_sigma_lattice(const Dev& d, int T, cudaStream_t s) {
  if (d.no != 1 || d.n_inst > kLatMaxK) return cudaErrorInvalidValue;
  const int nb = (T + kLatT) / kLatT + (d.r + kLatT - 1) / kLatT;
  const size_t smem = lat_smem(16);   // 35 KB
  if (d.prec) return launch_k(k_sigma_lattice<float2>, dim3(nb), 128, smem, s, d, T);
  return launch_k(k_sigma_lattice<double2>, dim3(nb), 128, smem, s, d, T);
}
cudaError_t launch_lattice_obs(const Dev& d, int t, double* out, cudaStream_t s) {
  if (d.no != 1 || d.n_inst > kLatMaxK) return cudaErrorInvalidValue;
  if (d.prec) k_lattice_obs<float2><<<1, kLatMaxK, 0, s>>>(d, t, out);
  else k_lattice_obs<double2><<<1, kLatMaxK, 0, s>>>(d, t, out);
  return cudaGetLastError();
}
cudaError_t launch_row_out(const Dev& d, int n, int T, double2* out_r, double2* out_l, cudaStream_t s) {
  HK_DISPATCH(d.no, (k_row_out<NO, S><<<(T + 128) / 128, 128, 0, s>>>(d, n, T, out_r, out_l)));
  return cudaGetLastError();
}

}  // namespace hk
