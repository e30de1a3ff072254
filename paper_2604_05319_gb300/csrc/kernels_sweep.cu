// The two Volterra sweeps of a time step (Eq. KBER retarded row, Eq. KBEL
// lesser column) for both storage forms (dense triangles, or HODLR with a
// ring of uncompressed rows), organised in 32-point chunks at fixed absolute
// positions.
//
// Within one chunk the unknowns couple through the near-diagonal part of the
// discretised equation: the BDF stencil, eps, and Sigma^R entries inside the
// chunk with their Gregory weights.  Row T of Sigma^R, the only one that the
// corrector iterations of step T change, multiplies known values there
// (retarded: y(T) = -i) or belongs to one unknown (lesser: x(T)), so the
// coefficients between the other unknowns are final before the step's first
// iteration.  k_inv_rows brings the inverses of these triangular systems up
// to date once per step and instance, one appended row at a time:
//   retarded chunk [a, a+32): points t' < T - 2k, whose integrals end in the
//     standard Gregory weights; the 2k points above them (the head: the start
//     block and the points of the k < n < 2k+1 rule) form a system of their
//     own, inverted anew for every T;
//   lesser chunk [a, a+32): rows t < T; chunk 0 holds rows 1..31 and begins
//     with the start block.  Row T (horizontal density matrix) is one point
//     solve at the end.
// A chunk's solve is then F times the inverse (retarded, row vector) or the
// inverse times F (lesser), where F holds everything outside the chunk (the
// far field), also for the chunk that is still growing, so no point waits
// for its neighbour.  Solving the growing chunks point by point in one warp
// (a chain of up to 64 FP64 point solves per sweep, and an LU of the start
// block) took 75 of the 89 thousand cycles of a retarded sweep at N_o = 1,
// T <= 64, and 820 of 1900 thousand at N_o = 4, T = 290; the two sweeps of
// those runs went from 89 to 35 us and from 1650 to 1040 us.
#include "bulk_copy.cuh"
#include "hodlr_util.cuh"

namespace hk {

namespace {

constexpr int CK = 32;   // chunk length
using Y = double2;       // element type of the row / column being solved
template <int NO> constexpr bool kStage = NO <= 2;   // chunk inverses staged in shared memory
template <int NO> constexpr size_t kStageBytes = kStage<NO> ? sizeof(zd) * CK * CK * NO * NO : 0;
// Bytes of a chunk inverse that are staged in shared memory by a bulk copy
// issued before the chunk's far field, so the copy overlaps that phase: the
// whole inverse (FP64, or the hi and lo matrices of the complex64 form, 16
// bytes per entry either way); 0 (read from global memory) for N_o > 2.
template <int NO, typename S>
constexpr uint32_t kInvStage = kStage<NO> ? (uint32_t)(CK * NO * CK * NO * sizeof(double2)) : 0u;
constexpr int kCopyWaitPolls = 1 << 20;   // bound of the wait for a staged inverse

// Sum over the 8 lanes of an aligned lane group of their history
// accumulators (every lane receives it).  Complex64 form: the compensated
// FP32 sums are combined in float-float, so the reduction runs on the FP32
// pipes; FP64 form: plain FP64.  val_of converts to FP64 (once, by the lane
// that uses the sum).
template <typename R>
__device__ __forceinline__ auto reduce8(const KAcc<R>& k) { return kacc_lanes(k, 1, 8); }

// Where a sweep keeps the row it solves: in place (FP64 storage), or in FP64
// next to the complex64 storage: the row's slot of the FP64 ring copies of the
// compressed form (which the TSVD later compresses), else the buffer
// row64[n][which] of the dense form.
template <int NO, typename S>
struct Row64 {
  static constexpr bool separate = true;
  __device__ static Y* get(const Dev& d, int n, int which, int T, S*) {
    if (d.ring64[which]) return el64<NO>(d, which, n, T, 0);
    return d.row64 + ((long long)n * 2 + which) * d.nt * (NO * NO);
  }
};
template <int NO>
struct Row64<NO, double2> {
  static constexpr bool separate = false;
  __device__ static Y* get(const Dev&, int, int, int, double2* p) { return p; }
};

// Inverse of chunk cc of sweep `which`, (32 N_o)^2 entries (rows of points not yet built: unused).  FP64
// storage form: complex128.  Complex64 form: the same 16 bytes per entry
// hold a complex64 pair hi + lo (hi = the inverse rounded to complex64, lo =
// the rounding of hi), [hi matrix][lo matrix].  The chunk's right-hand side
// splits into the far field (history sums, lesser source), whose image under
// the inverse is about h / a_0 times smaller than the row and needs FP32 only,
// and the BDF terms reaching across the chunk edge (k rows), which carry the
// implicit recursion and get hi + lo in float-float (about 48 bits); a plain
// complex64 inverse would put 2^-24 times the BDF amplitude a_j / h into
// every chunk and accumulate.
template <int NO>
__device__ __forceinline__ double2* Cinv(const Dev& d, int n, int cc, int which) {
  const long long nn = (long long)(CK * NO) * (CK * NO);
  return d.cinv + (((long long)n * d.nchunk + cc) * 2 + which) * nn;
}

// Projections of one block of Sigma^R for all N_o^2 orbital pairs in one pass
// (complex64 form, N_o <= 2, rank <= 64): out_p[q] = S_p[q] sum_{l in [l0, l1)}
// v_p(l) F_p(l, q) for q < rank_p, with F = U (ROWS: the retarded sweep, v_p =
// y_m, m = p / N_o) or F = conj(V) (the lesser sweep, v_p = w_l x_nn, nn =
// p % N_o); vf(l, i) returns the vector's component i at l.  A warp covers
// 32 / lpr rows per step, lpr = 8, 16 or 32 lanes per row (the smallest that
// holds the largest rank), so small ranks keep every lane loading; warps split
// the rows, and the pairs share the vector loads.  Partial sums (compensated
// FP32) are combined across a warp's rows in float-float and across warps in
// red ([8][N_o^2][64], shared memory).  Every thread calls it.
template <int NO, typename S, bool ROWS, typename VF>
__device__ __forceinline__ void proj_block(const Dev& d, int n, int blk, int lv, int slot, int l0, int l1, VF vf,
                                           zd* red) {
  constexpr int NO2 = NO * NO;
  using R = typename Bulk<S>::R;
  static_assert(sizeof(R) == sizeof(float), "the one-pass projections serve the complex64 form");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int rk[NO2];
  const S* F[NO2];
  int rkmax = 0;
#pragma unroll
  for (int p = 0; p < NO2; ++p) {
    rk[p] = *Rk<NO>(d, 2, n, blk, p);
    F[p] = ROWS ? Up<NO, S>(d, 2, n, blk, p) : Vp<NO, S>(d, 2, n, blk, p);
    rkmax = max(rkmax, rk[p]);
  }
  const int base = ROWS ? d.b_r0[blk] : d.b_c0[blk];
  const int lpr = rkmax <= 8 ? 8 : rkmax <= 16 ? 16 : 32;   // lanes per row
  const int rps = 32 / lpr, sub = lane / lpr, q0 = lane % lpr;
  const int stride = 8 * rps;                               // rows per CTA step
  KAcc<R> part[NO2][2];
  for (int sb = l0 + warp * rps + sub; sb < l1; sb += stride * FOLD) {
    cx<R> pp[NO2][2];
#pragma unroll
    for (int p = 0; p < NO2; ++p) pp[p][0] = pp[p][1] = cx<R>(0);
#pragma unroll
    for (int jj = 0; jj < FOLD; ++jj) {
      const int l = sb + stride * jj;
      if (l < l1) {
        cx<R> v[NO];
#pragma unroll
        for (int i = 0; i < NO; ++i) v[i] = vf(l, i);
#pragma unroll
        for (int p = 0; p < NO2; ++p) {
          const S* fr = F[p] + (long long)(l - base) * d.rmax;
          const cx<R> vp = v[ROWS ? p / NO : p % NO];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int q = q0 + lpr * u;
            if (q < rk[p]) {
              const cx<R> f = ROWS ? ldr<R>(fr + q) : ldr<R>(fr + q).conj();
              pp[p][u] = cfma(vp, f, pp[p][u]);
            }
          }
        }
      }
    }
#pragma unroll
    for (int p = 0; p < NO2; ++p) {
      part[p][0].add(pp[p][0]);
      part[p][1].add(pp[p][1]);
    }
  }
#pragma unroll
  for (int p = 0; p < NO2; ++p)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const cff r = kacc_lanes(part[p][u], lpr, 32);
      const int q = q0 + lpr * u;
      if (sub == 0 && q < 64) red[(warp * NO2 + p) * 64 + q] = cff_val(r);
    }
  __syncthreads();
  for (int e = tid; e < NO2 * d.rmax; e += blockDim.x) {
    const int p = e / d.rmax, q = e % d.rmax;
    int rkp = 0;
#pragma unroll
    for (int pp2 = 0; pp2 < NO2; ++pp2)
      if (pp2 == p) rkp = rk[pp2];
    zd acc = zd();
    if (q < rkp)   // entries q >= the pair's rank are not written by every warp
      for (int w2 = 0; w2 < 8; ++w2) acc += red[(w2 * NO2 + p) * 64 + q];
    st(Pj<NO>(d, n, slot, lv, p) + q, q < rkp ? acc * Sp<NO>(d, 2, n, blk, p)[q] : zd());
  }
  __syncthreads();
}

// Sum over q < rk of P[q] * F[q] (or P[q] * conj(F[q])): the far field of one
// compressed block at one row or column, P its projection vector staged in
// shared memory, F the block's factor row in global memory.  Four threads
// share an output (q = sl, sl + 4, ...) and each keeps eight loads of F in
// flight, so the row streams instead of waiting on one load per term.
template <typename R, typename S, bool CONJ>
__device__ __forceinline__ cx<R> lr_dot4(const cx<R>* P, const S* F, int rk, int sl) {
  cx<R> acc = cx<R>(0);
  for (int q0 = sl; q0 < rk; q0 += 32) {
    cx<R> f[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int q = q0 + 4 * u;
      f[u] = q < rk ? ldr<R>(F + q) : cx<R>(0);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) acc = cfma(P[q0 + 4 * u < rk ? q0 + 4 * u : 0], CONJ ? f[u].conj() : f[u], acc);
  }
  return acc;
}

}  // namespace

// ---------------------------------------------------------------------------
// Retarded row, Eq. KBER: unknown y(t') = G^R(T, t') (row irow), solved for
// t' = T-1 .. 0; the start block t' >= T-k is solved together.
// ---------------------------------------------------------------------------
template <int NO, typename S>
__global__ void __launch_bounds__(256, (NO <= 2) ? 2 : 1) k_ret2(Dev d, int T, int staged) {
  constexpr int NO2 = NO * NO;
  using R = typename Bulk<S>::R;
  const int n = blockIdx.y, irow = blockIdx.x;
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = d.k, c = d.cdir, L = d.L;
  const double h = d.h;
  const DevW& W = d.w;
  __shared__ zd sB[10 * NO];     // right-hand side of the head
  __shared__ zd FB[64][NO];
  __shared__ zd pbuf[8][128];
  __shared__ zd Fs[CK][NO];
  __shared__ zd Fb[CK][NO];      // the BDF part of Fs (rows at the chunk edge; zero elsewhere)
  __shared__ zd Old[CK][NO];     // the chunk's previous iterate (convergence measure)
  __shared__ zf Ff[CK][NO];      // complex64 form: the far field (Fs - Fb) rounded to complex64
  __shared__ cff FbF[CK][NO];    // complex64 form: Fb in float-float
  __shared__ double serr;
  extern __shared__ __align__(16) zd ctile[];  // for each chunk its staged inverse (N_o <= 2);
                                 // at leaf entry (staged != 0) the block projections
                                 // [maxl][NO2][rmax]
  __shared__ __align__(8) uint64_t cbar;   // completion of the inverse's bulk copy
  __shared__ int s_stage;                  // 0 once a wait for a copy has timed out
  uint32_t cphase = 0;
  if (tid == 0) {
    serr = 0.0;
    s_stage = 1;
    if (kInvStage<NO, S>) mbar_init(&cbar);
  }
  // The row being solved lives in FP64 during the sweep (in the complex64
  // storage form a separate buffer), so the point-to-point recursion of the
  // sweep (BDF terms, point solves) does not accumulate storage rounding.
  // yp: the FP64 row; sp: its storage, written at the same time (rounded in
  // the complex64 form), which the FP32 bulk sums read; it holds the previous
  // iterate until an element is overwritten (the convergence measure).
  S* rowp = el<NO, S>(d.GR, d, n, T, 0);
  Y* rowy = Row64<NO, S>::get(d, n, 0, T, rowp);
  auto yp = [&](int tp) { return rowy + (long long)tp * NO2 + irow * NO; };
  auto sp = [&](int tp) { return rowp + (long long)tp * NO2 + irow * NO; };
  double myerr = 0.0;
  // ---- the head: points T-s, s = 1..hs, and y(T) = -i.  Its right-hand side
  // is row T of Sigma^R (and the derivative's y(T) term) alone; 8 threads per
  // element of the product with the head's inverse ----
  const int hs = min(2 * k, T), nh = hs * NO;
  for (int e = tid; e < nh; e += blockDim.x) {
    const int s = e / NO + 1, j = e % NO;
    zd cc = ld(el<NO, S>(d.SR, d, n, T, T - s) + irow * NO + j) * (-h * (s <= k ? W.I0[s][0] : rule_w(W, s, 0)));
    if (s <= k && irow == j) cc += zd(0, W.D[s][0] / h);
    sB[e] = zd(0, 1) * cc;
  }
  __syncthreads();
  {
    const double2* Hi = d.hinv + (long long)n * (4 * k * k * NO2);
    for (int o8 = tid; o8 < nh * 8; o8 += blockDim.x) {
      const int o = o8 >> 3, sl = o8 & 7, s = o / NO + 1, j = o % NO;
      const int nb = max(s, min(k, hs)) * NO;   // the inverse is lower triangular below the start block
      zd y = zd();
      for (int b = sl; b < nb; b += 8) y = cfma(ld(Hi + (long long)o * nh + b), sB[b], y);
      const unsigned grp = 0xffu << (lane & 24);
#pragma unroll
      for (int off = 1; off < 8; off <<= 1)
        y += zd(__shfl_xor_sync(grp, y.re, off), __shfl_xor_sync(grp, y.im, off));
      if (sl == 0) {
        myerr = fmax(myerr, (y - ld(sp(T - s) + j)).abs2());
        st(yp(T - s) + j, y);
        if constexpr (Row64<NO, S>::separate) st(sp(T - s) + j, y);
      }
    }
  }
  if (tid < NO) {
    const zd v = (tid == irow) ? zd(0, -1) : zd();
    myerr = fmax(myerr, (ld(sp(T) + tid) - v).abs2());
    st(yp(T) + tid, v);
    if constexpr (Row64<NO, S>::separate) st(sp(T) + tid, v);
  }
  __syncthreads();
  const int top = T - 2 * k - 1;   // the highest point of the chunks (none while T <= 2k)
  for (int cc = top >= 0 ? top / CK : -1; cc >= 0; --cc) {
    const int a = cc * CK, b = min(a + CK, top + 1), cn = b - a;
    const bool comp = (c > 0 && b <= c);
    const int jl = comp ? a / L : 0, A = jl * L, E = comp ? (jl + 1) * L : 0;
    if (comp && (b == E || b == top + 1)) {   // (the top chunk may end inside its leaf)
      // Entering leaf jl from above.  (1) projections pi_B = sum_s y(s) U_B(s,:) S_B
      // of the blocks whose columns end at E, rows summed in 4 slices.
      for (int lv = 0; lv < d.maxl; ++lv) {
        const int blk = d.colblk[jl * d.maxl + lv];
        if (blk < 0 || d.b_c1[blk] != E) continue;
        const int r0 = d.b_r0[blk], rl = min(d.b_r1[blk], c);
        if constexpr (kStage<NO> && Row64<NO, S>::separate) {   // complex64 form: all pairs in one
          if (d.rmax <= 64) {                                     // pass (ctile is free here)
            proj_block<NO, S, true>(d, n, blk, lv, irow, r0, rl,
                                    [&](int s2, int m) { return ldr<R>(sp(s2) + m); }, ctile);
            continue;
          }
        }
        for (int p = 0; p < NO2; ++p) {
          const int m = p / NO;
          const int rk = *Rk<NO>(d, 2, n, blk, p);
          const S* U = Up<NO, S>(d, 2, n, blk, p);
          KAcc<R> part[4];
          for (int s0 = r0 + warp; s0 < rl; s0 += 8 * FOLD) {  // warps over rows, lanes over rank
            cx<R> pp[4] = {cx<R>(0), cx<R>(0), cx<R>(0), cx<R>(0)};
#pragma unroll
            for (int jj = 0; jj < FOLD; ++jj) {
              const int s2 = s0 + 8 * jj;
              if (s2 < rl) {
                const cx<R> yv = ldr<R>(sp(s2) + m);
                const S* ur = U + (long long)(s2 - r0) * d.rmax;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const int q = lane + 32 * u;
                  if (q < rk) pp[u] = cfma(yv, ldr<R>(ur + q), pp[u]);
                }
              }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) part[u].add(pp[u]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) pbuf[warp][lane + 32 * u] = part[u].get();
          __syncthreads();
          if (tid < d.rmax) {
            zd acc = zd();
            for (int w2 = 0; w2 < 8; ++w2) acc += pbuf[w2][tid];
            st(Pj<NO>(d, n, irow, lv, p) + tid, tid < rk ? acc * Sp<NO>(d, 2, n, blk, p)[tid] : zd());
          }
          __syncthreads();
        }
      }
      __syncthreads();
      // projections of every block over this leaf's columns, staged in shared
      // memory for the far-field loop below (the buffer of the chunk
      // inverses, whose copies are issued only after it)
      cx<R>* Ps = reinterpret_cast<cx<R>*>(ctile);
      if (staged) {
        const int per = NO2 * d.rmax;
        for (int e = tid; e < d.maxl * per; e += blockDim.x) {
          const int lv = e / per, p = (e / d.rmax) % NO2, q = e % d.rmax;
          const int blk = d.colblk[jl * d.maxl + lv];
          Ps[e] = (blk >= 0 && d.b_r0[blk] < c) ? ldr<R>(Pj<NO>(d, n, irow, lv, p) + q) : cx<R>(0);
        }
        __syncthreads();
      }
      // (2) for every column of the leaf: uncompressed rows s in [c, T], the
      // blocks below the leaf (weight 1) and the near-diagonal corrections;
      // 4 threads per column.
      {
        const int col = tid >> 2, sl = tid & 3;
        zd acc[NO];
#pragma unroll
        for (int j = 0; j < NO; ++j) acc[j] = zd();
        KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
        const int tp = A + col;
        if (col < L) {
          for (int s0 = c + sl; s0 <= T; s0 += 4 * FOLD) {
            cx<R> pa[NO];
#pragma unroll
            for (int j = 0; j < NO; ++j) pa[j] = cx<R>(0);
#pragma unroll
            for (int jj = 0; jj < FOLD; ++jj) {
              const int s2 = s0 + 4 * jj;
              if (s2 <= T) {
                const R ws = rule_wr<R>(W, T - tp, T - s2);
                const S* yl = sp(s2);
                const S* sr = el<NO, S>(d.SR, d, n, s2, tp);
#pragma unroll
                for (int m = 0; m < NO; ++m) {
                  const cx<R> ym = ldr<R>(yl + m) * ws;
#pragma unroll
                  for (int j = 0; j < NO; ++j) pa[j] = cfma(ym, ldr<R>(sr + m * NO + j), pa[j]);
                }
              }
            }
#pragma unroll
            for (int j = 0; j < NO; ++j) ka[j].add(pa[j]);
          }
          for (int lv = 0; lv < d.maxl; ++lv) {
            const int blk = d.colblk[jl * d.maxl + lv];
            if (blk < 0 || d.b_r0[blk] >= c) continue;
            const int c0 = d.b_c0[blk];
#pragma unroll
            for (int p = 0; p < NO2; ++p) {
              const int j = p % NO;
              const int rk = *Rk<NO>(d, 2, n, blk, p);
              const S* V = Vp<NO, S>(d, 2, n, blk, p) + (long long)(tp - c0) * d.rmax;
              cx<R> pb = cx<R>(0);
              if (staged) {
                pb = lr_dot4<R, S, true>(Ps + (lv * NO2 + p) * d.rmax, V, rk, sl);
              } else {
                const double2* P = Pj<NO>(d, n, irow, lv, p);
                for (int q = sl; q < rk; q += 4) pb = cfma(ldr<R>(P + q), ldr<R>(V + q).conj(), pb);
              }
              ka[j].add(pb);
            }
          }
          for (int s2 = E + sl; s2 <= tp + k && s2 < c; s2 += 4) {
            const double ws = rule_w(W, T - tp, T - s2) - 1.0;
            const S* bd = Bd<NO, S>(d, n, s2, s2 - tp);
            const Y* yl = yp(s2);
#pragma unroll
            for (int m = 0; m < NO; ++m) {
              const zd ym = ld(yl + m) * ws;
#pragma unroll
              for (int j = 0; j < NO; ++j) acc[j] = cfma(ym, ld(bd + m * NO + j), acc[j]);
            }
          }
        }
#pragma unroll
        for (int j = 0; j < NO; ++j) acc[j] += ka[j].get();
#pragma unroll
        for (int j = 0; j < NO; ++j) {
          acc[j] += zd(__shfl_xor_sync(FULL, acc[j].re, 1), __shfl_xor_sync(FULL, acc[j].im, 1));
          acc[j] += zd(__shfl_xor_sync(FULL, acc[j].re, 2), __shfl_xor_sync(FULL, acc[j].im, 2));
        }
        if (sl == 0 && col < L)
#pragma unroll
          for (int j = 0; j < NO; ++j) FB[col][j] = acc[j];
      }
      __syncthreads();
    }
    // the inverse of this chunk into shared memory, overlapping the far field
    const bool stage_now = kInvStage<NO, S> && s_stage;
    if (stage_now && tid == 0) bulk_g2s(ctile, Cinv<NO>(d, n, cc, 0), kInvStage<NO, S>, &cbar);
    // ---- far field of the chunk: rows s >= b not covered above; 8 threads per column ----
    {
      const int col = tid >> 3, sl = tid & 7;
      const int tp = a + col;
      zd acc[NO];
#pragma unroll
      for (int j = 0; j < NO; ++j) acc[j] = zd();
        KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
      if (col < cn) {
        const int s_end = comp ? E : T + 1;   // compressed: the rest of the leaf; else every later row
        for (int s0 = b + sl; s0 < s_end; s0 += 8 * FOLD) {
          cx<R> pa[NO];
#pragma unroll
          for (int j = 0; j < NO; ++j) pa[j] = cx<R>(0);
#pragma unroll
          for (int jj = 0; jj < FOLD; ++jj) {
            const int s2 = s0 + 8 * jj;
            if (s2 < s_end) {
              const R ws = rule_wr<R>(W, T - tp, T - s2);
              const S* yl = sp(s2);
              const S* sr = comp ? Lf<NO, S>(d, 2, n, jl, s2, tp) : el<NO, S>(d.SR, d, n, s2, tp);
#pragma unroll
              for (int m = 0; m < NO; ++m) {
                const cx<R> ym = ldr<R>(yl + m) * ws;
#pragma unroll
                for (int j = 0; j < NO; ++j) pa[j] = cfma(ym, ldr<R>(sr + m * NO + j), pa[j]);
              }
            }
          }
#pragma unroll
          for (int j = 0; j < NO; ++j) ka[j].add(pa[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < NO; ++j) {
        const auto r = reduce8(ka[j]);
        if (sl == 0) acc[j] = val_of(r);
      }
      if (sl == 0 && col < cn) {
        zd F[NO];
        zd Fbd[NO];
#pragma unroll
        for (int j = 0; j < NO; ++j) {
          F[j] = (acc[j] + (comp ? FB[tp - A][j] : zd())) * h;
          Fbd[j] = zd();
        }
        for (int jj = 1; jj <= k; ++jj) {  // BDF terms reaching above the chunk: (-i a_j / h) y(s2)
          const int s2 = tp + jj;
          if (s2 < b) continue;
          const double cj = W.ah[jj];
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            const zd y = ld(yp(s2) + m);
            Fbd[m] = zd(fma(cj, y.im, Fbd[m].re), fma(-cj, y.re, Fbd[m].im));
          }
        }
#pragma unroll
        for (int j = 0; j < NO; ++j) {
          Fs[col][j] = F[j] + Fbd[j];
          Fb[col][j] = Fbd[j];
          Ff[col][j] = zf((float)F[j].re, (float)F[j].im);
          FbF[col][j] = cff_of(Fbd[j]);
        }
      }
      if (sl == 1 && col < cn)
#pragma unroll
        for (int j = 0; j < NO; ++j) Old[col][j] = ld(sp(tp) + j);
    }
    __syncthreads();
    {
      // y = F C^-1 (row vector times the chunk's inverse, lower triangular),
      // 8 threads per output element
      const double2* Mi = Cinv<NO>(d, n, cc, 0);
      bool smem_inv = false;
      if (stage_now) {
        smem_inv = mbar_wait(&cbar, cphase, kCopyWaitPolls);
        cphase ^= 1u;
        if (!smem_inv) {
          s_stage = 0;
          atomicAdd(d.status + 2, 1);
        }
      }
      const double2* Mg = smem_inv ? reinterpret_cast<const double2*>(ctile) : Mi;
      constexpr int LD = CK * NO;
      for (int o8 = tid; o8 < CK * NO * 8; o8 += blockDim.x) {
        const int o = o8 >> 3, sl = o8 & 7, ti = o / NO, j = o % NO;
        zd sacc = zd();
        if constexpr (Row64<NO, S>::separate) {
          // complex64 form: far field x hi in FP32, the k edge rows x (hi + lo)
          // in float-float, reduced over the 8 lanes in float-float
          const float2* Mh = reinterpret_cast<const float2*>(Mg);
          const float2* Ml = Mh + LD * LD;
          zf s32 = zf(0);
          for (int si = (ti & ~7) + sl; si < cn; si += 8)
#pragma unroll
            for (int m = 0; m < NO; ++m)
              s32 = cfma(Ff[si][m], ldr<float>(Mh + (long long)(si * NO + m) * LD + ti * NO + j), s32);
          cff sf = cff_of(s32);
          for (int si = max(cn - k, 0) + sl; si < cn; si += 8)
#pragma unroll
            for (int m = 0; m < NO; ++m) {
              const long long e = (long long)(si * NO + m) * LD + ti * NO + j;
              const float2 hv = Mh[e], lv = Ml[e];
              sf = cff_add(sf, cff_mul(FbF[si][m], cff{{hv.x, lv.x}, {hv.y, lv.y}}));
            }
#pragma unroll
          for (int off = 1; off < 8; off <<= 1) sf = cff_add(sf, cff_shfl_xor(sf, off));
          if (sl == 0) sacc = cff_val(sf);
        } else {
          for (int si = (ti & ~7) + sl; si < cn; si += 8)
#pragma unroll
            for (int m = 0; m < NO; ++m) sacc = cfma(Fs[si][m], ld(Mg + (long long)(si * NO + m) * LD + ti * NO + j), sacc);
#pragma unroll
          for (int off = 1; off < 8; off <<= 1)
            sacc += zd(__shfl_xor_sync(FULL, sacc.re, off), __shfl_xor_sync(FULL, sacc.im, off));
        }
        if (sl == 0 && ti < cn) {
          myerr = fmax(myerr, (sacc - Old[ti][j]).abs2());
          st(yp(a + ti) + j, sacc);
          if constexpr (Row64<NO, S>::separate) st(sp(a + ti) + j, sacc);
        }
      }
    }
    __syncthreads();
  }
  myerr = sqrt(warp_max(myerr));
  if (lane == 0 && myerr > 0) atomic_max_nonneg(&serr, myerr);
  __syncthreads();
  if (tid == 0) atomic_max_nonneg(d.err + n, serr);
  // after a timed-out wait, a copy may still be in flight into this CTA's
  // shared memory: wait for it (bounded) before the CTA exits
  if (kInvStage<NO, S> && tid == 0 && !s_stage) mbar_wait(&cbar, cphase ^ 1u, kCopyWaitPolls);
}

// ---------------------------------------------------------------------------
// Lesser column, Eq. KBEL: unknown x(t) = G^<(t, T) (column jc), t = 0..T.
// ---------------------------------------------------------------------------
template <int NO, typename S>
__global__ void __launch_bounds__(256, (NO <= 2) ? 2 : 1) k_les2(Dev d, int T, int staged) {
  constexpr int NO2 = NO * NO;
  using R = typename Bulk<S>::R;
  const int n = blockIdx.y, jc = blockIdx.x;
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = d.k, c = d.cdir, L = d.L;
  const double h = d.h;
  const DevW& W = d.w;
  __shared__ zd FB[64][NO];
  __shared__ zd pbuf[8][128];
  __shared__ zd Fs[CK][NO];
  __shared__ zd Fb[CK][NO];      // the BDF part of Fs (rows at the chunk edge; zero elsewhere)
  __shared__ zd Old[CK][NO];     // the chunk's previous iterate (convergence measure)
  __shared__ zf Ff[CK][NO];      // complex64 form: the far field (Fs - Fb) rounded to complex64
  __shared__ cff FbF[CK][NO];    // complex64 form: Fb in float-float
  __shared__ double serr;
  extern __shared__ __align__(16) zd ctile[];  // for each chunk its staged inverse (N_o <= 2);
                                 // at leaf entry (staged != 0) the block projections
                                 // [maxl][NO2][rmax]
  __shared__ __align__(8) uint64_t cbar;   // completion of the inverse's bulk copy
  __shared__ int s_stage;                  // 0 once a wait for a copy has timed out
  uint32_t cphase = 0;
  if (tid == 0) {
    serr = 0.0;
    s_stage = 1;
    if (kInvStage<NO, S>) mbar_init(&cbar);
  }
  // FP64 column during the sweep (see k_ret2); xp: as solved, sp: storage
  S* colp = el<NO, S>(d.GL, d, n, T, 0);
  Y* coly = Row64<NO, S>::get(d, n, 1, T, colp);
  auto xp = [&](int t) { return coly + (long long)t * NO2; };  // element [m*NO + jc]
  auto sp = [&](int t) { return colp + (long long)t * NO2; };
  const double2* qs = d.qsrc + (long long)n * d.nt * NO2;
  double myerr = 0.0;
  const int last = (d.rho_mode == 1) ? T - 1 : T;
  if (warp == 0 && lane < NO) {  // x(0) = -[G^tv(T, 0+)]^dagger
    const int m = lane;
    zd v = ld(d.x0 + (long long)n * NO2 + m * NO + jc);
    myerr = fmax(myerr, (v - ld(sp(0) + m * NO + jc)).abs2());
    st(xp(0) + m * NO + jc, v);
    if constexpr (Row64<NO, S>::separate) st(sp(0) + m * NO + jc, v);
  }
  __syncthreads();
  for (int cc = 0; cc * CK <= last; ++cc) {
    const int a = (cc == 0) ? 1 : cc * CK, b = min((cc + 1) * CK, last + 1), cn = b - a;
    if (cn <= 0) break;
    const bool comp = (c > 0 && b <= c);
    const int jl = comp ? a / L : 0, A = jl * L;
    if (comp && cc * CK == A) {
      // Entering leaf jl.  (1) rho_B = S_B sum_l w_l conj(V_B(l,:)) x(l) for the
      // blocks whose rows start at A (w_l = omega_l for l <= k, else 1).
      for (int lv = 0; lv < d.maxl && jl > 0; ++lv) {
        const int blk = d.rowblk[jl * d.maxl + lv];
        if (blk < 0 || d.b_r0[blk] != A) continue;
        const int c0 = d.b_c0[blk], c1 = d.b_c1[blk];
        if constexpr (kStage<NO> && Row64<NO, S>::separate) {   // complex64 form: all pairs in one
          if (d.rmax <= 64) {                                     // pass (ctile is free here)
            proj_block<NO, S, false>(d, n, blk, lv, jc, c0, c1, [&](int l, int nn) {
              const R wl = (l <= k) ? (R)W.omega[l] : (R)1;
              return ldr<R>(sp(l) + nn * NO + jc) * wl;
            }, ctile);
            continue;
          }
        }
        for (int p = 0; p < NO2; ++p) {
          const int nn = p % NO;
          const int rk = *Rk<NO>(d, 2, n, blk, p);
          const S* V = Vp<NO, S>(d, 2, n, blk, p);
          KAcc<R> part[4];
          for (int l0 = c0 + warp; l0 < c1; l0 += 8 * FOLD) {  // warps over columns, lanes over rank
            cx<R> pp[4] = {cx<R>(0), cx<R>(0), cx<R>(0), cx<R>(0)};
#pragma unroll
            for (int jj = 0; jj < FOLD; ++jj) {
              const int l = l0 + 8 * jj;
              if (l < c1) {
                const R wl = (l <= k) ? (R)W.omega[l] : (R)1;
                const cx<R> xv = ldr<R>(sp(l) + nn * NO + jc) * wl;
                const S* vr = V + (long long)(l - c0) * d.rmax;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const int q = lane + 32 * u;
                  if (q < rk) pp[u] = cfma(ldr<R>(vr + q).conj(), xv, pp[u]);
                }
              }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) part[u].add(pp[u]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) pbuf[warp][lane + 32 * u] = part[u].get();
          __syncthreads();
          if (tid < d.rmax) {
            zd acc = zd();
            for (int w2 = 0; w2 < 8; ++w2) acc += pbuf[w2][tid];
            st(Pj<NO>(d, n, jc, lv, p) + tid, tid < rk ? acc * Sp<NO>(d, 2, n, blk, p)[tid] : zd());
          }
          __syncthreads();
        }
      }
      __syncthreads();
      // projections of every block left of this leaf's rows, staged in shared
      // memory for the loop below (the buffer of the chunk inverses, whose
      // copies are issued only after it)
      cx<R>* Ps = reinterpret_cast<cx<R>*>(ctile);
      if (staged) {
        const int per = NO2 * d.rmax;
        for (int e = tid; e < d.maxl * per; e += blockDim.x) {
          const int lv = e / per, p = (e / d.rmax) % NO2, q = e % d.rmax;
          const int blk = d.rowblk[jl * d.maxl + lv];
          Ps[e] = blk >= 0 ? ldr<R>(Pj<NO>(d, n, jc, lv, p) + q) : cx<R>(0);
        }
        __syncthreads();
      }
      // (2) every row of the leaf: blocks left of it and near-diagonal corrections
      {
        const int row = tid >> 2, sl = tid & 3;
        const int t = A + row;
        zd acc[NO];
#pragma unroll
        for (int m = 0; m < NO; ++m) acc[m] = zd();
        KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
        if (row < L) {
          for (int lv = 0; lv < d.maxl; ++lv) {
            const int blk = d.rowblk[jl * d.maxl + lv];
            if (blk < 0) continue;
            const int r0 = d.b_r0[blk];
#pragma unroll
            for (int p = 0; p < NO2; ++p) {
              const int m = p / NO;
              const int rk = *Rk<NO>(d, 2, n, blk, p);
              const S* U = Up<NO, S>(d, 2, n, blk, p) + (long long)(t - r0) * d.rmax;
              cx<R> pb = cx<R>(0);
              if (staged) {
                pb = lr_dot4<R, S, false>(Ps + (lv * NO2 + p) * d.rmax, U, rk, sl);
              } else {
                const double2* P = Pj<NO>(d, n, jc, lv, p);
                for (int q = sl; q < rk; q += 4) pb = cfma(ldr<R>(U + q), ldr<R>(P + q), pb);
              }
              ka[m].add(pb);
            }
          }
          for (int l = max(t - k, 0) + sl; l < A; l += 4) {
            const double wl = rule_w(W, t, l) - 1.0;
            const S* bd = Bd<NO, S>(d, n, t, t - l);
#pragma unroll
            for (int y = 0; y < NO; ++y) {
              const zd xy = ld(xp(l) + y * NO + jc) * wl;
#pragma unroll
              for (int m = 0; m < NO; ++m) acc[m] = cfma(ld(bd + m * NO + y), xy, acc[m]);
            }
          }
        }
#pragma unroll
        for (int m = 0; m < NO; ++m) acc[m] += ka[m].get();
#pragma unroll
        for (int m = 0; m < NO; ++m) {
          acc[m] += zd(__shfl_xor_sync(FULL, acc[m].re, 1), __shfl_xor_sync(FULL, acc[m].im, 1));
          acc[m] += zd(__shfl_xor_sync(FULL, acc[m].re, 2), __shfl_xor_sync(FULL, acc[m].im, 2));
        }
        if (sl == 0 && row < L)
#pragma unroll
          for (int m = 0; m < NO; ++m) FB[row][m] = acc[m];
      }
      __syncthreads();
    }
    const int fn = min(b, T) - a;   // rows solved with the chunk's inverse; row T, if it is here, follows them
    // the inverse of this chunk into shared memory, overlapping the far field
    const bool stage_now = kInvStage<NO, S> && fn > 0 && s_stage;
    if (stage_now && tid == 0) bulk_g2s(ctile, Cinv<NO>(d, n, cc, 1), kInvStage<NO, S>, &cbar);
    // ---- far field F(t) = q(t) - sum_{l < a} C(t,l) x(l); 8 threads per row ----
    {
      const int row = tid >> 3, sl = tid & 7;
      const int t = a + row;
      zd acc[NO], fbo[NO];   // fbo: this lane's BDF part (only the owner lane's is nonzero)
#pragma unroll
      for (int m = 0; m < NO; ++m) acc[m] = fbo[m] = zd();
        KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
      if (row < cn) {
        if (t <= k) {
          if (sl == 0) {  // start rows: only l = 0 lies left of chunk 0 (a derivative term: kept in Fb)
            zd fb[NO];
#pragma unroll
            for (int m = 0; m < NO; ++m) fb[m] = zd();
            for (int y = 0; y < NO; ++y) {
              const zd xv = ld(xp(0) + y * NO + jc);
#pragma unroll
              for (int m = 0; m < NO; ++m) {
                zd cf = srx_any<NO, S>(d, n, t, 0, m, y) * (-h * W.I0[t][0]);
                if (m == y) cf += zd(0, W.D[t][0] / h);
                fb[m] -= cf * xv;
              }
            }
#pragma unroll
            for (int m = 0; m < NO; ++m) {
              fbo[m] = fb[m];
              Fb[row][m] = fb[m];
            }
          }
        } else {
          const int l0 = comp ? A : 0;
          const S* srow = comp ? nullptr : el<NO, S>(d.SR, d, n, t, 0);
          const R hr = (R)h;
          for (int lb = l0 + sl; lb < a; lb += 8 * FOLD) {
            cx<R> pa[NO];
#pragma unroll
            for (int m = 0; m < NO; ++m) pa[m] = cx<R>(0);
#pragma unroll
            for (int jj = 0; jj < FOLD; ++jj) {
              const int l = lb + 8 * jj;
              if (l < a) {
                const R wl = hr * rule_wr<R>(W, t, l);
                const S* sr = comp ? Lf<NO, S>(d, 2, n, jl, t, l) : srow + (long long)l * NO2;
#pragma unroll
                for (int y = 0; y < NO; ++y) {
                  const cx<R> xy = ldr<R>(sp(l) + y * NO + jc) * wl;
#pragma unroll
                  for (int m = 0; m < NO; ++m) pa[m] = cfma(ldr<R>(sr + m * NO + y), xy, pa[m]);
                }
              }
            }
#pragma unroll
            for (int m = 0; m < NO; ++m) ka[m].add(pa[m]);
          }
          if (sl == 1) {  // BDF terms reaching left of the chunk, kept apart in Fb
            zd fb[NO];
#pragma unroll
            for (int m = 0; m < NO; ++m) fb[m] = zd();
            for (int jj = 1; jj <= k; ++jj) {   // (-i a_j / h) x(t - j)
              if (t - jj >= a) continue;
              const double cj = W.ah[jj];
#pragma unroll
              for (int m = 0; m < NO; ++m) {
                const zd x = ld(xp(t - jj) + m * NO + jc);
                fb[m] = zd(fma(cj, x.im, fb[m].re), fma(-cj, x.re, fb[m].im));
              }
            }
#pragma unroll
            for (int m = 0; m < NO; ++m) {
              fbo[m] = fb[m];
              Fb[row][m] = fb[m];
            }
          }
        }
      }
      // the BDF part from its owner lane (sl 0 for the start rows, else sl 1)
      const int owner = (lane & ~7) | (t <= k ? 0 : 1);
#pragma unroll
      for (int m = 0; m < NO; ++m) {
        const auto r = reduce8(ka[m]);
        const zd fbm(__shfl_sync(FULL, fbo[m].re, owner), __shfl_sync(FULL, fbo[m].im, owner));
        if (sl == 0 && row < cn) {
          const zd far = val_of(r) + (comp && t > k ? FB[t - A][m] * h : zd()) +
                         ld(qs + (long long)t * NO2 + m * NO + jc);
          Fs[row][m] = far + fbm;
          Ff[row][m] = zf((float)far.re, (float)far.im);
          FbF[row][m] = cff_of(fbm);
        }
      }
      (void)acc;
      if (sl == 1 && row < cn)
#pragma unroll
        for (int m = 0; m < NO; ++m) Old[row][m] = ld(sp(t) + m * NO + jc);
    }
    __syncthreads();
    if (fn > 0) {
      const double2* Mi = Cinv<NO>(d, n, cc, 1);
      bool smem_inv = false;
      if (stage_now) {
        smem_inv = mbar_wait(&cbar, cphase, kCopyWaitPolls);
        cphase ^= 1u;
        if (!smem_inv) {
          s_stage = 0;
          atomicAdd(d.status + 2, 1);
        }
      }
      const double2* Mg = smem_inv ? reinterpret_cast<const double2*>(ctile) : Mi;
      constexpr int LD = CK * NO;
      for (int o8 = tid; o8 < CK * NO * 8; o8 += blockDim.x) {
        const int o = o8 >> 3, sl = o8 & 7, ti = o / NO, m = o % NO;
        zd sacc = zd();
        if constexpr (Row64<NO, S>::separate) {
          // complex64 form: far field x hi in FP32, the k edge rows x (hi + lo) in
          // float-float, reduced over the 8 lanes in float-float
          const float2* Mh = reinterpret_cast<const float2*>(Mg);
          const float2* Ml = Mh + LD * LD;
          cff sf = cff_of(zf(0));
          if (ti < fn) {
            zf s32 = zf(0);
            for (int li = sl; li < max(ti + 1, min(k, fn)); li += 8)
#pragma unroll
              for (int y = 0; y < NO; ++y)
                s32 = cfma(ldr<float>(Mh + (long long)(ti * NO + m) * LD + li * NO + y), Ff[li][y], s32);
            sf = cff_of(s32);
            for (int li = sl; li < k && li < fn; li += 8)
#pragma unroll
              for (int y = 0; y < NO; ++y) {
                const long long e = (long long)(ti * NO + m) * LD + li * NO + y;
                const float2 hv = Mh[e], lv = Ml[e];
                sf = cff_add(sf, cff_mul(cff{{hv.x, lv.x}, {hv.y, lv.y}}, FbF[li][y]));
              }
          }
#pragma unroll
          for (int off = 1; off < 8; off <<= 1) sf = cff_add(sf, cff_shfl_xor(sf, off));
          if (sl == 0) sacc = cff_val(sf);
        } else {
          if (ti < fn)
            for (int li = sl; li < max(ti + 1, min(k, fn)); li += 8)
#pragma unroll
              for (int y = 0; y < NO; ++y)
                sacc = cfma(ld(Mg + (long long)(ti * NO + m) * LD + li * NO + y), Fs[li][y], sacc);
#pragma unroll
          for (int off = 1; off < 8; off <<= 1)
            sacc += zd(__shfl_xor_sync(FULL, sacc.re, off), __shfl_xor_sync(FULL, sacc.im, off));
        }
        if (sl == 0 && ti < fn) {
          myerr = fmax(myerr, (sacc - Old[ti][m]).abs2());
          st(xp(a + ti) + m * NO + jc, sacc);
          if constexpr (Row64<NO, S>::separate) st(sp(a + ti) + m * NO + jc, sacc);
        }
      }
    }
    if (fn < cn) {
      // row T (horizontal density matrix): x(T) from the rows of its chunk and
      // the current Sigma^R(T, .), one lane of warp 0 per row
      __syncthreads();
      if (warp == 0) {
        zd f[NO];
#pragma unroll
        for (int m = 0; m < NO; ++m) f[m] = zd();
        if (lane < fn) {
          const int l = a + lane, dd = T - l;
          const double wl = h * rule_w(W, T, l);
          const S* sr = el<NO, S>(d.SR, d, n, T, l);
#pragma unroll
          for (int y = 0; y < NO; ++y) {
            const zd x = ld(xp(l) + y * NO + jc), xw = x * wl;
#pragma unroll
            for (int m = 0; m < NO; ++m) f[m] = cfma(ld(sr + m * NO + y), xw, f[m]);
            if (dd <= k) f[y] += zd(W.ah[dd] * x.im, -W.ah[dd] * x.re);   // (-i a_d / h) x(l)
          }
        }
        warp_sum<NO>(f);
        if (lane == 0) {
          const double wt = h * rule_w(W, T, T);
          const S* sd = el<NO, S>(d.SR, d, n, T, T);
          const double2* ep = epsp<NO>(d, n, T);
          M<NO> Mm;
          zd x[NO];
#pragma unroll
          for (int x2 = 0; x2 < NO; ++x2) {
            f[x2] += Fs[fn][x2];
#pragma unroll
            for (int y = 0; y < NO; ++y)
              Mm.a[x2][y] = (x2 == y ? zd(0, W.a[0] / h) : zd()) - ld(ep + x2 * NO + y) - ld(sd + x2 * NO + y) * wt;
          }
          solve_col<NO>(Mm, f, x);
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            myerr = fmax(myerr, (x[m] - Old[fn][m]).abs2());
            st(xp(T) + m * NO + jc, x[m]);
            if constexpr (Row64<NO, S>::separate) st(sp(T) + m * NO + jc, x[m]);
          }
        }
      }
    }
    __syncthreads();
  }
  myerr = sqrt(warp_max(myerr));
  if (lane == 0 && myerr > 0) atomic_max_nonneg(&serr, myerr);
  __syncthreads();
  if (tid == 0) atomic_max_nonneg(d.err + n, serr);
  // after a timed-out wait, a copy may still be in flight into this CTA's
  // shared memory: wait for it (bounded) before the CTA exits
  if (kInvStage<NO, S> && tid == 0 && !s_stage) mbar_wait(&cbar, cphase ^ 1u, kCopyWaitPolls);
}

// ---------------------------------------------------------------------------
// Inverses of the sweeps' triangular systems, brought up to date once per time
// step (before its first iteration), one CTA per (instance, system):
//   system 0, retarded chunks: points s in [r0, r1).  C[(s,m),(t',j)] =
//     (i/h) a_{s-t'} [0 <= s-t' <= k] delta_mj - delta_{s t'} eps(t')_mj
//     - h w(s-t') Sigma^R(s,t')_mj, w(d) = omega_d (d <= k) else 1;
//   system 1, lesser chunks: rows t in [l0, l1) of E[(t,m),(l,y)] = (i/h)
//     a_{t-l} delta - delta_{tl} eps(t) - h w^(t)_l Sigma^R(t,l); rows t <= k
//     are the start equations with D and I_{0,t,.}, inverted together;
//   system 2, the retarded head of step T: unknowns y(T-s), s = 1..min(2k,T),
//     H[(s,j),(l,m)] = C[l,s]_mj of Eq. KBER: the start block s <= k with D and
//     I_{0,s,.}, then rows with w^(s)_l, s <= 2k.
// Each matrix is block lower triangular (below its start block), so a new row
// s of an inverse M follows from the rows before it,
//   M(s, c) = -A(s,s)^-1 sum_{c <= u < s} A(s, u) M(u, c),  M(s,s) = A(s,s)^-1,
// and a completed chunk is never touched again.  All FP64; the complex64 form
// keeps the growing chunk's rows in FP64 (cinv_ws) and writes their hi + lo
// pair into the chunk's slot.
// One launch per step, bound by the chain of the head's small inverse: 36 us at
// N_o = 1, 88 us at N_o = 2, 270 us at N_o = 4 (16 instances).  A Gauss-Jordan
// of the whole chunk every 32 steps took 0.2 ms (N_o = 1) to 7 ms (N_o = 4) and
// left the growing chunks without an inverse.
// ---------------------------------------------------------------------------
// In-place Gauss-Jordan inverse with partial pivoting of the n x n matrix A
// (leading dimension ld, shared memory, n <= 20); every thread calls it.
__device__ void gj_inverse(int n, zd* A, int ld) {
  __shared__ zd col[20];
  __shared__ int prow[20];
  const int tid = threadIdx.x;
  for (int c = 0; c < n; ++c) {
    if (tid < 32) {
      double v = (tid >= c && tid < n) ? A[tid * ld + c].abs2() : -1.0;
      int p = tid;
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        const double v2 = __shfl_xor_sync(FULL, v, off);
        const int p2 = __shfl_xor_sync(FULL, p, off);
        if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
      }
      if (p != c && tid < n) { const zd t = A[c * ld + tid]; A[c * ld + tid] = A[p * ld + tid]; A[p * ld + tid] = t; }
      if (tid == 0) prow[c] = p;
      __syncwarp();
      if (tid < n) col[tid] = tid == c ? cdiv(zd(1.0), A[c * ld + c]) : A[tid * ld + c];
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

// Row s of an inverse: Mi(s, .) from the coefficients crow[u][m][p] = A(s,u)_mp,
// u = 0..s (diagonal block last), and the rows u < s of Mi (leading dimension
// ld_m, columns u N_o + p; the first sb rows are a full start block).  out(m,
// col, value) stores.  Every thread calls it.
template <int NO, typename P, typename OUT>
__device__ void append_row(int s, int sb, const zd* crow, const P* Mi, int ld_m, zd* part, zd* dinv, OUT out) {
  constexpr int NO2 = NO * NO, SL = NO == 1 ? 8 : NO == 2 ? 2 : 1;   // slices of the sum over u
  const int tid = threadIdx.x, nc = s * NO, tps = blockDim.x / SL, slice = tid / tps;
  if (tid == 0) {
    M<NO> D;
#pragma unroll
    for (int q = 0; q < NO2; ++q) D.a[q / NO][q % NO] = crow[s * NO2 + q];
    const M<NO> I = solve_left<NO>(D, M<NO>::eye(zd(1.0)));
#pragma unroll
    for (int q = 0; q < NO2; ++q) dinv[q] = I.a[q / NO][q % NO];
  }
  for (int e = tid % tps; e < NO * nc; e += tps) {
    const int m = e / nc, col = e % nc;
    zd acc = zd();
    for (int u = (col < sb * NO ? 0 : col / NO) + slice; u < s; u += SL)
#pragma unroll
      for (int p = 0; p < NO; ++p) acc = cfma(crow[u * NO2 + m * NO + p], ldr<double>(Mi + (long long)(u * NO + p) * ld_m + col), acc);
    part[slice * (NO * nc) + e] = acc;
  }
  __syncthreads();
  for (int e = tid; e < NO * (nc + NO); e += blockDim.x) {
    const int m = e / (nc + NO), col = e % (nc + NO);
    zd v = zd();
    if (col >= nc) {
      v = dinv[m * NO + col - nc];
    } else {
#pragma unroll
      for (int q = 0; q < NO; ++q) {
        zd w = zd();
#pragma unroll
        for (int sl = 0; sl < SL; ++sl) w += part[sl * (NO * nc) + q * nc + col];
        v -= dinv[m * NO + q] * w;
      }
    }
    out(m, col, v);
  }
  __syncthreads();
}

template <int NO, typename S>
__global__ void __launch_bounds__(256) k_inv_rows(Dev d, int T, int r0, int r1, int l0, int l1) {
  constexpr int NO2 = NO * NO, LD = CK * NO, NH = 10 * NO;
  const int n = blockIdx.y, sys = blockIdx.x, tid = threadIdx.x;
  if (T > d.last[n]) return;   // the instance has ended
  const int k = d.k;
  const double h = d.h;
  const DevW& W = d.w;
  __shared__ zd part[NO <= 2 ? 256 : CK * NO2];
  __shared__ zd crow[CK * NO2];
  __shared__ zd dinv[NO2];
  __shared__ zd Hm[NH * NH];       // the head, or the lesser start block
  if (sys == 2) {
    const int hs = min(2 * k, T), kb = min(k, hs), nh = hs * NO, nb = kb * NO;
    auto coef = [&](int s, int l, int j, int m) {   // H[(s,j),(l,m)]
      const double wl = s <= k ? W.I0[s][l] : rule_w(W, s, l);
      zd v = srx_any<NO, S>(d, n, T - l, T - s, m, j) * (-h * wl);
      if (m == j) v += zd(0, s <= k ? W.D[s][l] / h : s - l <= k ? W.ah[s - l] : 0.0);
      if (l == s) v -= ld(epsp<NO>(d, n, T - s) + m * NO + j);
      return v;
    };
    for (int e = tid; e < nh * nh; e += blockDim.x) {
      const int row = e / nh, col = e % nh;
      Hm[e] = (row < nb && col < nb) ? coef(row / NO + 1, col / NO + 1, row % NO, col % NO) : zd();
    }
    __syncthreads();
    gj_inverse(nb, Hm, nh);
    for (int s = kb; s < hs; ++s) {
      for (int e = tid; e < (s + 1) * NO2; e += blockDim.x)
        crow[e] = coef(s + 1, e / NO2 + 1, (e % NO2) / NO, e % NO);
      __syncthreads();
      append_row<NO>(s, kb, crow, Hm, nh, part, dinv, [&](int m, int col, const zd& v) { Hm[(s * NO + m) * nh + col] = v; });
    }
    double2* Hi = d.hinv + (long long)n * (4 * k * k * NO2);
    for (int e = tid; e < nh * nh; e += blockDim.x) st(Hi + e, Hm[e]);
    return;
  }
  // chunk rows (systems 0 and 1)
  constexpr bool f64 = sizeof(S) == sizeof(double2);
  double2* wsm = d.cinv_ws + ((long long)n * 2 + sys) * (LD * LD);
  const int q0 = sys == 0 ? r0 : l0, q1 = sys == 0 ? r1 : l1;
  for (int s = q0; s < q1; ++s) {
    const int cc = s / CK, a = (sys == 1 && cc == 0) ? 1 : cc * CK;
    double2* slot = Cinv<NO>(d, n, cc, sys);
    double2* Mi = f64 ? slot : wsm;
    auto put = [&](int row, int col, const zd& v) {
      st(Mi + (long long)row * LD + col, v);
      if constexpr (!f64) {   // complex64 form: hi and lo matrices (see Cinv)
        float2* Oh = reinterpret_cast<float2*>(slot);
        const float2 hi = make_float2((float)v.re, (float)v.im);
        Oh[(long long)row * LD + col] = hi;
        Oh[(long long)LD * LD + (long long)row * LD + col] =
            make_float2((float)(v.re - (double)hi.x), (float)(v.im - (double)hi.y));
      }
    };
    if (sys == 1 && s == 1) {   // the lesser start block, rows 1..k together
      const int nb = k * NO;
      for (int e = tid; e < nb * nb; e += blockDim.x) {
        const int row = e / nb, col = e % nb;
        const int t = row / NO + 1, m = row % NO, l = col / NO + 1, y = col % NO;
        zd v = srx_any<NO, S>(d, n, t, l, m, y) * (-h * W.I0[t][l]);
        if (m == y) v += zd(0, W.D[t][l] / h);
        if (l == t) v -= ld(epsp<NO>(d, n, t) + m * NO + y);
        Hm[e] = v;
      }
      __syncthreads();
      gj_inverse(nb, Hm, nb);
      for (int e = tid; e < nb * nb; e += blockDim.x) put(e / nb, e % nb, Hm[e]);
      __syncthreads();
      s = k;
      continue;
    }
    const int ri = s - a;
    for (int e = tid; e < (ri + 1) * NO2; e += blockDim.x) {
      const int u = a + e / NO2, m = (e % NO2) / NO, p = e % NO, dd = s - u;
      const double wl = sys == 1 ? rule_w(W, s, u) : dd <= k ? W.omega[dd] : 1.0;
      zd v = sr_any<NO, S>(d, n, s, u, m, p) * (-h * wl);
      if (dd <= k && m == p) v += zd(0, W.ah[dd]);
      if (dd == 0) v -= ld(epsp<NO>(d, n, s) + m * NO + p);
      crow[e] = v;
    }
    __syncthreads();
    const int sb = sys == 1 && cc == 0 ? k : 0;   // rows of the start block in this chunk: full columns
    append_row<NO>(ri, sb, crow, Mi, LD, part, dinv, [&](int m, int col, const zd& v) { put(ri * NO + m, col, v); });
  }
}

#define HK_DISPATCH(NOV, CALL)                                                  \
  switch ((NOV) * 2 + d.prec) {                                                 \
    case 2: { constexpr int NO = 1; using S = double2; CALL; break; }           \
    case 3: { constexpr int NO = 1; using S = float2; CALL; break; }            \
    case 4: { constexpr int NO = 2; using S = double2; CALL; break; }           \
    case 5: { constexpr int NO = 2; using S = float2; CALL; break; }            \
    case 6: { constexpr int NO = 3; using S = double2; CALL; break; }           \
    case 7: { constexpr int NO = 3; using S = float2; CALL; break; }            \
    case 8: { constexpr int NO = 4; using S = double2; CALL; break; }           \
    case 9: { constexpr int NO = 4; using S = float2; CALL; break; }            \
    default: return cudaErrorInvalidValue;                                      \
  }

// Static plus dynamic shared memory above the 48 KB default needs an opt-in
// per kernel (the static arrays of the sweeps take 24-31 KB).
template <typename K>
static cudaError_t allow_smem(K kern, size_t bytes) {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, kern);
  if (e != cudaSuccess) return e;
  if (a.sharedSizeBytes + bytes <= 48 * 1024) return cudaSuccess;
  if (a.sharedSizeBytes + bytes > 227 * 1024) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
// Dynamic shared memory of a sweep: the staged chunk inverse (N_o <= 2)
// and, in the compressed form, the staged block projections, which share one
// buffer; staging is used when it fits in 64 KiB.
template <int NO, typename S>
static size_t sweep_smem(const Dev& d, int* staged) {
  using R = typename Bulk<S>::R;
  const size_t ps = d.ring ? (size_t)d.maxl * NO * NO * d.rmax * sizeof(cx<R>) : 0;
  *staged = (d.ring && ps <= 65536) ? 1 : 0;
  return std::max(kStageBytes<NO>, *staged ? ps : (size_t)0);
}
template <int NO, typename S>
static cudaError_t sweep_ret(const Dev& d, int T, cudaStream_t s) {
  int staged = 0;
  const size_t bytes = sweep_smem<NO, S>(d, &staged);
  cudaError_t e = allow_smem(k_ret2<NO, S>, bytes);
  if (e != cudaSuccess) return e;
  k_ret2<NO, S><<<dim3(d.no, d.n_inst), 256, bytes, s>>>(d, T, staged);
  return cudaGetLastError();
}
template <int NO, typename S>
static cudaError_t sweep_les(const Dev& d, int T, cudaStream_t s) {
  int staged = 0;
  const size_t bytes = sweep_smem<NO, S>(d, &staged);
  cudaError_t e = allow_smem(k_les2<NO, S>, bytes);
  if (e != cudaSuccess) return e;
  k_les2<NO, S><<<dim3(d.no, d.n_inst), 256, bytes, s>>>(d, T, staged);
  return cudaGetLastError();
}
cudaError_t launch_ret_h(const Dev& d, int T, cudaStream_t s) {
  HK_DISPATCH(d.no, return (sweep_ret<NO, S>(d, T, s)));
  return cudaSuccess;
}
cudaError_t launch_les_h(const Dev& d, int T, cudaStream_t s) {
  HK_DISPATCH(d.no, return (sweep_les<NO, S>(d, T, s)));
  return cudaSuccess;
}
cudaError_t launch_inv_rows(const Dev& d, int T, int r0, int r1, int l0, int l1, cudaStream_t s) {
  HK_DISPATCH(d.no, (k_inv_rows<NO, S><<<dim3(3, d.n_inst), 256, 0, s>>>(d, T, r0, r1, l0, l1)));
  return cudaGetLastError();
}

}  // namespace hk
