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
#include <algorithm>
#include <type_traits>

#include "bulk_copy.cuh"
#include "hodlr_util.cuh"
#include "mixed_nodes.cuh"

namespace hk {

namespace {

constexpr int CK = 32;   // chunk length
using Y = double2;       // element type of the row / column being solved
template <int NO> constexpr bool kStage = NO <= 2;   // chunk inverses staged in shared memory
// Bytes of a chunk inverse that are staged in shared memory by a bulk copy
// issued before the chunk's far field, so the copy overlaps it: the whole
// inverse (FP64, or the hi and lo matrices of the complex64 form, 16 bytes
// per entry either way); 0 (read from global memory) for N_o > 2.
template <int NO>
constexpr uint32_t kInvStage = kStage<NO> ? (uint32_t)(CK * NO * CK * NO * sizeof(double2)) : 0u;
// Orbital pairs that one pass of proj_block takes, and the bytes of its
// cross-warp partial sums (which share the buffer of the staged inverse).
template <int NO> constexpr int kPG = NO == 1 ? 1 : NO == 3 ? 3 : 4;
template <int NO>
constexpr size_t kBufBytes = std::max((size_t)kInvStage<NO>, (size_t)8 * kPG<NO> * 64 * 16);
// Leaf rows (of four per thread) that a chunk's far field keeps in flight.
template <int NO, typename S> constexpr int kLB = NO == 1 ? 4 : NO == 2 ? (sizeof(S) == 8 ? 4 : 2) : 1;
constexpr int kCopyWaitPolls = 1 << 20;   // bound of the wait for a staged inverse
constexpr int kSplitRows = 192;           // compressed rows from which a sweep is split (see split_les)

// What a sweep's launch covers: everything, or (see split_les) only the
// uncompressed rows (retarded: with the head) or only the compressed leaves.
enum { kAll = 0, kTop = 1, kLeaves = 2 };

// Sum over the 8 lanes of an aligned lane group of their history
// accumulators (every lane receives it).  Complex64 form: the compensated
// FP32 sums are combined in float-float, so the reduction runs on the FP32
// pipes; FP64 form: plain FP64.
template <typename R>
__device__ __forceinline__ auto reduce8(const KAcc<R>& k) { return kacc_lanes(k, 1, 8); }

// m: the largest |new - old|^2 of a thread, old a stored element; its root is the
// measure of the iteration's change.  It sits at the end of every chunk of the
// chain, so it stays one register: fmax would drop a NaN, and in FP64 a change that
// is not finite goes to the CTA's measure serr at once; the complex64 form compares
// the bits, in which a NaN is above infinity (change_out tells an overflow of the
// square apart).  Bits in FP64 cost 1.5% (1 x 64: 10.15 -> 10.30 ms), a root per
// element or a way of its own for large changes in the complex64 form 2%
// (N_o = 2, 1 x 1089) and 1.0% (128 x 600).
__device__ __forceinline__ void fold_change(double& m, const zd& a, const zd& o, double* serr) {
  const double d = (a - o).abs2();
  m = fmax(m, d);
  if ((__double2hiint(d) & 0x7fffffff) >= 0x7ff00000) atomic_max_nonneg(serr, INFINITY);
}
__device__ __forceinline__ void fold_change(float& m, const cff& a, const zf& o, double*) {
  const float x = (a.re.hi - o.re) + a.re.lo, y = (a.im.hi - o.im) + a.im.lo;
  m = __int_as_float(max(__float_as_int(m), __float_as_int(x * x + y * y) & 0x7fffffff));
}
// The warp's measure: bits in which a NaN is kept (complex64 form), or numbers.
__device__ __forceinline__ double change_warp(double m) { return sqrt(warp_max(m)); }
__device__ __forceinline__ double change_warp(float m) {
  return sqrt((double)__int_as_float(__reduce_max_sync(FULL, __float_as_int(m))));
}
// The CTA's measure, by one thread: where a square left FP32 but every element of
// the row (one component, elements `step` apart) is finite, the change was large,
// at least the root of the largest square, and the step goes on.
template <int NO, typename S>
__device__ __forceinline__ double change_out(double e, const S* row, int T, int step) {
  if constexpr (sizeof(S) == sizeof(float2)) {
    if (!(e < INFINITY)) {
      bool finite = true;
      for (int t = 0; t <= T; ++t)
        for (int j = 0; j < NO; ++j) {
          const float2 v = row[(long long)t * NO * NO + j * step];
          finite &= isfinite(v.x) && isfinite(v.y);
        }
      if (finite) e = 1.8446743e19;
    }
  }
  return e;
}
__device__ __forceinline__ void vstore(double2* p, const zd& v) { st(p, v); }
__device__ __forceinline__ void vstore(float2* p, const cff& v) { *p = make_float2(v.re.hi, v.im.hi); }
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

// Inverse of chunk cc of sweep `which`, (32 N_o)^2 entries (rows of points not
// yet built: unused).  FP64
// storage form: complex128.  Complex64 form: the same 16 bytes per entry
// hold a complex64 pair hi + lo (hi = the inverse rounded to complex64, lo =
// the rounding of hi), [hi matrix][lo matrix].  The chunk's right-hand side
// splits into the far field (history sums, lesser source), whose image under
// the inverse is about h / a_0 times smaller than the row and needs FP32 only,
// and the BDF terms reaching across the chunk edge (k rows), which carry the
// implicit recursion and get hi + lo in float-float (about 48 bits); a plain
// complex64 inverse would put 2^-24 times the BDF amplitude a_j / h into
// every chunk and accumulate.  In a chunk that is still growing the far field
// goes through hi + lo too: the next steps' BDF terms come from its points (rms
// error of the density matrix against FP64, N_o = 1, runs of 40 points: 5.7e-8
// with the FP32 product, 4.5e-8 so; no time: 99.1 -> 99.3 ms at 304 x 384, 158.1 ->
// 158.0 at N_o = 2, 128 x 600).
template <int NO>
__device__ __forceinline__ double2* Cinv(const Dev& d, int n, int cc, int which) {
  const long long nn = (long long)(CK * NO) * (CK * NO);
  return d.cinv + (((long long)n * d.nchunk + cc) * 2 + which) * nn;
}

// Dynamic shared memory of a sweep: the buffer of the staged inverse, the
// projections Ps[slot][rmax] of the blocks that cover the current leaf (slot =
// (target m or j, level, other index), target-major), the same packed without
// the gaps between ranks (Pk, and the factor entry Off each belongs to), and
// per slot its factor base and first packed entry; per slot and level the rank
// and the block with its geometry, for this leaf and the next.
struct LeafBlk {
  long long uoff, voff;
  int b, r0, r1, c0, c1, pad;
};
template <int NO, typename R>
struct SweepMem {
  cx<R>*Ps, *Pk;
  long long* base;
  LeafBlk* blk;   // [2][maxl]
  unsigned* off;
  int *start, *rk;
  int nslot;
  __host__ __device__ static size_t bytes(int maxl, int rmax) {
    const size_t ns = (size_t)maxl * NO * NO;
    return ns * rmax * (2 * sizeof(cx<R>) + 4) + ns * 8 + 2 * maxl * sizeof(LeafBlk) + (3 * ns + 1) * 4 + 16;
  }
  __device__ SweepMem(char* p, int maxl, int rmax) {
    nslot = maxl * NO * NO;
    Ps = reinterpret_cast<cx<R>*>(p);
    Pk = Ps + (size_t)nslot * rmax;
    base = reinterpret_cast<long long*>(Pk + (size_t)nslot * rmax);
    blk = reinterpret_cast<LeafBlk*>(base + nslot);
    off = reinterpret_cast<unsigned*>(blk + 2 * maxl);
    start = reinterpret_cast<int*>(off + (size_t)nslot * rmax);
    rk = start + nslot + 1;
  }
};

// Projections of one block of Sigma^R for all N_o^2 orbital pairs: P_p[q] =
// S_p[q] sum_{l in [l0, l1)} v_p(l) F_p(l, q) for q < rank_p, with F = U
// (ROWS: the retarded sweep, v_p = y_m, m = p / N_o) or F = conj(V) (the
// lesser sweep, v_p = w_l x_nn, nn = p % N_o); vf(l, i) returns the vector's
// component i at l.  A warp covers 32 / lpr rows per step, lpr = 8, 16 or 32
// lanes per row (the smallest that holds the largest rank), so small ranks
// keep every lane loading; warps split the rows, and the pairs of a group
// share the vector loads.  Partial sums (compensated FP32, or FP64) are
// combined across a warp's rows by shuffles and across warps in red
// ([8][group][64], shared memory).  out(p, q, value).  Every thread calls it.
template <int NO, typename S, bool ROWS, typename VF, typename RK, typename OUT>
__device__ __forceinline__ void proj_block(const Dev& d, int n, const LeafBlk& B, int l0, int l1, VF vf, RK rank_of,
                                           void* buf, OUT out) {
  constexpr int NO2 = NO * NO, PG = kPG<NO>;
  using R = typename Bulk<S>::R;
  using V = typename Val<S>::t;
  V* red = static_cast<V*>(buf);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int base = ROWS ? B.r0 : B.c0, len = ROWS ? B.r1 - B.r0 : B.c1 - B.c0;
  const S* Fb = static_cast<const S*>(ROWS ? d.hod[2].U : d.hod[2].V) +
                ((long long)n * (ROWS ? d.utot : d.vtot) + (ROWS ? B.uoff : B.voff)) * d.rmax;
#pragma unroll 1
  for (int p0 = 0; p0 < NO2; p0 += PG) {
    int rk[PG], rkmax = 0;
    const S* F[PG];
#pragma unroll
    for (int g = 0; g < PG; ++g) {
      rk[g] = rank_of(p0 + g);
      F[g] = Fb + (long long)(p0 + g) * len * d.rmax;
      rkmax = max(rkmax, rk[g]);
    }
    for (int qb = 0; qb < rkmax; qb += 64) {   // 64 entries of the rank at a time
      const int rem = min(rkmax - qb, 64), lpr = rem <= 8 ? 8 : rem <= 16 ? 16 : 32;   // lanes per row
      const int rps = 32 / lpr, sub = lane / lpr, q0 = qb + lane % lpr;
      const int stride = 8 * rps;   // rows per CTA step
      double sv = 0.0;              // the singular value this thread multiplies at the end
      if (tid < PG * 64) {
        const int g = tid >> 6, q = qb + (tid & 63);
        if (q < d.rmax) sv = Sp<NO>(d, 2, n, B.b, p0 + g)[q];
      }
      KAcc<R> part[PG][2];
      for (int sb = l0 + warp * rps + sub; sb < l1; sb += stride * FOLD) {
        cx<R> pp[PG][2];
#pragma unroll
        for (int g = 0; g < PG; ++g) pp[g][0] = pp[g][1] = cx<R>(0);
#pragma unroll
        for (int jj = 0; jj < FOLD; ++jj) {
          const int l = sb + stride * jj;
          if (l < l1) {
            cx<R> v[NO];
#pragma unroll
            for (int i = 0; i < NO; ++i) v[i] = vf(l, i);
#pragma unroll
            for (int g = 0; g < PG; ++g) {
              const S* fr = F[g] + (long long)(l - base) * d.rmax;
              const cx<R> vp = pick(v, ROWS ? (p0 + g) / NO : (p0 + g) % NO);
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int q = q0 + lpr * u;
                if (q < rk[g]) {
                  const cx<R> f = ROWS ? ldr<R>(fr + q) : ldr<R>(fr + q).conj();
                  pp[g][u] = cfma(vp, f, pp[g][u]);
                }
              }
            }
          }
        }
#pragma unroll
        for (int g = 0; g < PG; ++g) {
          part[g][0].add(pp[g][0]);
          part[g][1].add(pp[g][1]);
        }
      }
#pragma unroll
      for (int g = 0; g < PG; ++g)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int q = q0 + lpr * u - qb;
          if (lpr * u < rem) {
            const V r = kacc_lanes(part[g][u], lpr, 32);
            if (sub == 0 && q < 64) red[(warp * PG + g) * 64 + q] = r;
          }
        }
      __syncthreads();
      if (tid < PG * 64) {
        const int g = tid >> 6, q = tid & 63;
        if (q < min(pick(rk, g) - qb, 64)) {   // (entries past rem are not written by the warps)
          V a[8];
#pragma unroll
          for (int w2 = 0; w2 < 8; ++w2) a[w2] = red[(w2 * PG + g) * 64 + q];
#pragma unroll
          for (int s2 = 4; s2; s2 >>= 1)
#pragma unroll
            for (int w2 = 0; w2 < s2; ++w2) a[w2] = vadd(a[w2], a[w2 + s2]);
          out(p0 + g, qb + q, a[0], sv);
        }
      }
      __syncthreads();
    }
  }
}
__device__ __forceinline__ zd scale_sv(const zd& a, double s) { return a * s; }
__device__ __forceinline__ zf scale_sv(const cff& a, double s) {
  const ffl f = ff_of(s);
  return zf(ff_mul(a.re, f).hi, ff_mul(a.im, f).hi);
}

// Geometry of block b (b < 0: none), where it is not kept in shared memory.
__device__ __forceinline__ LeafBlk block_at(const Dev& d, int b) {
  if (b < 0) return {0, 0, -1, 0, 0, 0, 0, 0};
  return {d.b_uoff[b], d.b_voff[b], b, d.b_r0[b], d.b_r1[b], d.b_c0[b], d.b_c1[b], 0};
}

// The blocks of Sigma^R that cover leaf jl (retarded: over its columns, only
// blocks with built rows; lesser: over its rows), their geometry and ranks, into
// blk and rk.  The kernels read them a leaf ahead.
template <int NO, typename R>
__device__ __forceinline__ void leaf_table(const Dev& d, int n, int jl, bool cols, int* rk, LeafBlk* blk, int t0) {
  constexpr int NO2 = NO * NO;
  const int* tab = cols ? d.colblk : d.rowblk;
  for (int e = t0; e < d.maxl * NO2; e += blockDim.x) {
    // slot order: target-major (retarded: target j = p % N_o; lesser: m = p / N_o)
    const int tg = e / (d.maxl * NO), lv = (e / NO) % d.maxl, oth = e % NO, p = cols ? oth * NO + tg : tg * NO + oth;
    int b = tab[jl * d.maxl + lv];
    if (b >= 0 && cols && d.b_r0[b] >= d.cdir) b = -1;
    rk[e] = b >= 0 ? *Rk<NO>(d, 2, n, b, p) : 0;
    if (tg == 0 && oth == 0) {
      blk[lv].b = b;
      if (b >= 0) blk[lv] = {d.b_uoff[b], d.b_voff[b], b, d.b_r0[b], d.b_r1[b], d.b_c0[b], d.b_c1[b], 0};
    }
  }
}
// Pack the projections of the current leaf: entry e of target tg belongs to
// e in [start[tg maxl NO], start[(tg + 1) maxl NO]).  Every thread calls it.
template <int NO, typename R>
__device__ __forceinline__ void leaf_pack(const Dev& d, int A, bool cols, const SweepMem<NO, R>& sm, const int* rk,
                                          const LeafBlk* blk) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp == 0) {   // first packed entry of each slot
    int carry = 0;
    for (int s0 = 0; s0 < sm.nslot; s0 += 32) {
      const int r = s0 + lane < sm.nslot ? rk[s0 + lane] : 0;
      int x = r;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
      }
      if (s0 + lane < sm.nslot) sm.start[s0 + lane] = carry + x - r;
      carry += __shfl_sync(FULL, x, 31);
    }
    if (lane == 0) sm.start[sm.nslot] = carry;
  }
  __syncthreads();
  for (int s = warp; s < sm.nslot; s += 8) {
    const int r = rk[s];
    if (!r) continue;
    const int tg = s / (d.maxl * NO), lv = (s / NO) % d.maxl, oth = s % NO, p = cols ? oth * NO + tg : tg * NO + oth;
    const LeafBlk& B = blk[lv];
    const long long base = cols ? (B.voff + (long long)p * (B.c1 - B.c0) + (A - B.c0)) * d.rmax
                                : (B.uoff + (long long)p * (B.r1 - B.r0) + (A - B.r0)) * d.rmax;
    for (int q = lane; q < r; q += 32) {
      sm.Pk[sm.start[s] + q] = sm.Ps[(size_t)s * d.rmax + q];
      sm.off[sm.start[s] + q] = (unsigned)(base + q);
    }
  }
  __syncthreads();
}

}  // namespace

// ---------------------------------------------------------------------------
// Retarded row, Eq. KBER: unknown y(t') = G^R(T, t') (row irow), solved for
// t' = T-1 .. 0; the 2k points of the head are solved together.
//
// One CTA per (instance, orbital row) walks the chunks; its time is the
// dependency chain of their phases, not bandwidth.  What keeps a phase short:
// the last 64 solved points stay in shared memory (the far field of the lower
// half of a leaf, the BDF terms and the band read them there), the chunks of the
// complex64 form compute on the FP32 pipes but for the scaling of projections by
// their singular values (FP64 copies of the row are written a phase later, off
// the chain; the head and row T of the lesser column are FP64), the ranks of the
// next leaf are read while this one is worked on, and the factors of all blocks
// over a leaf are read as one packed list with eight loads in flight per thread
// (one block and pair after the other, each waited for its rank and then for its
// row).
// Both sweeps of an iteration, before and after these: 1.05 -> 0.53 ms (N_o = 2,
// complex64, 128 instances, T = 600), 1.34 -> 0.69 ms (one instance, T = 1089),
// 0.75 -> 0.43 ms (N_o = 2, FP64, 16 instances, T = 300).
// ---------------------------------------------------------------------------
// MIX: the CTAs after the first N_o of an instance compute its mixed component.
template <int NO, typename S, bool MIX>
__global__ void __launch_bounds__(256, (NO <= 2) ? 2 : 1) k_ret2(Dev d, int T, int staged, int part) {
  pdl_start();
  constexpr int NO2 = NO * NO;
  constexpr bool MX = Row64<NO, S>::separate;
  using R = typename Bulk<S>::R;
  using V = typename Val<S>::t;
  const int n = blockIdx.y, irow = blockIdx.x;
  if constexpr (MIX) {
    if (irow >= NO) {
      mixed_nodes<NO, S, kNodesFew<NO>>(d, T, irow - NO, n);
      return;
    }
  }
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int k = d.k, c = d.cdir, L = d.L;
  const double h = d.h;
  const DevW& W = d.w;
  __shared__ zd sB[10 * NO];      // right-hand side of the head
  __shared__ V FB[64][NO];        // far field of the leaf's columns from the rows beyond the leaf
  __shared__ V Yl[64][NO];        // the last 64 solved points, y(t') in slot t' mod 64
  __shared__ cx<R> yr[kRingRows][NO];   // y on the uncompressed rows, times the weights at the end T
  __shared__ cx<R> Ff[CK][NO];    // the chunk's far field (FP64 form: with its BDF part)
  __shared__ V Fb[CK][NO];        // the BDF terms reaching beyond the chunk (complex64 form)
  __shared__ cx<R> Old[CK][NO];   // the chunk's previous iterate (convergence measure)
  __shared__ double serr;
  extern __shared__ __align__(16) char dyn[];
  zd* ctile = reinterpret_cast<zd*>(dyn);
  SweepMem<NO, R> sm(dyn + kBufBytes<NO>, d.maxl, d.rmax);
  __shared__ __align__(8) uint64_t cbar;   // completion of the inverse's bulk copy
  __shared__ int s_stage;                  // 0 once a wait for a copy has timed out
  uint32_t cphase = 0;
  const int top = T - 2 * k - 1;   // the highest point of the chunks (none while T <= 2k)
  int buf = 0;                     // table buffer of the current leaf
  if (tid == 0) {
    serr = 0.0;
    s_stage = 1;
    if (kInvStage<NO>) mbar_init(&cbar);
  }
  // The row being solved lives in FP64 during the sweep (in the complex64
  // storage form a separate buffer), so the point-to-point recursion of the
  // sweep (BDF terms, chunk solves) does not accumulate storage rounding.
  // yp: the FP64 row; sp: its storage, written at the same time (rounded in
  // the complex64 form), which the FP32 bulk sums read; it holds the previous
  // iterate until an element is overwritten (the convergence measure).
  S* rowp = el<NO, S>(d.GR, d, n, T, 0);
  Y* rowy = Row64<NO, S>::get(d, n, 0, T, rowp);
  auto yp = [&](int tp) { return rowy + (long long)tp * NO2 + irow * NO; };
  auto sp = [&](int tp) { return rowp + (long long)tp * NO2 + irow * NO; };
  std::conditional_t<MX, float, double> myerr = 0;
  const bool below = part != kTop, above = part != kLeaves;   // the compressed columns; the head and the others
  if (staged && below && top >= 0 && c > 0)
    leaf_table<NO, R>(d, n, (min(c, top + 1) - 1) / L, true, sm.rk, sm.blk, tid);
  // ---- the head: points T-s, s = 1..hs, and y(T) = -i.  Its right-hand side
  // is row T of Sigma^R (and the derivative's y(T) term) alone; 8 threads per
  // element of the product with the head's inverse ----
  const int hs = above ? min(2 * k, T) : 0, nh = hs * NO;
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
        V v;
        vset(v, y);
        fold_change(myerr, v, ldr<R>(sp(T - s) + j), &serr);
        Yl[(T - s) & 63][j] = v;
        st(yp(T - s) + j, y);
        if constexpr (MX) vstore(sp(T - s) + j, v);
      }
    }
  }
  if (above && tid < NO) {
    V v;
    vset(v, (tid == irow) ? zd(0, -1) : zd());
    fold_change(myerr, v, ldr<R>(sp(T) + tid), &serr);
    st(yp(T) + tid, v64(v));
    if constexpr (MX) vstore(sp(T) + tid, v);
  }
  __syncthreads();
  // FP64 copies of the points [wa, wa + wn) (complex64 form), by the last threads first
  auto write64 = [&](int wa, int wn) {
    if constexpr (MX)
      for (int e = blockDim.x - 1 - tid; e < wn * NO; e += blockDim.x)
        st(yp(wa + e / NO) + e % NO, cff_val(Yl[(wa + e / NO) & 63][e % NO]));
  };
  bool first_comp = part == kAll;
  int wa = 0, wn = 0;
  if (part == kLeaves) {   // the points solved last by the part before
    const int b0 = min(c, top + 1);
    for (int e = tid; e < 64 * NO; e += blockDim.x) {
      const int tp = b0 + e / NO;
      if (tp > T) continue;
      if constexpr (MX) Yl[tp & 63][e % NO] = cff_of(ld(yp(tp) + e % NO));   // (hi rounded: it is used by itself too)
      else Yl[tp & 63][e % NO] = ld(yp(tp) + e % NO);
    }
    __syncthreads();
  }
  const V* fr = reinterpret_cast<const V*>(d.fring) + ((long long)n * NO + irow) * d.nt * NO;
  const int cstart = part == kLeaves ? min(c, top + 1) - 1 : top;
  for (int cc = cstart >= 0 ? cstart / CK : -1; cc >= 0; --cc) {
    const int a = cc * CK, b = min(a + CK, top + 1), cn = b - a;
    const bool comp = (c > 0 && b <= c);
    if (comp && !below) break;
    const int jl = comp ? a / L : 0, A = jl * L, E = comp ? (jl + 1) * L : 0;
    if (comp && (b == E || b == top + 1)) {   // (the top chunk may end inside its leaf)
      // Entering leaf jl from above.
      const int* rk = sm.rk + buf * sm.nslot;
      const LeafBlk* blks = sm.blk + buf * d.maxl;
      const int nr = part == kAll ? T + 1 - c : 0;   // uncompressed rows to sum here
      if (first_comp) {   // the uncompressed rows with their weights at the end T
        first_comp = false;
        for (int e = tid; e < nr * NO; e += blockDim.x) {
          const int s2 = c + e / NO;
          const cx<R> v = ldr<R>(sp(s2) + e % NO);
          yr[e / NO][e % NO] = T - s2 <= k ? v * rule_wr<R>(W, T + 2 * k + 1, T - s2) : v;
        }
      }
      // (1) projections pi_B = sum_s y(s) U_B(s,:) S_B of the blocks whose columns end at E
      for (int lv = 0; lv < d.maxl; ++lv) {
        const LeafBlk B = staged ? blks[lv] : block_at(d, d.colblk[jl * d.maxl + lv]);
        if (B.b < 0 || B.c1 != E || B.r0 >= c) continue;
        auto slot = [&](int p) { return ((p % NO) * d.maxl + lv) * NO + p / NO; };
        proj_block<NO, S, true>(
            d, n, B, B.r0, min(B.r1, c), [&](int s2, int m) { return ldr<R>(sp(s2) + m); },
            [&](int p) { return staged ? rk[slot(p)] : *Rk<NO>(d, 2, n, B.b, p); }, dyn,
            [&](int p, int q, const V& v, double sv) {
              if (staged) sm.Ps[(size_t)slot(p) * d.rmax + q] = scale_sv(v, sv);
              else reinterpret_cast<cx<R>*>(Pj<NO>(d, n, irow, lv, p))[q] = scale_sv(v, sv);
            });
      }
      __syncthreads();
      if (staged) leaf_pack<NO, R>(d, A, true, sm, rk, blks);
      // (2) for every column of the leaf: uncompressed rows s in [c, T], the
      // blocks below the leaf (weight 1) and the near-diagonal corrections;
      // 256 / L threads per column.
      if (staged && jl > 0)
        leaf_table<NO, R>(d, n, jl - 1, true, sm.rk + (buf ^ 1) * sm.nslot, sm.blk + (buf ^ 1) * d.maxl, blockDim.x - 1 - tid);
      {
        const int lpc = blockDim.x / L, col = tid / lpc, sl = tid % lpc, tp = A + col;
        KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
        V fr0[NO];        // the uncompressed rows' part, if a kernel before this one has it
#pragma unroll
        for (int j = 0; j < NO; ++j) {
          vset(fr0[j], zd());
          if (part == kLeaves && sl == 0) fr0[j] = fr[(long long)tp * NO + j];
        }
        constexpr int RB = NO == 1 ? 8 : NO == 2 ? (MX ? 4 : 2) : 1;   // rows in flight
        const S* Sr = static_cast<const S*>(d.SR) + ((long long)n * d.ring * d.nt + tp) * NO2;
        const int s0 = c % d.ring;
        for (int i0 = sl; i0 < nr; i0 += lpc * RB) {
          cx<R> sv[RB][NO2];
#pragma unroll
          for (int u = 0; u < RB; ++u) {
            const int i = i0 + lpc * u;
            int slot = s0 + i;
            if (slot >= d.ring) slot -= d.ring;
            const S* s = Sr + (long long)slot * d.nt * NO2;
#pragma unroll
            for (int q = 0; q < NO2; ++q) sv[u][q] = i < nr ? ldr<R>(s + q) : cx<R>(0);
          }
          cx<R> pa[NO];
#pragma unroll
          for (int j = 0; j < NO; ++j) pa[j] = cx<R>(0);
#pragma unroll
          for (int u = 0; u < RB; ++u) {
            const int i = min(i0 + lpc * u, nr - 1), dd = c + i - tp;
            const R wd = dd <= k && dd >= 0 ? rule_wr<R>(W, 2 * k + 1 + dd, dd) : (R)1;
#pragma unroll
            for (int m = 0; m < NO; ++m) {
              const cx<R> ym = yr[i][m] * wd;
#pragma unroll
              for (int j = 0; j < NO; ++j) pa[j] = cfma(ym, sv[u][m * NO + j], pa[j]);
            }
          }
#pragma unroll
          for (int j = 0; j < NO; ++j) ka[j].add(pa[j]);
        }
        if (staged) {
          const S* Vb = static_cast<const S*>(d.hod[2].V) + (long long)n * d.vtot * d.rmax + (long long)col * d.rmax;
#pragma unroll
          for (int j = 0; j < NO; ++j) {
            const int e1 = sm.start[(j + 1) * d.maxl * NO];
            for (int e0 = sm.start[j * d.maxl * NO] + sl; e0 < e1; e0 += lpc * FOLD) {
              cx<R> f[FOLD], pb = cx<R>(0);
#pragma unroll
              for (int u = 0; u < FOLD; ++u) {
                const int e = e0 + lpc * u;
                f[u] = e < e1 ? ldr<R>(Vb + sm.off[e]) : cx<R>(0);
              }
#pragma unroll
              for (int u = 0; u < FOLD; ++u) pb = cfma(sm.Pk[min(e0 + lpc * u, e1 - 1)], f[u].conj(), pb);
              ka[j].add(pb);
            }
          }
        } else {
          for (int lv = 0; lv < d.maxl; ++lv) {
            const int blk = d.colblk[jl * d.maxl + lv];
            if (blk < 0 || d.b_r0[blk] >= c) continue;
#pragma unroll
            for (int p = 0; p < NO2; ++p) {
              const int rkp = *Rk<NO>(d, 2, n, blk, p);
              const S* Vr = Vp<NO, S>(d, 2, n, blk, p) + (long long)(tp - d.b_c0[blk]) * d.rmax;
              const cx<R>* P = reinterpret_cast<const cx<R>*>(Pj<NO>(d, n, irow, lv, p));
              cx<R> pb = cx<R>(0);
              for (int q = sl; q < rkp; q += lpc) pb = cfma(P[q], ldr<R>(Vr + q).conj(), pb);
              ka[p % NO].add(pb);
            }
          }
        }
        V acc[NO];
#pragma unroll
        for (int j = 0; j < NO; ++j) vset(acc[j], zd());
        if (E < c && __any_sync(FULL, tp + k >= E))
          for (int s2 = E + sl; s2 <= tp + k && s2 < c; s2 += lpc) {   // (w - 1) of the band's entries
            const S* bd = Bd<NO, S>(d, n, s2, s2 - tp);
#pragma unroll
            for (int m = 0; m < NO; ++m) {
              const V ym = vreal(Yl[s2 & 63][m], W.omega[s2 - tp] - 1.0, W.wm1f[s2 - tp]);
#pragma unroll
              for (int j = 0; j < NO; ++j) {
                if constexpr (MX) acc[j] = cff_add(acc[j], cff_mul(ym, cff_of(ldr<R>(bd + m * NO + j))));
                else acc[j] = cfma(ym, ld(bd + m * NO + j), acc[j]);
              }
            }
          }
#pragma unroll
        for (int j = 0; j < NO; ++j) {
          V r = kacc_lanes(ka[j], 1, lpc);
          if (E < c && __any_sync(FULL, tp + k >= E)) {
            for (int off = 1; off < lpc; off <<= 1) acc[j] = vadd(acc[j], vshfl_xor(acc[j], off));
            r = vadd(r, acc[j]);
          }
          if (sl == 0) FB[col][j] = vadd(r, fr0[j]);
        }
      }
      buf ^= 1;
      __syncthreads();
    }
    const bool full = MX && cc >= d.nfrozR;   // still growing: all of its right-hand side in float-float
    // the inverse of this chunk into shared memory, overlapping the far field
    const bool stage_now = kInvStage<NO> && s_stage;
    if (stage_now && tid == 0) bulk_g2s(ctile, Cinv<NO>(d, n, cc, 0), kInvStage<NO>, &cbar);
    // ---- far field of the chunk: rows s >= b not covered above; 8 threads per column ----
    {
      const int col = tid >> 3, sl = tid & 7;
      const int tp = a + col;
      KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
      cx<R> old = cx<R>(0);
      if (sl < NO && col < cn) old = ldr<R>(sp(tp) + sl);
      if (col < cn) {
        if (comp) {   // the rest of the leaf (at most 32 points, solved last)
          const S* lf = static_cast<const S*>(d.hod[2].leaf) +
                        ((long long)n * d.leaftot + (long long)jl * ((long long)L * (L + 1) / 2) + (tp - A)) * NO2;
          cx<R> pa[NO];
#pragma unroll
          for (int j = 0; j < NO; ++j) pa[j] = cx<R>(0);
#pragma unroll
          for (int u0 = 0; u0 < 4; u0 += kLB<NO, S>) {
            cx<R> sv[kLB<NO, S>][NO2];
#pragma unroll
            for (int u = 0; u < kLB<NO, S>; ++u) {
              const int s2 = b + sl + 8 * (u0 + u);
#pragma unroll
              for (int q = 0; q < NO2; ++q) sv[u][q] = s2 < E ? ldr<R>(lf + tri(s2 - A) * NO2 + q) : cx<R>(0);
            }
#pragma unroll
            for (int u = 0; u < kLB<NO, S>; ++u) {
              const int s2 = b + sl + 8 * (u0 + u);
              if (s2 < E) {
                const R ws = rule_wr<R>(W, T - tp, T - s2);
#pragma unroll
                for (int m = 0; m < NO; ++m) {
                  const cx<R> ym = vbulk(Yl[s2 & 63][m]) * ws;
#pragma unroll
                  for (int j = 0; j < NO; ++j) pa[j] = cfma(ym, sv[u][m * NO + j], pa[j]);
                }
              }
            }
          }
#pragma unroll
          for (int j = 0; j < NO; ++j) ka[j].add(pa[j]);
        } else {
          for (int s0 = b + sl; s0 <= T; s0 += 8 * FOLD) {
            cx<R> pa[NO];
#pragma unroll
            for (int j = 0; j < NO; ++j) pa[j] = cx<R>(0);
#pragma unroll
            for (int jj = 0; jj < FOLD; ++jj) {
              const int s2 = s0 + 8 * jj;
              if (s2 <= T) {
                const bool end = T - s2 <= k || s2 - tp <= k;   // (weight 1 elsewhere: no product)
                const R ws = end ? rule_wr<R>(W, T - tp, T - s2) : (R)1;
                const S* yl = sp(s2);
                const S* sr = el<NO, S>(d.SR, d, n, s2, tp);
#pragma unroll
                for (int m = 0; m < NO; ++m) {
                  cx<R> ym = ldr<R>(yl + m);
                  if (end) ym = ym * ws;
#pragma unroll
                  for (int j = 0; j < NO; ++j) pa[j] = cfma(ym, ldr<R>(sr + m * NO + j), pa[j]);
                }
              }
            }
#pragma unroll
            for (int j = 0; j < NO; ++j) ka[j].add(pa[j]);
          }
        }
      }
      V r[NO];
#pragma unroll
      for (int j = 0; j < NO; ++j) r[j] = reduce8(ka[j]);
      if (sl < NO && col < cn) {   // lane sl of the group finishes component sl
        V F = pick(r, sl), fb;
        if (comp) F = vadd(F, FB[tp - A][sl]);
        F = vreal(F, h, W.hf);
        vset(fb, zd());
        if (col >= cn - k)   // BDF terms reaching above the chunk: (-i a_j / h) y(s2)
          for (int jj = b - tp; jj <= k; ++jj) fb = vbdf(fb, Yl[(tp + jj) & 63][sl], W, jj);
        if constexpr (MX) {
          Ff[col][sl] = vbulk(F);
          Fb[col][sl] = full ? vadd(F, fb) : fb;
        } else {
          Ff[col][sl] = F + fb;
        }
        Old[col][sl] = old;
      }
    }
    write64(wa, wn);
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
        V out;
        if constexpr (MX) {
          // complex64 form: far field x hi in FP32, the k edge rows x (hi + lo)
          // in float-float, reduced over the 8 lanes in float-float
          const float2* Mh = reinterpret_cast<const float2*>(Mg);
          const float2* Ml = Mh + LD * LD;
          zf s32 = zf(0);
          for (int si = (ti & ~7) + sl; si < cn && !full; si += 8)
#pragma unroll
            for (int m = 0; m < NO; ++m)
              s32 = cfma(Ff[si][m], ldr<float>(Mh + (long long)(si * NO + m) * LD + ti * NO + j), s32);
          out = cff_of(s32);
          for (int si = (full ? ti & ~7 : max(cn - k, 0)) + sl; si < cn; si += 8)
#pragma unroll
            for (int m = 0; m < NO; ++m) {
              const long long e = (long long)(si * NO + m) * LD + ti * NO + j;
              const float2 hv = Mh[e], lv = Ml[e];
              out = cff_add(out, cff_mul(Fb[si][m], cff{{hv.x, lv.x}, {hv.y, lv.y}}));
            }
        } else {
          out = zd();
          for (int si = (ti & ~7) + sl; si < cn; si += 8)
#pragma unroll
            for (int m = 0; m < NO; ++m) out = cfma(Ff[si][m], ld(Mg + (long long)(si * NO + m) * LD + ti * NO + j), out);
        }
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) out = vadd(out, vshfl_xor(out, off));
        if (sl == 0 && ti < cn) {
          fold_change(myerr, out, Old[ti][j], &serr);
          Yl[(a + ti) & 63][j] = out;
          vstore(sp(a + ti) + j, out);
        }
      }
      wa = a;
      wn = cn;
    }
    __syncthreads();
  }
  write64(wa, wn);
  const double e1 = change_warp(myerr);
  if (lane == 0 && !(e1 <= 0)) atomic_max_nonneg(&serr, e1);
  __syncthreads();
  if (tid == 0) atomic_max_nonneg(d.err + n, change_out<NO, S>(serr, sp(0), T, 1));
  // after a timed-out wait, a copy may still be in flight into this CTA's
  // shared memory: wait for it (bounded) before the CTA exits
  if (kInvStage<NO> && tid == 0 && !s_stage) mbar_wait(&cbar, cphase ^ 1u, kCopyWaitPolls);
}

// ---------------------------------------------------------------------------
// Lesser column, Eq. KBEL: unknown x(t) = G^<(t, T) (column jc), t = 0..T; the
// same phases as the retarded sweep, upwards.
// ---------------------------------------------------------------------------
template <int NO, typename S>
__global__ void __launch_bounds__(256, (NO <= 2) ? 2 : 1) k_les2(Dev d, int T, int staged, int part) {
  pdl_start();
  constexpr int NO2 = NO * NO;
  constexpr bool MX = Row64<NO, S>::separate;
  using R = typename Bulk<S>::R;
  using V = typename Val<S>::t;
  const int n = blockIdx.y, jc = blockIdx.x;
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = d.k, c = d.cdir, L = d.L;
  const double h = d.h;
  const DevW& W = d.w;
  __shared__ V FB[64][NO];        // far field of the leaf's rows from the columns before the leaf
  __shared__ V Xl[64][NO];        // the last 64 solved points, x(t) in slot t mod 64
  __shared__ V FT[NO];            // right-hand side of row T
  __shared__ cx<R> Ff[CK][NO];    // the chunk's far field (FP64 form: with its BDF part)
  __shared__ V Fb[CK][NO];        // the BDF terms reaching beyond the chunk (complex64 form)
  __shared__ cx<R> Old[CK][NO];   // the chunk's previous iterate (convergence measure)
  __shared__ double serr;
  extern __shared__ __align__(16) char dyn[];
  zd* ctile = reinterpret_cast<zd*>(dyn);
  SweepMem<NO, R> sm(dyn + kBufBytes<NO>, d.maxl, d.rmax);
  __shared__ __align__(8) uint64_t cbar;   // completion of the inverse's bulk copy
  __shared__ int s_stage;                  // 0 once a wait for a copy has timed out
  uint32_t cphase = 0;
  int buf = 0;
  if (tid == 0) {
    serr = 0.0;
    s_stage = 1;
    if (kInvStage<NO>) mbar_init(&cbar);
  }
  __syncwarp();   // (serr, for the lanes that fold x(0))
  // FP64 column during the sweep (see k_ret2); xp: as solved, sp: storage
  S* colp = el<NO, S>(d.GL, d, n, T, 0);
  Y* coly = Row64<NO, S>::get(d, n, 1, T, colp);
  auto xp = [&](int t) { return coly + (long long)t * NO2; };  // element [m*NO + jc]
  auto sp = [&](int t) { return colp + (long long)t * NO2; };
  const double2* qs = d.qsrc + (long long)n * d.nt * NO2;
  std::conditional_t<MX, float, double> myerr = 0;
  const int last = (d.rho_mode == 1) ? T - 1 : T;
  if (staged && c > 0 && part != kTop) leaf_table<NO, R>(d, n, 0, false, sm.rk, sm.blk, tid);
  if (part == kTop) {   // the points solved last by the part before
    for (int e = tid; e < 64 * NO; e += blockDim.x) {
      const int t = c - 1 - e / NO, m = e % NO;
      if (t < 0) continue;
      if constexpr (MX) Xl[t & 63][m] = cff_of(ld(xp(t) + m * NO + jc));
      else Xl[t & 63][m] = ld(xp(t) + m * NO + jc);
    }
  } else if (tid < NO) {  // x(0) = -[G^tv(T, 0+)]^dagger
    const int m = tid;
    const zd x = ld(d.x0 + (long long)n * NO2 + m * NO + jc);
    V v;
    vset(v, x);
    fold_change(myerr, v, ldr<R>(sp(0) + m * NO + jc), &serr);
    Xl[0][m] = v;
    st(xp(0) + m * NO + jc, x);
    if constexpr (MX) vstore(sp(0) + m * NO + jc, v);
  }
  __syncthreads();
  auto write64 = [&](int wa, int wn) {
    if constexpr (MX)
      for (int e = blockDim.x - 1 - tid; e < wn * NO; e += blockDim.x)
        st(xp(wa + e / NO) + (e % NO) * NO + jc, cff_val(Xl[(wa + e / NO) & 63][e % NO]));
  };
  int wa = 0, wn = 0;
  const V* fl = reinterpret_cast<const V*>(d.fring) + ((long long)d.n_inst * d.nt + (long long)n * kRingRows) * NO2;
  const int chi = part == kLeaves ? c : last + 1;   // points below this
  for (int cc = part == kTop ? c / CK : 0; cc * CK < chi; ++cc) {
    const int a = (cc == 0) ? 1 : cc * CK, b = min((cc + 1) * CK, last + 1), cn = b - a;
    if (cn <= 0) break;
    const bool comp = (c > 0 && b <= c);
    const int jl = comp ? a / L : 0, A = jl * L;
    if (comp && cc * CK == A) {
      const int* rk = sm.rk + buf * sm.nslot;
      const LeafBlk* blks = sm.blk + buf * d.maxl;
      // Entering leaf jl.  (1) rho_B = S_B sum_l w_l conj(V_B(l,:)) x(l) for the
      // blocks whose rows start at A (w_l = omega_l for l <= k, else 1).
      for (int lv = 0; lv < d.maxl && jl > 0; ++lv) {
        const LeafBlk B = staged ? blks[lv] : block_at(d, d.rowblk[jl * d.maxl + lv]);
        if (B.b < 0 || B.r0 != A) continue;
        auto slot = [&](int p) { return ((p / NO) * d.maxl + lv) * NO + p % NO; };
        proj_block<NO, S, false>(
            d, n, B, B.c0, B.c1,
            [&](int l, int nn) {
              const cx<R> x = ldr<R>(sp(l) + nn * NO + jc);
              return l <= k ? x * (R)W.omega[l] : x;
            },
            [&](int p) { return staged ? rk[slot(p)] : *Rk<NO>(d, 2, n, B.b, p); }, dyn,
            [&](int p, int q, const V& v, double sv) {
              if (staged) sm.Ps[(size_t)slot(p) * d.rmax + q] = scale_sv(v, sv);
              else reinterpret_cast<cx<R>*>(Pj<NO>(d, n, jc, lv, p))[q] = scale_sv(v, sv);
            });
      }
      __syncthreads();
      if (staged) leaf_pack<NO, R>(d, A, false, sm, rk, blks);
      // (2) every row of the leaf: blocks left of it and near-diagonal corrections
      if (staged && (jl + 1) * L < c)
        leaf_table<NO, R>(d, n, jl + 1, false, sm.rk + (buf ^ 1) * sm.nslot, sm.blk + (buf ^ 1) * d.maxl, blockDim.x - 1 - tid);
      {
        const int lpc = blockDim.x / L, row = tid / lpc, sl = tid % lpc;
        const int t = A + row;
        KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
        if (staged) {
          const S* Ub = static_cast<const S*>(d.hod[2].U) + (long long)n * d.utot * d.rmax + (long long)row * d.rmax;
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            const int e1 = sm.start[(m + 1) * d.maxl * NO];
            for (int e0 = sm.start[m * d.maxl * NO] + sl; e0 < e1; e0 += lpc * FOLD) {
              cx<R> f[FOLD], pb = cx<R>(0);
#pragma unroll
              for (int u = 0; u < FOLD; ++u) {
                const int e = e0 + lpc * u;
                f[u] = e < e1 ? ldr<R>(Ub + sm.off[e]) : cx<R>(0);
              }
#pragma unroll
              for (int u = 0; u < FOLD; ++u) pb = cfma(sm.Pk[min(e0 + lpc * u, e1 - 1)], f[u], pb);
              ka[m].add(pb);
            }
          }
        } else {
          for (int lv = 0; lv < d.maxl; ++lv) {
            const int blk = d.rowblk[jl * d.maxl + lv];
            if (blk < 0) continue;
#pragma unroll
            for (int p = 0; p < NO2; ++p) {
              const int rkp = *Rk<NO>(d, 2, n, blk, p);
              const S* Ur = Up<NO, S>(d, 2, n, blk, p) + (long long)(t - d.b_r0[blk]) * d.rmax;
              const cx<R>* P = reinterpret_cast<const cx<R>*>(Pj<NO>(d, n, jc, lv, p));
              cx<R> pb = cx<R>(0);
              for (int q = sl; q < rkp; q += lpc) pb = cfma(ldr<R>(Ur + q), P[q], pb);
              ka[p / NO].add(pb);
            }
          }
        }
        V acc[NO];
#pragma unroll
        for (int m = 0; m < NO; ++m) vset(acc[m], zd());
        const bool band = jl > 0 && __any_sync(FULL, t - k < A);
        if (band)
          for (int l = max(t - k, 0) + sl; l < A; l += lpc) {
            const S* bd = Bd<NO, S>(d, n, t, t - l);
#pragma unroll
            for (int y = 0; y < NO; ++y) {
              const V xy = vreal(Xl[l & 63][y], W.omega[t - l] - 1.0, W.wm1f[t - l]);
#pragma unroll
              for (int m = 0; m < NO; ++m) {
                if constexpr (MX) acc[m] = cff_add(acc[m], cff_mul(cff_of(ldr<R>(bd + m * NO + y)), xy));
                else acc[m] = cfma(ld(bd + m * NO + y), xy, acc[m]);
              }
            }
          }
#pragma unroll
        for (int m = 0; m < NO; ++m) {
          V r = kacc_lanes(ka[m], 1, lpc);
          if (band) {
            for (int off = 1; off < lpc; off <<= 1) acc[m] = vadd(acc[m], vshfl_xor(acc[m], off));
            r = vadd(r, acc[m]);
          }
          if (sl == 0) FB[row][m] = r;
        }
      }
      buf ^= 1;
      __syncthreads();
    }
    const int fn = min(b, T) - a;   // rows solved with the chunk's inverse; row T, if it is here, follows them
    const bool full = MX && cc >= d.nfrozL;   // still growing: all of its right-hand side in float-float
    // the inverse of this chunk into shared memory, overlapping the far field
    const bool stage_now = kInvStage<NO> && fn > 0 && s_stage;
    if (stage_now && tid == 0) bulk_g2s(ctile, Cinv<NO>(d, n, cc, 1), kInvStage<NO>, &cbar);
    // ---- far field F(t) = q(t) - sum_{l < a} C(t,l) x(l); 8 threads per row ----
    {
      const int row = tid >> 3, sl = tid & 7;
      const int t = a + row;
      KAcc<R> ka[NO];   // FP32 history sums, compensated (FP64 in the FP64 form)
      cx<R> old = cx<R>(0);
      V q;
      if (sl < NO && row < cn) {
        old = ldr<R>(sp(t) + sl * NO + jc);
        q = ldv<S>(qs + (long long)t * NO2 + sl * NO + jc);
      }
      if (row < cn && t > k) {
        if (comp) {   // the leaf's rows before the chunk (at most 32 points, solved last)
          const S* lf = static_cast<const S*>(d.hod[2].leaf) +
                        ((long long)n * d.leaftot + (long long)jl * ((long long)L * (L + 1) / 2) + tri(t - A)) * NO2;
          cx<R> pa[NO];
#pragma unroll
          for (int m = 0; m < NO; ++m) pa[m] = cx<R>(0);
#pragma unroll
          for (int u0 = 0; u0 < 4; u0 += kLB<NO, S>) {
            cx<R> sv[kLB<NO, S>][NO2];
#pragma unroll
            for (int u = 0; u < kLB<NO, S>; ++u) {
              const int l = A + sl + 8 * (u0 + u);
#pragma unroll
              for (int e = 0; e < NO2; ++e) sv[u][e] = l < a ? ldr<R>(lf + (l - A) * NO2 + e) : cx<R>(0);
            }
#pragma unroll
            for (int u = 0; u < kLB<NO, S>; ++u) {
              const int l = A + sl + 8 * (u0 + u);
              if (l < a) {
                const R wl = rule_wr<R>(W, t, l);
#pragma unroll
                for (int y = 0; y < NO; ++y) {
                  const cx<R> xy = vbulk(Xl[l & 63][y]) * wl;
#pragma unroll
                  for (int m = 0; m < NO; ++m) pa[m] = cfma(sv[u][m * NO + y], xy, pa[m]);
                }
              }
            }
          }
#pragma unroll
          for (int m = 0; m < NO; ++m) ka[m].add(pa[m]);
        } else {
          const S* srow = el<NO, S>(d.SR, d, n, t, 0);
          for (int lb = (part == kTop ? c : 0) + sl; lb < a; lb += 8 * FOLD) {
            cx<R> pa[NO];
#pragma unroll
            for (int m = 0; m < NO; ++m) pa[m] = cx<R>(0);
#pragma unroll
            for (int jj = 0; jj < FOLD; ++jj) {
              const int l = lb + 8 * jj;
              if (l < a) {
                const bool end = l <= k || t - l <= k || t < 2 * k + 1;
                const R wl = end ? rule_wr<R>(W, t, l) : (R)1;
                const S* sr = srow + (long long)l * NO2;
#pragma unroll
                for (int y = 0; y < NO; ++y) {
                  cx<R> xy = ldr<R>(sp(l) + y * NO + jc);
                  if (end) xy = xy * wl;
#pragma unroll
                  for (int m = 0; m < NO; ++m) pa[m] = cfma(ldr<R>(sr + m * NO + y), xy, pa[m]);
                }
              }
            }
#pragma unroll
            for (int m = 0; m < NO; ++m) ka[m].add(pa[m]);
          }
        }
      }
      V r[NO];
#pragma unroll
      for (int m = 0; m < NO; ++m) r[m] = reduce8(ka[m]);
      if (sl < NO && row < cn) {   // lane sl of the group finishes component sl
        V F = pick(r, sl), fb;
        if (comp && t > k) F = vadd(F, FB[t - A][sl]);
        if (part == kTop) F = vadd(F, fl[((t - c) * NO + sl) * NO + jc]);   // the compressed columns
        F = vadd(vreal(F, h, W.hf), q);
        vset(fb, zd());
        if (t <= k) {   // start rows: only l = 0 lies left of chunk 0 (a derivative term: kept in Fb)
          zd f0 = zd();
          for (int y = 0; y < NO; ++y) {
            zd cf = srx_any<NO, S>(d, n, t, 0, sl, y) * (-h * W.I0[t][0]);
            if (sl == y) cf += zd(0, W.D[t][0] / h);
            f0 -= cf * ld(d.x0 + (long long)n * NO2 + y * NO + jc);
          }
          vset(fb, f0);
        } else if (row < k) {   // BDF terms reaching left of the chunk: (-i a_j / h) x(t - j)
          for (int jj = t - a + 1; jj <= k; ++jj) fb = vbdf(fb, Xl[(t - jj) & 63][sl], W, jj);
        }
        if (t == T) FT[sl] = vadd(F, fb);
        if constexpr (MX) {
          Ff[row][sl] = vbulk(F);
          Fb[row][sl] = full ? vadd(F, fb) : fb;
        } else {
          Ff[row][sl] = F + fb;
        }
        Old[row][sl] = old;
      }
    }
    write64(wa, wn);
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
        const int le = ti < fn ? max(ti + 1, min(k, fn)) : 0;   // lower triangular below the start block
        V out;
        if constexpr (MX) {
          // complex64 form: far field x hi in FP32, the k edge rows x (hi + lo) in
          // float-float, reduced over the 8 lanes in float-float
          const float2* Mh = reinterpret_cast<const float2*>(Mg);
          const float2* Ml = Mh + LD * LD;
          zf s32 = zf(0);
          for (int li = sl; li < le && !full; li += 8)
#pragma unroll
            for (int y = 0; y < NO; ++y)
              s32 = cfma(ldr<float>(Mh + (long long)(ti * NO + m) * LD + li * NO + y), Ff[li][y], s32);
          out = cff_of(s32);
          for (int li = sl; li < (full ? le : min(k, le)); li += 8)
#pragma unroll
            for (int y = 0; y < NO; ++y) {
              const long long e = (long long)(ti * NO + m) * LD + li * NO + y;
              const float2 hv = Mh[e], lv = Ml[e];
              out = cff_add(out, cff_mul(cff{{hv.x, lv.x}, {hv.y, lv.y}}, Fb[li][y]));
            }
        } else {
          out = zd();
          for (int li = sl; li < le; li += 8)
#pragma unroll
            for (int y = 0; y < NO; ++y) out = cfma(ld(Mg + (long long)(ti * NO + m) * LD + li * NO + y), Ff[li][y], out);
        }
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) out = vadd(out, vshfl_xor(out, off));
        if (sl == 0 && ti < fn) {
          fold_change(myerr, out, Old[ti][m], &serr);
          Xl[(a + ti) & 63][m] = out;
          vstore(sp(a + ti) + m * NO + jc, out);
        }
      }
    }
    wa = a;
    wn = fn;
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
            const zd x = v64(Xl[l & 63][y]), xw = x * wl;
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
            f[x2] += v64(FT[x2]);
#pragma unroll
            for (int y = 0; y < NO; ++y)
              Mm.a[x2][y] = (x2 == y ? zd(0, W.a[0] / h) : zd()) - ld(ep + x2 * NO + y) - ld(sd + x2 * NO + y) * wt;
          }
          solve_col<NO>(Mm, f, x);
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            V v;
            vset(v, x[m]);
            fold_change(myerr, v, Old[fn][m], &serr);
            st(xp(T) + m * NO + jc, x[m]);
            if constexpr (MX) vstore(sp(T) + m * NO + jc, v);
          }
        }
      }
    }
    __syncthreads();
  }
  write64(wa, wn);
  const double e1 = change_warp(myerr);
  if (lane == 0 && !(e1 <= 0)) atomic_max_nonneg(&serr, e1);
  __syncthreads();
  if (tid == 0) atomic_max_nonneg(d.err + n, change_out<NO, S>(serr, sp(0) + jc, T, NO));
  // after a timed-out wait, a copy may still be in flight into this CTA's
  // shared memory: wait for it (bounded) before the CTA exits
  if (kInvStage<NO> && tid == 0 && !s_stage) mbar_wait(&cbar, cphase ^ 1u, kCopyWaitPolls);
}

// ---------------------------------------------------------------------------
// Between the two launches of a split sweep: the products of the uncompressed
// rows of Sigma^R with the points the first launch has solved, which no later
// point changes.  In the sweep's own chain they were its longest phases: an
// SM's share of rows read one chunk (lesser) or leaf (retarded) at a time.
// ---------------------------------------------------------------------------
// Retarded: F(t')_ij = sum_{s in [c, T]} w_s y_i(s) Sigma^R(s, t') for t' < c, all
// orbital rows i; 32 columns per CTA (adjacent elements of every row along the
// lanes), the rows s over the 8 warps.
template <int NO, typename S>
__global__ void __launch_bounds__(256) k_ret_ring(Dev d, int T) {
  pdl_start();
  constexpr int NO2 = NO * NO;
  using R = typename Bulk<S>::R;
  using V = typename Val<S>::t;
  const int n = blockIdx.y;
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = d.cdir, k = d.k, nr = T + 1 - c;
  const DevW& W = d.w;
  extern __shared__ __align__(16) char dyn[];
  V* red = reinterpret_cast<V*>(dyn);                           // [8][NO2][32]
  cx<R>* ys = reinterpret_cast<cx<R>*>(red + 8 * NO2 * 32);     // [kRingRows][i][m] y with its weight at the end T
  const S* yrow = el<NO, S>(d.GR, d, n, T, 0);
  for (int e = tid; e < nr * NO2; e += blockDim.x) {
    const int s2 = c + e / NO2;
    const cx<R> v = ldr<R>(yrow + (long long)c * NO2 + e);
    ys[e] = T - s2 <= k ? v * rule_wr<R>(W, T + 2 * k + 1, T - s2) : v;
  }
  __syncthreads();
  const int tp = blockIdx.x * 32 + lane;
  const S* Sr = static_cast<const S*>(d.SR) + ((long long)n * d.ring * d.nt + tp) * NO2;
  const int s0 = c % d.ring;
  KAcc<R> ka[NO2];
  for (int i0 = warp; i0 < nr; i0 += 8 * FOLD) {
    cx<R> pa[NO2];
#pragma unroll
    for (int q = 0; q < NO2; ++q) pa[q] = cx<R>(0);
#pragma unroll
    for (int jj = 0; jj < FOLD; ++jj) {
      const int i = i0 + 8 * jj;
      if (i < nr) {
        int slot = s0 + i;
        if (slot >= d.ring) slot -= d.ring;
        const S* sr = Sr + (long long)slot * d.nt * NO2;
        const int dd = c + i - tp;
        const bool near = dd <= k;
        const R wd = near ? rule_wr<R>(W, 2 * k + 1 + dd, dd) : (R)1;
#pragma unroll
        for (int m = 0; m < NO; ++m)
#pragma unroll
          for (int j = 0; j < NO; ++j) {
            cx<R> sv = ldr<R>(sr + m * NO + j);
            if (near) sv = sv * wd;
#pragma unroll
            for (int x = 0; x < NO; ++x) pa[x * NO + j] = cfma(ys[(i * NO + x) * NO + m], sv, pa[x * NO + j]);
          }
      }
    }
#pragma unroll
    for (int q = 0; q < NO2; ++q) ka[q].add(pa[q]);
  }
#pragma unroll
  for (int q = 0; q < NO2; ++q) red[(warp * NO2 + q) * 32 + lane] = kacc_lanes(ka[q], 32, 32);
  __syncthreads();
  V* fr = reinterpret_cast<V*>(d.fring) + (long long)n * NO * d.nt * NO;
  for (int e = tid; e < 32 * NO2; e += blockDim.x) {   // e: orbital row, column, j
    const int x = e / (32 * NO), tt = (e / NO) % 32, j = e % NO;
    V a[8];
#pragma unroll
    for (int w2 = 0; w2 < 8; ++w2) a[w2] = red[(w2 * NO2 + x * NO + j) * 32 + tt];
#pragma unroll
    for (int s2 = 4; s2; s2 >>= 1)
#pragma unroll
      for (int w2 = 0; w2 < s2; ++w2) a[w2] = vadd(a[w2], a[w2 + s2]);
    fr[((long long)x * d.nt + blockIdx.x * 32 + tt) * NO + j] = a[0];
  }
}

// Lesser: F(t)_mj = sum_{l < c} w^(t)_l Sigma^R(t, l) x_j(l) for the uncompressed
// rows t >= c, all orbital columns j; 4 warps per row.
template <int NO, typename S>
__global__ void __launch_bounds__(256) k_les_ring(Dev d, int T) {
  pdl_start();
  constexpr int NO2 = NO * NO;
  using R = typename Bulk<S>::R;
  using V = typename Val<S>::t;
  const int n = blockIdx.y;
  if (!d.active[n]) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = d.cdir, k = d.k;
  const DevW& W = d.w;
  __shared__ V red[8][NO2];
  const int t = c + blockIdx.x * 2 + (warp >> 2), i = tid & 127;
  const bool row = t <= T;
  const S* sr = el<NO, S>(d.SR, d, n, row ? t : T, 0);
  const S* xr = el<NO, S>(d.GL, d, n, T, 0);
  KAcc<R> ka[NO2];
  for (int l0 = i; row && l0 < c; l0 += 128 * FOLD) {
    cx<R> pa[NO2];
#pragma unroll
    for (int q = 0; q < NO2; ++q) pa[q] = cx<R>(0);
#pragma unroll
    for (int jj = 0; jj < FOLD; ++jj) {
      const int l = l0 + 128 * jj;
      if (l < c) {
        const bool end = l <= k || t - l <= k;
        const R wl = end ? rule_wr<R>(W, t, l) : (R)1;
        cx<R> x[NO2];
#pragma unroll
        for (int q = 0; q < NO2; ++q) {
          x[q] = ldr<R>(xr + (long long)l * NO2 + q);
          if (end) x[q] = x[q] * wl;
        }
#pragma unroll
        for (int m = 0; m < NO; ++m)
#pragma unroll
          for (int y = 0; y < NO; ++y) {
            const cx<R> sv = ldr<R>(sr + (long long)l * NO2 + m * NO + y);
#pragma unroll
            for (int j = 0; j < NO; ++j) pa[m * NO + j] = cfma(sv, x[y * NO + j], pa[m * NO + j]);
          }
      }
    }
#pragma unroll
    for (int q = 0; q < NO2; ++q) ka[q].add(pa[q]);
  }
#pragma unroll
  for (int q = 0; q < NO2; ++q) {
    const V v = kacc_lanes(ka[q], 1, 32);
    if (lane == 0) red[warp][q] = v;
  }
  __syncthreads();
  if (row && i < NO2) {
    const int w0 = warp & 4;
    const V v = vadd(vadd(red[w0][i], red[w0 + 1][i]), vadd(red[w0 + 2][i], red[w0 + 3][i]));
    reinterpret_cast<V*>(d.fring)[((long long)d.n_inst * d.nt + (long long)n * kRingRows + (t - c)) * NO2 + i] = v;
  }
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
// Row s of an inverse: Mi(s, .) from the coefficients crow[m][u N_o + p] =
// A(s,u)_mp, u < s (leading dimension ld_c), the inverse dinv of A(s,s), and the
// rows u < s of Mi (leading dimension ld_m, columns u N_o + p; the first sb rows
// are a full start block).  out(m, col, value) stores.  Every thread calls it.
template <int NO, typename P, typename OUT>
__device__ __forceinline__ void append_row(int s, int sb, const zd* crow, int ld_c, const zd* dinv, const P* Mi, int ld_m,
                                           zd* part, OUT out) {
  constexpr int SL = NO == 1 ? 8 : NO == 2 ? 2 : 1;   // slices of the sum over u
  const int tid = threadIdx.x, nc = s * NO, tps = blockDim.x / SL, slice = tid / tps;
  for (int e = tid % tps; e < NO * nc; e += tps) {
    const int m = e / nc, col = e % nc;
    zd acc = zd();
    for (int u = (col < sb * NO ? 0 : col / NO) + slice; u < s; u += SL)
#pragma unroll
      for (int p = 0; p < NO; ++p) acc = cfma(crow[m * ld_c + u * NO + p], ldr<double>(Mi + (long long)(u * NO + p) * ld_m + col), acc);
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
  pdl_start();
  constexpr int NO2 = NO * NO, LD = CK * NO, NH = 10 * NO;
  const int n = blockIdx.y, sys = blockIdx.x, tid = threadIdx.x;
  if (T > d.last[n]) return;   // the instance has ended
  const int k = d.k;
  const double h = d.h;
  const DevW& W = d.w;
  __shared__ zd part[NO <= 2 ? 256 : CK * NO2];
  __shared__ zd crow[NO * (CK * NO)];
  __shared__ zd dinv[8][NO2], dtmp[8][NO2], diag[8][NO2];
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
      // the start block, and below it the rows s > k up to their diagonal
      Hm[e] = (row < nb ? col < nb : col / NO <= row / NO) ? coef(row / NO + 1, col / NO + 1, row % NO, col % NO) : zd();
    }
    __syncthreads();
    {   // the diagonal blocks' inverses of the rows s > k, a warp each (k <= 5 rows)
      const int w = tid >> 5, l = tid & 31, s = kb + w;
      if (s < hs) {
        if (l < NO2) diag[w][l] = Hm[(s * NO + l / NO) * nh + s * NO + l % NO];
        __syncwarp();
        warp_inv<NO>(diag[w], dtmp[w], dinv[w]);
      }
    }
    gj_inverse(nb, Hm, nh);
    for (int s = kb; s < hs; ++s)
      append_row<NO>(s, kb, Hm + s * NO * nh, nh, dinv[s - kb], Hm, nh, part,
                     [&](int m, int col, const zd& v) { Hm[(s * NO + m) * nh + col] = v; });
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
      if (dd == 0) {
        v -= ld(epsp<NO>(d, n, s) + m * NO + p);
        diag[0][m * NO + p] = v;
      } else {
        crow[m * LD + (u - a) * NO + p] = v;
      }
    }
    __syncthreads();
    if (tid < 32) warp_inv<NO>(diag[0], dtmp[0], dinv[0]);   // (read after append_row's barrier)
    const int sb = sys == 1 && cc == 0 ? k : 0;   // rows of the start block in this chunk: full columns
    append_row<NO>(ri, sb, crow, LD, dinv[0], Mi, LD, part, [&](int m, int col, const zd& v) { put(ri * NO + m, col, v); });
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

// Dynamic shared memory of a sweep: the buffer of the staged inverse and, in
// the compressed form, the projections of the blocks over a leaf, unless ranks
// and levels make them larger than 200 KB in all, or than the kernels' static
// arrays leave room for (4 to 27 KB of them; then they stay in global memory).
template <int NO, typename S>
static size_t sweep_smem(const Dev& d, int* staged) {
  const size_t b = kBufBytes<NO> + (d.ring ? SweepMem<NO, typename Bulk<S>::R>::bytes(d.maxl, d.rmax) : 0);
  const bool off32 = std::max(d.utot, d.vtot) * d.rmax < (1ll << 32);
  *staged = (d.ring && b <= std::min<size_t>(200 * 1024, d.sweep_room) && off32) ? 1 : 0;
  return *staged ? b : kBufBytes<NO>;
}
// In small batches the retarded sweep and the mixed component, in small node
// groups, are one launch: the sweep is a chain on a few SMs, and the nodes need
// the others.  In FP64 up to a CTA per SM (3 instances, T = 256: 97.0 -> 91.6 ms
// a pass); beyond that the nodes hold FP64 pipes that the sweeps wait for (20 x
// 150: 40.4 -> 41.9; N_o = 2, 10 x 150: 40.1 -> 44.5).  In complex64 up to four
// (60 x 150: 22.4 -> 20.9; N_o = 4, 16 x 290: 111.3 -> 108.1); large batches fill
// the SMs in large groups (N_o = 2, 128 x 600: 158 -> 179 in one launch).
bool ret_takes_mixed(const Dev& d) {
  const int ni = d.no == 1 ? kNodesFew<1> : d.no == 2 ? kNodesFew<2> : kNodesFew<3>;
  return (long long)(d.no + (d.r + ni - 1) / ni) * d.n_inst <= (d.prec ? 4 : 1) * kSMs;
}
// A sweep runs as two launches with its ring kernel between them once kSplitRows
// rows are compressed: before that, the ring's products in the chain cost less
// than two more launches (complex64, T = 150, 64 to 128 rows: 4.4 -> 4.8 ms of
// lesser sweeps in 49 steps).  From there on, the lesser sweep: 35 -> 31 ms (128
// instances, N_o = 2, T = 600), 43.5 -> 38.4 (1, FP64, T = 384).  The retarded
// sweep, whose ring phases are shorter, gains only while its CTAs leave SMs
// idle: 43 -> 36 ms (1, FP64, T = 384), but 19.7 -> 21.6 (304, complex64).
static bool split_les(const Dev& d) { return d.cdir >= kSplitRows; }
static bool split_ret(const Dev& d) { return d.cdir >= kSplitRows && d.no * d.n_inst <= kSMs; }
int ret_launches(const Dev& d) { return split_ret(d) ? 3 : 1; }
int les_launches(const Dev& d) { return split_les(d) ? 3 : 1; }
// A sweep comes early (see pdl_start) in the dense form with up to four CTAs: 1 x
// 64, FP64, 10.7 -> 10.2 ms; 3 x 256 91.5 -> 90.8; 4 x 200 58.6 -> 57.6. Compressed
// forms gain nothing there (4 x 300, FP64, 55.9 -> 56.6), and more CTAs end up two
// to an SM next to the kernel before them (N_o = 2, 8 x 300, FP64, 79.8 -> 112.8).
static bool early_sweep(const Dev& d) { return !d.ring && d.no * d.n_inst <= 4; }
template <int NO, typename S>
static cudaError_t sweep_ret(const Dev& d, int T, cudaStream_t s) {
  int staged = 0;
  const size_t bytes = sweep_smem<NO, S>(d, &staged);
  const bool with = ret_takes_mixed(d);
  auto kern = with ? k_ret2<NO, S, true> : k_ret2<NO, S, false>;
  cudaError_t e;
  if (d.ring && T + 1 - d.cdir > kRingRows && d.cdir > 0) return cudaErrorInvalidValue;
  const int mix = with ? (d.r + kNodesFew<NO> - 1) / kNodesFew<NO> : 0;
  const bool split = split_ret(d);
  if ((e = launch_on(early_sweep(d), kern, dim3(NO + mix, d.n_inst), 256, bytes, s, d, T, staged, split ? (int)kTop : (int)kAll)) !=
          cudaSuccess ||
      !split)
    return e;
  const size_t rb = NO * NO * (8 * 32 * 16 + kRingRows * sizeof(S));
  if ((e = launch_k(k_ret_ring<NO, S>, dim3(d.cdir / 32, d.n_inst), 256, rb, s, d, T)) != cudaSuccess) return e;
  return launch_on(early_sweep(d), k_ret2<NO, S, false>, dim3(NO, d.n_inst), 256, bytes, s, d, T, staged, (int)kLeaves);
}
template <int NO, typename S>
static cudaError_t sweep_les(const Dev& d, int T, cudaStream_t s) {
  int staged = 0;
  const size_t bytes = sweep_smem<NO, S>(d, &staged);
  cudaError_t e;
  const bool split = split_les(d);
  const int rows = T + 1 - d.cdir;
  if (split && rows > kRingRows) return cudaErrorInvalidValue;
  if ((e = launch_on(early_sweep(d), k_les2<NO, S>, dim3(NO, d.n_inst), 256, bytes, s, d, T, staged,
                     split ? (int)kLeaves : (int)kAll)) != cudaSuccess ||
      !split)
    return e;
  if ((e = launch_k(k_les_ring<NO, S>, dim3((rows + 1) / 2, d.n_inst), 256, 0, s, d, T)) != cudaSuccess) return e;
  return launch_on(early_sweep(d), k_les2<NO, S>, dim3(NO, d.n_inst), 256, bytes, s, d, T, staged, (int)kTop);
}
cudaError_t open_sweeps(Dev& d) {
  cudaError_t e = cudaErrorInvalidValue;
  int ring = 1 << 30;
  d.sweep_room = 1 << 30;
  HK_DISPATCH(d.no, {
    if ((e = open_smem(k_ret2<NO, S, true>, &d.sweep_room)) == cudaSuccess &&
        (e = open_smem(k_ret2<NO, S, false>, &d.sweep_room)) == cudaSuccess &&
        (e = open_smem(k_les2<NO, S>, &d.sweep_room)) == cudaSuccess)
      e = open_smem(k_ret_ring<NO, S>, &ring);
  })
  return e;
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
  HK_DISPATCH(d.no, return launch_k(k_inv_rows<NO, S>, dim3(3, d.n_inst), 256, 0, s, d, T, r0, r1, l0, l1));
  return cudaSuccess;
}

}  // namespace hk
