// Ragged batch of independent LPs solved by r^2HPDHG (Algorithm 1) in ONE
// persistent kernel launch.
//
// The paper batches same-shape instances by vectorising the solver (Sec. 3.2).
// Here instances may differ in size: they are packed back to back as one
// block-diagonal problem, so the device transpose and the Ruiz/Pock-Chambolle
// scaling (row- and column-local operations) of the single-problem path apply
// unchanged.  The iteration itself runs in one launch: each CTA takes the next
// unsolved instance from an atomic work counter and runs the whole restarted
// loop for it -- power iteration, initial primal weight, half-steps, relative
// KKT checks, restarts, primal-weight updates, termination -- with the two
// gathered vectors of the instance (y for the SpMV^T, the reflected primal point
// for the SpMV) held in shared memory, or, for an instance too large for that,
// in global memory (the same code through generic pointers).  All reductions are fixed-order CTA
// trees in FP64; no instance waits on another, so no grid-wide synchronisation
// exists and a finished CTA simply takes the next instance.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/mpax.h"
#include "batch_work.h"
#include "problem.cuh"

namespace mpax {

// Threads of the CTA that solves one instance.  FP64: 512 at 128 registers, one CTA per SM
// (300 instances of 50 to 2,000 rows 33 ms; two CTAs of 512 at 64 registers, which spill,
// 40 ms).  FP32: one CTA of 1024 at 64 registers, or two of 512 where there are more
// instances than such CTAs and they are small, at most kSmallCols columns on average and
// kSmallVec rows and columns each: their slices of 32 rows leave many of 32 warps idle.
// Measured, 640 iterations, 1024 / 2 x 512 threads: 2,000 instances of 320 columns on average
// 27.3 / 17.7 ms, 1,500 of 900 38.7 / 32.3, 1,000 of 1,200 34.9 / 31.1; in whole solves 2,000 of
// 2,050 56 / 71 and 100 of 620 3.2 / 3.7.
template <typename T>
constexpr int kBatchThreads = sizeof(T) == 4 ? 1024 : 512;
constexpr int kBatchSmallThreads = 512;
constexpr int kSmallCols = 1400;
constexpr int kSmallVec = 25000;  // rows + columns: the vectors of two CTAs fit in one SM
constexpr double kBatchMaxSeconds = 600.0;
// Partial sums of a row: entries 0, 2, 4, ... and 1, 3, 5, ..., added at the end.  In CSR
// (RowsCsr) two lanes hold them.  Rows of the batch recipe hold ~1-40 nonzeros: measured on 4096 instances, 2 lanes per
// row (0.325 s per batch mixed, 0.450 s FP64) beat 8 (0.490 / 0.956 s) and 1
// (0.521 / 0.597 s) -- with 8 lanes a row's shuffle reduction and its one-lane
// epilogue cost more than its two or three loads per lane.
constexpr int kLPR = 2;
// Iterations whose Halpern weights the CTA forms at a time.  A double-precision division
// takes tens of instructions, each 16 cycles of the SM's FP64 pipe per warp, so the
// weights are formed by one warp or two for 64 iterations and not by every thread in
// each (512 ragged LPs, FP32: the launch 38.4 -> 35.2 ms together with reciprocal
// scaling factors in the checks; 64 grid LPs in FP64: an iteration 13.3 -> 11.9 us).
constexpr int kCoefs = 64;

template <typename T>
struct BatchArgs {
  int B;
  const long long* m_off;
  const long long* n_off;
  const int* rp;      // A (block diagonal, global columns)
  const int* col;
  const T* val;
  const int* rpt;     // A^T (columns are global rows of A)
  const int* colt;
  const T* valt;
  const T *c, *l, *u, *lc, *uc;                 // scaled data
  const double *c0, *l0, *u0, *lc0, *uc0, *Dr, *Dc, *iDr, *iDc;  // originals, scaling, inverses
  T *w, *xa, *xhat, *ya, *yhat, *gbuf;          // iterate storage
  double *xout, *yout;
  int* status;
  long long* iters;
  long long* restarts;
  double *relkkt, *pobj, *secs;
  int* next;
  // Rows by length (k_sort_rows): the vectors and scaled data of an instance lie in its
  // sorted order; permm / permn give the original (local) index.  An instance whose zs
  // range is empty keeps the original order and the CSR arrays above.
  const int *permm, *permn;
  const unsigned short *lenm, *lenn;   // row lengths, sorted order
  const int *soffm, *soffn;            // slice offsets; instance b's start at slice_base
  const long long *zsa, *zst;          // B + 1: storage of the sorted matrices
  const T *sval, *svalt;
  const unsigned short *scol, *scolt;  // sorted local indices of the gathered vector
  // Shared-memory pool of a CTA: smem_vec elements for the instance's two
  // gathered vectors (y, m_b entries, then the primal vector, n_b entries).  An instance
  // with m_b + n_b > smem_vec keeps both vectors in global memory instead (gys, gxs: its
  // slices of two m- and n-vectors).
  int smem_vec;
  T* gys;
  T* gxs;
  double eps_abs, eps_rel, r_suff, r_nec, r_art, pw_smooth, step_safety, power_tol;
  long long iter_limit;
  long long time_limit_ns;  // from the start of the launch, on the device clock
  int check_every, power_max_iter;
  const int* todo;  // instances of this launch (nullptr: all B, in order)
  int n_todo;       // work items of this launch
  int warm;         // 1: start from the returned points (xout, yout) instead of zero
  double power_cap; // certified bound on ||A~_b||_2 (1 after Pock-Chambolle, else inf)
  int stall_limit;  // > 0: end an instance whose KKT error stops improving (FP32 floor)
  long long stage_cap;  // bytes of the shared pool an instance may stage whole (0: none)
};

// A thread's share of a sum over an instance.  The order of the sum is that of a CTA of
// kBatchThreads threads whatever the launch: with half of them (kFold = 2) a thread keeps the
// shares of two, so an instance's result does not depend on the batch it is in.
template <int kFold>
struct Share {
  double v[kFold] = {};
  // x of the item that this thread takes in its pass number `pass`
  __device__ __forceinline__ void add(int pass, double x) {
    if constexpr (kFold == 1) {
      v[0] += x;
    } else {
      if (pass & 1) v[1] += x;
      else v[0] += x;
    }
  }
};

// The sum over the block, to every thread.  Warps without a share skip theirs: a step of the
// tree takes the FP64 pipe 16 cycles a warp.
template <int kFold>
__device__ __forceinline__ double bsum(const Share<kFold>& s, double* sh) {
  __shared__ double bc;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, warps = blockDim.x >> 5;
  double part[kFold];
#pragma unroll
  for (int f = 0; f < kFold; ++f) {
    const bool any = __any_sync(0xffffffffu, __double_as_longlong(s.v[f]) != 0);
    part[f] = any ? warp_sum(s.v[f]) : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int f = 0; f < kFold; ++f)
    if (lane == 0) sh[w + f * warps] = part[f];
  __syncthreads();
  if (w == 0) {
    const double v = warp_sum(lane < kFold * warps ? sh[lane] : 0.0);
    if (lane == 0) bc = v;
  }
  __syncthreads();
  return bc;
}

template <typename T>
__device__ __forceinline__ T group_sum(T v) {
#pragma unroll
  for (int o = kLPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, kLPR);
  return v;
}

__device__ __forceinline__ double bound_val(double lo, double hi) {
  const bool fl = isfinite(lo), fu = isfinite(hi);
  if (fl && fu) return (fabs(lo) >= fabs(hi)) ? lo : hi;
  if (fl) return lo;
  if (fu) return hi;
  return 0.0;
}

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---- the rows of one matrix of an instance ----------------------------------------
// each(vec, pre, row): for every row i, s = the row times vec; pre(i) is called before the
// row's loads (it returns the operands of row's epilogue, which travel with them) and
// row(i, s, operands) on one thread after.

// CSR, two lanes per row: for instances whose vectors do not fit in shared memory or
// whose rows are too uneven to sort.
template <typename T>
struct RowsCsr {
  int rows;
  const int* rp;
  const T* val;
  const int* col;
  int off;  // columns are global: less off
  template <class Pre, class Row>
  __device__ __forceinline__ void each(const T* vec, Pre pre, Row row) const {
    const int grp = threadIdx.x / kLPR, gl = threadIdx.x % kLPR;
    const int G = blockDim.x / kLPR;
    for (int i0 = 0; i0 < rows; i0 += G) {
      const int i = i0 + grp;
      const bool in = i < rows;
      const int pe = in ? rp[i + 1] : 0;
      decltype(pre(0)) q{};
      if (gl == 0 && in) q = pre(i);
      T s = 0;
      for (int p = in ? rp[i] + gl : 0; p < pe; p += kLPR) s += val[p] * vec[col[p] - off];
      s = group_sum(s);
      if (gl == 0 && in) row(i, s, q);
    }
  }
};

// Rows sorted by length, longest first, in slices of 32 stored entry-major: a thread per
// row, so that a warp's loads of values and 16-bit columns are consecutive, its epilogues
// use every lane (an FP64 instruction costs the same 16 cycles for one lane as for 32)
// and rows of a warp end together.  In CSR with two lanes per row a warp load touched
// 16 rows' sectors and every second lane idled in the epilogue: 2.7 warp instructions per
// nonzero and pass.  The sums are the same: even and odd entries, then their sum.
// What bounds it now: the round trips to L2 of a row's eight entries at a time (4 in
// flight: 1% slower), in FP64 the FP64 pipe.  Whole solves, CSR -> sorted:
// 512 LPs of 50 to 2,000 rows 45 -> 19 ms in FP32, 300 of them 85 -> 33 ms in FP64; 64 grid
// LPs of 144 rows staged in shared memory 6.8 -> 5.1 ms in FP64.
template <typename T>
struct RowsSorted {
  int rows;
  const int* soff;
  const unsigned short* len;
  const T* val;
  const unsigned short* col;
  template <class Pre, class Row>
  __device__ __forceinline__ void each(const T* vec, Pre pre, Row row) const {
    const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
    for (int sl = threadIdx.x >> 5; sl * 32 < rows; sl += W) {
      const int i = sl * 32 + lane;
      const bool in = i < rows;
      const int o = soff[sl], w = (soff[sl + 1] - o) >> 5;
      const int n = in ? (int)len[i] : 0;
      decltype(pre(0)) q{};
      if (in) q = pre(i);
      const T* v = val + o + lane;
      const unsigned short* c = col + o + lane;
      T e = 0, d = 0;
      constexpr int U = 8;  // entries in flight (padded entries are zeros of column 0)
      int t = 0;
      for (; t + U <= w; t += U) {
        T x[U];
        int k[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          x[u] = v[(t + u) * 32];
          k[u] = c[(t + u) * 32];
        }
#pragma unroll
        for (int u = 0; u < U; u += 2) {
          const T ge = vec[k[u]], go = vec[k[u + 1]];
          if (t + u < n) e += x[u] * ge;
          if (t + u + 1 < n) d += x[u + 1] * go;
        }
      }
      for (; t < w; t += 2) {
        const T x0 = v[t * 32], ge = vec[c[t * 32]];
        if (t < n) e += x0 * ge;
        if (t + 1 < w) {
          const T x1 = v[(t + 1) * 32], go = vec[c[(t + 1) * 32]];
          if (t + 1 < n) d += x1 * go;
        }
      }
      if (in) row(i, e + d, q);
    }
  }
};

// Slices of k rows; first slice offset of an instance whose rows start at r0 (every
// instance has one entry more than slices).
__host__ __device__ __forceinline__ int n_slices(int k) { return (k + 31) / 32; }
__host__ __device__ __forceinline__ long long slice_base(long long r0, int b) {
  return r0 / 32 + 2LL * b;
}

// Shared-memory pool of an instance run with kStage (T elements, ints, then 16-bit):
// ys[mb] xs[nb] val[za] valt[zt] c l u w xa xhat gbuf [nb each] lc uc ya yhat [mb each]
// | soffm[slices + 1] soffn[slices + 1] | col[za] colt[zt] lenm[mb] lenn[nb], za and zt the
// stored entries of the sorted matrices.
__host__ __device__ __forceinline__ long long stage_bytes(long long mb, long long nb, long long za,
                                                          long long zt, int tsize) {
  return tsize * (5 * mb + 8 * nb + za + zt) + 4 * (n_slices((int)mb) + n_slices((int)nb) + 2) +
         2 * (za + zt + mb + nb);
}

// The vectors of one instance as the loop reads them, indexed locally in the instance's
// row order.  In place, every array is the kernel parameter's pointer plus the instance
// offset (no register holds it); staged, it is the pool position that mb, nb and the
// matrix sizes fix.
template <typename T, bool kStage>
struct Inst {
  const BatchArgs<T>& a;
  int m0, n0, mb, nb;
  T* sp;  // staged: the pool after the matrices
#define MPAX_INST_ARR(Type, name, staged, inplace) \
  __device__ __forceinline__ Type* name() const {    \
    if constexpr (kStage) return staged;             \
    else return inplace;                             \
  }
  MPAX_INST_ARR(const T, c, sp, a.c + n0)
  MPAX_INST_ARR(const T, l, sp + nb, a.l + n0)
  MPAX_INST_ARR(const T, u, sp + 2 * nb, a.u + n0)
  MPAX_INST_ARR(T, w, sp + 3 * nb, a.w + n0)
  MPAX_INST_ARR(T, xa, sp + 4 * nb, a.xa + n0)
  MPAX_INST_ARR(T, xhat, sp + 5 * nb, a.xhat + n0)
  MPAX_INST_ARR(T, gbuf, sp + 6 * nb, a.gbuf + n0)
  MPAX_INST_ARR(const T, lc, sp + 7 * nb, a.lc + m0)
  MPAX_INST_ARR(const T, uc, sp + 7 * nb + mb, a.uc + m0)
  MPAX_INST_ARR(T, ya, sp + 7 * nb + 2 * mb, a.ya + m0)
  MPAX_INST_ARR(T, yhat, sp + 7 * nb + 3 * mb, a.yhat + m0)
#undef MPAX_INST_ARR
};

// kStage: the whole instance -- both matrices, the scaled data and every
// iterate vector -- is copied into the shared pool first, so the loop touches
// global memory only at checks (the unscaled data) and at the end.  Otherwise
// the two gathered vectors sit at ys, xs (shared or global) and the rest is
// read in place.  kSorted: rows by length (RowsSorted), else CSR.  kFold: see Share.
template <typename T, bool kStage, bool kSorted, int kFold>
__device__ __forceinline__ void solve_instance(const BatchArgs<T>& a, int b, T* ys, T* xs,
                                               double* sh, unsigned long long t_launch) {
  static_assert(kSorted || !kStage, "only sorted instances are staged");
  const unsigned long long t_start = gtimer();
  __shared__ int s_late;
  __shared__ T s_coef[kCoefs + 1];
  const int m0 = (int)a.m_off[b], mb = (int)(a.m_off[b + 1] - a.m_off[b]);
  const int n0 = (int)a.n_off[b], nb = (int)(a.n_off[b + 1] - a.n_off[b]);
  const long long za0 = a.zsa[b], zt0 = a.zst[b];
  const int za = (int)(a.zsa[b + 1] - za0), zt = (int)(a.zst[b + 1] - zt0);
  Inst<T, kStage> v{a, m0, n0, mb, nb, xs + nb + za + zt};
  using Rows = std::conditional_t<kSorted, RowsSorted<T>, RowsCsr<T>>;
  Rows A, At;
  if constexpr (kSorted) {
    A = Rows{mb, a.soffm + slice_base(m0, b), a.lenm + m0, a.sval + za0, a.scol + za0};
    At = Rows{nb, a.soffn + slice_base(n0, b), a.lenn + n0, a.svalt + zt0, a.scolt + zt0};
  } else {
    A = Rows{mb, a.rp + m0, a.val, a.col, n0};
    At = Rows{nb, a.rpt + n0, a.valt, a.colt, m0};
  }
  if constexpr (kStage) {
    // ys (the pool's start) and xs = ys + mb come first; copy the rest in
    T* sval = xs + nb;
    T* svalt = sval + za;
    int* sm = reinterpret_cast<int*>(v.sp + 7 * nb + 4 * mb);
    int* sn = sm + n_slices(mb) + 1;
    unsigned short* scol = reinterpret_cast<unsigned short*>(sn + n_slices(nb) + 1);
    unsigned short* scolt = scol + za;
    unsigned short* slm = scolt + zt;
    unsigned short* sln = slm + mb;
    for (int i = threadIdx.x; i <= n_slices(mb); i += blockDim.x) sm[i] = A.soff[i];
    for (int j = threadIdx.x; j <= n_slices(nb); j += blockDim.x) sn[j] = At.soff[j];
    for (int p = threadIdx.x; p < za; p += blockDim.x) {
      sval[p] = A.val[p];
      scol[p] = A.col[p];
    }
    for (int p = threadIdx.x; p < zt; p += blockDim.x) {
      svalt[p] = At.val[p];
      scolt[p] = At.col[p];
    }
    T* sc = const_cast<T*>(v.c());
    T* sl = const_cast<T*>(v.l());
    T* su = const_cast<T*>(v.u());
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
      sc[j] = a.c[n0 + j];
      sl[j] = a.l[n0 + j];
      su[j] = a.u[n0 + j];
      sln[j] = At.len[j];
    }
    T* slc = const_cast<T*>(v.lc());
    T* suc = const_cast<T*>(v.uc());
    for (int i = threadIdx.x; i < mb; i += blockDim.x) {
      slc[i] = a.lc[m0 + i];
      suc[i] = a.uc[m0 + i];
      slm[i] = A.len[i];
    }
    __syncthreads();
    A = Rows{mb, sm, slm, sval, scol};
    At = Rows{nb, sn, sln, svalt, scolt};
  }
  // original (global) row and column of a place in the instance's order
  auto row_of = [&](int i) { return m0 + (kSorted ? a.permm[m0 + i] : i); };
  auto col_of = [&](int j) { return n0 + (kSorted ? a.permn[n0 + j] : j); };
  auto none = [](int) { return 0; };
  // a product of the scaled matrix in the unscaled space: one rounding in FP64; a product of
  // FP32 sums takes the stored reciprocal, whose rounding lies 2^29 below theirs
  auto unscale = [](double s, double d, double inv) {
    if constexpr (sizeof(T) == 8) return s / d;
    else return s * inv;
  };
  // the pass in which a thread meets coordinate i in a loop over the block, and row i in each()
  constexpr int kT = kBatchThreads<T> / kFold;
  auto pass = [](int i) { return i / kT; };
  auto row_pass = [](int i) { return i / (kSorted ? kT : kT / kLPR); };
  const bool has_rows = a.rp[m0 + mb] > a.rp[m0];

  // ---- power iteration for ||A~_b||_2 from the common start vector ----------
  Share<kFold> ss0;
  for (int j = threadIdx.x; j < nb; j += blockDim.x) {
    const double r = power_start_raw(j);
    ss0.add(pass(j), r * r);
  }
  const double inv0 = 1.0 / sqrt(fmax(bsum(ss0, sh), 1e-300));
  for (int j = threadIdx.x; j < nb; j += blockDim.x)
    xs[j] = (T)(power_start_raw(col_of(j) - n0) * inv0);
  __syncthreads();
  double nA = 0.0, nu_prev = 0.0, d_prev = 0.0;
  if (has_rows && a.power_max_iter == 0) nA = a.power_cap;  // the certified bound
  for (int t = 1; has_rows && t <= a.power_max_iter; ++t) {
    A.each(xs, none, [&](int i, T s, int) { ys[i] = s; });
    __syncthreads();
    Share<kFold> acc;
    At.each(ys, none, [&](int j, T s, int) {
      v.gbuf()[j] = s;
      acc.add(row_pass(j), (double)s * (double)s);
    });
    const double nrm = sqrt(bsum(acc, sh));
    if (nrm == 0.0) {
      nA = 0.0;
      break;
    }
    const double nu = sqrt(nrm);
    for (int j = threadIdx.x; j < nb; j += blockDim.x) xs[j] = (T)((double)v.gbuf()[j] / nrm);
    __syncthreads();
    nA = nu;
    double est = nu;
    if (t > 1 && power_stop(nu, nu_prev, &d_prev, a.power_tol, a.power_cap, &est)) {
      nA = est;
      break;
    }
    if (t == a.power_max_iter && isfinite(a.power_cap)) nA = a.power_cap;
    nu_prev = nu;
  }

  // ---- initial primal weight, norms of the unscaled data ------------------
  Share<kFold> s_cs, s_bs, s_c, s_b;
  for (int j = threadIdx.x; j < nb; j += blockDim.x) {
    const double cs = (double)v.c()[j];
    s_cs.add(pass(j), cs * cs);
    s_c.add(pass(j), a.c0[n0 + j] * a.c0[n0 + j]);
  }
  for (int i = threadIdx.x; i < mb; i += blockDim.x) {
    const double bs = bound_val((double)v.lc()[i], (double)v.uc()[i]);
    const double bo = bound_val(a.lc0[m0 + i], a.uc0[m0 + i]);
    s_bs.add(pass(i), bs * bs);
    s_b.add(pass(i), bo * bo);
  }
  const double ncs = sqrt(bsum(s_cs, sh)), nbs = sqrt(bsum(s_bs, sh));
  const double c_norm = sqrt(bsum(s_c, sh)), b_norm = sqrt(bsum(s_b, sh));
  double omega = (ncs > 1e-10 && nbs > 1e-10) ? ncs / nbs : 1.0;
  const double eta = nA > 0.0 ? a.step_safety / nA : 1.0;
  double tau = eta / omega, sigma = eta * omega;

  // ---- start at zero, or (warm) at the returned point of an earlier launch,
  // taken back into the scaled space: anchor, reflected point, duals ---------
  for (int j = threadIdx.x; j < nb; j += blockDim.x) {
    const T x = a.warm ? (T)(a.xout[col_of(j)] / a.Dc[col_of(j)]) : (T)0;
    v.xa()[j] = x;
    v.w()[j] = x;
    v.xhat()[j] = x;
  }
  for (int i = threadIdx.x; i < mb; i += blockDim.x) {
    const T y = a.warm ? (T)(a.yout[row_of(i)] / a.Dr[row_of(i)]) : (T)0;
    ys[i] = y;
    v.ya()[i] = y;
    v.yhat()[i] = y;
  }
  __syncthreads();

  long long total = 0, k = 0, restarts = 0;
  double r_anchor = 0.0, r_prev = 0.0, rel = INFINITY, pobj = 0.0;
  bool have_anchor = false;
  int term = 0;
  long long checks = 0, stall_count = 0;
  double best_rel = INFINITY;
  while (true) {
    const int len = (int)min((long long)a.check_every, a.iter_limit - total);
    const T tt = (T)tau, ss = (T)sigma, iss = (T)(1.0 / sigma);
    // Iteration `it` of the block.  The last one, which the check follows, is code of its own:
    // the sums of the restart rule take registers that the others' loads need.
    struct Sums {
      Share<kFold> p0, p1, q0, q1;  // columns, then rows
    };
    auto iterate = [&](int it, auto last, Sums& sq) {
      constexpr bool chk = decltype(last)::value;
      // weights 1/(k+1) and 1/(k+2) of this and the next iterations
      if (it % kCoefs == 0) {
        if (threadIdx.x <= min(kCoefs, len - it)) s_coef[threadIdx.x] = (T)(1.0 / (double)(k + 1 + threadIdx.x));
        __syncthreads();
      }
      const T rb = s_coef[it % kCoefs];      // rebuild weight of x^{n,k}
      const T hb = s_coef[it % kCoefs + 1];  // Halpern weight of the anchor
      // primal half-step over the rows of A^T (eq. 3, first line)
      struct Col {
        T x0, w, c, l, u;
      };
      At.each(
          ys, [&](int j) { return Col{v.xa()[j], v.w()[j], v.c()[j], v.l()[j], v.u()[j]}; },
          [&](int j, T s, const Col& q) {
            const T x = (k == 0) ? q.x0 : q.w + rb * (q.x0 - q.w);
            const T xh = clampv<T>(x - tt * (q.c - s), q.l, q.u);
            const T wn = (T)2 * xh - x;
            v.w()[j] = wn;
            xs[j] = wn;
            if constexpr (chk) {
              v.xhat()[j] = xh;
              const double d0 = (double)xh - (double)x, d1 = (double)xh - (double)q.x0;
              sq.p0.add(row_pass(j), d0 * d0);
              sq.p1.add(row_pass(j), d1 * d1);
            }
          });
      __syncthreads();
      // dual half-step over the rows of A (eq. 3, second line) and Halpern (eq. 4)
      struct Row {
        T ya, lc, uc;
      };
      A.each(
          xs, [&](int i) { return Row{v.ya()[i], v.lc()[i], v.uc()[i]}; },
          [&](int i, T s, const Row& q) {
            const T y0 = ys[i];
            const T t = y0 * iss - s;
            const T yh = ss * (t - clampv<T>(t, -q.uc, -q.lc));
            const T z = (T)2 * yh - y0;
            ys[i] = z + hb * (q.ya - z);
            if constexpr (chk) {
              v.yhat()[i] = yh;
              const double d0 = (double)yh - (double)y0, d1 = (double)yh - (double)q.ya;
              sq.q0.add(row_pass(i), d0 * d0);
              sq.q1.add(row_pass(i), d1 * d1);
            }
          });
      __syncthreads();
      ++k;
      ++total;
    };
    Sums sq;
    for (int it = 0; it + 1 < len; ++it) iterate(it, std::false_type{}, sq);
    if (len > 0) iterate(len - 1, std::true_type{}, sq);
    const double P0 = bsum(sq.p0, sh), P1 = bsum(sq.p1, sh);
    const double D0 = bsum(sq.q0, sh), D1 = bsum(sq.q1, sh);
    // ---- check: relative KKT error of (x^, y^) on the unscaled problem ----
    for (int j = threadIdx.x; j < nb; j += blockDim.x) xs[j] = v.xhat()[j];
    __syncthreads();
    Share<kFold> r0, r1;
    A.each(xs, none, [&](int i, T s, int) {
      const int g = row_of(i);
      const double ax = unscale((double)s, a.Dr[g], a.iDr[g]);
      const double lo = a.lc0[g], hi = a.uc0[g];
      const double r = ax - fmin(fmax(ax, lo), hi);
      r0.add(row_pass(i), r * r);
      const double y = a.Dr[g] * (double)v.yhat()[i];
      if (y > 0.0 && isfinite(lo)) r1.add(row_pass(i), lo * y);
      if (y < 0.0 && isfinite(hi)) r1.add(row_pass(i), hi * y);
    });
    const double K0 = bsum(r0, sh), K1 = bsum(r1, sh);
    Share<kFold> c0, c1, c2;
    At.each(v.yhat(), none, [&](int j, T s, int) {
      const int g = col_of(j);
      const double aty = unscale((double)s, a.Dc[g], a.iDc[g]);
      const double x = a.Dc[g] * (double)xs[j];
      const double lam = a.c0[g] - aty;
      const double lo = a.l0[g], hi = a.u0[g];
      const bool lf = isfinite(lo), uf = isfinite(hi);
      const double lh = (lf && uf) ? lam : lf ? fmax(lam, 0.0) : uf ? fmin(lam, 0.0) : 0.0;
      const double rd = lam - lh;
      c0.add(row_pass(j), rd * rd);
      c1.add(row_pass(j), a.c0[g] * x);
      c2.add(row_pass(j), (lf ? lo * fmax(lh, 0.0) : 0.0) + (uf ? hi * fmin(lh, 0.0) : 0.0));
    });
    const double C0 = bsum(c0, sh), C1 = bsum(c1, sh), C2 = bsum(c2, sh);
    const double nrp = sqrt(K0), nrd = sqrt(C0);
    pobj = C1;
    const double dobj = K1 + C2;
    const double gap = fabs(pobj - dobj);
    rel = fmax(fmax(nrp / (1.0 + b_norm), nrd / (1.0 + c_norm)),
               gap / (1.0 + fabs(pobj) + fabs(dobj)));
    const bool conv = nrp <= a.eps_abs + a.eps_rel * b_norm &&
                      nrd <= a.eps_abs + a.eps_rel * c_norm &&
                      gap <= a.eps_abs + a.eps_rel * (fabs(pobj) + fabs(dobj));
    if (!isfinite(rel) || !isfinite(P0) || !isfinite(D0)) term = MPAX_TERM_NUMERICAL_ERROR;
    else if (conv) term = MPAX_TERM_OPTIMAL;
    else if (total >= a.iter_limit) term = MPAX_TERM_ITERATION_LIMIT;
    // one thread reads the clock so that the decision is uniform over the block
    if (threadIdx.x == 0) s_late = (long long)(gtimer() - t_launch) >= a.time_limit_ns;
    __syncthreads();
    if (!term && s_late) term = MPAX_TERM_TIME_LIMIT;
    __syncthreads();
    // the FP32 floor: no 10% improvement of the KKT error over stall_limit
    // checks.  Unlike the single-problem rule the window does not grow: a batch
    // instance is small and latency-bound, FP64 costs it about twice per
    // iteration, and an FP32 run that keeps finding slightly lower minima while
    // it drifts would otherwise run on.  Every quantity here is uniform over the
    // block.
    ++checks;
    if (!term && a.stall_limit > 0) {
      const long long window = a.stall_limit;
      if (rel < 0.9 * best_rel) {
        best_rel = rel;
        stall_count = 0;
      } else if (++stall_count >= window) {
        term = kTermStalled;
      }
    }
    if (term) break;
    // restart rule and primal weight (the same rule as the single-problem path)
    const double r = sqrt(omega * P0 + D0 / omega);
    const bool restart = !have_anchor || r <= a.r_suff * r_anchor ||
                         (r <= a.r_nec * r_anchor && r > r_prev) ||
                         (double)k >= a.r_art * (double)total;
    if (restart) {
      const double dx = sqrt(P1), dy = sqrt(D1);
      if (dx > 1e-10 && dy > 1e-10)
        omega = exp(a.pw_smooth * log(dy / dx) + (1.0 - a.pw_smooth) * log(omega));
      tau = eta / omega;
      sigma = eta * omega;
      have_anchor = true;
      r_anchor = r;
      r_prev = r;
      k = 0;
      ++restarts;
      for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const T x = v.xhat()[j];
        v.xa()[j] = x;
        v.w()[j] = x;
      }
      for (int i = threadIdx.x; i < mb; i += blockDim.x) {
        const T y = v.yhat()[i];
        v.ya()[i] = y;
        ys[i] = y;
      }
    } else {
      r_prev = r;
    }
    __syncthreads();
  }
  // ---- returned point (x^, y^), unscaled; per-instance statistics ---------
  for (int j = threadIdx.x; j < nb; j += blockDim.x)
    a.xout[col_of(j)] = a.Dc[col_of(j)] * (double)v.xhat()[j];
  for (int i = threadIdx.x; i < mb; i += blockDim.x)
    a.yout[row_of(i)] = a.Dr[row_of(i)] * (double)v.yhat()[i];
  if (threadIdx.x == 0) {
    // a warm launch continues an instance: its counts and time add to the earlier ones
    a.status[b] = term;
    a.iters[b] = (a.warm ? a.iters[b] : 0) + total;
    a.restarts[b] = (a.warm ? a.restarts[b] : 0) + restarts;
    a.relkkt[b] = rel;
    a.pobj[b] = pobj;
    a.secs[b] = (a.warm ? a.secs[b] : 0.0) + (double)(gtimer() - t_start) * 1e-9;
  }
  __syncthreads();
}

// kStaging: the launch may stage whole instances (a separate instantiation, so
// that the many-instance kernel carries only the two in-place call sites).
template <typename T, bool kStaging, int kThreads>
__global__ void __launch_bounds__(kThreads, kBatchThreads<T> / kThreads)
    batch_lp_kernel(BatchArgs<T> a) {
  constexpr int kFold = kBatchThreads<T> / kThreads;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ double sh[32];
  __shared__ int s_inst;
  T* pool = reinterpret_cast<T*>(sm);
  const unsigned long long t_launch = gtimer();  // used by thread 0 only
  while (true) {
    if (threadIdx.x == 0) s_inst = atomicAdd(a.next, 1);
    __syncthreads();
    const int w = s_inst;
    __syncthreads();
    if (w >= a.n_todo) return;
    const int b = a.todo ? a.todo[w] : w;
    const int mb = (int)(a.m_off[b + 1] - a.m_off[b]), nb = (int)(a.n_off[b + 1] - a.n_off[b]);
    const long long za = a.zsa[b + 1] - a.zsa[b], zt = a.zst[b + 1] - a.zst[b];
    // call sites: the whole instance in shared memory; its two gathered vectors in
    // shared memory (shared loads for the gathers), sorted rows or CSR; everything global
    if (kStaging && za > 0 && stage_bytes(mb, nb, za, zt, (int)sizeof(T)) <= a.stage_cap)
      solve_instance<T, kStaging, true, kFold>(a, b, pool, pool + mb, sh, t_launch);
    else if (za > 0)
      solve_instance<T, false, true, kFold>(a, b, pool, pool + mb, sh, t_launch);
    else if (mb + nb <= a.smem_vec)
      solve_instance<T, false, false, kFold>(a, b, pool, pool + mb, sh, t_launch);
    else
      solve_instance<T, false, false, kFold>(a, b, a.gys + a.m_off[b], a.gxs + a.n_off[b], sh, t_launch);
  }
}

// ---- rows by length -------------------------------------------------------------------
constexpr int kLenBins = 1024;  // rows of kLenBins - 1 or more entries share a bin
constexpr int kPadSlack = 4096;

// Stable order of one matrix's rows by falling length, by one warp: perm[place] = row,
// inv[row] = place, the lengths and the slices' offsets in sorted order.  Returns the
// stored entries (32 times the longest row of each slice).
__device__ __forceinline__ long long sort_rows(const int* rp, int rows, int* bins, int* perm,
                                               int* inv, unsigned short* len, int* soff) {
  const int lane = threadIdx.x & 31;
  for (int k = lane; k < kLenBins; k += 32) bins[k] = 0;
  __syncwarp();
  for (int i = lane; i < rows; i += 32) atomicAdd(&bins[min(rp[i + 1] - rp[i], kLenBins - 1)], 1);
  __syncwarp();
  int run = 0;  // first place of each bin, longest first: 32 bins at a time
  for (int k = kLenBins - 32; k >= 0; k -= 32) {
    const int bin = k + 31 - lane, c = bins[bin];
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    bins[bin] = run + x - c;
    run += __shfl_sync(0xffffffffu, x, 31);
  }
  __syncwarp();
  for (int i0 = 0; i0 < rows; i0 += 32) {
    const int i = i0 + lane;
    const int bin = i < rows ? min(rp[i + 1] - rp[i], kLenBins - 1) : -1;
    const unsigned same = __match_any_sync(0xffffffffu, bin);
    const int rank = __popc(same & ((1u << lane) - 1u));
    const int base = bin >= 0 ? bins[bin] : 0;
    __syncwarp();
    if (bin >= 0) {
      perm[base + rank] = i;
      inv[i] = base + rank;
      len[base + rank] = (unsigned short)min(rp[i + 1] - rp[i], 65535);
      if (rank == 0) bins[bin] = base + __popc(same);
    }
    __syncwarp();
  }
  long long o = 0;
  for (int sl = 0; sl * 32 < rows; ++sl) {
    const int i = sl * 32 + lane;
    const int w = (int)__reduce_max_sync(0xffffffffu, i < rows ? (unsigned)len[i] : 0u);
    if (lane == 0) soff[sl] = (int)min(o, 0x7fffffffLL);
    o += 32LL * w;
  }
  if (lane == 0) soff[n_slices(rows)] = (int)min(o, 0x7fffffffLL);
  return o;
}

// A warp per instance.  size[b], size[B + b]: stored entries of its sorted A and A^T, or zero
// when it keeps CSR: its vectors do not fit in shared memory (mb + nb > vec_cap, which is
// below 2^16), or padding would store more than twice its nonzeros.
__global__ void k_sort_rows(const long long* __restrict__ m_off, const long long* __restrict__ n_off,
                            int B, const int* __restrict__ rp, const int* __restrict__ rpt,
                            int vec_cap, int* __restrict__ permm, int* __restrict__ permn,
                            int* __restrict__ invm, int* __restrict__ invn,
                            unsigned short* __restrict__ lenm, unsigned short* __restrict__ lenn,
                            int* __restrict__ soffm, int* __restrict__ soffn,
                            long long* __restrict__ size) {
  __shared__ int bins[kLenBins];
  const int b = blockIdx.x, lane = threadIdx.x;
  const int m0 = (int)m_off[b], mb = (int)(m_off[b + 1] - m0);
  const int n0 = (int)n_off[b], nb = (int)(n_off[b + 1] - n0);
  const long long z = rp[m0 + mb] - rp[m0];
  long long za = 0, zt = 0;
  if (z > 0 && mb + nb <= vec_cap) {
    za = sort_rows(rp + m0, mb, bins, permm + m0, invm + m0, lenm + m0, soffm + slice_base(m0, b));
    __syncwarp();
    zt = sort_rows(rpt + n0, nb, bins, permn + n0, invn + n0, lenn + n0, soffn + slice_base(n0, b));
    if (za > 2 * z + kPadSlack || zt > 2 * z + kPadSlack) za = zt = 0;
  }
  if (za == 0) {
    for (int i = lane; i < mb; i += 32) permm[m0 + i] = i;
    for (int j = lane; j < nb; j += 32) permn[n0 + j] = j;
  }
  if (lane == 0) {
    size[b] = za;
    size[B + b] = zt;
  }
}

// One matrix of every sorted instance into its slices: values cast to T (through src when
// given: A^T's entries in A), columns as places of the gathered vector; padding is zeros of
// column 0.  Block (b, y): every gridDim.y-th group of slices of instance b.
template <typename T>
__global__ void k_fill_sorted(const long long* __restrict__ r_off, const int* __restrict__ rp, const int* __restrict__ col,
                              const double* __restrict__ val, const int* __restrict__ src,
                              const int* __restrict__ perm, const int* __restrict__ inv,
                              const int* __restrict__ soff, const long long* __restrict__ zs,
                              T* __restrict__ sval, unsigned short* __restrict__ scol) {
  const int b = blockIdx.x;
  const long long z0 = zs[b];
  if (zs[b + 1] == z0) return;
  const int r0 = (int)r_off[b], rows = (int)(r_off[b + 1] - r0);
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  const int* so = soff + slice_base(r0, b);
  for (int sl = blockIdx.y * W + (threadIdx.x >> 5); sl * 32 < rows; sl += gridDim.y * W) {
    const int i = sl * 32 + lane;
    const int r = i < rows ? r0 + perm[r0 + i] : 0;
    const int p0 = i < rows ? rp[r] : 0, n = i < rows ? rp[r + 1] - p0 : 0;
    const int o = so[sl], w = (so[sl + 1] - o) >> 5;
    for (int t = 0; t < w; ++t) {
      const long long e = z0 + o + t * 32 + lane;
      T x = (T)0;
      int k = 0;
      if (t < n) {
        x = (T)(src ? val[src[p0 + t]] : val[p0 + t]);
        k = inv[col[p0 + t]];
      }
      sval[e] = x;
      scol[e] = (unsigned short)k;
    }
  }
}

// Scaled data in every instance's row order: dst_i = src_g * d_g (or / d_g), g the original
// index of place i of instance b (a block per instance and chunk).
template <typename T>
__global__ void k_scale_perm(const long long* __restrict__ off, const int* __restrict__ perm,
                             const double* __restrict__ src, const double* __restrict__ d,
                             bool divide, T* __restrict__ dst) {
  const int b = blockIdx.x;
  const long long o = off[b];
  const int k = (int)(off[b + 1] - o);
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < k; i += gridDim.y * blockDim.x) {
    const long long g = o + perm[o + i];
    dst[o + i] = (T)(divide ? src[g] / d[g] : src[g] * d[g]);
  }
}

// row -> instance via binary search in m_off; global column = n_off[b] + local
__global__ void k_globalize_cols(const long long* __restrict__ m_off,
                                 const long long* __restrict__ n_off, int B,
                                 const long long* __restrict__ rp, int rows,
                                 int* __restrict__ col, int* flags) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= rows) return;
  int lo = 0, hi = B;  // find b with m_off[b] <= i < m_off[b+1]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (m_off[mid] <= i) lo = mid;
    else hi = mid;
  }
  const long long nb = n_off[lo + 1] - n_off[lo];
  for (long long p = rp[i]; p < rp[i + 1]; ++p) {
    const int c = col[p];
    if (c < 0 || c >= nb) atomicOr(flags, 1);
    col[p] = (int)(n_off[lo] + c);
  }
}

// ---- B copies of one LP's constraints (the replicated batch) -----------------
__global__ void k_rep_rowptr(const long long* __restrict__ rp, int m, long long nnz, int B,
                             long long* __restrict__ out) {
  const long long total = (long long)B * m;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / m, i = t - b * m;
    out[t + 1] = rp[i + 1] + b * nnz;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) out[0] = 0;
}

template <typename V>
__global__ void k_tile(const V* __restrict__ src, long long len, int B, V* __restrict__ dst) {
  const long long total = len * B;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x)
    dst[t] = src[t % len];
}

// ---- SPO+ (Sec. 3.4): the surrogate loss of predicted costs ------------------
// c' = 2 c_hat - c_true, the costs of the solve that gives x~.
__global__ void k_spo_costs(const double* __restrict__ c_hat, const double* __restrict__ c_true,
                            long long len, double* __restrict__ out) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < len;
       t += (long long)gridDim.x * blockDim.x)
    out[t] = 2.0 * c_hat[t] - c_true[t];
}

// One block per instance b (coordinates [off[b], off[b+1]), or b*n.. with off
// null): loss_b = -c'^T x~ + 2 c_hat^T x* - z*_b and grad = 2 (x* - x~), where
// x~ minimises c'^T x (Elmachtoub and Grigas 2022).  Fixed-order FP64 sums.
__global__ void k_spo_loss(const long long* __restrict__ off, int n, const double* __restrict__ cp,
                           const double* __restrict__ c_hat, const double* __restrict__ x_true,
                           const double* __restrict__ z_true, const double* __restrict__ x_tl,
                           double* __restrict__ loss, double* __restrict__ grad) {
  __shared__ double sh[32];
  const int b = blockIdx.x;
  const long long j0 = off ? off[b] : (long long)b * n, j1 = off ? off[b + 1] : j0 + n;
  double v = 0.0, t = 0.0;
  for (long long j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
    const double xt = x_tl[j], xs = x_true[j];
    v += cp[j] * xt;
    t += c_hat[j] * xs;
    grad[j] = 2.0 * (xs - xt);
  }
  v = block_sum(v, sh);
  __syncthreads();
  t = block_sum(t, sh);
  if (threadIdx.x == 0) loss[b] = -v + 2.0 * t - z_true[b];
}

}  // namespace mpax

// ============================================================================

using namespace mpax;

struct mpax_batch {
  mpax_problem* prob = nullptr;  // the block-diagonal problem
  int B = 0;
  long long* m_off = nullptr;  // device
  long long* n_off = nullptr;
  std::vector<long long> h_moff, h_noff;
  int max_m = 0, max_n = 0;
  int* next = nullptr;
  int* status = nullptr;
  long long* iters = nullptr;
  long long* restarts = nullptr;
  double *relkkt = nullptr, *pobj = nullptr, *secs = nullptr, *xout = nullptr, *yout = nullptr;
  void* work = nullptr;  // iterate storage and scaled data (precision dependent)
  size_t work_bytes = 0;
  bool solved = false;
  double solve_seconds = 0.0;
  long long launches = 0;
  int* todo = nullptr;     // device list of instances continued in FP64
  int fp64_instances = 0;  // instances of the last solve continued in FP64
  double* spo = nullptr;   // SPO+ staging of host arguments: 3 sum(n) + B doubles
  // rows by length (k_sort_rows): orders, lengths, slice offsets and storage ranges in
  // one buffer, the stored matrices (precision dependent) in another
  void* rows = nullptr;
  void* sell = nullptr;
  size_t sell_bytes = 0;
};

namespace mpax {
// defined in api.cu
ProblemData* problem_data(mpax_problem* p);
cudaStream_t problem_stream(mpax_problem* p);
void problem_order_after_user(mpax_problem* p);
void problem_order_user_after(mpax_problem* p);
}  // namespace mpax

namespace {

mpax_status bfail(mpax_status s, const std::string& m) {
  set_last_error(m.c_str());
  return s;
}

// Bytes of shared memory an instance's two vectors may take (larger instances
// keep them in global memory).
constexpr long long kBatchVecBytes = 200 * 1024;
// Shared-memory bytes an instance may stage whole (matrices, data and iterates)
// when the launch has at most one instance per SM.  With more instances nothing
// is staged whole: a pool of that size shrinks the L1 share of every CTA, and
// on 4096 instances of the ragged recipe (about 15% small enough at 100 KB)
// the batch took 0.57 s against 0.35 s without.
constexpr long long kStageFew = 200 * 1024;

// The arguments and shared-memory size of one batch launch in precision T.
template <typename T>
struct BatchLaunch {
  BatchArgs<T> a;
  size_t smem = 0;
};

// Scaled data and iterate storage of the launch in T (in *work, grown to fit),
// its arguments and its shared-memory pool; allow_stage: whole instances may be
// staged.
template <typename T>
mpax_status batch_prepare(mpax_batch* bt, const mpax_options* o, long long* launches,
                          const int* todo, const int* todo_host, int n_todo, int warm,
                          int stall_limit, bool allow_stage, void** work, size_t* work_bytes,
                          BatchLaunch<T>* L) {
  ProblemData& P = *problem_data(bt->prob);
  cudaStream_t s = P.s;
  const int m = P.m, n = P.n, nnz = P.nnz;
  // scaled data and iterate storage in the iteration precision
  const BatchWork at((size_t)m, (size_t)n, (size_t)nnz + kPad);
  const size_t need = sizeof(T) * at.total;
  if (*work_bytes < need) {
    if (*work) cudaFree(*work);
    *work = nullptr;
    *work_bytes = 0;
    if (cudaMalloc(work, need) != cudaSuccess) return bfail(MPAX_ERR_OUT_OF_MEMORY, "batch work");
    *work_bytes = need;
  }
  T* p = reinterpret_cast<T*>(*work);
  T *valA = p + at.val, *valAt = p + at.valt;
  T *c = p + at.c, *l = p + at.l, *u = p + at.u, *lc = p + at.lc, *uc = p + at.uc;
  T *w = p + at.w, *xa = p + at.xa, *xhat = p + at.xhat, *gbuf = p + at.gbuf;
  T *ya = p + at.ya, *yhat = p + at.yhat, *gys = p + at.gys, *gxs = p + at.gxs;
  // ---- rows by length: orders, slices and, per instance, what they store -------------
  const int B = bt->B;
  const long long vec_cap = kBatchVecBytes / (long long)sizeof(T);
  const size_t slm = (size_t)m / 32 + 2 * (size_t)B + 2, sln = (size_t)n / 32 + 2 * (size_t)B + 2;
  if (!bt->rows) {
    const size_t bytes = sizeof(long long) * (4 * (size_t)B + 2) +
                         sizeof(int) * (2 * ((size_t)m + n) + slm + sln) +
                         sizeof(unsigned short) * ((size_t)m + n + 8);
    if (cudaMalloc(&bt->rows, bytes) != cudaSuccess)
      return bfail(MPAX_ERR_OUT_OF_MEMORY, "batch row orders");
  }
  long long* size = reinterpret_cast<long long*>(bt->rows);  // 2 B
  long long *zsa = size + 2 * (size_t)B, *zst = zsa + B + 1;
  int *permm = reinterpret_cast<int*>(zst + B + 1), *permn = permm + m, *invm = permn + n,
      *invn = invm + m, *soffm = invn + n, *soffn = soffm + slm;
  unsigned short *lenm = reinterpret_cast<unsigned short*>(soffn + sln), *lenn = lenm + m;
  k_sort_rows<<<B, 32, 0, s>>>(bt->m_off, bt->n_off, B, P.A.rp, P.At.rp, (int)vec_cap, permm, permn,
                               invm, invn, lenm, lenn, soffm, soffn, size);
  std::vector<long long> hsize(2 * (size_t)B), hz(2 * (size_t)B + 2, 0);
  cudaError_t e = cudaGetLastError();
  if (!e) e = cudaMemcpyAsync(hsize.data(), size, sizeof(long long) * 2 * B, cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaStreamSynchronize(s);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  std::vector<char> run(B, todo_host ? 0 : 1);  // instances of this launch
  for (int w = 0; todo_host && w < n_todo; ++w) run[todo_host[w]] = 1;
  long long *hza = hz.data(), *hzt = hza + B + 1;
  bool csr = false;  // an instance of the launch reads the CSR arrays
  for (int b = 0; b < B; ++b) {
    hza[b + 1] = hza[b] + (run[b] ? hsize[b] : 0);
    hzt[b + 1] = hzt[b] + (run[b] ? hsize[B + b] : 0);
    csr = csr || (run[b] && hsize[b] == 0);
  }
  const long long ZA = hza[B], ZT = hzt[B];
  const size_t sell_need = (sizeof(T) + sizeof(unsigned short)) * ((size_t)ZA + ZT) + 256;
  if (bt->sell_bytes < sell_need) {
    if (bt->sell) cudaFree(bt->sell);
    bt->sell = nullptr;
    bt->sell_bytes = 0;
    if (cudaMalloc(&bt->sell, sell_need) != cudaSuccess)
      return bfail(MPAX_ERR_OUT_OF_MEMORY, "batch rows by length");
    bt->sell_bytes = sell_need;
  }
  T *sval = reinterpret_cast<T*>(bt->sell), *svalt = sval + ZA;
  unsigned short *scol = reinterpret_cast<unsigned short*>(svalt + ZT), *scolt = scol + ZA;
  if ((e = cudaMemcpyAsync(zsa, hz.data(), sizeof(long long) * (2 * (size_t)B + 2),
                           cudaMemcpyHostToDevice, s)))
    return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  // blocks per instance of the fills: about 16 per SM in all, at most 8
  const int fy = std::max(1, std::min(8, (16 * 152 + B - 1) / B));
  if (ZA > 0) {
    k_fill_sorted<T><<<dim3(B, fy), 256, 0, s>>>(bt->m_off, P.A.rp, P.A.col, P.val_s, nullptr, permm, invn, soffm, zsa, sval, scol);
    k_fill_sorted<T><<<dim3(B, fy), 256, 0, s>>>(bt->n_off, P.At.rp, P.At.col, P.val_s,
                                                 P.permT, permn, invm, soffn, zst, svalt, scolt);
  }
  if (csr) {
    if ((e = cast_vec<T>(P.val_s, valA, nnz, s))) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
    if ((e = gather_cast<T>(P.val_s, P.permT, valAt, nnz, s)))
      return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  }
  const dim3 gp(B, fy);
  if (n) {
    k_scale_perm<T><<<gp, 256, 0, s>>>(bt->n_off, permn, P.c, P.Dc, false, c);
    k_scale_perm<T><<<gp, 256, 0, s>>>(bt->n_off, permn, P.l, P.Dc, true, l);
    k_scale_perm<T><<<gp, 256, 0, s>>>(bt->n_off, permn, P.u, P.Dc, true, u);
  }
  if (m) {
    k_scale_perm<T><<<gp, 256, 0, s>>>(bt->m_off, permm, P.lc, P.Dr, false, lc);
    k_scale_perm<T><<<gp, 256, 0, s>>>(bt->m_off, permm, P.uc, P.Dr, false, uc);
  }
  *launches += 8 + (csr ? 2 : 0);
  BatchArgs<T>& a = L->a;
  a.B = bt->B;
  a.m_off = bt->m_off;
  a.n_off = bt->n_off;
  a.rp = P.A.rp;
  a.col = P.A.col;
  a.val = valA;
  a.rpt = P.At.rp;
  a.colt = P.At.col;
  a.valt = valAt;
  a.c = c;
  a.l = l;
  a.u = u;
  a.lc = lc;
  a.uc = uc;
  a.c0 = P.c;
  a.l0 = P.l;
  a.u0 = P.u;
  a.lc0 = P.lc;
  a.uc0 = P.uc;
  a.Dr = P.Dr;
  a.Dc = P.Dc;
  a.iDr = P.invDr;
  a.iDc = P.invDc;
  a.w = w;
  a.xa = xa;
  a.xhat = xhat;
  a.ya = ya;
  a.yhat = yhat;
  a.gbuf = gbuf;
  a.xout = bt->xout;
  a.yout = bt->yout;
  a.status = bt->status;
  a.iters = bt->iters;
  a.restarts = bt->restarts;
  a.relkkt = bt->relkkt;
  a.pobj = bt->pobj;
  a.secs = bt->secs;
  a.next = bt->next;
  a.gys = gys;
  a.gxs = gxs;
  a.permm = permm;
  a.permn = permn;
  a.lenm = lenm;
  a.lenn = lenn;
  a.soffm = soffm;
  a.soffn = soffn;
  a.zsa = zsa;
  a.zst = zst;
  a.sval = sval;
  a.svalt = svalt;
  a.scol = scol;
  a.scolt = scolt;
  a.eps_abs = o->eps_abs;
  a.eps_rel = o->eps_rel;
  a.r_suff = o->restart_sufficient;
  a.r_nec = o->restart_necessary;
  a.r_art = o->restart_artificial;
  a.pw_smooth = o->primal_weight_smoothing;
  a.step_safety = o->step_safety;
  a.power_tol = o->power_tol;
  a.iter_limit = o->iteration_limit;
  // the whole batch is one launch: it always ends, at the latest kBatchMaxSeconds
  // after it starts, even with no iteration or time limit given
  a.time_limit_ns = (long long)(std::min(o->time_limit, kBatchMaxSeconds) * 1e9);
  a.check_every = o->check_every;
  a.power_max_iter = o->power_max_iter;
  a.power_cap = o->pock_chambolle ? 1.0 : INFINITY;
  // the shared pool fits the largest instance of this launch that fits in
  // kBatchVecBytes; larger instances run from global memory
  long long vmax = 0;
  for (int w = 0; w < n_todo; ++w) {
    const int b = todo_host ? todo_host[w] : w;
    const long long v = (bt->h_moff[b + 1] - bt->h_moff[b]) + (bt->h_noff[b + 1] - bt->h_noff[b]);
    if (v <= vec_cap) vmax = std::max(vmax, v);
  }
  a.smem_vec = (int)((vmax + 3) / 4 * 4);
  const size_t smem = sizeof(T) * (size_t)a.smem_vec;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // whole-instance staging when every instance of the launch has an SM of its own
  const long long cap = (allow_stage && o->batch_stage && n_todo <= sms) ? kStageFew : 0;
  long long smax = 0;
  for (int w = 0; w < n_todo; ++w) {
    const int b = todo_host ? todo_host[w] : w;
    const long long need = stage_bytes(bt->h_moff[b + 1] - bt->h_moff[b],
                                       bt->h_noff[b + 1] - bt->h_noff[b], hsize[b], hsize[B + b],
                                       (int)sizeof(T));
    if (hsize[b] > 0 && need <= cap) smax = std::max(smax, need);
  }
  a.stage_cap = smax;
  L->smem = std::max(smem, (size_t)((smax + 15) / 16 * 16));
  a.todo = todo;
  a.n_todo = n_todo;
  a.warm = warm;
  a.stall_limit = stall_limit;
  if ((e = cudaGetLastError())) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  return MPAX_OK;
}

// Resident CTAs of `kernel` on the whole GPU (at least one per SM).
template <class K>
int batch_grid(K kernel, int threads, size_t smem, int n_todo) {
  int occ = 0, dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem);
  return std::min(n_todo, std::max(1, occ) * sms);
}

template <typename T>
mpax_status run_batch(mpax_batch* bt, const mpax_options* o, long long* launches,
                      const int* todo, const int* todo_host, int n_todo, int warm,
                      int stall_limit) {
  BatchLaunch<T> L;
  mpax_status st = batch_prepare<T>(bt, o, launches, todo, todo_host, n_todo, warm, stall_limit,
                                    true, &bt->work, &bt->work_bytes, &L);
  if (st) return st;
  cudaStream_t s = problem_data(bt->prob)->s;
  constexpr int kT = kBatchThreads<T>;
  auto kernel = L.a.stage_cap > 0 ? batch_lp_kernel<T, true, kT> : batch_lp_kernel<T, false, kT>;
  int threads = kT;
  if constexpr (kT > kBatchSmallThreads) {
    // by the batch's sizes; the results do not depend on it (Share)
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    bool small = bt->B > 2 * sms && bt->h_noff[bt->B] <= (long long)kSmallCols * bt->B;
    for (int b = 0; b < bt->B && small; ++b)
      small = bt->h_moff[b + 1] - bt->h_moff[b] + bt->h_noff[b + 1] - bt->h_noff[b] <= kSmallVec;
    if (small) {
      kernel = batch_lp_kernel<T, false, kBatchSmallThreads>;  // more instances than are staged
      threads = kBatchSmallThreads;
    }
  }
  const int grid = batch_grid(kernel, threads, L.smem, n_todo);
  cudaMemsetAsync(bt->next, 0, sizeof(int), s);
  kernel<<<grid, threads, L.smem, s>>>(L.a);
  *launches += 1;
  cudaError_t e = cudaGetLastError();
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  return MPAX_OK;
}

}  // namespace

extern "C" {

mpax_status mpax_lp_batch_create(int32_t B, const int64_t* m_off, const int64_t* n_off,
                                 const int64_t* row_ptr, const int32_t* col_idx,
                                 const double* val, const double* c, const double* lc,
                                 const double* uc, const double* l, const double* u,
                                 mpax_mem_kind kind, void* cuda_stream, mpax_batch** out) {
  if (!out) return bfail(MPAX_ERR_INVALID_ARGUMENT, "out must not be NULL");
  *out = nullptr;
  if (B < 1) return bfail(MPAX_ERR_INVALID_ARGUMENT, "B must be >= 1");
  if (!m_off || !n_off || !row_ptr) return bfail(MPAX_ERR_INVALID_ARGUMENT, "NULL offsets");
  std::vector<long long> hm(B + 1), hn(B + 1);
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyHostToHost : cudaMemcpyDeviceToHost;
  if (cudaMemcpy(hm.data(), m_off, sizeof(long long) * (B + 1), k) != cudaSuccess ||
      cudaMemcpy(hn.data(), n_off, sizeof(long long) * (B + 1), k) != cudaSuccess)
    return bfail(MPAX_ERR_CUDA, "copy of the offsets failed");
  if (hm[0] != 0 || hn[0] != 0) return bfail(MPAX_ERR_INVALID_ARGUMENT, "offsets must start at 0");
  int max_m = 0, max_n = 0;
  for (int b = 0; b < B; ++b) {
    if (hm[b + 1] < hm[b] || hn[b + 1] < hn[b])
      return bfail(MPAX_ERR_INVALID_ARGUMENT, "offsets must be non-decreasing");
    max_m = std::max<long long>(max_m, hm[b + 1] - hm[b]);
    max_n = std::max<long long>(max_n, hn[b + 1] - hn[b]);
  }
  if (hm[B] >= (1LL << 31) || hn[B] >= (1LL << 31))
    return bfail(MPAX_ERR_UNSUPPORTED, "total rows and columns must be < 2^31");
  const int m = (int)hm[B], n = (int)hn[B];
  long long nnz = 0;
  if (cudaMemcpy(&nnz, row_ptr + m, sizeof(long long), k) != cudaSuccess)
    return bfail(MPAX_ERR_CUDA, "copy of row_ptr failed");
  // device copies of the structure with columns made global
  long long *d_moff = nullptr, *d_noff = nullptr, *d_rp = nullptr;
  int *d_col = nullptr, *flags = nullptr;
  cudaError_t e = cudaMalloc(&d_moff, sizeof(long long) * (B + 1));
  if (!e) e = cudaMalloc(&d_noff, sizeof(long long) * (B + 1));
  if (!e) e = cudaMalloc(&d_rp, sizeof(long long) * (m + 1));
  if (!e) e = cudaMalloc(&d_col, sizeof(int) * std::max<long long>(nnz, 1));
  if (!e) e = cudaMalloc(&flags, sizeof(int));
  if (!e) e = cudaMemcpy(d_moff, hm.data(), sizeof(long long) * (B + 1), cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(d_noff, hn.data(), sizeof(long long) * (B + 1), cudaMemcpyHostToDevice);
  const cudaMemcpyKind kin = kind == MPAX_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  if (!e) e = cudaMemcpy(d_rp, row_ptr, sizeof(long long) * (m + 1), kin);
  if (!e && nnz > 0) e = cudaMemcpy(d_col, col_idx, sizeof(int) * nnz, kin);
  if (!e) e = cudaMemset(flags, 0, sizeof(int));
  if (!e && m > 0) k_globalize_cols<<<(m + 255) / 256, 256>>>(d_moff, d_noff, B, d_rp, m, d_col, flags);
  int hf = 0;
  if (!e) e = cudaMemcpy(&hf, flags, sizeof(int), cudaMemcpyDeviceToHost);
  mpax_problem* prob = nullptr;
  mpax_status st = MPAX_OK;
  if (!e && hf) st = bfail(MPAX_ERR_INVALID_ARGUMENT, "a column index is outside its instance");
  if (!e && !hf) {
    // values and vectors go through the single-problem create (copy + validation);
    // host inputs are staged on the device first so that every pointer is device memory
    const double* dv[6] = {val, c, lc, uc, l, u};
    const long long cnt[6] = {nnz, n, m, m, n, n};
    double* tmp[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    if (kind == MPAX_MEM_HOST) {
      for (int q = 0; q < 6 && !e; ++q) {
        e = cudaMalloc(&tmp[q], sizeof(double) * std::max<long long>(cnt[q], 1));
        if (!e && cnt[q] > 0) e = cudaMemcpy(tmp[q], dv[q], sizeof(double) * cnt[q], cudaMemcpyHostToDevice);
        dv[q] = tmp[q];
      }
    }
    if (!e)
      st = mpax_lp_create(m, n, nnz, (const int64_t*)d_rp, d_col, dv[0], dv[1], dv[2], dv[3],
                          dv[4], dv[5], MPAX_MEM_DEVICE, cuda_stream, &prob);
    for (double* t : tmp)
      if (t) cudaFree(t);
  }
  cudaFree(d_rp);
  cudaFree(d_col);
  cudaFree(flags);
  if (e) {
    cudaFree(d_moff);
    cudaFree(d_noff);
    return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  }
  if (st) {
    cudaFree(d_moff);
    cudaFree(d_noff);
    return st;
  }
  mpax_batch* bt = new mpax_batch();
  e = cudaMalloc(&bt->next, sizeof(int));
  if (!e) e = cudaMalloc(&bt->status, sizeof(int) * B);
  if (!e) e = cudaMalloc(&bt->iters, sizeof(long long) * B);
  if (!e) e = cudaMalloc(&bt->restarts, sizeof(long long) * B);
  if (!e) e = cudaMalloc(&bt->relkkt, sizeof(double) * B);
  if (!e) e = cudaMalloc(&bt->pobj, sizeof(double) * B);
  if (!e) e = cudaMalloc(&bt->secs, sizeof(double) * B);
  if (!e) e = cudaMalloc(&bt->xout, sizeof(double) * std::max(n, 1));
  if (!e) e = cudaMalloc(&bt->yout, sizeof(double) * std::max(m, 1));
  bt->prob = prob;
  bt->B = B;
  bt->m_off = d_moff;
  bt->n_off = d_noff;
  bt->h_moff = hm;
  bt->h_noff = hn;
  bt->max_m = max_m;
  bt->max_n = max_n;
  if (e) {
    mpax_batch_destroy(bt);
    return bfail(MPAX_ERR_OUT_OF_MEMORY, "batch output arrays");
  }
  *out = bt;
  return MPAX_OK;
}

mpax_status mpax_batch_solve(mpax_batch* bt, const mpax_options* o) {
  if (!bt || !o) return bfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  if (o->reflection_gamma != 1.0)
    return bfail(MPAX_ERR_UNSUPPORTED, "the batch path implements reflection_gamma = 1");
  if (o->check_every < 1 || o->iteration_limit < 1 || o->ruiz_iters < 0 ||
      !(o->step_safety > 0 && o->step_safety < 1) || o->power_max_iter < 0 ||
      (o->power_max_iter == 0 && !o->pock_chambolle) ||
      !(o->time_limit >= 0) || (o->batch_stage != 0 && o->batch_stage != 1))
    return bfail(MPAX_ERR_INVALID_ARGUMENT, "invalid options");
  if (o->precision != MPAX_PREC_FP64 && o->precision != MPAX_PREC_MIXED)
    return bfail(MPAX_ERR_INVALID_ARGUMENT, "bad precision");
  const auto t0 = std::chrono::steady_clock::now();
  ProblemData& P = *problem_data(bt->prob);
  cudaStream_t s = P.s;
  problem_order_after_user(bt->prob);
  long long launches = 0;
  cudaError_t e = transpose_csr(P.A, P.At, P.permT, P.tmp_rows, P.tmp_scan, P.val_s, s);
  if (!e) e = compute_scaling(P, o->ruiz_iters, o->pock_chambolle != 0);
  launches += 6 + 5 * o->ruiz_iters + 8;
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  const bool cont = o->precision == MPAX_PREC_MIXED && o->fp64_continuation;
  mpax_status st =
      o->precision == MPAX_PREC_FP64
          ? run_batch<double>(bt, o, &launches, nullptr, nullptr, bt->B, 0, 0)
          : run_batch<float>(bt, o, &launches, nullptr, nullptr, bt->B, 0,
                             cont ? o->stall_checks : 0);
  if (st) return st;
  if (cont) {
    // FP64 continuation of the instances that stalled in FP32, warm-started
    // from their returned points, in one more persistent launch
    std::vector<int> hs(bt->B), todo;
    e = cudaMemcpyAsync(hs.data(), bt->status, sizeof(int) * bt->B, cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
    for (int b = 0; b < bt->B; ++b)
      if (hs[b] == kTermStalled) todo.push_back(b);
    bt->fp64_instances = (int)todo.size();
    if (!todo.empty()) {
      if (!bt->todo && (e = cudaMalloc(&bt->todo, sizeof(int) * bt->B)))
        return bfail(MPAX_ERR_OUT_OF_MEMORY, "batch continuation list");
      e = cudaMemcpyAsync(bt->todo, todo.data(), sizeof(int) * todo.size(),
                          cudaMemcpyHostToDevice, s);
      if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
      st = run_batch<double>(bt, o, &launches, bt->todo, todo.data(), (int)todo.size(), 1, 0);
      if (st) return st;
    }
  }
  e = cudaStreamSynchronize(s);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  problem_order_user_after(bt->prob);
  bt->solved = true;
  bt->launches = launches;
  bt->solve_seconds =
      std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  return MPAX_OK;
}

mpax_status mpax_batch_get_solution(const mpax_batch* bt, double* x, double* y,
                                    mpax_mem_kind kind) {
  if (!bt) return bfail(MPAX_ERR_INVALID_ARGUMENT, "NULL batch");
  if (!bt->solved) return bfail(MPAX_ERR_NOT_SOLVED, "call mpax_batch_solve first");
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  const long long n = bt->h_noff[bt->B], m = bt->h_moff[bt->B];
  cudaError_t e = cudaSuccess;
  if (x && n) e = cudaMemcpy(x, bt->xout, sizeof(double) * n, k);
  if (!e && y && m) e = cudaMemcpy(y, bt->yout, sizeof(double) * m, k);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  return MPAX_OK;
}

mpax_status mpax_batch_get_stats(const mpax_batch* bt, mpax_batch_stats* stats, int32_t* status,
                                 int64_t* iterations, double* rel_kkt, double* primal_obj,
                                 double* seconds) {
  if (!bt || !stats) return bfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  if (!bt->solved) return bfail(MPAX_ERR_NOT_SOLVED, "call mpax_batch_solve first");
  const int B = bt->B;
  std::vector<int> hs(B);
  std::vector<long long> hi(B), hr(B);
  std::vector<double> hk(B), hp(B), ht(B);
  cudaError_t e = cudaMemcpy(hs.data(), bt->status, sizeof(int) * B, cudaMemcpyDeviceToHost);
  if (!e) e = cudaMemcpy(hi.data(), bt->iters, sizeof(long long) * B, cudaMemcpyDeviceToHost);
  if (!e) e = cudaMemcpy(hr.data(), bt->restarts, sizeof(long long) * B, cudaMemcpyDeviceToHost);
  if (!e) e = cudaMemcpy(hk.data(), bt->relkkt, sizeof(double) * B, cudaMemcpyDeviceToHost);
  if (!e) e = cudaMemcpy(hp.data(), bt->pobj, sizeof(double) * B, cudaMemcpyDeviceToHost);
  if (!e) e = cudaMemcpy(ht.data(), bt->secs, sizeof(double) * B, cudaMemcpyDeviceToHost);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  std::memset(stats, 0, sizeof(*stats));
  stats->B = B;
  std::vector<double> sorted = ht;
  std::sort(sorted.begin(), sorted.end());
  for (int b = 0; b < B; ++b) {
    stats->n_optimal += hs[b] == MPAX_TERM_OPTIMAL;
    stats->iterations_total += hi[b];
    stats->iterations_max = std::max<long long>(stats->iterations_max, hi[b]);
    stats->restarts_total += hr[b];
    stats->rel_kkt_max = std::max(stats->rel_kkt_max, hk[b]);
  }
  auto pct = [&](double q) {
    const size_t i = std::min<size_t>(sorted.size() - 1, (size_t)std::ceil(q * sorted.size()) - 1);
    return sorted[i];
  };
  stats->instance_seconds_p50 = pct(0.50);
  stats->instance_seconds_p99 = pct(0.99);
  stats->instance_seconds_max = sorted.back();
  stats->solve_seconds = bt->solve_seconds;
  stats->kernel_launches = bt->launches;
  stats->fp64_instances = bt->fp64_instances;
  for (int b = 0; b < B; ++b) {
    if (status) status[b] = hs[b];
    if (iterations) iterations[b] = hi[b];
    if (rel_kkt) rel_kkt[b] = hk[b];
    if (primal_obj) primal_obj[b] = hp[b];
    if (seconds) seconds[b] = ht[b];
  }
  return MPAX_OK;
}

mpax_status mpax_lp_batch_create_replicated(int32_t B, int32_t m, int32_t n, int64_t nnz,
                                            const int64_t* row_ptr, const int32_t* col_idx,
                                            const double* val, const double* lc,
                                            const double* uc, const double* l, const double* u,
                                            mpax_mem_kind kind, void* cuda_stream,
                                            mpax_batch** out) {
  if (!out) return bfail(MPAX_ERR_INVALID_ARGUMENT, "out must not be NULL");
  *out = nullptr;
  if (B < 1 || m < 0 || n < 0 || nnz < 0)
    return bfail(MPAX_ERR_INVALID_ARGUMENT, "B >= 1 and non-negative sizes required");
  if (!row_ptr || (nnz > 0 && (!col_idx || !val)) || (m > 0 && (!lc || !uc)) ||
      (n > 0 && (!l || !u)))
    return bfail(MPAX_ERR_INVALID_ARGUMENT, "a required array pointer is NULL");
  if ((long long)B * m >= (1LL << 31) || (long long)B * n >= (1LL << 31) ||
      (long long)B * nnz >= (1LL << 31))
    return bfail(MPAX_ERR_UNSUPPORTED, "B copies must hold < 2^31 rows, columns and nonzeros");
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  // one copy of the set on the device, then B copies of it (columns stay local)
  const long long Bm = (long long)B * m, Bn = (long long)B * n, Bz = (long long)B * nnz;
  long long *rp1 = nullptr, *rpB = nullptr, *moff = nullptr, *noff = nullptr;
  int *col1 = nullptr, *colB = nullptr;
  double* v1 = nullptr;  // nnz + 2m + 2n
  double* vB = nullptr;  // B (nnz + 3n + 2m): values, c (zero), lc, uc, l, u
  cudaError_t e = cudaMalloc(&rp1, sizeof(long long) * (m + 1));
  if (!e) e = cudaMalloc(&rpB, sizeof(long long) * (Bm + 1));
  if (!e) e = cudaMalloc(&moff, sizeof(long long) * (B + 1));
  if (!e) e = cudaMalloc(&noff, sizeof(long long) * (B + 1));
  if (!e) e = cudaMalloc(&col1, sizeof(int) * std::max<long long>(nnz, 1));
  if (!e) e = cudaMalloc(&colB, sizeof(int) * std::max<long long>(Bz, 1));
  if (!e) e = cudaMalloc(&v1, sizeof(double) * std::max<long long>(nnz + 2LL * m + 2LL * n, 1));
  if (!e) e = cudaMalloc(&vB, sizeof(double) * std::max<long long>(Bz + 3 * Bn + 2 * Bm, 1));
  double* valB = vB;
  double* cB = vB + Bz;
  double* lcB = cB + Bn;
  double* ucB = lcB + Bm;
  double* lB = ucB + Bm;
  double* uB = lB + Bn;
  if (!e) e = cudaMemcpyAsync(rp1, row_ptr, sizeof(long long) * (m + 1), k, s);
  if (!e && nnz) e = cudaMemcpyAsync(col1, col_idx, sizeof(int) * nnz, k, s);
  if (!e && nnz) e = cudaMemcpyAsync(v1, val, sizeof(double) * nnz, k, s);
  if (!e && m) e = cudaMemcpyAsync(v1 + nnz, lc, sizeof(double) * m, k, s);
  if (!e && m) e = cudaMemcpyAsync(v1 + nnz + m, uc, sizeof(double) * m, k, s);
  if (!e && n) e = cudaMemcpyAsync(v1 + nnz + 2LL * m, l, sizeof(double) * n, k, s);
  if (!e && n) e = cudaMemcpyAsync(v1 + nnz + 2LL * m + n, u, sizeof(double) * n, k, s);
  std::vector<long long> hm(B + 1), hn(B + 1);
  for (int b = 0; b <= B; ++b) {
    hm[b] = (long long)b * m;
    hn[b] = (long long)b * n;
  }
  if (!e) e = cudaMemcpyAsync(moff, hm.data(), sizeof(long long) * (B + 1), cudaMemcpyHostToDevice, s);
  if (!e) e = cudaMemcpyAsync(noff, hn.data(), sizeof(long long) * (B + 1), cudaMemcpyHostToDevice, s);
  if (!e) {
    const int g = 1024;
    k_rep_rowptr<<<g, 256, 0, s>>>(rp1, m, nnz, B, rpB);
    if (nnz) k_tile<int><<<g, 256, 0, s>>>(col1, nnz, B, colB);
    if (nnz) k_tile<double><<<g, 256, 0, s>>>(v1, nnz, B, valB);
    if (m) k_tile<double><<<g, 256, 0, s>>>(v1 + nnz, m, B, lcB);
    if (m) k_tile<double><<<g, 256, 0, s>>>(v1 + nnz + m, m, B, ucB);
    if (n) k_tile<double><<<g, 256, 0, s>>>(v1 + nnz + 2LL * m, n, B, lB);
    if (n) k_tile<double><<<g, 256, 0, s>>>(v1 + nnz + 2LL * m + n, n, B, uB);
    if (Bn) e = cudaMemsetAsync(cB, 0, sizeof(double) * Bn, s);
    if (!e) e = cudaGetLastError();
    if (!e) e = cudaStreamSynchronize(s);
  }
  mpax_status st = MPAX_ERR_CUDA;
  if (!e)
    st = mpax_lp_batch_create(B, (const int64_t*)moff, (const int64_t*)noff,
                              (const int64_t*)rpB, colB, valB, cB, lcB, ucB, lB, uB,
                              MPAX_MEM_DEVICE, cuda_stream, out);
  cudaStreamSynchronize(s);
  for (void* p : {(void*)rp1, (void*)rpB, (void*)moff, (void*)noff, (void*)col1, (void*)colB,
                  (void*)v1, (void*)vB})
    if (p) cudaFree(p);
  if (e) return bfail(e == cudaErrorMemoryAllocation ? MPAX_ERR_OUT_OF_MEMORY : MPAX_ERR_CUDA,
                      cudaGetErrorString(e));
  return st;
}

mpax_status mpax_batch_set_costs(mpax_batch* bt, const double* c, mpax_mem_kind kind) {
  if (!bt || !c) return bfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  ProblemData& P = *problem_data(bt->prob);
  const long long n = bt->h_noff[bt->B];
  problem_order_after_user(bt->prob);
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  cudaError_t e = n ? cudaMemcpyAsync(P.c, c, sizeof(double) * n, k, P.s) : cudaSuccess;
  if (!e) e = cudaStreamSynchronize(P.s);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  problem_order_user_after(bt->prob);
  bt->solved = false;
  return MPAX_OK;
}

mpax_status mpax_batch_get_objective(const mpax_batch* bt, double* v, mpax_mem_kind kind) {
  if (!bt || !v) return bfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  if (!bt->solved) return bfail(MPAX_ERR_NOT_SOLVED, "call mpax_batch_solve first");
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  const cudaError_t e = cudaMemcpy(v, bt->pobj, sizeof(double) * bt->B, k);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  return MPAX_OK;
}

mpax_status mpax_batch_spo_plus(mpax_batch* bt, const mpax_options* o, const double* c_hat,
                                const double* c_true, const double* x_true,
                                const double* z_true, double* loss, double* grad,
                                mpax_mem_kind kind) {
  if (!bt || !o || !c_hat || !c_true || !x_true || !z_true || !loss || !grad)
    return bfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  ProblemData& P = *problem_data(bt->prob);
  cudaStream_t s = P.s;
  const int B = bt->B;
  const long long n = bt->h_noff[B];
  problem_order_after_user(bt->prob);
  cudaError_t e = cudaSuccess;
  if (kind == MPAX_MEM_HOST) {
    // stage the host arguments: c_hat, c_true, x_true (sum n each), z_true (B)
    if (!bt->spo) e = cudaMalloc(&bt->spo, sizeof(double) * (3 * std::max<long long>(n, 1) + B));
    double* d = bt->spo;
    if (!e && n) e = cudaMemcpyAsync(d, c_hat, sizeof(double) * n, cudaMemcpyHostToDevice, s);
    if (!e && n) e = cudaMemcpyAsync(d + n, c_true, sizeof(double) * n, cudaMemcpyHostToDevice, s);
    if (!e && n)
      e = cudaMemcpyAsync(d + 2 * n, x_true, sizeof(double) * n, cudaMemcpyHostToDevice, s);
    if (!e) e = cudaMemcpyAsync(d + 3 * n, z_true, sizeof(double) * B, cudaMemcpyHostToDevice, s);
    c_hat = d;
    c_true = d + n;
    x_true = d + 2 * n;
    z_true = d + 3 * n;
  }
  if (!e && n) {
    k_spo_costs<<<(int)std::min<long long>(4096, (n + 255) / 256), 256, 0, s>>>(c_hat, c_true,
                                                                              n, P.c);
    e = cudaGetLastError();
  }
  if (!e) e = cudaStreamSynchronize(s);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  problem_order_user_after(bt->prob);
  bt->solved = false;
  mpax_status st = mpax_batch_solve(bt, o);
  if (st) return st;
  problem_order_after_user(bt->prob);
  double* dl = loss;
  double* dg = grad;
  if (kind == MPAX_MEM_HOST) {
    // results go through the work area of the staged inputs (c_true is no longer needed)
    dg = bt->spo + n;
    dl = bt->spo + 3 * n;  // z_true is read before loss is written, block by block
  }
  k_spo_loss<<<B, 256, 0, s>>>(bt->n_off, 0, P.c, c_hat, x_true, z_true, bt->xout, dl, dg);
  e = cudaGetLastError();
  if (!e && kind == MPAX_MEM_HOST) {
    if (n) e = cudaMemcpyAsync(grad, dg, sizeof(double) * n, cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaMemcpyAsync(loss, dl, sizeof(double) * B, cudaMemcpyDeviceToHost, s);
  }
  if (!e) e = cudaStreamSynchronize(s);
  if (e) return bfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  problem_order_user_after(bt->prob);
  return MPAX_OK;
}

void mpax_batch_destroy(mpax_batch* bt) {
  if (!bt) return;
  if (bt->prob) mpax_destroy(bt->prob);
  void* bufs[] = {bt->m_off, bt->n_off, bt->next, bt->status, bt->iters, bt->restarts,
                  bt->relkkt, bt->pobj, bt->secs, bt->xout, bt->yout, bt->work, bt->todo,
                  bt->spo, bt->rows, bt->sell};
  for (void* b : bufs)
    if (b) cudaFree(b);
  delete bt;
}

}  // extern "C"
