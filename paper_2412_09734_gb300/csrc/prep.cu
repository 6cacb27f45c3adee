// Preprocessing on the device: Ruiz and Pock-Chambolle diagonal scaling
// (Sec. 3 names both and applies them by default), the rescaled problem data,
// and the norms that set the initial primal weight and the relative KKT test.
#include <algorithm>

#include "problem.cuh"

namespace mpax {

// ---- rows by lane groups ------------------------------------------------------------
// A warp takes four consecutive rows of at most kGroupRow entries side by side, eight lanes
// each.  With a warp per row most lanes idled on rows of a few entries (a fifth of a million
// rows of one or two in a power-law matrix), and each row paid a five-step tree of the whole
// warp.  Longer rows come from a list (LongRows), a warp each: they often stand together (the
// coupling rows of a model), and one warp that took four of them in turn held up the launch
// (preparation of an LP of 20 rows of 100,000 entries 67.8 -> 20.4 ms).
constexpr int kGroup = 8, kGroupRows = 32 / kGroup, kGroupRow = 64;

// The rows of a matrix with more than kGroupRow entries, in no particular order.
struct LongRows {
  const int* n;    // their number, on the device; nullptr: there are none
  const int* row;
};

// Rows i of the block's threads with more than kGroupRow entries are appended to n, row.
__device__ __forceinline__ void append_long(const int* __restrict__ rp, int rows, long long i,
                                            int* n, int* row) {
  const bool is_long = i < rows && rp[i + 1] - rp[i] > kGroupRow;
  const unsigned longs = __ballot_sync(0xffffffffu, is_long);
  if (longs == 0) return;
  const int lane = threadIdx.x & 31;
  int at = lane == 0 ? atomicAdd(n, __popc(longs)) : 0;
  at = __shfl_sync(0xffffffffu, at, 0);
  if (is_long) row[at + __popc(longs & ((1u << lane) - 1u))] = (int)i;
}
__global__ void find_long(const int* __restrict__ rp, int rows, int* n, int* row) {
  append_long(rp, rows, (long long)blockIdx.x * blockDim.x + threadIdx.x, n, row);
}

// f(i, p, k) on every entry p of this warp's rows i; k = (entry's place in its row) / 8 % 4
// tells which of the row's 32 strided partial sums it belongs to.  done(i, valid, wide) ends
// row i: called by all lanes, for a short row of the lane's group (wide = false) or one row
// of the whole warp.
template <class F, class Done>
__device__ __forceinline__ void for_rows(const int* __restrict__ rp, int rows, LongRows lr, F f,
                                         Done done) {
  const int lane = threadIdx.x & 31, gl = lane & (kGroup - 1);
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const int nl = lr.n ? *lr.n : 0;
  for (long long r0 = (long long)warp * kGroupRows; r0 < rows; r0 += (long long)nw * kGroupRows) {
    const bool in = r0 + lane / kGroup < rows;
    const int i = in ? (int)r0 + lane / kGroup : 0;
    const int b = in ? rp[i] : 0, e = in ? rp[i + 1] : 0;
    const bool is_long = e - b > kGroupRow;
    if (!is_long) {
      for (int p = b + gl, t = 0; p < e; p += kGroup, ++t) f(i, p, t & 3);
    }
    __syncwarp();
    done(i, !is_long && in, false);
  }
  for (int t = warp; t < nl; t += nw) {
    const int i = lr.row[t], e = rp[i + 1];
    for (int p = rp[i] + lane; p < e; p += 32) f(i, p, 0);
    __syncwarp();
    done(i, true, true);
  }
}

// Sum of a row in the order of a warp per row (lane i adds entries i, i + 32, ...; then
// halves are added, 16 apart, 8, 4, 2, 1), whichever lanes hold it: a group's lane l
// keeps the four partial sums l, l + 8, l + 16, l + 24.
struct RowSum {
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  __device__ __forceinline__ double total(bool wide) const {
    double s;
    int o;
    if (wide) {
      s = a[0];
      o = 16;
    } else {
      s = (a[0] + a[2]) + (a[1] + a[3]);
      o = kGroup / 2;
    }
    for (; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  }
  __device__ __forceinline__ void clear() { a[0] = a[1] = a[2] = a[3] = 0.0; }
};

// Sum of |K_ij| over the rows; values through `perm` (columns of A as rows of A^T).
__global__ void row_abssum(const int* __restrict__ rp, const double* __restrict__ val,
                           const int* __restrict__ perm, int rows, LongRows lr,
                           double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  RowSum sum;
  for_rows(
      rp, rows, lr,
      [&](int, int p, int k) {
        const double v = fabs(val[perm[p]]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (k == q) sum.a[q] += v;
      },
      [&](int i, bool valid, bool wide) {
        const double t = sum.total(wide);
        if (valid && (wide ? lane == 0 : (lane & (kGroup - 1)) == 0)) out[i] = t;
        if (valid) sum.clear();
      });
}

// One pass over the rows of A for a scaling round.  With the previous round's
// factors (dr, dc non-null) the values are first rescaled in place,
// v <- (v * dr_i) * dc_j; then |v| is reduced to its row norm (maximum, or sum
// when SUM, in a fixed order) and, for the maximum, to its column maximum.  Maxima are
// taken on the bit patterns: non-negative doubles order like them, so the result is
// exact in any order (columns by integer atomics; colmax must start at +0.0) and keeps
// off the FP64 pipe.  10M entries in 500,000 power-law rows: 401 us with a warp per row,
// 182 us by groups, 132 us with the long rows apart; 2M entries in 100,000 rows of about 20:
// 59 -> 25 us.
template <bool SUM>
__global__ void scale_pass(const int* __restrict__ rp, const int* __restrict__ col,
                           double* __restrict__ val, int rows, LongRows lr,
                           const double* __restrict__ dr, const double* __restrict__ dc,
                           double* __restrict__ rownorm,
                           unsigned long long* __restrict__ colmax) {
  const int lane = threadIdx.x & 31;
  RowSum sum;
  unsigned long long mx = 0ull;
  for_rows(
      rp, rows, lr,
      [&](int i, int p, int k) {
        double v = val[p];
        if (SUM ? dr != nullptr : true) {
          const int j = col[p];
          if (dr) {
            v = (v * dr[i]) * dc[j];
            val[p] = v;
          }
          if constexpr (!SUM) {
            const unsigned long long a =
                (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
            mx = a > mx ? a : mx;
            atomicMax(colmax + j, a);
          }
        }
        if constexpr (SUM) {
          const double a = fabs(v);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (k == q) sum.a[q] += a;
        }
      },
      [&](int i, bool valid, bool wide) {
        const bool first = wide ? lane == 0 : (lane & (kGroup - 1)) == 0;
        if constexpr (SUM) {
          const double t = sum.total(wide);
          if (valid && first) rownorm[i] = t;
          if (valid) sum.clear();
        } else {
          unsigned long long t = mx;
          for (int o = wide ? 16 : kGroup / 2; o > 0; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, t, o);
            t = x > t ? x : t;
          }
          if (valid && first) rownorm[i] = __longlong_as_double((long long)t);
          if (valid) mx = 0ull;
        }
      });
}

// d_i = 1/sqrt(norm_i) (1 for an empty row/column); D_i *= d_i.  d overwrites norm.
// Rows (m of rnorm, Dr) then columns (n of cnorm, Dc).  With qdiag (QP columns) the
// current scaled diagonal D_j^2 qdiag_j joins the norm first: max with it (Ruiz, SUM =
// false) or added to it (Pock-Chambolle).
template <bool SUM>
__global__ void factor_update(double* __restrict__ rnorm, int m, double* __restrict__ Dr,
                              double* __restrict__ cnorm, int n, double* __restrict__ Dc,
                              const double* __restrict__ qdiag) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)m + n) return;
  const bool row = t < m;
  const int i = (int)(row ? t : t - m);
  double* norm = row ? rnorm : cnorm;
  double* D = row ? Dr : Dc;
  double v = norm[i];
  if (qdiag && !row) {
    const double q = D[i] * D[i] * qdiag[i];
    v = SUM ? v + q : fmax(v, q);
  }
  const double d = (v > 0.0) ? 1.0 / sqrt(v) : 1.0;
  norm[i] = d;
  D[i] *= d;
}

// K_ij <- (K_ij * dr_i) * dc_j  (src may differ from dst: start from the original;
// dc may be nullptr = all ones)
__global__ void apply_scale(const int* __restrict__ rp, const int* __restrict__ col,
                            const double* __restrict__ src, double* __restrict__ dst, int rows,
                            LongRows lr, const double* __restrict__ dr,
                            const double* __restrict__ dc) {
  for_rows(
      rp, rows, lr,
      [&](int i, int p, int) { dst[p] = dc ? (src[p] * dr[i]) * dc[col[p]] : src[p] * dr[i]; },
      [](int, bool, bool) {});
}

// diag(Q)_j = D_j + sum_r F_jr^2 for Q = diag(D) + F F^T
__global__ void q_diagonal(const int* __restrict__ frp, const double* __restrict__ fval,
                           const double* __restrict__ D, int n, double* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  double s = D[j];
  for (int p = frp[j]; p < frp[j + 1]; ++p) s += fval[p] * fval[p];
  out[j] = s;
}

// diag(Q)_j += Q_jj for a general sparse Q (entries of row j in column j)
__global__ void q_diagonal_add(const int* __restrict__ qrp, const int* __restrict__ qcol,
                               const double* __restrict__ qval, int n, double* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  double s = 0.0;
  for (int p = qrp[j]; p < qrp[j + 1]; ++p)
    if (qcol[p] == j) s += qval[p];
  out[j] += s;
}

// D = 1, and the long rows of A and A^T (nl: their two numbers, zero before; nullptr: none).
__global__ void scaling_start(int m, double* __restrict__ Dr, int n, double* __restrict__ Dc,
                              const int* __restrict__ rp, const int* __restrict__ rpt, int* nl,
                              int* lm, int* ln) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < m) Dr[t] = 1.0;
  if (t < n) Dc[t] = 1.0;
  if (nl) {
    append_long(rp, m, t, nl, lm);
    append_long(rpt, n, t, nl + 1, ln);
  }
}

__global__ void inv_vec(const double* __restrict__ a, double* __restrict__ b, int k) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < k) b[i] = 1.0 / a[i];
}

// D~ = (Dc * Dc) * D
__global__ void scale_diag(const double* __restrict__ D, const double* __restrict__ Dc, int k,
                           double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < k) out[i] = (Dc[i] * Dc[i]) * D[i];
}

static int grid_for(long long k) { return (int)std::max(1LL, (k + 255) / 256); }
// Four rows per warp (up to 2^21 warps, then grid-stride): every row's dependent load
// chain (row pointer, values and columns, the gathered factor) is in flight at once.  Few
// rows get a warp each, should they be long.
constexpr int kFewRows = 152 * 64;  // one warp each fills the GPU
static int warp_grid(int rows) {
  const int warps = std::max((rows + kGroupRows - 1) / kGroupRows, std::min(rows, kFewRows));
  return (std::max(1, std::min(warps, 1 << 21)) + 7) / 8;
}

cudaError_t compute_scaling(ProblemData& P, int ruiz_iters, bool pock_chambolle) {
  cudaStream_t s = P.s;
  const int m = P.m, n = P.n;
  const bool have = (P.nnz > 0 && m > 0 && n > 0);
  // tmp_rows: the numbers of long rows of A and A^T, then the rows
  int *nl = P.tmp_rows, *lm = nl + 2, *ln = lm + m;
  if (have) cudaMemsetAsync(nl, 0, 2 * sizeof(int), s);
  scaling_start<<<grid_for(std::max(m, n)), 256, 0, s>>>(m, P.Dr, n, P.Dc, P.A.rp, P.At.rp,
                                                         have ? nl : nullptr, lm, ln);
  const LongRows la{nl, lm}, lat{nl + 1, ln};
  if (P.nnz) cudaMemcpyAsync(P.val_s, P.val, sizeof(double) * P.nnz, cudaMemcpyDeviceToDevice, s);
  const int mf = have ? m : 0;  // rows whose factors change
  const double* qd = nullptr;
  if (P.is_qp && n) {
    q_diagonal<<<grid_for(n), 256, 0, s>>>(P.F.rp, P.fval, P.D, n, P.qdiag);
    if (P.q_general)
      q_diagonal_add<<<grid_for(n), 256, 0, s>>>(P.Q.rp, P.Q.col, P.qval, n, P.qdiag);
    qd = P.qdiag;
  }
  // Round t's norms are taken in the pass that applies round t-1's factors, so a
  // round costs one pass over A: (rowred, colred) hold the factors of the last
  // finished round, (rowred2, colred2) receive the next round's norms.
  double *fr = P.rowred, *fc = P.colred, *nr = P.rowred2, *nc = P.colred2;
  bool pending = false;  // factors in (fr, fc) not yet applied to val_s
  for (int t = 0; (have || qd) && t < ruiz_iters; ++t) {
    cudaMemsetAsync(nc, 0, sizeof(double) * n, s);
    if (have)
      scale_pass<false><<<warp_grid(m), 256, 0, s>>>(
          P.A.rp, P.A.col, P.val_s, m, la, pending ? fr : nullptr, pending ? fc : nullptr, nr,
          reinterpret_cast<unsigned long long*>(nc));
    std::swap(fr, nr);
    std::swap(fc, nc);
    factor_update<false><<<grid_for((long long)mf + n), 256, 0, s>>>(fr, mf, P.Dr, fc, n, P.Dc, qd);
    pending = have;
  }
  if ((have || qd) && pock_chambolle) {
    if (have) {
      // apply the last Ruiz factors while summing rows; columns through A^T
      scale_pass<true><<<warp_grid(m), 256, 0, s>>>(P.A.rp, P.A.col, P.val_s, m, la,
                                                    pending ? fr : nullptr,
                                                    pending ? fc : nullptr, nr, nullptr);
      row_abssum<<<warp_grid(n), 256, 0, s>>>(P.At.rp, P.val_s, P.permT, n, lat, nc);
    } else {
      cudaMemsetAsync(nc, 0, sizeof(double) * n, s);
    }
    factor_update<true><<<grid_for((long long)mf + n), 256, 0, s>>>(nr, mf, P.Dr, nc, n, P.Dc, qd);
  }
  // the scaled matrix from the original values and the accumulated factors
  if (have)
    apply_scale<<<warp_grid(m), 256, 0, s>>>(P.A.rp, P.A.col, P.val, P.val_s, m, la, P.Dr, P.Dc);
  if (m) inv_vec<<<grid_for(m), 256, 0, s>>>(P.Dr, P.invDr, m);
  if (n) inv_vec<<<grid_for(n), 256, 0, s>>>(P.Dc, P.invDc, n);
  if (P.is_qp) {
    if (n) scale_diag<<<grid_for(n), 256, 0, s>>>(P.D, P.Dc, n, P.D_s);
    auto scale = [&](const Csr& K, const double* src, double* dst, const double* dc) {
      if (K.cols > kGroupRow) {  // its long rows, in place of those of A
        cudaMemsetAsync(nl, 0, sizeof(int), s);
        find_long<<<grid_for(n), 256, 0, s>>>(K.rp, n, nl, nl + 1);
      }
      apply_scale<<<warp_grid(n), 256, 0, s>>>(
          K.rp, K.col, src, dst, n, LongRows{K.cols > kGroupRow ? nl : nullptr, nl + 1}, P.Dc, dc);
    };
    if (P.f_nnz) scale(P.F, P.fval, P.fval_s, nullptr);                  // F~ = diag(Dc) F
    if (P.q_general && P.Q.nnz) scale(P.Q, P.qval, P.qval_s, P.Dc);      // diag(Dc) Q diag(Dc)
  }
  return cudaGetLastError();
}

// ---- norms of the cost and of the row-bound vector, scaled and unscaled ----

__device__ __forceinline__ double bound_of(double lo, double hi) {
  const bool fl = isfinite(lo), fu = isfinite(hi);
  if (fl && fu) return (fabs(lo) >= fabs(hi)) ? lo : hi;
  if (fl) return lo;
  if (fu) return hi;
  return 0.0;
}

__global__ void norms_partial(const double* __restrict__ c, const double* __restrict__ lc,
                              const double* __restrict__ uc, const double* __restrict__ Dr,
                              const double* __restrict__ Dc, int m, int n,
                              double* __restrict__ part) {
  __shared__ double sh[32];
  double s0 = 0, s1 = 0, s2 = 0, s3 = 0;
  const int stride = gridDim.x * blockDim.x;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
    const double cs = Dc[j] * c[j];
    s0 += cs * cs;
    s2 += c[j] * c[j];
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
    const double b = bound_of(lc[i], uc[i]);
    const double bs = bound_of(Dr[i] * lc[i], Dr[i] * uc[i]);
    s1 += bs * bs;
    s3 += b * b;
  }
  const double r0 = block_sum(s0, sh);
  const double r1 = block_sum(s1, sh);
  const double r2 = block_sum(s2, sh);
  const double r3 = block_sum(s3, sh);
  if (threadIdx.x == 0) {
    part[0 * gridDim.x + blockIdx.x] = r0;
    part[1 * gridDim.x + blockIdx.x] = r1;
    part[2 * gridDim.x + blockIdx.x] = r2;
    part[3 * gridDim.x + blockIdx.x] = r3;
  }
}

__global__ void finalize_sqrt_sums(const double* __restrict__ part, int nb, int nq,
                                   double* __restrict__ out) {
  __shared__ double sh[32];
  for (int q = 0; q < nq; ++q) {
    double v = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) v += part[q * nb + b];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) out[q] = sqrt(v);
  }
}

cudaError_t bound_and_cost_norms(ProblemData& P) {
  norms_partial<<<kRedBlocks, 256, 0, P.s>>>(P.c, P.lc, P.uc, P.Dr, P.Dc, P.m, P.n, P.red);
  finalize_sqrt_sums<<<1, 256, 0, P.s>>>(P.red, kRedBlocks, 4, P.red_out);
  return cudaGetLastError();
}

// ---- casts ----

template <typename T>
__global__ void k_gather_cast(const double* __restrict__ src, const int* __restrict__ perm,
                              T* __restrict__ dst, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    dst[i] = (T)(perm ? src[perm[i]] : src[i]);
}

template <typename T>
__global__ void k_scale_cast(const double* __restrict__ src, const double* __restrict__ d,
                             bool divide, T* __restrict__ dst, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double v = src[i];
    if (d) v = divide ? v / d[i] : v * d[i];
    dst[i] = (T)v;
  }
}

template <typename T>
cudaError_t gather_cast(const double* src, const int* perm, T* dst, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_gather_cast<T><<<std::min(4096, grid_for(n)), 256, 0, s>>>(src, perm, dst, n);
  return cudaGetLastError();
}
template <typename T>
cudaError_t cast_vec(const double* src, T* dst, int n, cudaStream_t s) {
  return gather_cast<T>(src, nullptr, dst, n, s);
}
template <typename T>
cudaError_t scale_cast(const double* src, const double* d, bool divide, T* dst, int n,
                       cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_scale_cast<T><<<std::min(4096, grid_for(n)), 256, 0, s>>>(src, d, divide, dst, n);
  return cudaGetLastError();
}

template cudaError_t gather_cast<double>(const double*, const int*, double*, int, cudaStream_t);
template cudaError_t gather_cast<float>(const double*, const int*, float*, int, cudaStream_t);
template cudaError_t cast_vec<double>(const double*, double*, int, cudaStream_t);
template cudaError_t cast_vec<float>(const double*, float*, int, cudaStream_t);
template cudaError_t scale_cast<double>(const double*, const double*, bool, double*, int,
                                        cudaStream_t);
template cudaError_t scale_cast<float>(const double*, const double*, bool, float*, int,
                                       cudaStream_t);

}  // namespace mpax
