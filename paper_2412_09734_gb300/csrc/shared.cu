// Batch of LPs sharing one dense constraint matrix: B instances
//     min c_k^T x  s.t.  lc <= A x <= uc,  l <= x <= u,   k = 0..B-1,
// solved together by r^2HPDHG (Algorithm 1) with per-instance step sizes,
// primal weights, restarts and termination.  Stacking the instances' iterates
// as the columns of X (n x B) and Y (m x B) turns the two matrix-vector products
// of every iteration into dense GEMMs, A X and A^T Y (the paper batches
// same-shape instances by vectorisation, Sec. 3.2; with a shared A the batched
// product is a dense contraction), which run on the tensor cores.
//
// Precision: the scaled matrix and the iterates are split into BF16 pairs
// v = v_hi + v_lo (v_hi = bf16(v), v_lo = bf16(v - v_hi)); each product is the
// sum of three BF16 GEMMs with FP32 accumulation, A_hi X_lo + A_lo X_hi +
// A_hi X_hi: each operand keeps about 16 significant bits and the dropped
// A_lo X_lo term is of order 2^-16 relative, so a product is accurate to about
// 2^-16 relative per term (an FP32 product: 2^-24).  The split of
// the iterates is written by the fused update kernels, so a GEMM reads BF16
// operands only.  The products are the kernels of umma.cuh; the PDHG update,
// projection, Halpern step, splitting and the FP64 check reductions are this
// file's kernels.  The plain FP32 products (sgemm.cuh) run on the FP32 pipes.
//
// Layout: A is row-major m x n, i.e. column-major n x m; X, Y and every
// per-instance vector are column-major (column k = instance k).
#include <cuda_bf16.h>

#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/mpax.h"
#include "umma_host.h"
#include "common.cuh"
#include "float_pair.h"
#include "rules.h"
#include "sgemm.cuh"

namespace mpax {

namespace {

int g1(long long k) { return (int)std::max(1LL, std::min(8192LL, (k + 255) / 256)); }
// Grid of the per-instance elementwise kernels: x over `len` coordinates (256
// threads, up to 4 coordinates each), y over the B instances (65,535 at most; the
// kernels loop over the rest).
dim3 grid2d(long long len, int B) {
  const long long bx = std::max(1LL, std::min(1024LL, (len + 1023) / 1024));
  return dim3((unsigned)bx, (unsigned)std::max(1, std::min(B, 65535)));
}

// Threads of a block that walks the `len` items of one instance: whole warps, no more than
// there are items.  A block of a small instance holds its SM for one chain of memory round
// trips however few of its threads work, so the blocks in flight count: 20,000 instances of
// 8 x 12, 640 iterations, 48.0 ms with 256 threads, 37.5 ms with a warp.
int row_threads(long long len, int most) {
  return (int)std::max(32LL, std::min((long long)most, (len + 31) / 32 * 32));
}
// Grid of the updates: V coordinates per thread and pass, x over the coordinates of an
// instance, y over the instances.
dim3 update_grid(long long len, int B, int V, int threads) {
  const long long per = (long long)threads * V;
  const long long bx = std::max(1LL, std::min(1024LL, (len + per - 1) / per));
  return dim3((unsigned)bx, (unsigned)std::max(1, std::min(B, 65535)));
}
// Chunks of the check reductions of B instances of `len` coordinates: blocks of at
// least 2048 coordinates, about eight per SM in all.
int check_chunks(long long len, int B) {
  const long long want = (8LL * 152 + B - 1) / B;
  return (int)std::max(1LL, std::min(want, (len + 2047) / 2048));
}

mpax_status sfail(mpax_status s, const std::string& m) {
  set_last_error(m.c_str());
  return s;
}

// ---- per-instance state --------------------------------------------------------
struct Inst {
  double tau, sigma, omega, r_anchor, r_prev, rel, pobj, dobj, c_norm, best_rel;
  long long k, total, restarts, done_at, checks, stall_count;
  int done, status, restart, have_anchor, stalled;
};

__device__ __forceinline__ void split_store(float v, __nv_bfloat16* hi, __nv_bfloat16* lo,
                                            size_t e) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  hi[e] = h;
  lo[e] = __float2bfloat16_rn(v - __bfloat162float(h));
}

template <int V>
__device__ __forceinline__ void ld_vec(const float* p, size_t e, float* v) {
  if constexpr (V == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p + e);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
  } else {
    v[0] = p[e];
  }
}
template <int V>
__device__ __forceinline__ void st_vec(float* p, size_t e, const float* v) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(p + e) = make_float4(v[0], v[1], v[2], v[3]);
  else p[e] = v[0];
}
template <int V>
__device__ __forceinline__ void split_vec(const float* v, __nv_bfloat16* hi, __nv_bfloat16* lo,
                                          size_t e) {
  if constexpr (V == 4) {
    __nv_bfloat16 h[4], r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      h[i] = __float2bfloat16_rn(v[i]);
      r[i] = __float2bfloat16_rn(v[i] - __bfloat162float(h[i]));
    }
    *reinterpret_cast<uint2*>(hi + e) = *reinterpret_cast<const uint2*>(h);
    *reinterpret_cast<uint2*>(lo + e) = *reinterpret_cast<const uint2*>(r);
  } else {
    split_store(v[0], hi, lo, e);
  }
}
// ---- dense scaling (row-major m x n): Ruiz and Pock-Chambolle rounds -------------
// One pass over A per Ruiz round: it applies the last round's factors, writes the
// rescaled value and reduces its row and column maximum.  A tile is kDenseRows rows by
// 256 V columns; a thread keeps its V column maxima in registers down the tile, a row's
// V values are reduced across the warp.  Maxima are exact in any order and go through
// integer atomics on the bit patterns of the non-negative floats.
//
// The pass is bound by HBM (one read, and one write from the second round on) only if
// it keeps off the FP64 pipe (two lanes per SM and cycle), so the scaled value
// fl32((a r) c), r and c in FP64, is formed from float pairs (float_pair.h): the result is
// that of the FP64 products, bit for bit (the BF16 splits of the products that follow turn
// any other last bit into a 2^-17 one).
// Measured on 8192 x 16384 (0.54 GB): row maxima 0.79 ms, column maxima 1.88 ms and
// scaling 1.00 ms before; one pass 0.16 ms (6.5 TB/s) now.
constexpr int kDenseRows = 64;  // rows of a tile
struct DensePass {
  const float* src;
  float* dst;
  int m, n;
  int ctiles;                   // column tiles; block b takes tile (b / ctiles, b % ctiles)
  const float2 *fr, *fc;        // factors as float pairs
  const double *dr, *dc;        // the same in FP64
  unsigned *rowmax, *colmax;    // norms of a Ruiz round (float bits, start at 0)
  __nv_bfloat16 *hi, *lo;       // BF16 split of the result (rows of ldh)
  long long ldh;
};

template <int V, bool kFactor, bool kMax, bool kWrite, bool kSplit>
__global__ void __launch_bounds__(256) k_dense_pass(DensePass a) {
  __shared__ unsigned srow[kDenseRows];
  const int ct = blockIdx.x % a.ctiles, rt = blockIdx.x / a.ctiles;
  const int j = (ct * 256 + threadIdx.x) * V;
  const int r0 = rt * kDenseRows, r1 = min(a.m, r0 + kDenseRows);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool in = j < a.n;  // V = 4: n is a multiple of 4
  if (kMax && threadIdx.x < kDenseRows) srow[threadIdx.x] = 0u;
  if (kMax) __syncthreads();
  float2 fc[V];
  float cmax[V];
#pragma unroll
  for (int i = 0; i < V; ++i) {
    fc[i] = (kFactor && in) ? a.fc[j + i] : make_float2(1.0f, 0.0f);
    cmax[i] = 0.0f;
  }
  constexpr int U = 4;  // rows in flight
  for (int rb = r0; rb < r1; rb += U) {
    float v[U][V];
#pragma unroll
    for (int t = 0; t < U; ++t) {
#pragma unroll
      for (int i = 0; i < V; ++i) v[t][i] = 0.0f;
      if (in && rb + t < r1) ld_vec<V>(a.src, (size_t)(rb + t) * a.n + j, v[t]);
    }
#pragma unroll
    for (int t = 0; t < U; ++t) {
      const int r = rb + t;
      if (r >= r1) break;
      if constexpr (kFactor) {
        const float2 fr = a.fr[r];
#pragma unroll
        for (int i = 0; i < V; ++i)
          if (in) v[t][i] = scale_pair(v[t][i], fr, fc[i], a.dr + r, a.dc + j + i);
      }
      if (kWrite && in) st_vec<V>(a.dst, (size_t)r * a.n + j, v[t]);
      if constexpr (kSplit) {
        if (in) split_vec<V>(v[t], a.hi, a.lo, (size_t)r * a.ldh + j);
      }
      if constexpr (kMax) {
        float rm = 0.0f;
#pragma unroll
        for (int i = 0; i < V; ++i) {
          const float w = fabsf(v[t][i]);
          rm = fmaxf(rm, w);
          cmax[i] = fmaxf(cmax[i], w);
        }
        const unsigned wm = __reduce_max_sync(0xffffffffu, __float_as_uint(rm));
        if (lane == 0) atomicMax(&srow[r - r0], wm);
      }
    }
  }
  if constexpr (kMax) {
#pragma unroll
    for (int i = 0; i < V; ++i)
      if (in) atomicMax(a.colmax + j + i, __float_as_uint(cmax[i]));
    __syncthreads();
    if (threadIdx.x < r1 - r0) atomicMax(a.rowmax + r0 + threadIdx.x, srow[threadIdx.x]);
  }
}

// Pock-Chambolle norms in FP64: row sums, a block per row (each thread every 256th
// value, then a fixed tree), and column sums, a thread per column down the rows in
// blocks of kColThreads.  The column sums are bound by the FP64 pipe of the SMs that
// hold a block (a conversion and an addition per value), hence blocks narrower than
// 256, and by the loads in flight, hence 32 unconditional ones per thread: 0.75 ms on
// 8192 x 16384 (1.88 ms with 256 threads and one row at a time; one-warp blocks would
// reach every SM but read 128 bytes a row, 3.7 ms).  The row sums take 0.53 ms, their
// FP64 pipe time.
constexpr int kColThreads = 128;
__global__ void k_row_sum(const float* __restrict__ A, int m, int n, double* __restrict__ out) {
  __shared__ double sh[32];
  for (int i = blockIdx.x; i < m; i += gridDim.x) {
    double acc = 0.0;
    const float* r = A + (size_t)i * n;
#pragma unroll 4
    for (int j = threadIdx.x; j < n; j += blockDim.x) acc += fabs((double)r[j]);
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) out[i] = acc;
    __syncthreads();
  }
}
__global__ void __launch_bounds__(kColThreads) k_col_sum(const float* __restrict__ A, int m,
                                                         int n, double* __restrict__ out) {
  constexpr int U = 32;
  const int j = blockIdx.x * kColThreads + threadIdx.x;
  if (j >= n) return;
  double acc = 0.0;
  const float* p = A + j;
  int i = 0;
  for (; i + U <= m; i += U, p += (size_t)U * n) {
    float v[U];
#pragma unroll
    for (int t = 0; t < U; ++t) v[t] = p[(size_t)t * n];
#pragma unroll
    for (int t = 0; t < U; ++t) acc += fabs((double)v[t]);
  }
  for (; i < m; ++i, p += n) acc += fabs((double)*p);
  out[j] = acc;
}

// The factors of a finished round, d = 1/sqrt(norm) (1 for an empty row or column),
// rows then columns: D *= d; d (over dr, dc) and its float pair are stored.  Norms are
// the float bits nmax (reset to zero for the next round) or, without them, dr and dc.
__global__ void k_dense_factor(int m, int n, unsigned* __restrict__ nmax, double* __restrict__ Dr,
                               double* __restrict__ Dc, double* __restrict__ dr,
                               double* __restrict__ dc, float2* __restrict__ fr,
                               float2* __restrict__ fc) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m + n) return;
  const bool row = t < m;
  const int i = row ? t : t - m;
  const double v = nmax ? (double)__uint_as_float(nmax[t]) : (row ? dr : dc)[i];
  if (nmax) nmax[t] = 0u;
  const double d = v > 0.0 ? 1.0 / sqrt(v) : 1.0;
  (row ? Dr : Dc)[i] *= d;
  (row ? dr : dc)[i] = d;
  (row ? fr : fc)[i] = float_pair<float2>(d);
}

// The accumulated factors (rows then columns): float pairs and inverses.
__global__ void k_dense_final(int m, int n, const double* __restrict__ Dr,
                              const double* __restrict__ Dc, float2* __restrict__ fr,
                              float2* __restrict__ fc, double* __restrict__ iDr,
                              double* __restrict__ iDc) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m + n) return;
  const bool row = t < m;
  const int i = row ? t : t - m;
  const double d = (row ? Dr : Dc)[i];
  (row ? fr : fc)[i] = float_pair<float2>(d);
  (row ? iDr : iDc)[i] = 1.0 / d;
}

// D = 1, maxima = 0 at the start of a scaling
__global__ void k_dense_init(int m, int n, double* __restrict__ Dr, double* __restrict__ Dc,
                             unsigned* __restrict__ nmax) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m + n) return;
  if (t < m) Dr[t] = 1.0;
  else Dc[t - m] = 1.0;
  nmax[t] = 0u;
}

// Four columns per thread where every row starts on 16 bytes (the buffers are the
// library's own), else one.
int dense_col_tiles(int n) { return (int)(n % 4 == 0 ? (n + 1023LL) / 1024 : (n + 255LL) / 256); }

template <bool kFactor, bool kMax, bool kWrite, bool kSplit>
void dense_pass(const DensePass& a, cudaStream_t s) {
  const unsigned g = (unsigned)a.ctiles * (unsigned)((a.m + kDenseRows - 1) / kDenseRows);
  if (a.n % 4 == 0) k_dense_pass<4, kFactor, kMax, kWrite, kSplit><<<g, 256, 0, s>>>(a);
  else k_dense_pass<1, kFactor, kMax, kWrite, kSplit><<<g, 256, 0, s>>>(a);
}

// ---- fused updates ----------------------------------------------------------------
struct Vecs {
  int m, n, B;
  const float *ct, *l, *u, *lc, *uc;  // scaled: ct n x B, l/u n, lc/uc m
  float *w, *xa, *xhat, *xprev, *T;     // n x B
  float *y, *ya, *yhat, *yprev, *S;     // m x B
  __nv_bfloat16 *xh_hi, *xh_lo, *y_hi, *y_lo;  // BF16 splits: B rows of ldx / ldy
  Inst* inst;
  const float4* step;                    // per instance: tau, sigma, 1/sigma, running (1 or 0)
  long long ldx, ldy;                    // row strides of the splits (n, m rounded to 8)
};

// Step sizes and Halpern weights of every instance in the precision the updates
// use them in: step[k] = (tau, sigma, 1/sigma, running), and for the iterations
// it0 .. it0 + len - 1 of the block halpern[t * B + k] = (1/(k'+1), 1/(k'+2)), k' the
// instance's counter at iteration it0 + t.  The updates are bound by HBM (24 bytes per
// coordinate), and a double-precision division costs tens of instructions of a pipe
// that takes 16 cycles for a warp, so none may run per coordinate.  Measured on 512
// instances of 8192 x 16384: with the divisions in the updates 124 us (primal) and
// 109 us (dual), from this table with 128-bit accesses 32 us (6.3 TB/s) and 13.7 us.
constexpr int kCoefIters = 256;  // iterations per table, at most
// Iterations per table of B instances: many instances get a shorter table (a launch of it
// costs little beside their updates), or it would take 2 KB of memory for each.
int coef_iters(int B) { return std::max(1, std::min(kCoefIters, (1 << 22) / B)); }
__global__ void k_coefs(const Inst* __restrict__ inst, int B, int it0, int len,
                        float4* __restrict__ step, float2* __restrict__ halpern) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= B * len) return;
  const int k = t % B;
  const Inst& I = inst[k];
  const long long c = I.k + it0 + t / B;
  halpern[t] = make_float2((float)(1.0 / (double)(c + 1)), (float)(1.0 / (double)(c + 2)));
  if (t < B)
    step[k] = make_float4((float)I.tau, (float)I.sigma, (float)(1.0 / I.sigma), I.done ? 0.f : 1.f);
}

// The sum of `chunks` partial vectors of length len at coordinate e, in order (B = 1:
// the matrix-vector product's partials), the loads of kPartsAhead chunks in flight at once.
// One instance has too few coordinates to hide them otherwise: 1000 x 100,000, primal
// and dual update 7.6 and 6.0 us with eight, 6.2 and 4.6 us with sixteen.
constexpr int kPartsAhead = 16;
template <int V>
__device__ __forceinline__ void sum_parts(const float* part, int chunks, int len, int e, float* t) {
#pragma unroll
  for (int i = 0; i < V; ++i) t[i] = 0.0f;
  int c = 0;
  for (; c + kPartsAhead <= chunks; c += kPartsAhead) {
    float q[kPartsAhead][V];
#pragma unroll
    for (int u = 0; u < kPartsAhead; ++u) ld_vec<V>(part, (size_t)(c + u) * len + e, q[u]);
#pragma unroll
    for (int u = 0; u < kPartsAhead; ++u)
#pragma unroll
      for (int i = 0; i < V; ++i) t[i] += q[u][i];
  }
  for (; c < chunks; ++c) {
    float q[V];
    ld_vec<V>(part, (size_t)c * len + e, q);
#pragma unroll
    for (int i = 0; i < V; ++i) t[i] += q[i];
  }
}

// primal: T = A~^T Y; x = w + (anchor - w)/(k+1); x^ = proj(x - tau (c~ - T));
// w <- 2 x^ - x (BF: also split for the next product).  Check iterations store x^ and x.
// tpart (B = 1 only): T is the sum of the GEMV's tchunks partials, in order.
// Grid: x over V coordinates of an instance per thread, y over instances (update_grid).
template <int V, bool BF>
__global__ void k_primal(Vecs v, const float2* __restrict__ halpern, int check,
                         const float* __restrict__ tpart, int tchunks) {
  for (int k = blockIdx.y; k < v.B; k += gridDim.y) {
    const float4 st = v.step[k];
    if (st.w == 0.0f) continue;
    const float rb = halpern[k].x;  // 1 exactly when the anchor is the iterate
    for (int j = (blockIdx.x * blockDim.x + threadIdx.x) * V; j < v.n;
         j += gridDim.x * blockDim.x * V) {
      const size_t e = (size_t)k * v.n + j;
      float t[V], x0[V], wv[V], c[V], lo[V], hi[V], x[V], xh[V], wn[V];
      if (tpart) sum_parts<V>(tpart, tchunks, v.n, j, t);
      else ld_vec<V>(v.T, e, t);
      ld_vec<V>(v.xa, e, x0);
      ld_vec<V>(v.w, e, wv);
      ld_vec<V>(v.ct, e, c);
      ld_vec<V>(v.l, j, lo);
      ld_vec<V>(v.u, j, hi);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        x[i] = (rb == 1.0f) ? x0[i] : wv[i] + rb * (x0[i] - wv[i]);
        xh[i] = fminf(fmaxf(x[i] - st.x * (c[i] - t[i]), lo[i]), hi[i]);
        wn[i] = 2.0f * xh[i] - x[i];
      }
      st_vec<V>(v.w, e, wn);
      if constexpr (BF) split_vec<V>(wn, v.xh_hi, v.xh_lo, (size_t)k * v.ldx + j);
      if (check) {
        st_vec<V>(v.xhat, e, xh);
        st_vec<V>(v.xprev, e, x);
      }
    }
  }
}

// dual: S = A~ xbar; y^ = sigma (v - proj_[-uc,-lc](v)), v = y/sigma - S;
// y <- z + (anchor - z)/(k+2), z = 2 y^ - y (BF: also split)
// spart (B = 1 only): S is the sum of the GEMV's schunks partials, in order.
template <int V, bool BF>
__global__ void k_dual(Vecs v, const float2* __restrict__ halpern, int check,
                       const float* __restrict__ spart, int schunks) {
  for (int k = blockIdx.y; k < v.B; k += gridDim.y) {
    const float4 st = v.step[k];
    if (st.w == 0.0f) continue;
    const float hb = halpern[k].y;
    for (int i0 = (blockIdx.x * blockDim.x + threadIdx.x) * V; i0 < v.m;
         i0 += gridDim.x * blockDim.x * V) {
      const size_t e = (size_t)k * v.m + i0;
      float s[V], y0[V], ya[V], lc[V], uc[V], yh[V], yn[V];
      if (spart) sum_parts<V>(spart, schunks, v.m, i0, s);
      else ld_vec<V>(v.S, e, s);
      ld_vec<V>(v.y, e, y0);
      ld_vec<V>(v.ya, e, ya);
      ld_vec<V>(v.lc, i0, lc);
      ld_vec<V>(v.uc, i0, uc);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const float vv = y0[i] * st.z - s[i];
        yh[i] = st.y * (vv - fminf(fmaxf(vv, -uc[i]), -lc[i]));
        const float z = 2.0f * yh[i] - y0[i];
        yn[i] = z + hb * (ya[i] - z);
      }
      st_vec<V>(v.y, e, yn);
      if constexpr (BF) split_vec<V>(yn, v.y_hi, v.y_lo, (size_t)k * v.ldy + i0);
      if (check) {
        st_vec<V>(v.yhat, e, yh);
        st_vec<V>(v.yprev, e, y0);
      }
    }
  }
}

// Launches of the two updates: four coordinates per thread where every row of
// the iterates starts on 16 bytes.
void launch_primal(const Vecs& v, bool bf, const float2* halpern, int check, const float* tpart,
                   int tchunks, cudaStream_t s) {
  const int V = v.n % 4 == 0 ? 4 : 1, t = row_threads((v.n + V - 1) / V, 256);
  const dim3 g = update_grid(v.n, v.B, V, t);
  auto kernel = V == 4 ? (bf ? k_primal<4, true> : k_primal<4, false>)
                       : (bf ? k_primal<1, true> : k_primal<1, false>);
  kernel<<<g, t, 0, s>>>(v, halpern, check, tpart, tchunks);
}
void launch_dual(const Vecs& v, bool bf, const float2* halpern, int check, const float* spart,
                 int schunks, cudaStream_t s) {
  const int V = v.m % 4 == 0 ? 4 : 1, t = row_threads((v.m + V - 1) / V, 256);
  const dim3 g = update_grid(v.m, v.B, V, t);
  auto kernel = V == 4 ? (bf ? k_dual<4, true> : k_dual<4, false>)
                       : (bf ? k_dual<1, true> : k_dual<1, false>);
  kernel<<<g, t, 0, s>>>(v, halpern, check, spart, schunks);
}

// Partial sums of a check in FP64: block (c, k) takes chunk c of the coordinates and
// rows of instance k and writes part[(q * chunks + c) * B + k]:
//   q 0-4: |r_d|^2, c x, bound terms, |r_p|^2, row terms of the KKT test at (x^, y^)
//          (S = A~ x^ and T = A~^T y^ were formed by the caller);
//   q 5-8: |x^-x|^2, |x^-anchor|^2, |y^-y|^2, |y^-anchor|^2 of the restart rule.
// With one block per instance a single instance of 100,000 columns took 1.17 ms a
// check on its one SM (0.10 of the dense knapsack's solve); the chunks give every SM a
// part of it.  512 instances of 8192 x 16384: 0.60 ms, bound by the FP64 pipe (about
// 12 operations per coordinate at two lanes per SM and cycle).
constexpr int kCheckParts = 9;
struct CheckArgs {
  int m, n, B, chunks;
  const float *xhat, *yhat, *S, *T, *xprev, *xa, *yprev, *ya;
  const double *Dr, *Dc, *iDr, *iDc, *c0, *lc0, *uc0, *l0, *u0;  // c0: n x B unscaled costs
  double* part;
};

__global__ void k_check_part(CheckArgs a, const Inst* inst) {
  __shared__ double sh[32];
  const int c = blockIdx.x;
  const int np = (a.n + a.chunks - 1) / a.chunks, mp = (a.m + a.chunks - 1) / a.chunks;
  for (int k = blockIdx.y; k < a.B; k += gridDim.y) {
    if (inst[k].done) continue;
    const size_t on = (size_t)k * a.n, om = (size_t)k * a.m;
    double rd2 = 0, cx = 0, bt = 0, p0 = 0, p1 = 0;
    for (int j = c * np + threadIdx.x; j < min(a.n, (c + 1) * np); j += blockDim.x) {
      const double xh = (double)a.xhat[on + j];
      const double aty = (double)a.T[on + j] * a.iDc[j];
      const double x = a.Dc[j] * xh;
      const double cc = a.c0[on + j];
      const double lam = cc - aty;
      const double lo = a.l0[j], hi = a.u0[j];
      const bool lf = isfinite(lo), uf = isfinite(hi);
      const double lh = (lf && uf) ? lam : lf ? fmax(lam, 0.0) : uf ? fmin(lam, 0.0) : 0.0;
      rd2 += (lam - lh) * (lam - lh);
      cx += cc * x;
      bt += (lf ? lo * fmax(lh, 0.0) : 0.0) + (uf ? hi * fmin(lh, 0.0) : 0.0);
      const double d0 = xh - (double)a.xprev[on + j], d1 = xh - (double)a.xa[on + j];
      p0 += d0 * d0;
      p1 += d1 * d1;
    }
    double rp2 = 0, yt = 0, d0 = 0, d1 = 0;
    for (int i = c * mp + threadIdx.x; i < min(a.m, (c + 1) * mp); i += blockDim.x) {
      const double yh = (double)a.yhat[om + i];
      const double ax = (double)a.S[om + i] * a.iDr[i];
      const double lo = a.lc0[i], hi = a.uc0[i];
      const double r = ax - fmin(fmax(ax, lo), hi);
      rp2 += r * r;
      const double y = a.Dr[i] * yh;
      if (y > 0.0 && isfinite(lo)) yt += lo * y;
      if (y < 0.0 && isfinite(hi)) yt += hi * y;
      const double e0 = yh - (double)a.yprev[om + i], e1 = yh - (double)a.ya[om + i];
      d0 += e0 * e0;
      d1 += e1 * e1;
    }
    const double v[kCheckParts] = {rd2, cx, bt, rp2, yt, p0, p1, d0, d1};
#pragma unroll
    for (int q = 0; q < kCheckParts; ++q) {
      const double s = block_sum(v[q], sh);
      if (threadIdx.x == 0) a.part[((size_t)q * a.chunks + c) * a.B + k] = s;
    }
  }
}

struct CheckParams {
  double eps_abs, eps_rel, r_suff, r_nec, r_art, pw_smooth, eta, b_norm;
  long long iter_limit, now_ns, time_limit_ns;
  int B, len, chunks, stall_limit;
};

// The check of every instance after a block of p.len iterations (which advance its
// counters here), from the chunk sums of k_check_part in chunk order.
__global__ void k_check_finalize(Inst* inst, const double* part, CheckParams p) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= p.B) return;
  Inst& I = inst[k];
  I.restart = 0;
  if (I.done) return;
  I.k += p.len;
  I.total += p.len;
  double t[kCheckParts];
#pragma unroll
  for (int q = 0; q < kCheckParts; ++q) t[q] = 0.0;
#pragma unroll 4
  for (int c = 0; c < p.chunks; ++c)
#pragma unroll
    for (int q = 0; q < kCheckParts; ++q) t[q] += part[((size_t)q * p.chunks + c) * p.B + k];
  const double rd2 = t[0], cx = t[1], bt = t[2], rp2 = t[3], yt = t[4], P0 = t[5], P1 = t[6],
               D0 = t[7], D1 = t[8];
  const double nrp = sqrt(rp2), nrd = sqrt(rd2), pobj = cx, dobj = yt + bt;
  const double gap = fabs(pobj - dobj);
  const double rel = fmax(fmax(nrp / (1.0 + p.b_norm), nrd / (1.0 + I.c_norm)),
                          gap / (1.0 + fabs(pobj) + fabs(dobj)));
  I.rel = rel;
  I.pobj = pobj;
  I.dobj = dobj;
  const bool conv = nrp <= p.eps_abs + p.eps_rel * p.b_norm &&
                    nrd <= p.eps_abs + p.eps_rel * I.c_norm &&
                    gap <= p.eps_abs + p.eps_rel * (fabs(pobj) + fabs(dobj));
  int term = 0;
  if (!isfinite(rel)) term = MPAX_TERM_NUMERICAL_ERROR;
  else if (conv) term = MPAX_TERM_OPTIMAL;
  else if (I.total >= p.iter_limit) term = MPAX_TERM_ITERATION_LIMIT;
  else if (p.now_ns >= p.time_limit_ns) term = MPAX_TERM_TIME_LIMIT;
  if (term) {
    I.done = 1;
    I.status = term;
    I.done_at = p.now_ns;
    return;
  }
  // the BF16x3 floor (the single-problem rule): no 10% improvement of the KKT
  // error over max(stall_limit, checks / 4) checks marks the instance stalled;
  // the host then continues the batch with FP32 products
  I.checks += 1;
  if (p.stall_limit > 0 && !I.stalled) {
    const long long window = p.stall_limit > I.checks / 4 ? (long long)p.stall_limit : I.checks / 4;
    if (rel < 0.9 * I.best_rel) {
      I.best_rel = rel;
      I.stall_count = 0;
    } else if (++I.stall_count >= window) {
      I.stalled = 1;
    }
  }
  const double r = sqrt(I.omega * P0 + D0 / I.omega);
  const bool restart = !I.have_anchor || r <= p.r_suff * I.r_anchor ||
                       (r <= p.r_nec * I.r_anchor && r > I.r_prev) ||
                       (double)I.k >= p.r_art * (double)I.total;
  if (restart) {
    const double dx = sqrt(P1), dy = sqrt(D1);
    if (dx > 1e-10 && dy > 1e-10)
      I.omega = exp(p.pw_smooth * log(dy / dx) + (1.0 - p.pw_smooth) * log(I.omega));
    I.tau = p.eta / I.omega;
    I.sigma = p.eta * I.omega;
    I.have_anchor = 1;
    I.r_anchor = r;
    I.r_prev = r;
    I.k = 0;
    I.restarts += 1;
    I.restart = 1;
  } else {
    I.r_prev = r;
  }
}

__global__ void k_restart_apply(Vecs v, int bf) {
  const int tot = v.n + v.m;
  for (int k = blockIdx.y; k < v.B; k += gridDim.y) {
    if (!v.inst[k].restart) continue;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += gridDim.x * blockDim.x) {
      if (t < v.n) {
        const size_t e = (size_t)k * v.n + t;
        const float xh = v.xhat[e];
        v.xa[e] = xh;
        v.w[e] = xh;
        if (bf) split_store(xh, v.xh_hi, v.xh_lo, (size_t)k * v.ldx + t);
      } else {
        const size_t f = (size_t)k * v.m + (t - v.n);
        const float yh = v.yhat[f];
        v.ya[f] = yh;
        v.y[f] = yh;
        if (bf) split_store(yh, v.y_hi, v.y_lo, (size_t)k * v.ldy + (t - v.n));
      }
    }
  }
}

__global__ void k_init_inst(Inst* inst, int B, const double* cnorm_s, const double* cnorm,
                            double bnorm_s, double eta) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= B) return;
  Inst I;
  memset(&I, 0, sizeof(I));
  const double nc = cnorm_s[k];
  I.omega = (nc > 1e-10 && bnorm_s > 1e-10) ? nc / bnorm_s : 1.0;
  I.tau = eta / I.omega;
  I.sigma = eta * I.omega;
  I.c_norm = cnorm[k];
  I.rel = INFINITY;
  I.best_rel = INFINITY;
  inst[k] = I;
}

// ||column k||_2 of an n x B column-major double matrix, optionally scaled by D
__global__ void k_colnorm(const double* __restrict__ Cm, const double* __restrict__ D, int n,
                          double* __restrict__ out) {
  __shared__ double sh[32];
  const int k = blockIdx.x;
  double s = 0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double v = Cm[(size_t)k * n + j] * (D ? D[j] : 1.0);
    s += v * v;
  }
  s = block_sum(s, sh);
  if (threadIdx.x == 0) out[k] = sqrt(s);
}

__global__ void k_scale_costs(const double* __restrict__ C0, const double* __restrict__ Dc, int n,
                              size_t total, float* __restrict__ ct) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x)
    ct[e] = (float)(C0[e] * Dc[e % n]);
}

__global__ void k_scale_vec(const double* __restrict__ v, const double* __restrict__ D, int div,
                            int n, float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (float)(div ? v[i] / D[i] : v[i] * D[i]);
}

__global__ void k_unscale_out(const float* __restrict__ v, const double* __restrict__ D, int n,
                              size_t total, double* __restrict__ out) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x)
    out[e] = D[e % n] * (double)v[e];
}

__global__ void k_bound_norm(const double* lc, const double* uc, const double* Dr, int m,
                             double* out) {
  __shared__ double sh[32];
  double s = 0, ss = 0;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const double lo = lc[i], hi = uc[i];
    auto bnd = [](double a, double b) {
      const bool fa = isfinite(a), fb = isfinite(b);
      if (fa && fb) return fabs(a) >= fabs(b) ? a : b;
      if (fa) return a;
      if (fb) return b;
      return 0.0;
    };
    const double b = bnd(lo, hi), bs = bnd(lo * Dr[i], hi * Dr[i]);
    s += b * b;
    ss += bs * bs;
  }
  s = block_sum(s, sh);
  __syncthreads();
  ss = block_sum(ss, sh);
  if (threadIdx.x == 0) {
    out[0] = sqrt(s);
    out[1] = sqrt(ss);
  }
}

// ---- power iteration for ||A~||_2 on the device ------------------------------------
// A round is w = A~ v, g = A~^T w (the matrix-vector kernels below), v = g / ||g||; its
// norm, stop rule and estimate stay on the device, so the host reads the state once
// every kPowerBatch rounds.  Rounds launched past the last return at once.
// Bound by the two reads of A per round (0.54 GB at 8192 x 16384: 80 us each); with the
// norm in one block, the rescaling and a host round trip per round a round took 205 us.
constexpr int kPowerBatch = 8;
constexpr int kPowerBlocks = 512;  // at most: every block of k_power_scale adds all partials
struct PowerState {
  double nu, prev, d_prev;
  int done;    // the round that ended the iteration, 0 while it runs
  int rounds;  // rounds taken
};

// Sum of the block partials part[0..nb) in a fixed order, returned to every thread.
__device__ __forceinline__ double sum_to_all(const double* __restrict__ part, int nb, double* sh) {
  double s = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) s += part[b];
  s = block_sum(s, sh);
  __shared__ double all;
  if (threadIdx.x == 0) all = s;
  __syncthreads();
  return all;
}

// Start vector (power_start_raw): squares per block, then v = raw / ||raw||.
__global__ void k_power_start_sq(int n, double* __restrict__ part, PowerState* st) {
  __shared__ double sh[32];
  const int j0 = blockIdx.x * blockDim.x + threadIdx.x;
  double q = 0.0;
  for (int j = j0; j < n; j += gridDim.x * blockDim.x) {
    const double r = power_start_raw(j);
    q += r * r;
  }
  const double s = block_sum(q, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
  if (j0 == 0) *st = PowerState{0.0, 0.0, 0.0, 0, 0};
}
__global__ void k_power_start_vec(int n, const double* __restrict__ part, float* __restrict__ v) {
  __shared__ double sh[32];
  const double ss = sum_to_all(part, gridDim.x, sh);
  const double inv = 1.0 / sqrt(ss > 0.0 ? ss : 1.0);
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    v[j] = (float)(power_start_raw(j) * inv);
}

// g_j = the sum of the product's chunk partials in order; squares of g per block.
__global__ void k_power_sum(const float* __restrict__ gpart, int chunks, int n,
                            float* __restrict__ g, double* __restrict__ part,
                            const PowerState* st) {
  __shared__ double sh[32];
  if (st->done) return;
  double q = 0.0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    float t = 0.0f;
#pragma unroll 8
    for (int c = 0; c < chunks; ++c) t += gpart[(size_t)c * n + j];
    g[j] = t;
    q += (double)t * (double)t;
  }
  const double s = block_sum(q, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// End of round t: v = g / ||g||, and in block 0 the stop rule (power_stop) and the
// estimate.  Block 0 may set `done` to t while other blocks start, hence the rule that
// takes no notice of this launch's own round.
__global__ void k_power_scale(float* __restrict__ v, int n, const double* __restrict__ part,
                              PowerState* st, int t, int max_iter, double tol, double cap) {
  __shared__ double sh[32];
  if (power_round_over(st->done, t)) return;
  const double nrm = sqrt(sum_to_all(part, gridDim.x, sh));
  const double inv = nrm > 0 ? 1.0 / nrm : 0.0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    v[j] = (float)((double)v[j] * inv);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->rounds = t;
    if (nrm == 0.0) {  // the previous estimate stands
      st->done = t;
      return;
    }
    double nu = sqrt(nrm), est = nu, d = st->d_prev;
    bool stop = t > 1 && power_stop(nu, st->prev, &d, tol, cap, &est);
    if (stop) nu = est;
    else if (t == max_iter && isfinite(cap)) nu = cap;
    st->d_prev = d;
    st->prev = nu;
    st->nu = nu;
    if (stop || t == max_iter) st->done = t;
  }
}

// SPO+ (Sec. 3.4): c' = 2 c_hat - c_true; per instance k (one block),
// loss_k = -c'_k^T x~_k + 2 c_hat_k^T x*_k - z*_k and grad_k = 2 (x*_k - x~_k),
// fixed-order FP64 sums (Elmachtoub and Grigas 2022).
__global__ void k_spo_costs2(const double* __restrict__ c_hat, const double* __restrict__ c_true,
                             size_t len, double* __restrict__ out) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < len;
       t += (size_t)gridDim.x * blockDim.x)
    out[t] = 2.0 * c_hat[t] - c_true[t];
}
__global__ void k_spo_loss2(int n, const double* __restrict__ cp, const double* __restrict__ c_hat,
                            const double* __restrict__ x_true, const double* __restrict__ z_true,
                            const double* __restrict__ x_tl, double* __restrict__ loss,
                            double* __restrict__ grad) {
  __shared__ double sh[32];
  const size_t j0 = (size_t)blockIdx.x * n;
  double v = 0.0, t = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double xt = x_tl[j0 + j], xs = x_true[j0 + j];
    v += cp[j0 + j] * xt;
    t += c_hat[j0 + j] * xs;
    grad[j0 + j] = 2.0 * (xs - xt);
  }
  v = block_sum(v, sh);
  __syncthreads();
  t = block_sum(t, sh);
  if (threadIdx.x == 0) loss[blockIdx.x] = -v + 2.0 * t - z_true[blockIdx.x];
}
__global__ void k_inst_pobj(const Inst* __restrict__ inst, int B, double* __restrict__ v) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < B) v[k] = inst[k].pobj;
}

}  // namespace
}  // namespace mpax

using namespace mpax;

struct mpax_shared {
  int m = 0, n = 0, B = 0;
  cudaStream_t user = nullptr, s = nullptr;
  float* A0 = nullptr;   // original FP32, row-major m x n
  float* As = nullptr;   // scaled FP32
  __nv_bfloat16 *Ahi = nullptr, *Alo = nullptr;
  double *C0 = nullptr, *lc = nullptr, *uc = nullptr, *l = nullptr, *u = nullptr;
  double *Dr = nullptr, *Dc = nullptr, *red_m = nullptr, *red_n = nullptr, *scal = nullptr;
  float *ct = nullptr, *lf = nullptr, *uf = nullptr, *lcf = nullptr, *ucf = nullptr;
  float *w = nullptr, *xa = nullptr, *xhat = nullptr, *T = nullptr, *xprev = nullptr;
  float *y = nullptr, *ya = nullptr, *yhat = nullptr, *S = nullptr, *yprev = nullptr;
  __nv_bfloat16 *xh_hi = nullptr, *xh_lo = nullptr, *y_hi = nullptr, *y_lo = nullptr;
  double *part = nullptr, *cn = nullptr, *cns = nullptr;
  double *iDr = nullptr, *iDc = nullptr;  // 1 / Dr, 1 / Dc
  float2 *fr = nullptr, *fc = nullptr;    // scaling factors of a pass as float pairs
  unsigned* nmax = nullptr;               // row then column maxima of a Ruiz round
  int ctiles = 1;                         // column tiles of a scaling pass
  PowerState* pstate = nullptr;           // power iteration: state and block partials
  double* ppart = nullptr;
  float4* step = nullptr;                 // per-instance step sizes (k_coefs)
  float2* halpern = nullptr;              // Halpern weights of coef_iters iterations (k_coefs)
  int chunks = 1;                         // chunks of the check reductions
  Inst* inst = nullptr;
  double *Xout = nullptr, *Yout = nullptr;
  bool solved = false;
  double solve_seconds = 0.0, norm_A = 0.0;
  long long launches = 0, gemms = 0;
  double gemm_flops = 0.0;
  long long switch_iter = -1;  // last solve: iteration of the switch to FP32 products
  int switch_active = 0;       // last solve: instances still running at the switch
  std::vector<Inst> h_inst;
  // B = 1: partial sums of the A^T y product over gemv_chunks row chunks and of
  // the A w product over gemv_nchunks column chunks
  float* gpart = nullptr;
  float* gpart_n = nullptr;
  double* spo = nullptr;  // SPO+ staging of host arguments: 3 n B + B doubles
  // tensor-core products: BF16 splits are stored with row strides n8, m8 (n, m
  // rounded up to 8, as TMA wants 16-byte strides; the pad columns stay zero)
  long long n8 = 0, m8 = 0;
  UmmaPlan plan_dual, plan_primal;  // S = A~ X (K = n), T = A~^T Y (K = m)
  int* uerr = nullptr;              // set by a bounded wait of the product kernel
  float shape_ms[2][2] = {{0, 0}, {0, 0}};  // tuner: [dual, primal][K block 64, 32] ms
  double prep_seconds = 0.0;   // last solve: scaling, splits, plans, power iteration
  int power_rounds = 0;        // last solve: rounds of the power iteration
  // profile_kernels: event pairs of the iteration products and their sums
  struct ProdEvent {
    cudaEvent_t e0, e1;
    int trans;
  };
  bool profiling = false;
  std::vector<ProdEvent> prof_events;
  double prof_ms[2] = {0, 0};  // [primal (A~^T Y), dual (A~ X)]
  long long prof_n[2] = {0, 0};
  int gemv_chunks = 1, gemv_nchunks = 1;
  long long gemv_launches = 0;
};

namespace {

void free_shared(mpax_shared* sh) {
  if (!sh) return;
  if (sh->s) cudaStreamSynchronize(sh->s);
  void* bufs[] = {sh->A0,  sh->As,   sh->Ahi,   sh->Alo,   sh->C0,   sh->lc,   sh->uc,
                  sh->l,   sh->u,    sh->Dr,    sh->Dc,    sh->red_m, sh->red_n, sh->scal,
                  sh->ct,  sh->lf,   sh->uf,    sh->lcf,   sh->ucf,  sh->w,    sh->xa,
                  sh->xhat, sh->T,   sh->xprev, sh->y,     sh->ya,   sh->yhat, sh->S,
                  sh->yprev, sh->xh_hi, sh->xh_lo, sh->y_hi, sh->y_lo, sh->part, sh->cn,
                  sh->cns, sh->inst, sh->Xout, sh->Yout, sh->gpart, sh->gpart_n, sh->spo,
                  sh->uerr, sh->iDr, sh->iDc, sh->step, sh->halpern, sh->fr, sh->fc,
                  sh->nmax, sh->pstate, sh->ppart};
  for (void* b : bufs)
    if (b) cudaFree(b);
  if (sh->s) cudaStreamDestroy(sh->s);
  delete sh;
}

}  // namespace

// Template kernels sit in a named namespace: the host stubs generated for a
// template kernel name its enclosing unnamed namespace, which is ambiguous in
// this file (mpax's and the global one).
namespace mpax_gemv {

// ---- single instance (B = 1, FP32 products): the two matrix-vector products --------
// With one cost vector each product reads A once and is bound by HBM.  Both are
// plain FP32 sums in a fixed order (no atomics), so results do not depend on the
// schedule.  V = 4: float4 loads (n % 4 == 0 and 16-byte aligned rows), else 1.
constexpr int kGemvThreads = 256;

// part[s][j] = sum_{i in chunk s} A_ij y_i: block (bx, s) covers V * 256 columns
// from bx * V * 256 and the rows [s * rows_per, (s + 1) * rows_per), four rows
// in flight per thread.
template <int V>
__global__ void __launch_bounds__(kGemvThreads) k_gemv_t_part(const float* __restrict__ A, int m,
                                                              int n, const float* __restrict__ y,
                                                              int rows_per,
                                                              float* __restrict__ part,
                                                              const int* skip) {
  if (skip && *skip) return;
  const int j0 = (blockIdx.x * kGemvThreads + threadIdx.x) * V;
  if (j0 >= n) return;
  const int r0 = blockIdx.y * rows_per, r1 = min(m, r0 + rows_per);
  float acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = 0.0f;
  int i = r0;
  for (; i + 4 <= r1; i += 4) {
    float a[4][V];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float* row = A + (size_t)(i + k) * n + j0;
      if constexpr (V == 4) {
        const float4 q = __ldcs(reinterpret_cast<const float4*>(row));
        a[k][0] = q.x;
        a[k][1] = q.y;
        a[k][2] = q.z;
        a[k][3] = q.w;
      } else {
        a[k][0] = __ldcs(row);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float yk = __ldg(y + i + k);
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v] = fmaf(a[k][v], yk, acc[v]);
    }
  }
  for (; i < r1; ++i) {
    const float yk = __ldg(y + i);
    const float* row = A + (size_t)i * n + j0;
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = fmaf(__ldcs(row + v), yk, acc[v]);
  }
  float* out = part + (size_t)blockIdx.y * n + j0;
#pragma unroll
  for (int v = 0; v < V; ++v) out[v] = acc[v];
}

// T_j = sum_s part[s][j], s in order.
__global__ void k_gemv_t_sum(const float* __restrict__ part, int chunks, int n,
                             float* __restrict__ T, const int* skip = nullptr) {
  if (skip && *skip) return;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    float t = 0.0f;
    for (int c = 0; c < chunks; ++c) t += part[(size_t)c * n + j];
    T[j] = t;
  }
}

// part[c][i] = sum_{j in column chunk c} A_ij w_j for R rows per block: block
// (bx, c) covers rows [bx R, bx R + R) and the columns [c cols_per, (c + 1)
// cols_per) (cols_per a multiple of 4).  Each float4 of w is loaded once and used
// for the R rows, so every thread keeps R independent loads of A in flight; the
// R sums are reduced over the block in a fixed order.
constexpr int kGemvRows = 8;
template <int V>
__global__ void __launch_bounds__(kGemvThreads) k_gemv_n_part(const float* __restrict__ A, int m,
                                                              int n, const float* __restrict__ w,
                                                              int cols_per,
                                                              float* __restrict__ part,
                                                              const int* skip) {
  if (skip && *skip) return;
  constexpr int R = kGemvRows;
  __shared__ float sh[R][kGemvThreads / 32];
  const int r0 = blockIdx.x * R;
  const int j0 = blockIdx.y * cols_per, j1 = min(n, j0 + cols_per);
  float acc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = 0.0f;
  const float* rows[R];
#pragma unroll
  for (int r = 0; r < R; ++r) rows[r] = A + (size_t)min(r0 + r, m - 1) * n;  // valid row
  if constexpr (V == 4) {
    for (int q = j0 / 4 + threadIdx.x; q < j1 / 4; q += kGemvThreads) {
      const float4 wv = __ldg(reinterpret_cast<const float4*>(w) + q);
      float4 a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = __ldcs(reinterpret_cast<const float4*>(rows[r]) + q);
#pragma unroll
      for (int r = 0; r < R; ++r)
        acc[r] = fmaf(a[r].x, wv.x, fmaf(a[r].y, wv.y, fmaf(a[r].z, wv.z, fmaf(a[r].w, wv.w, acc[r]))));
    }
  } else {
    for (int j = j0 + threadIdx.x; j < j1; j += kGemvThreads) {
      const float wv = __ldg(w + j);
      float a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = __ldcs(rows[r] + j);
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fmaf(a[r], wv, acc[r]);
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float t = mpax::warp_sum(acc[r]);
    if (lane == 0) sh[r][wid] = t;
  }
  __syncthreads();
  if (threadIdx.x < R && r0 + threadIdx.x < m) {
    float t = 0.0f;
#pragma unroll
    for (int k = 0; k < kGemvThreads / 32; ++k) t += sh[threadIdx.x][k];
    part[(size_t)blockIdx.y * m + r0 + threadIdx.x] = t;
  }
}

}  // namespace mpax_gemv

namespace {

using namespace mpax_gemv;

// B = 1, FP32 products: the partial-sum kernel of one product, trans = 1: A v
// into gpart_n (column chunks), trans = 0: A^T v into gpart (row chunks).  A set
// device flag *skip (nullable) turns the launch into a no-op.
void gemv_part(mpax_shared* sh, int trans, const float* vf, const float* Mf,
               const int* skip = nullptr) {
  const int m = sh->m, n = sh->n;
  const bool v4 = (n % 4 == 0) && ((reinterpret_cast<uintptr_t>(Mf) & 15) == 0) &&
                  ((reinterpret_cast<uintptr_t>(vf) & 15) == 0);
  if (trans) {
    const dim3 grid((m + kGemvRows - 1) / kGemvRows, sh->gemv_nchunks);
    const int cols_per = ((n + sh->gemv_nchunks - 1) / sh->gemv_nchunks + 3) / 4 * 4;
    if (v4) k_gemv_n_part<4><<<grid, kGemvThreads, 0, sh->s>>>(Mf, m, n, vf, cols_per, sh->gpart_n, skip);
    else k_gemv_n_part<1><<<grid, kGemvThreads, 0, sh->s>>>(Mf, m, n, vf, cols_per, sh->gpart_n, skip);
  } else {
    const int V = v4 ? 4 : 1;
    const dim3 grid((n + V * kGemvThreads - 1) / (V * kGemvThreads), sh->gemv_chunks);
    const int rows_per = (m + sh->gemv_chunks - 1) / sh->gemv_chunks;
    if (v4) k_gemv_t_part<4><<<grid, kGemvThreads, 0, sh->s>>>(Mf, m, n, vf, rows_per, sh->gpart, skip);
    else k_gemv_t_part<1><<<grid, kGemvThreads, 0, sh->s>>>(Mf, m, n, vf, rows_per, sh->gpart, skip);
  }
  sh->gemv_launches += 1;
  sh->gemms += 1;
  sh->gemm_flops += 2.0 * m * (double)n;
}

// C (rows x B, col-major) = op(M) V, M the stored column-major n x m matrix
// (A row-major).  trans = 1: C = M^T V (= A V, rows = m, K = n); trans = 0:
// C = M V (= A^T V, rows = n, K = m).  BF16x3 or FP32.
cudaError_t product_impl(mpax_shared* sh, int trans, const __nv_bfloat16* vhi,
                         const __nv_bfloat16* vlo, const float* vf, float* C, bool bf16x3,
                         const float* Mf);

// With profile_kernels set, every iteration product is bracketed by CUDA events
// on the solve's stream; the host sums the times after each check block.
cudaError_t product(mpax_shared* sh, int trans, const __nv_bfloat16* vhi,
                    const __nv_bfloat16* vlo, const float* vf, float* C, bool bf16x3,
                    const float* Mf) {
  if (!sh->profiling) return product_impl(sh, trans, vhi, vlo, vf, C, bf16x3, Mf);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaEventRecord(e0, sh->s);
  const cudaError_t e = product_impl(sh, trans, vhi, vlo, vf, C, bf16x3, Mf);
  cudaEventRecord(e1, sh->s);
  sh->prof_events.push_back({e0, e1, trans});
  return e;
}

void collect_product_times(mpax_shared* sh) {
  for (const auto& pe : sh->prof_events) {
    float ms = 0.f;
    cudaEventSynchronize(pe.e1);
    cudaEventElapsedTime(&ms, pe.e0, pe.e1);
    sh->prof_ms[pe.trans] += ms;
    sh->prof_n[pe.trans] += 1;
    cudaEventDestroy(pe.e0);
    cudaEventDestroy(pe.e1);
  }
  sh->prof_events.clear();
}

cudaError_t product_impl(mpax_shared* sh, int trans, const __nv_bfloat16* vhi,
                         const __nv_bfloat16* vlo, const float* vf, float* C, bool bf16x3,
                         const float* Mf) {
  const int m = sh->m, n = sh->n, B = sh->B;
  const int rows = trans ? m : n, K = trans ? n : m;
  if (!bf16x3 && B == 1) {
    gemv_part(sh, trans, vf, Mf);
    if (trans) k_gemv_t_sum<<<g1(m), 256, 0, sh->s>>>(sh->gpart_n, sh->gemv_nchunks, m, C);
    else k_gemv_t_sum<<<g1(n), 256, 0, sh->s>>>(sh->gpart, sh->gemv_chunks, n, C);
    sh->gemv_launches += 1;
    return cudaGetLastError();
  }
  if (!bf16x3) {
    // FP32 on the CUDA cores: trans = 1 is A~ V (A~ [m][n] K-major), trans = 0
    // is A~^T V (the same storage read M-major)
    sh->gemms += 1;
    sh->gemm_flops += 2.0 * rows * (double)B * K;
    return trans ? sgemm<0>(Mf, n, vf, K, C, rows, rows, B, K, sh->s)
                 : sgemm<1>(Mf, n, vf, K, C, rows, rows, B, K, sh->s);
  }
  // A_hi V_lo + A_lo V_hi + A_hi V_hi in one tensor-core kernel (umma.cuh); the
  // plan of this direction holds the split buffers (vhi, vlo) and the output C
  (void)vhi;
  (void)vlo;
  const UmmaPlan& p = trans ? sh->plan_dual : sh->plan_primal;
  const cudaError_t e = umma_run(p, sh->s);
  sh->gemms += 1;
  sh->gemm_flops += p.flops;
  return e;
}

// The two products' plans.  Their pipeline shape (K block 64 with two stages,
// or 32 with four; the same sums in the same order) is chosen per direction by
// timing both on this solve's own buffers, once per (m, n, B) for the process.
std::mutex& shape_mutex() {
  static std::mutex mu;
  return mu;
}
std::map<std::tuple<int, int, int>, std::pair<int, int>>& shape_cache() {
  static std::map<std::tuple<int, int, int>, std::pair<int, int>> c;
  return c;
}

cudaError_t plan_products(mpax_shared* sh, bool tune) {
  const int m = sh->m, n = sh->n, B = sh->B;
  auto make = [&](UmmaPlan* p, int dir, int bk) {
    return dir == 0 ? umma_plan(p, sh->Ahi, sh->Alo, sh->n8, 0, sh->xh_hi, sh->xh_lo, sh->n8, m,
                                B, n, sh->S, m, sh->uerr, bk)
                    : umma_plan(p, sh->Ahi, sh->Alo, sh->n8, 1, sh->y_hi, sh->y_lo, sh->m8, n,
                                B, m, sh->T, n, sh->uerr, bk);
  };
  const auto key = std::make_tuple(m, n, B);
  std::pair<int, int> bk(32, 32);
  bool have;
  {
    std::lock_guard<std::mutex> g(shape_mutex());
    auto it = shape_cache().find(key);
    have = it != shape_cache().end();
    if (have) bk = it->second;
  }
  cudaError_t e;
  if (!have && tune) {
    // the products write S and T, scratch until the iteration starts
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int best[2] = {32, 32};
    for (int dir = 0; dir < 2; ++dir) {
      float tbest = INFINITY;
      for (int cand : {64, 32}) {
        UmmaPlan p;
        if ((e = make(&p, dir, cand))) return e;
        if ((e = umma_run(p, sh->s))) return e;
        cudaEventRecord(e0, sh->s);
        for (int r = 0; r < 2; ++r) umma_run(p, sh->s);
        cudaEventRecord(e1, sh->s);
        if ((e = cudaEventSynchronize(e1))) return e;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        sh->shape_ms[dir][cand == 64 ? 0 : 1] = ms / 2;
        if (ms < tbest) {
          tbest = ms;
          best[dir] = cand;
        }
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    bk = std::make_pair(best[0], best[1]);
    std::lock_guard<std::mutex> g(shape_mutex());
    shape_cache()[key] = bk;
  }
  if ((e = make(&sh->plan_dual, 0, bk.first))) return e;
  return make(&sh->plan_primal, 1, bk.second);
}

}  // namespace

extern "C" {

mpax_status mpax_lp_shared_create(int32_t m, int32_t n, int32_t B, const float* A,
                                  const double* C, const double* lc, const double* uc,
                                  const double* l, const double* u, mpax_mem_kind kind,
                                  void* cuda_stream, mpax_shared** out) {
  if (!out) return sfail(MPAX_ERR_INVALID_ARGUMENT, "out must not be NULL");
  *out = nullptr;
  if (m < 1 || n < 1 || B < 1) return sfail(MPAX_ERR_INVALID_ARGUMENT, "m, n, B must be >= 1");
  if (!A || !C || !lc || !uc || !l || !u)
    return sfail(MPAX_ERR_INVALID_ARGUMENT, "a required array pointer is NULL");
  mpax_shared* sh = new mpax_shared();
  sh->m = m;
  sh->n = n;
  sh->B = B;
  sh->user = (cudaStream_t)cuda_stream;
  const size_t mn = (size_t)m * n, nB = (size_t)n * B, mB = (size_t)m * B;
  cudaError_t e = cudaStreamCreateWithFlags(&sh->s, cudaStreamNonBlocking);
  auto al = [&](auto** p, size_t cnt) {
    if (!e) e = cudaMalloc((void**)p, sizeof(**p) * std::max<size_t>(cnt, 1));
  };
  al(&sh->A0, mn);
  al(&sh->As, mn);
  sh->n8 = ((long long)n + 7) / 8 * 8;
  sh->m8 = ((long long)m + 7) / 8 * 8;
  al(&sh->Ahi, (size_t)m * sh->n8);
  al(&sh->Alo, (size_t)m * sh->n8);
  al(&sh->C0, nB);
  al(&sh->lc, m);
  al(&sh->uc, m);
  al(&sh->l, n);
  al(&sh->u, n);
  al(&sh->Dr, m);
  al(&sh->Dc, n);
  al(&sh->red_m, m);
  al(&sh->red_n, n);
  al(&sh->scal, 8);
  al(&sh->ct, nB);
  al(&sh->lf, n);
  al(&sh->uf, n);
  al(&sh->lcf, m);
  al(&sh->ucf, m);
  for (float** p : {&sh->w, &sh->xa, &sh->xhat, &sh->T, &sh->xprev}) al(p, nB);
  for (float** p : {&sh->y, &sh->ya, &sh->yhat, &sh->S, &sh->yprev}) al(p, mB);
  al(&sh->xh_hi, (size_t)B * sh->n8);
  al(&sh->xh_lo, (size_t)B * sh->n8);
  al(&sh->y_hi, (size_t)B * sh->m8);
  al(&sh->y_lo, (size_t)B * sh->m8);
  al(&sh->uerr, 1);
  sh->chunks = check_chunks(std::max(m, n), B);
  al(&sh->part, (size_t)kCheckParts * sh->chunks * B);
  al(&sh->iDr, m);
  al(&sh->iDc, n);
  sh->ctiles = dense_col_tiles(n);
  al(&sh->fr, m);
  al(&sh->fc, n);
  al(&sh->nmax, (size_t)m + n);
  al(&sh->pstate, 1);
  al(&sh->ppart, kPowerBlocks);
  al(&sh->step, B);
  al(&sh->halpern, (size_t)coef_iters(B) * B);
  al(&sh->cn, B);
  al(&sh->cns, B);
  al(&sh->inst, B);
  al(&sh->Xout, nB);
  al(&sh->Yout, mB);
  {
    // (every B: the power iteration's matrix-vector products use them too)
    // row chunks of the A^T y product: about four blocks per SM in all
    const long long tiles = (n + 4LL * kGemvThreads - 1) / (4LL * kGemvThreads);
    const long long want = (4LL * 152 + tiles - 1) / tiles;
    sh->gemv_chunks = (int)std::max(1LL, std::min(want, std::max(1LL, (long long)m / 16)));
    al(&sh->gpart, (size_t)sh->gemv_chunks * n);
    // column chunks of the A w product (multiples of 1024 columns)
    const long long groups = (m + kGemvRows - 1) / kGemvRows;
    const long long want_n = (4LL * 152 + groups - 1) / groups;
    sh->gemv_nchunks = (int)std::max(1LL, std::min(want_n, (n + 1023LL) / 1024));
    al(&sh->gpart_n, (size_t)sh->gemv_nchunks * m);
  }
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  for (void* q : {(void*)sh->xh_hi, (void*)sh->xh_lo})
    if (!e) e = cudaMemset(q, 0, sizeof(__nv_bfloat16) * (size_t)B * sh->n8);
  for (void* q : {(void*)sh->y_hi, (void*)sh->y_lo})
    if (!e) e = cudaMemset(q, 0, sizeof(__nv_bfloat16) * (size_t)B * sh->m8);
  if (sh->n8 != n)  // the pad columns of the split matrix stay zero
    for (void* q : {(void*)sh->Ahi, (void*)sh->Alo})
      if (!e) e = cudaMemset(q, 0, sizeof(__nv_bfloat16) * (size_t)m * sh->n8);
  if (!e) e = cudaMemset(sh->uerr, 0, sizeof(int));
  if (!e) e = cudaMemcpy(sh->A0, A, sizeof(float) * mn, k);
  if (!e) e = cudaMemcpy(sh->C0, C, sizeof(double) * nB, k);
  if (!e) e = cudaMemcpy(sh->lc, lc, sizeof(double) * m, k);
  if (!e) e = cudaMemcpy(sh->uc, uc, sizeof(double) * m, k);
  if (!e) e = cudaMemcpy(sh->l, l, sizeof(double) * n, k);
  if (!e) e = cudaMemcpy(sh->u, u, sizeof(double) * n, k);
  if (e) {
    free_shared(sh);
    return sfail(e == cudaErrorMemoryAllocation ? MPAX_ERR_OUT_OF_MEMORY : MPAX_ERR_CUDA,
                 cudaGetErrorString(e));
  }
*out = sh;
  return MPAX_OK;
}

mpax_status mpax_shared_solve(mpax_shared* sh, const mpax_options* o, int32_t fp32_products) {
  if (!sh || !o) return sfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  if (o->reflection_gamma != 1.0 || o->check_every < 1 || o->iteration_limit < 1 ||
      !(o->time_limit >= 0) || o->power_max_iter < 0 ||
      (o->power_max_iter == 0 && !o->pock_chambolle))
    return sfail(MPAX_ERR_INVALID_ARGUMENT, "invalid options (reflection_gamma must be 1)");
  const auto t0 = std::chrono::steady_clock::now();
  const int m = sh->m, n = sh->n, B = sh->B;
  const size_t nB = (size_t)n * B, mB = (size_t)m * B;
  cudaStream_t s = sh->s;
  cudaEvent_t ev;
  cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  cudaEventRecord(ev, sh->user);
  cudaStreamWaitEvent(s, ev, 0);
  long long L = 0;
  sh->gemms = 0;
  sh->profiling = o->profile_kernels != 0;
  sh->prof_ms[0] = sh->prof_ms[1] = 0.0;
  sh->prof_n[0] = sh->prof_n[1] = 0;
  sh->gemm_flops = 0.0;
  sh->gemv_launches = 0;
  // ---- scaling of the shared matrix (Ruiz, Pock-Chambolle) ----------------------
  const int gf = (int)(((long long)m + n + 255) / 256);
  DensePass D{sh->A0, sh->As, m, n, sh->ctiles, sh->fr, sh->fc, sh->red_m, sh->red_n, sh->nmax,
              sh->nmax + m, sh->Ahi, sh->Alo, sh->n8};
  k_dense_init<<<gf, 256, 0, s>>>(m, n, sh->Dr, sh->Dc, sh->nmax);
  for (int t = 0; t < o->ruiz_iters; ++t) {
    if (t == 0) dense_pass<false, true, false, false>(D, s);
    else dense_pass<true, true, true, false>(D, s);
    if (t > 0) D.src = sh->As;
    k_dense_factor<<<gf, 256, 0, s>>>(m, n, sh->nmax, sh->Dr, sh->Dc, sh->red_m, sh->red_n,
                                      sh->fr, sh->fc);
    L += 2;
  }
  if (o->pock_chambolle) {
    if (o->ruiz_iters > 0) {
      dense_pass<true, false, true, false>(D, s);
      D.src = sh->As;
      L += 1;
    }
    k_row_sum<<<std::min(m, 4096), 256, 0, s>>>(D.src, m, n, sh->red_m);
    k_col_sum<<<(n + kColThreads - 1) / kColThreads, kColThreads, 0, s>>>(D.src, m, n, sh->red_n);
    k_dense_factor<<<gf, 256, 0, s>>>(m, n, nullptr, sh->Dr, sh->Dc, sh->red_m, sh->red_n, sh->fr,
                                      sh->fc);
    L += 3;
  }
  // the scaled matrix from the original values, with its split when the products use it
  k_dense_final<<<gf, 256, 0, s>>>(m, n, sh->Dr, sh->Dc, sh->fr, sh->fc, sh->iDr, sh->iDc);
  D.src = sh->A0;
  D.dr = sh->Dr;
  D.dc = sh->Dc;
  if (fp32_products) dense_pass<true, false, true, false>(D, s);
  else dense_pass<true, false, true, true>(D, s);
  {
    cudaError_t pe = plan_products(sh, !fp32_products);
    if (pe) {
      cudaEventDestroy(ev);
      return sfail(MPAX_ERR_CUDA, std::string("tensor-core product plan: ") +
                                      cudaGetErrorString(pe));
    }
  }
  k_scale_costs<<<g1(nB), 256, 0, s>>>(sh->C0, sh->Dc, n, nB, sh->ct);
  k_scale_vec<<<(n + 255) / 256, 256, 0, s>>>(sh->l, sh->Dc, 1, n, sh->lf);
  k_scale_vec<<<(n + 255) / 256, 256, 0, s>>>(sh->u, sh->Dc, 1, n, sh->uf);
  k_scale_vec<<<(m + 255) / 256, 256, 0, s>>>(sh->lc, sh->Dr, 0, m, sh->lcf);
  k_scale_vec<<<(m + 255) / 256, 256, 0, s>>>(sh->uc, sh->Dr, 0, m, sh->ucf);
  L += 8;
  // ---- ||A~||_2 by power iteration (FP32 products, FP64 norms) --------------------
  {
    float* v = sh->T;    // n (first column of T as scratch)
    float* wv = sh->S;   // m
    const int nb = std::min(kPowerBlocks, (n + 255) / 256);
    const double cap = o->pock_chambolle ? 1.0 : INFINITY;
    const int* skip = &sh->pstate->done;
    PowerState ps{};
    if (o->power_max_iter > 0) {
      k_power_start_sq<<<nb, 256, 0, s>>>(n, sh->ppart, sh->pstate);
      k_power_start_vec<<<nb, 256, 0, s>>>(n, sh->ppart, v);
      L += 2;
    }
    for (int t = 1; t <= o->power_max_iter; ++t) {
      // wv = A~ v, v = A~^T wv with this file's matrix-vector kernels
      gemv_part(sh, 1, v, sh->As, skip);
      if (sh->gemv_nchunks > 1) {
        k_gemv_t_sum<<<g1(m), 256, 0, s>>>(sh->gpart_n, sh->gemv_nchunks, m, wv, skip);
        L += 1;
      }
      gemv_part(sh, 0, sh->gemv_nchunks > 1 ? wv : sh->gpart_n, sh->As, skip);
      k_power_sum<<<nb, 256, 0, s>>>(sh->gpart, sh->gemv_chunks, n, v, sh->ppart, sh->pstate);
      k_power_scale<<<nb, 256, 0, s>>>(v, n, sh->ppart, sh->pstate, t, o->power_max_iter,
                                       o->power_tol, cap);
      L += 2;
      if (t % kPowerBatch == 0 || t == o->power_max_iter) {
        cudaMemcpyAsync(&ps, sh->pstate, sizeof(ps), cudaMemcpyDeviceToHost, s);
        if (cudaStreamSynchronize(s) != cudaSuccess || ps.done) break;
      }
    }
    sh->power_rounds = ps.rounds;
    sh->norm_A = o->power_max_iter == 0 ? 1.0 : ps.nu;  // 1: the Pock-Chambolle bound
  }
  const double eta = sh->norm_A > 0 ? o->step_safety / sh->norm_A : 1.0;
  cudaStreamSynchronize(s);
  sh->prep_seconds =
      std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  // ---- per-instance initial state --------------------------------------------------
  const int ct = row_threads(n, 1024);
  k_colnorm<<<B, ct, 0, s>>>(sh->C0, sh->Dc, n, sh->cns);
  k_colnorm<<<B, ct, 0, s>>>(sh->C0, nullptr, n, sh->cn);
  k_bound_norm<<<1, 512, 0, s>>>(sh->lc, sh->uc, sh->Dr, m, sh->scal);
  double bn[2];
  cudaMemcpyAsync(bn, sh->scal, sizeof(bn), cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  k_init_inst<<<(B + 255) / 256, 256, 0, s>>>(sh->inst, B, sh->cns, sh->cn, bn[1], eta);
  for (void* p : {(void*)sh->w, (void*)sh->xa, (void*)sh->xhat})
    cudaMemsetAsync(p, 0, sizeof(float) * nB, s);
  for (void* p : {(void*)sh->y, (void*)sh->ya, (void*)sh->yhat})
    cudaMemsetAsync(p, 0, sizeof(float) * mB, s);
  cudaMemsetAsync(sh->xh_hi, 0, sizeof(__nv_bfloat16) * B * sh->n8, s);
  cudaMemsetAsync(sh->xh_lo, 0, sizeof(__nv_bfloat16) * B * sh->n8, s);
  cudaMemsetAsync(sh->y_hi, 0, sizeof(__nv_bfloat16) * B * sh->m8, s);
  cudaMemsetAsync(sh->y_lo, 0, sizeof(__nv_bfloat16) * B * sh->m8, s);
  cudaMemsetAsync(sh->uerr, 0, sizeof(int), s);
  L += 4;
  bool bf = !fp32_products;
  long long switch_iter = -1;  // iteration at which BF16x3 gave way to FP32 products
  int switch_active = 0;
  Vecs V{m, n, B, sh->ct, sh->lf, sh->uf, sh->lcf, sh->ucf, sh->w, sh->xa, sh->xhat, sh->xprev,
         sh->T, sh->y, sh->ya, sh->yhat, sh->yprev, sh->S, sh->xh_hi, sh->xh_lo, sh->y_hi,
         sh->y_lo, sh->inst, sh->step, sh->n8, sh->m8};
  CheckArgs K{m, n, B, sh->chunks, sh->xhat, sh->yhat, sh->S, sh->T, sh->xprev, sh->xa,
              sh->yprev, sh->ya, sh->Dr, sh->Dc, sh->iDr, sh->iDc, sh->C0, sh->lc, sh->uc,
              sh->l, sh->u, sh->part};
  long long done_iters = 0;
  const int table = coef_iters(B);
  // time limit, checked at each KKT check against the host clock
  const long long tl_ns = o->time_limit >= 9.0e9 ? LLONG_MAX : (long long)(o->time_limit * 1e9);
  std::vector<Inst> hi(B);
  mpax_status result = MPAX_OK;
  while (true) {
    const int len = (int)std::min<long long>(o->check_every, o->iteration_limit - done_iters);
    for (int it = 0; it < len; ++it) {
      const int chk = (it == len - 1);
      const float2* hk = sh->halpern + (size_t)(it % table) * B;
      if (it % table == 0) {
        const int cl = std::min(table, len - it);
        k_coefs<<<(B * cl + 255) / 256, 256, 0, s>>>(sh->inst, B, it, cl, sh->step, sh->halpern);
        L += 1;
      }
      if (B == 1 && !bf) {
        // one instance, FP32: GEMV partials, summed inside the update kernels
        gemv_part(sh, 0, sh->y, sh->As);
        launch_primal(V, false, hk, chk, sh->gpart, sh->gemv_chunks, s);
        gemv_part(sh, 1, sh->w, sh->As);
        launch_dual(V, false, hk, chk, sh->gpart_n, sh->gemv_nchunks, s);
        L += 2;
        continue;
      }
      if (product(sh, 0, sh->y_hi, sh->y_lo, sh->y, sh->T, bf, sh->As)) {
        result = sfail(MPAX_ERR_CUDA, "matrix product launch failed");
        break;
      }
      launch_primal(V, bf, hk, chk, nullptr, 0, s);
      // the dual product reads the reflected point w (FP32) or its BF16 split
      if (product(sh, 1, sh->xh_hi, sh->xh_lo, sh->w, sh->S, bf, sh->As)) {
        result = sfail(MPAX_ERR_CUDA, "matrix product launch failed");
        break;
      }
      launch_dual(V, bf, hk, chk, nullptr, 0, s);
      L += 2;
    }
    if (result) break;
    done_iters += len;
    // KKT products at (x^, y^): S = A~ x^, T = A~^T y^ (BF16x3: the x^/y^ splits reuse
    // the iterates' buffers, which are rebuilt below)
    if (bf) {
      split_rows(sh->xhat, B, n, n, sh->xh_hi, sh->xh_lo, sh->n8, s);
      split_rows(sh->yhat, B, m, m, sh->y_hi, sh->y_lo, sh->m8, s);
      L += 2;
    }
    product(sh, 1, sh->xh_hi, sh->xh_lo, sh->xhat, sh->S, bf, sh->As);
    product(sh, 0, sh->y_hi, sh->y_lo, sh->yhat, sh->T, bf, sh->As);
    k_check_part<<<dim3((unsigned)sh->chunks, (unsigned)std::min(B, 65535)), 256, 0, s>>>(K,
                                                                                     sh->inst);
    CheckParams cp{o->eps_abs, o->eps_rel, o->restart_sufficient, o->restart_necessary,
                   o->restart_artificial, o->primal_weight_smoothing, eta, bn[0],
                   o->iteration_limit,
                   (long long)std::chrono::duration_cast<std::chrono::nanoseconds>(
                       std::chrono::steady_clock::now() - t0).count(),
                   tl_ns, B, len, sh->chunks, (bf && o->fp64_continuation) ? o->stall_checks : 0};
    k_check_finalize<<<(B + 255) / 256, 256, 0, s>>>(sh->inst, sh->part, cp);
    if (bf) {  // the BF16 splits of the iterates again (a restart copies x^, y^ into them)
      split_rows(sh->w, B, n, n, sh->xh_hi, sh->xh_lo, sh->n8, s);
      split_rows(sh->y, B, m, m, sh->y_hi, sh->y_lo, sh->m8, s);
      L += 2;
    }
    k_restart_apply<<<grid2d((long long)n + m, B), 256, 0, s>>>(V, bf);
    L += 3;
    cudaMemcpyAsync(hi.data(), sh->inst, sizeof(Inst) * B, cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    if (sh->profiling) collect_product_times(sh);
    int active = 0, stalled = 0;
    for (const Inst& I : hi) {
      active += !I.done;
      stalled += !I.done && I.stalled;
    }
    if (!active) break;
    if (bf && stalled) {
      // an instance reached the BF16x3 floor: the rest of the solve forms its
      // products in FP32 (the iterates are FP32 throughout, so nothing converts)
      bf = false;
      switch_iter = done_iters;
      switch_active = active;
    }
  }
  if (sh->profiling) collect_product_times(sh);
  cudaError_t e = cudaGetLastError();
  if (!result && e) result = sfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  {
    int herr = 0;
    cudaMemcpyAsync(&herr, sh->uerr, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    if (!result && herr)
      result = sfail(MPAX_ERR_DEVICE_TIMEOUT, "a bounded wait of the tensor-core product gave up");
  }
  k_unscale_out<<<g1(nB), 256, 0, s>>>(sh->xhat, sh->Dc, n, nB, sh->Xout);
  k_unscale_out<<<g1(mB), 256, 0, s>>>(sh->yhat, sh->Dr, m, mB, sh->Yout);
  L += 2;
  cudaStreamSynchronize(s);
  cudaEventRecord(ev, s);
  cudaStreamWaitEvent(sh->user, ev, 0);
  cudaEventDestroy(ev);
  sh->h_inst = hi;
  sh->launches = L + sh->gemv_launches;
  sh->switch_iter = switch_iter;
  sh->switch_active = switch_active;
  sh->solved = !result;
  sh->solve_seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  return result;
}

mpax_status mpax_shared_get_solution(const mpax_shared* sh, double* X, double* Y,
                                     mpax_mem_kind kind) {
  if (!sh) return sfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  if (!sh->solved) return sfail(MPAX_ERR_NOT_SOLVED, "call mpax_shared_solve first");
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  cudaError_t e = cudaSuccess;
  if (X) e = cudaMemcpy(X, sh->Xout, sizeof(double) * (size_t)sh->n * sh->B, k);
  if (!e && Y) e = cudaMemcpy(Y, sh->Yout, sizeof(double) * (size_t)sh->m * sh->B, k);
  if (e) return sfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  return MPAX_OK;
}

mpax_status mpax_shared_get_stats(const mpax_shared* sh, mpax_batch_stats* stats,
                                  int32_t* status, int64_t* iterations, double* rel_kkt,
                                  double* primal_obj, double* seconds, double* gemm_info) {
  if (!sh || !stats) return sfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  if (!sh->solved) return sfail(MPAX_ERR_NOT_SOLVED, "call mpax_shared_solve first");
  std::memset(stats, 0, sizeof(*stats));
  stats->B = sh->B;
  std::vector<double> secs(sh->B);
  for (int k = 0; k < sh->B; ++k) {
    const Inst& I = sh->h_inst[k];
    stats->n_optimal += I.status == MPAX_TERM_OPTIMAL;
    stats->iterations_total += I.total;
    stats->iterations_max = std::max<long long>(stats->iterations_max, I.total);
    stats->restarts_total += I.restarts;
    stats->rel_kkt_max = std::max(stats->rel_kkt_max, I.rel);
    secs[k] = I.done_at * 1e-9;
    if (status) status[k] = I.status;
    if (iterations) iterations[k] = I.total;
    if (rel_kkt) rel_kkt[k] = I.rel;
    if (primal_obj) primal_obj[k] = I.pobj;
    if (seconds) seconds[k] = secs[k];
  }
  std::vector<double> so = secs;
  std::sort(so.begin(), so.end());
  auto pct = [&](double q) {
    const size_t i = std::min<size_t>(so.size() - 1, (size_t)std::ceil(q * so.size()) - 1);
    return so[i];
  };
  stats->instance_seconds_p50 = pct(0.5);
  stats->instance_seconds_p99 = pct(0.99);
  stats->instance_seconds_max = so.back();
  stats->solve_seconds = sh->solve_seconds;
  stats->kernel_launches = sh->launches;
  stats->fp64_instances = sh->switch_active;
  if (gemm_info) {
    gemm_info[0] = (double)sh->gemms;
    gemm_info[1] = sh->gemm_flops;
    gemm_info[2] = sh->norm_A;
    gemm_info[3] = sh->plan_dual.bk;
    gemm_info[4] = sh->plan_primal.bk;
    gemm_info[5] = sh->prof_n[1] ? sh->prof_ms[1] / sh->prof_n[1] : 0.0;
    gemm_info[6] = sh->prof_n[0] ? sh->prof_ms[0] / sh->prof_n[0] : 0.0;
    gemm_info[7] = sh->prep_seconds;
    gemm_info[8] = sh->power_rounds;
  }
  return MPAX_OK;
}

mpax_status mpax_shared_set_costs(mpax_shared* sh, const double* C, mpax_mem_kind kind) {
  if (!sh || !C) return sfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  const cudaMemcpyKind k = kind == MPAX_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  cudaEvent_t ev;
  cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  cudaEventRecord(ev, sh->user);
  cudaStreamWaitEvent(sh->s, ev, 0);
  cudaError_t e = cudaMemcpyAsync(sh->C0, C, sizeof(double) * (size_t)sh->n * sh->B, k, sh->s);
  if (!e) e = cudaStreamSynchronize(sh->s);
  cudaEventDestroy(ev);
  if (e) return sfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  sh->solved = false;
  return MPAX_OK;
}

mpax_status mpax_shared_get_objective(const mpax_shared* sh, double* v, mpax_mem_kind kind) {
  if (!sh || !v) return sfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  if (!sh->solved) return sfail(MPAX_ERR_NOT_SOLVED, "call mpax_shared_solve first");
  cudaError_t e;
  if (kind == MPAX_MEM_HOST) {
    for (int k = 0; k < sh->B; ++k) v[k] = sh->h_inst[k].pobj;
    return MPAX_OK;
  }
  k_inst_pobj<<<(sh->B + 255) / 256, 256, 0, sh->s>>>(sh->inst, sh->B, v);
  e = cudaGetLastError();
  if (!e) e = cudaStreamSynchronize(sh->s);
  if (e) return sfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  return MPAX_OK;
}

mpax_status mpax_shared_spo_plus(mpax_shared* sh, const mpax_options* o, int32_t fp32_products,
                                 const double* C_hat, const double* C_true, const double* X_true,
                                 const double* z_true, double* loss, double* grad,
                                 mpax_mem_kind kind) {
  if (!sh || !o || !C_hat || !C_true || !X_true || !z_true || !loss || !grad)
    return sfail(MPAX_ERR_INVALID_ARGUMENT, "NULL argument");
  const int B = sh->B, n = sh->n;
  const size_t nB = (size_t)n * B;
  cudaStream_t s = sh->s;
  cudaEvent_t ev;
  cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  cudaEventRecord(ev, sh->user);
  cudaStreamWaitEvent(s, ev, 0);
  cudaEventDestroy(ev);
  cudaError_t e = cudaSuccess;
  if (kind == MPAX_MEM_HOST) {
    if (!sh->spo) e = cudaMalloc(&sh->spo, sizeof(double) * (3 * nB + B));
    double* d = sh->spo;
    if (!e) e = cudaMemcpyAsync(d, C_hat, sizeof(double) * nB, cudaMemcpyHostToDevice, s);
    if (!e) e = cudaMemcpyAsync(d + nB, C_true, sizeof(double) * nB, cudaMemcpyHostToDevice, s);
    if (!e) e = cudaMemcpyAsync(d + 2 * nB, X_true, sizeof(double) * nB, cudaMemcpyHostToDevice, s);
    if (!e) e = cudaMemcpyAsync(d + 3 * nB, z_true, sizeof(double) * B, cudaMemcpyHostToDevice, s);
    C_hat = d;
    C_true = d + nB;
    X_true = d + 2 * nB;
    z_true = d + 3 * nB;
  }
  if (!e) {
    k_spo_costs2<<<g1(nB), 256, 0, s>>>(C_hat, C_true, nB, sh->C0);
    e = cudaGetLastError();
  }
  if (!e) e = cudaStreamSynchronize(s);
  if (e) return sfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  mpax_status st = mpax_shared_solve(sh, o, fp32_products);
  if (st) return st;
  double* dl = loss;
  double* dg = grad;
  if (kind == MPAX_MEM_HOST) {
    dg = sh->spo + nB;      // C_true is no longer read
    dl = sh->spo + 3 * nB;  // each block reads z_true[k] before writing loss[k]
  }
  k_spo_loss2<<<B, 256, 0, s>>>(n, sh->C0, C_hat, X_true, z_true, sh->Xout, dl, dg);
  e = cudaGetLastError();
  if (!e && kind == MPAX_MEM_HOST) {
    e = cudaMemcpyAsync(grad, dg, sizeof(double) * nB, cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaMemcpyAsync(loss, dl, sizeof(double) * B, cudaMemcpyDeviceToHost, s);
  }
  if (!e) e = cudaStreamSynchronize(s);
  if (e) return sfail(MPAX_ERR_CUDA, cudaGetErrorString(e));
  return MPAX_OK;
}

void mpax_shared_destroy(mpax_shared* sh) { free_shared(sh); }

}  // extern "C"
