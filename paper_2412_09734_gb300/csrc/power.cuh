// The power iteration of a small or medium problem as ONE cooperative launch.
//
// A round is two products, a reduction and a few scalars; as launches it took two SpMVs,
// two small kernels and every eighth time a host round trip, and a problem may need 50 to
// 450 rounds (preparation of a 200 x 400 LP with 184 rounds 5.1 -> 2.9 ms, of a QP of 200,000
// variables 7.6 -> 6.0 ms, of a 1000 x 2000 LP 1.0 -> 0.7 ms, against the launched rounds on the
// same problem).  Here the grid stays resident, a barrier ends each product,
// a warp takes the same work items in every round (their matrix entries stay in L1) and
// the stop rule is evaluated on the device.  Every item is computed by spmv_item, as the
// launched kernels compute it, so the products are the same bits; the squares are added
// in another fixed order.
//
// v, w and g change during the launch and are read through L2; the matrices are constant
// and go through L1.  The scalars of a round are formed by one thread: a double division
// or root on every thread would take the FP64 pipe (16 cycles per warp instruction) longer
// than the products of a small problem.  The barrier is bounded: a wait that gives up sets
// the error word, its CTA returns, the others follow within their own limit (each decides by
// its own wait alone, so that its threads decide alike), the host restores the words and
// counters that the launch left behind, and the solve reports MPAX_ERR_DEVICE_TIMEOUT.
#pragma once

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "rules.h"
#include "sync.cuh"

namespace mpax {

constexpr int kRoundWarps = 16;  // one CTA per SM, 128 registers a thread
template <typename T>
constexpr int kRoundSmem = kRoundWarps * kSpmvBufLen<T> * (int)sizeof(T);
constexpr int kRoundMaxCtas = 1024;

// Words of the barrier, zero between launches: arrivals, CTAs that left, error.
struct GridBar {
  unsigned* w;
};
constexpr int kGridBarWords = 3;

// All CTAs of the grid (all resident: cooperative launch); phase counts this CTA's
// arrivals.  False when the wait gave up, after `limit_ns` of the device clock.
__device__ __forceinline__ bool grid_sync(const GridBar& b, unsigned& phase,
                                          unsigned long long limit_ns = kWaitNs) {
  __shared__ int s_ok;
  __syncthreads();
  if (gridDim.x == 1) return true;
  if (threadIdx.x == 0) {
    phase += gridDim.x;
    __threadfence();
    atomicAdd(b.w, 1u);
    int ok = 1;
    unsigned long long t0 = 0;
    for (unsigned n = 0;; ++n) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(b.w) : "memory");
      if (barrier_open(v, phase)) break;
      if ((n & 255u) == 255u) {
        const unsigned long long t = globaltimer_ns();
        if (t0 == 0) t0 = t;
        if (t - t0 > limit_ns) {
          atomicExch(b.w + 2, 1u);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// After its last barrier: the last CTA to leave zeroes the counters for the next launch.
__device__ __forceinline__ void grid_leave(const GridBar& b) {
  if (gridDim.x == 1 || threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(b.w + 1, 1u) == gridDim.x - 1) {
    b.w[0] = 0u;
    b.w[1] = 0u;
  }
}

// out_r = s * scale + diag_r * (din_r * dscale); partial [0] sum out^2.
template <typename T>
struct EpiRound {
  static constexpr int NQ = 1;
  struct Pre {
    T d, di;
  };
  T* out;
  const T* diag;  // nullable
  const T* din;
  T scale, dscale;
  int check;
  __device__ __forceinline__ bool skip() const { return false; }
  __device__ __forceinline__ void load() {}
  __device__ __forceinline__ void pre(int r, Pre& p) const {
    p.d = diag ? diag[r] : (T)0;
    p.di = diag ? __ldcg(din + r) : (T)0;
  }
  __device__ __forceinline__ void row(int r, T s, const Pre& p, double* acc) {
    T v = s * scale;
    if (diag) v += p.d * (p.di * dscale);
    out[r] = v;
    if (check) acc[0] += (double)v * (double)v;
  }
};

// This warp's items: warp w of CTA c takes w * CTAs + c, then every CTAs * warps further,
// so that few items spread over the SMs first.
template <typename T, class In, class Epi>
__device__ __forceinline__ void round_items(const SpmvArgs<T>& a, In in, Epi epi, T* buf) {
  const int stride = gridDim.x * kRoundWarps;
  for (int item = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; item < a.n_items; item += stride) {
    spmv_item<T, In, Epi, true>(a, in, epi, item, buf);
    __syncwarp();  // the next item rewrites the warp's buffer
  }
}

// Partials up to which every CTA adds them all; beyond, each CTA adds a chunk and a third
// barrier shares the chunks' sums.
constexpr int kRoundSumAll = 2048;

// two = 1: v -> w = K1 v -> g = K2 w (plus diag v when given); two = 0: g = K2 v.  The next
// round's v is g over its norm, the scale applied in the next product.  root: the norm is
// sqrt(||g||) (A~^T A~), else ||g||.  Every CTA comes to the same sums and decisions; CTA 0
// writes the state.  csum: a double per CTA.
template <typename T>
__global__ void __launch_bounds__(32 * kRoundWarps, 1)
    power_rounds(SpmvArgs<T> a1, SpmvArgs<T> a2, int two, T* v, T* g, T* w, const T* diag, int root,
                 double tol, double cap, int max_iter, double* csum, DevState* st, GridBar bar) {
  extern __shared__ __align__(16) unsigned char round_smem[];
  T* buf = reinterpret_cast<T*>(round_smem) + (threadIdx.x >> 5) * kSpmvBufLen<T>;
  __shared__ double sh[32];
  __shared__ double s_scale, s_nu;
  __shared__ int s_stop;
  unsigned phase = 0;
  double prev = 0.0, d_prev = 0.0;  // thread 0's
  if (threadIdx.x == 0) {
    s_scale = 1.0;
    s_stop = 0;
    s_nu = 0.0;
  }
  __syncthreads();
  int t = 1;
  for (; t <= max_iter; ++t) {
    const T scale = (T)s_scale;
    if (two) {
      round_items(a1, InPlain<T, true>{v}, EpiRound<T>{w, nullptr, nullptr, scale, (T)1, 0}, buf);
      if (!grid_sync(bar, phase)) return;
    }
    round_items(a2, InPlain<T, true>{two ? w : v},
                EpiRound<T>{g, diag, v, two ? (T)1 : scale, scale, 1}, buf);
    if (!grid_sync(bar, phase)) return;
    const double* part = a2.part;
    int np = a2.n_items;
    if (np > kRoundSumAll && gridDim.x > 1) {
      const int lo = (int)((long long)np * blockIdx.x / gridDim.x);
      const int hi = (int)((long long)np * (blockIdx.x + 1) / gridDim.x);
      double q = 0.0;
      for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) q += __ldcg(part + i);
      q = block_sum(q, sh);
      if (threadIdx.x == 0) csum[blockIdx.x] = q;
      if (!grid_sync(bar, phase)) return;
      part = csum;
      np = gridDim.x;
    }
    double q = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) q += __ldcg(part + i);
    q = block_sum(q, sh);
    if (threadIdx.x == 0) {
      const double nrm = sqrt(q);
      if (nrm == 0.0) {
        s_nu = 0.0;
        s_stop = 1;
      } else {
        const double nu = root ? sqrt(nrm) : nrm;
        double est = nu;
        s_scale = 1.0 / nrm;
        s_nu = nu;
        if (t > 1 && power_stop(nu, prev, &d_prev, tol, cap, &est)) {
          s_nu = est;
          s_stop = 1;
        } else if (t >= max_iter && isfinite(cap)) {
          s_nu = cap;  // out of rounds: the certified bound
        }
        prev = nu;
      }
    }
    __syncthreads();
    if (s_stop) break;
    T* sw = v;
    v = g;
    g = sw;
    // the partials are written again by the next round's second product, behind a barrier;
    // without a first product, or with chunk sums, that barrier is this one
    if (!two && !grid_sync(bar, phase)) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->pw_nu = s_nu;
    st->pw_iters = min(t, max_iter);
    st->pw_done = 1;
    if (root) st->norm_A = s_nu;
    else st->norm_Q = s_nu;
  }
  grid_leave(bar);
}

// ---- host side --------------------------------------------------------------------

// CTAs for products of at most `items` items: one while a CTA's barrier is cheaper than
// the grid's, then four items per CTA, at most one CTA per SM.
inline int round_ctas(int items, int sms) {
  if (items <= 8) return 1;
  return std::max(1, std::min(std::min(sms, kRoundMaxCtas), (items + 3) / 4));
}
// Items per warp up to which the single launch is taken; past it the launched kernels'
// occupancy (40 warps per SM) hides the gathers better.
constexpr int kRoundItemsPerWarp = 4;
inline bool round_fits(int items, int sms) {
  return items > 0 && items <= kRoundItemsPerWarp * kRoundWarps * sms;
}

template <class K, class... Args>
cudaError_t launch_cooperative(K kernel, int ctas, int threads, int smem, cudaStream_t s,
                               Args... args) {
  if (smem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace mpax
