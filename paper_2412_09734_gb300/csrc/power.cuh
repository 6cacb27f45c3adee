// The power iteration of a small or medium problem.
//
// A round is two products, a reduction and a few scalars; as launches of the general kernels
// it took two SpMVs, two small kernels and every eighth time a host round trip, and a problem
// may need 50 to 450 rounds.  Here every CTA of a round's first launch adds the partial sums
// that the round before left, for the scale of v, and one CTA more evaluates the stop rule
// meanwhile, so a round is two launches (one for a general Q); a problem of a few work items
// takes all its rounds in ONE launch of one CTA.  Microseconds per round, general kernels -> here, FP64 and FP32:
//   LP 200 x 400 (one CTA)      24.5 -> 12.4    23.3 -> 11.1
//   LP 20,000 x 40,000          32.5 -> 22.3    25.5 -> 18.2
//   LP 150,000 x 99,000         59.0 -> 38.9    36.6 -> 30.1
//   QP of 200,000, both norms    104 -> 73       66 -> 57
// What bounds them: two dependent launches, the gathers of an item and, with thousands of
// items, their partial sums on the FP64 pipe of every SM.
//
// One cooperative launch of all SMs with a grid barrier per product was as fast (12.4, 20.7,
// 42 and 75 us in FP64, 11.2, 17.8, 27.6 and 53 in FP32), but it starts only once all its CTAs
// fit at the same time: beside a batch that kept half of the SMs for 2 s an LP of 38 ms
// waited for the batch's end, and four threads with 20 solves each took 1.61 s against 0.98.
//
// Every item is computed by spmv_item, as the general kernels compute it, so the products are
// the same bits; the squares are added in another fixed order.  The scalars of a round are
// formed by one thread of each CTA: a double division or root on every thread would take the
// FP64 pipe (16 cycles per warp instruction) longer than the products of a small problem.
#pragma once

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "rules.h"

namespace mpax {

constexpr int kRoundWarps = 16;
template <typename T>
constexpr int kRoundSmem = kRoundWarps * kSpmvBufLen<T> * (int)sizeof(T);

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
  // nullable, read behind the matrix loads: a word that ends the launch when set, dscale
  const int* ended = nullptr;
  const double* ds = nullptr;
  __device__ __forceinline__ bool skip() const { return ended && *ended; }
  __device__ __forceinline__ void load() {
    if (ds) dscale = (T)*ds;
  }
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

// This warp's items: warp w of CTA c takes w * ctas + c, then every ctas * warps further,
// so that few items spread over the SMs first.  kResident: see spmv_item.
template <typename T, bool kResident, class In, class Epi>
__device__ __forceinline__ void round_items(const SpmvArgs<T>& a, int ctas, In in, Epi epi,
                                            T* buf) {
  for (int item = (threadIdx.x >> 5) * ctas + blockIdx.x; item < a.n_items;
       item += ctas * kRoundWarps) {
    spmv_item<T, In, Epi, kResident>(a, in, epi, item, buf);
    __syncwarp();  // the next item rewrites the warp's buffer
  }
}

// After a round: the estimate, its last increment, and 1 / ||g||, the scale of the next v.
struct RoundState {
  double nu = 0.0, d = 0.0, scale = 1.0;
};

// What the rounds have in common.  root: the norm is sqrt(||g||) (A~^T A~), else ||g||.
struct RoundRule {
  int root;
  double tol, cap;
  int max_iter;
};

// Round t gave q = ||g||^2 after state `was`; true when it is the last, with the norm.
__device__ __forceinline__ bool round_end(const RoundRule& rule, int t, double q,
                                          const RoundState& was, RoundState* now, double* norm) {
  const double nrm = sqrt(q);
  if (nrm == 0.0) {
    *norm = 0.0;
    return true;
  }
  const double nu = rule.root ? sqrt(nrm) : nrm;
  *now = RoundState{nu, was.d, 1.0 / nrm};
  *norm = nu;
  if (t > 1 && power_stop(nu, was.nu, &now->d, rule.tol, rule.cap, norm)) return true;
  if (t < rule.max_iter) return false;
  *norm = isfinite(rule.cap) ? rule.cap : nu;  // out of rounds: the certified bound
  return true;
}

__device__ __forceinline__ void store_norm(DevState* st, const RoundRule& rule, double norm, int t) {
  st->pw_nu = norm;
  st->pw_iters = t;
  if (rule.root) st->norm_A = norm;
  else st->norm_Q = norm;
}

// This thread's share of part[0..np), and the sum of the shares over the block (valid in
// thread 0).  Warps that have no share skip their tree: a step takes the FP64 pipe 16 cycles.
__device__ __forceinline__ double round_share(const double* part, int np) {
  double q = 0.0;
#pragma unroll 8
  for (int i = threadIdx.x; i < np; i += 32 * kRoundWarps) q += __ldcg(part + i);
  return q;
}
__device__ __forceinline__ double round_sum(double q, int np, double* sh) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w * 32 < np) q = warp_sum(q);
  if (np <= 32) return q;
  if (lane == 0) sh[w] = q;
  __syncthreads();
  if (w == 0) q = warp_sum(lane < kRoundWarps ? sh[lane] : 0.0);
  return q;
}

// All rounds by one CTA.  two = 1: v -> w = K1 v -> g = K2 w (plus diag v when given); two = 0:
// g = K2 v.  v, w and g change during the launch and are read through L2; the matrices are
// constant and stay in L1.
template <typename T>
__global__ void __launch_bounds__(32 * kRoundWarps, 1)
    power_rounds(SpmvArgs<T> a1, SpmvArgs<T> a2, int two, T* v, T* g, T* w, const T* diag,
                 RoundRule rule, DevState* st) {
  extern __shared__ __align__(16) unsigned char round_smem[];
  T* buf = reinterpret_cast<T*>(round_smem) + (threadIdx.x >> 5) * kSpmvBufLen<T>;
  __shared__ double sh[kRoundWarps];
  __shared__ double s_scale;
  __shared__ int s_stop;
  RoundState was;  // thread 0's
  if (threadIdx.x == 0) s_scale = 1.0;
  __syncthreads();
  for (int t = 1;; ++t) {
    const T scale = (T)s_scale;
    if (two) {
      round_items<T, true>(a1, 1, InPlain<T, true>{v},
                           EpiRound<T>{w, nullptr, nullptr, scale, (T)1, 0}, buf);
      __syncthreads();
    }
    round_items<T, true>(a2, 1, InPlain<T, true>{two ? w : v},
                         EpiRound<T>{g, diag, v, two ? (T)1 : scale, scale, 1}, buf);
    __syncthreads();
    const double q = round_sum(round_share(a2.part, a2.n_items), a2.n_items, sh);
    if (threadIdx.x == 0) {
      RoundState now;
      double norm;
      s_stop = round_end(rule, t, q, was, &now, &norm);
      s_scale = now.scale;
      was = now;
      if (s_stop) store_norm(st, rule, norm, t);
    }
    __syncthreads();
    if (s_stop) return;
    T* sw = v;
    v = g;
    g = sw;
  }
}

// Round t as launches.  kFirst: the round's first product, w = K1 v (or its only one,
// g = K2 v, which also leaves partial sums: check = 1).  Before it, every CTA adds the np
// partial sums `part` of round t - 1 for the scale of v.  The last CTA has no items: it ends
// round t - 1, reading the state rs[(t - 1) & 1] and writing rs[t & 1], while the others
// multiply; when that round was the last it writes pw_done = t, of which its own launch takes
// no notice (power_round_over) and with which all later ones return.  The host sees launch
// and end in mapped memory.  Else the second product,
// g = K2 w (plus diag v when given).  Launch max_iter + 1 is the last CTA alone.
template <typename T, bool kFirst>
__global__ void __launch_bounds__(32 * kRoundWarps, 1)
    power_step(SpmvArgs<T> a, const T* in, T* out, const T* diag, const T* v, int check, int t,
               const double* part, int np, RoundRule rule, RoundState* rs, DevState* st,
               HostStatus* host) {
  extern __shared__ __align__(16) unsigned char round_smem[];
  T* buf = reinterpret_cast<T*>(round_smem) + (threadIdx.x >> 5) * kSpmvBufLen<T>;
  if constexpr (kFirst) {
    __shared__ double sh[kRoundWarps];
    __shared__ double s_scale;
    const int done = st->pw_done;
    double q = t > 1 ? round_share(part, np) : 0.0;
    if (power_round_over(done, t)) return;
    if (t > 1) q = round_sum(q, np, sh);
    if (blockIdx.x == gridDim.x - 1) {
      if (threadIdx.x != 0) return;
      RoundState now;
      if (t > 1) {
        double norm;
        if (round_end(rule, t - 1, q, rs[(t - 1) & 1], &now, &norm)) {
          store_norm(st, rule, norm, t - 1);
          st->pw_done = t;
          host->power_done = 1;
        }
      }
      rs[t & 1] = now;
      host->power_launch = t;
      return;
    }
    if (threadIdx.x == 0) s_scale = t > 1 && q > 0.0 ? 1.0 / sqrt(q) : 1.0;
    __syncthreads();
    round_items<T, false>(a, gridDim.x - 1, InPlain<T>{in},
                          EpiRound<T>{out, nullptr, nullptr, (T)s_scale, (T)1, check}, buf);
  } else {
    round_items<T, false>(
        a, gridDim.x, InPlain<T>{in},
        EpiRound<T>{out, diag, v, (T)1, (T)1, 1, &st->pw_done, diag ? &rs[t & 1].scale : nullptr}, buf);
  }
}

// ---- host side --------------------------------------------------------------------

// CTAs for a product of `items` items: four items each, at most one per SM (a second one on
// any would run when the first has left).
inline int round_ctas(int items, int sms) { return std::max(1, std::min(sms, (items + 3) / 4)); }
// Work items up to which one CTA takes all rounds: a CTA's barrier is cheaper than a launch.
constexpr int kOneCtaItems = 8;
// Items per warp up to which these rounds are taken; past it the general kernels' occupancy
// (40 warps per SM) hides the gathers better.
constexpr int kRoundItemsPerWarp = 4;
inline bool round_fits(int items, int sms) {
  return items > 0 && items <= kRoundItemsPerWarp * kRoundWarps * sms;
}

template <class K>
cudaError_t allow_smem(K kernel, int smem) {
  return smem > 48 * 1024
             ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
             : cudaSuccess;
}

}  // namespace mpax
