// FP32 products of the shared-matrix batch on the CUDA cores:
//   C[n][m] = sum_k A_op[m][k] V[n][k]
// for the B instances' vectors V (rows of ldv): A_op = A~ stored [M][K] (A_MN = 0, the
// dual step's A~ X) or A~^T of an A~ stored [K][M] (A_MN = 1, the primal step's A~^T Y).
// Every output is one chain of fused multiply-adds in increasing k, whatever the tile, so
// the choice of a tile changes no bit of a result.
//
// Tiles: a CTA forms BM x BN outputs, a thread TM x TN of them from float4 fragments of
// slabs of BK k values that lie k-major in shared memory.  Slabs arrive by cp.async, one
// value each (the operands' rows are k-contiguous, so a transposing copy has no wider
// unit), STAGES - 1 slabs ahead of the one being multiplied, with one barrier per slab.
#pragma once

#include <cuda_runtime.h>

namespace mpax_gemv {

template <int BM, int BN, int TM, int TN, int BK, int STAGES>
struct SgShape {
  static constexpr int kThreads = (BM / TM) * (BN / TN);
  static constexpr int kLdA = BM + 4, kLdV = BN + 4;  // 16-byte rows, 4-bank shift per k
  static constexpr int kLoadA = BM * BK / kThreads, kLoadV = BN * BK / kThreads;
  static constexpr int kStage = BK * (kLdA + kLdV);  // floats
  static constexpr int kSmem = STAGES * kStage * 4;
  static_assert(TM % 4 == 0 && TN % 4 == 0, "float4 fragments");
  static_assert(kThreads % 32 == 0 && BM * BK % kThreads == 0 && BN * BK % kThreads == 0, "");
};

// 4 bytes from global to shared memory; zero when !ok (src must still be a valid address).
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}

// Element t of this thread of a slab of R rows with k contiguous in memory: a warp takes
// four rows by eight k (32-byte pieces of a row), so that its stores [k][row] hit all 32
// banks (rows shift by one bank, k by four).
template <int R, int BK, int THREADS>
__device__ __forceinline__ void sg_kmajor(int tid, int t, int& row, int& k) {
  const int e = tid + t * THREADS;
  const int lane = e & 31, w = e >> 5;
  row = (w % (R / 4)) * 4 + (lane >> 3);
  k = (w / (R / 4)) * 8 + (lane & 7);
}

template <int A_MN, int BM, int BN, int TM, int TN, int BK, int STAGES>
__global__ void __launch_bounds__(SgShape<BM, BN, TM, TN, BK, STAGES>::kThreads)
    k_sgemm(const float* __restrict__ A, long long lda, const float* __restrict__ V, long long ldv,
            float* __restrict__ Cm, long long ldc, int M, int N, int K) {
  using S = SgShape<BM, BN, TM, TN, BK, STAGES>;
  extern __shared__ __align__(16) float sg_smem[];
  const int tid = threadIdx.x;
  const int tm = tid % (BM / TM), tn = tid / (BM / TM);
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;
  const int slabs = (K + BK - 1) / BK;
  auto load = [&](int slab) {
    if (slab < slabs) {
      float* as = sg_smem + (slab % STAGES) * S::kStage;
      float* vs = as + BK * S::kLdA;
      const int k0 = slab * BK;
#pragma unroll
      for (int t = 0; t < S::kLoadA; ++t) {
        int r, k;
        if constexpr (A_MN) {
          const int e = tid + t * S::kThreads;
          r = e % BM;
          k = e / BM;
        } else {
          sg_kmajor<BM, BK, S::kThreads>(tid, t, r, k);
        }
        const bool ok = m0 + r < M && k0 + k < K;
        const long long gm = ok ? m0 + r : 0, gk = ok ? k0 + k : 0;
        cp_async4(as + k * S::kLdA + r, A_MN ? A + gk * lda + gm : A + gm * lda + gk, ok);
      }
#pragma unroll
      for (int t = 0; t < S::kLoadV; ++t) {
        int r, k;
        sg_kmajor<BN, BK, S::kThreads>(tid, t, r, k);
        const bool ok = n0 + r < N && k0 + k < K;
        const long long gn = ok ? n0 + r : 0, gk = ok ? k0 + k : 0;
        cp_async4(vs + k * S::kLdV + r, V + gn * ldv + gk, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) load(s);
  for (int s = 0; s < slabs; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();  // slab s is in; everyone has left the stage that is refilled next
    load(s + STAGES - 1);
    const float* as = sg_smem + (s % STAGES) * S::kStage;
    const float* vs = as + BK * S::kLdA;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      // fragments of four rows (instances) each, BM / (TM / 4) apart so that neighbouring
      // threads read neighbouring 16 bytes
      float a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; i += 4)
        *reinterpret_cast<float4*>(a + i) = *reinterpret_cast<const float4*>(
            as + kk * S::kLdA + (i / 4) * (BM * 4 / TM) + tm * 4);
#pragma unroll
      for (int j = 0; j < TN; j += 4)
        *reinterpret_cast<float4*>(b + j) = *reinterpret_cast<const float4*>(
            vs + kk * S::kLdV + (j / 4) * (BN * 4 / TN) + tn * 4);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int gn = n0 + (j / 4) * (BN * 4 / TN) + tn * 4 + j % 4;
    if (gn >= N) continue;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int gm = m0 + (i / 4) * (BM * 4 / TM) + tm * 4 + i % 4;
      if (gm < M) Cm[(long long)gn * ldc + gm] = acc[i][j];
    }
  }
}

// Launch with the largest tile that still gives most SMs a CTA: large tiles reuse their
// fragments most, but idle SMs cost more.  At 1018 x 2050 x 100 a k step takes a CTA 28 ns with
// 32 x 32 tiles (two warps), 31 with 64 x 32 (four) and 116 with 128 x 128 (eight): the few
// warps' issue slots and four-byte copies, not the chain of an output, which a dependent FMA
// lengthens by about 2 ns a step.  Measured, microseconds of A~ V / A~^T V (128 x 128 tiles of the
// register-staged kernel before: first column):
//   1018 x 2050 x 100    317 / 158    32 x 32: 57 / 35    64 x 32: 64 / 31    128 x 128: 238 / 113
//   2036 x 4100 x 500    660 / 666    32 x 32: 356 / 352  64 x 32: 330 / 312  128 x 128: 441 / 431
//   4096 x 8192 x 512   1457 / 1378   32 x 32: 1358 / 1228  64 x 32: 1171 / 1028  128 x 128: 907 / 863
template <int A_MN, int BM, int BN, int TM, int TN, int BK, int STAGES>
cudaError_t sgemm_tile(const float* A, long long lda, const float* V, long long ldv, float* C,
                       long long ldc, int M, int N, int K, cudaStream_t s) {
  using S = SgShape<BM, BN, TM, TN, BK, STAGES>;
  auto kernel = k_sgemm<A_MN, BM, BN, TM, TN, BK, STAGES>;
  if (S::kSmem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmem);
    if (e) return e;
  }
  const dim3 g((unsigned)((M + BM - 1) / BM), (unsigned)((N + BN - 1) / BN));
  kernel<<<g, S::kThreads, S::kSmem, s>>>(A, lda, V, ldv, C, ldc, M, N, K);
  return cudaGetLastError();
}

template <int A_MN>
cudaError_t sgemm(const float* A, long long lda, const float* V, long long ldv, float* C,
                  long long ldc, int M, int N, int K, cudaStream_t s) {
  auto tiles = [&](int bm, int bn) {
    return (long long)((M + bm - 1) / bm) * ((N + bn - 1) / bn);
  };
  if (tiles(128, 128) >= 100)
    return sgemm_tile<A_MN, 128, 128, 8, 8, 16, 4>(A, lda, V, ldv, C, ldc, M, N, K, s);
  if (tiles(64, 32) >= 128)
    return sgemm_tile<A_MN, 64, 32, 4, 4, 32, 3>(A, lda, V, ldv, C, ldc, M, N, K, s);
  return sgemm_tile<A_MN, 32, 32, 4, 4, 16, 6>(A, lda, V, ldv, C, ldc, M, N, K, s);
}

}  // namespace mpax_gemv
