// FP32 GEMM for the OPQ rotation steps (Sec. 3 "OPQ": z = x R, the Procrustes
// product Y^T Zhat and the polar iteration).  C = alpha * op(A) * B + beta * C,
// op(A) = A or A^T, all row-major with explicit leading dimensions.  The general
// kernel has 64 x 64 output tiles, K in steps of 16, each of 256 threads
// accumulating 4 x 4 in FP32 FFMA.  Large K is split over CTAs (split-K) with
// FP32 atomics into C; the caller then owns a C that was pre-scaled by beta.
// Products of many rows take gemm_rows_kernel.
#include <algorithm>

#include "devutil.cuh"
#include "internal.cuh"

namespace adn {

namespace {
constexpr int TM = 64, TN = 64, TK = 16;

template <bool TA>
__global__ void __launch_bounds__(256) gemm_f32_kernel(int M, int N, int K, float alpha,
                                                        const float *__restrict__ A, int lda,
                                                        const float *__restrict__ B, int ldb,
                                                        float *__restrict__ C, int ldc, int kslice,
                                                        bool atomic_out) {
  __shared__ float As[TK][TM + 4];
  __shared__ float Bs[TK][TN + 4];
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int k_beg = blockIdx.z * kslice;
  const int k_end = min(K, k_beg + kslice);
  float acc[4][4] = {};
  for (int k0 = k_beg; k0 < k_end; k0 += TK) {
    // A tile: TM x TK elements of op(A)
    for (int e = tid; e < TM * TK; e += 256) {
      int mm, kk;
      if (TA) { kk = e / TM; mm = e % TM; } else { mm = e / TK; kk = e % TK; }
      const int gm = m0 + mm, gk = k0 + kk;
      float v = 0.f;
      if (gm < M && gk < k_end) v = TA ? A[(int64_t)gk * lda + gm] : A[(int64_t)gm * lda + gk];
      As[kk][mm] = v;
    }
    for (int e = tid; e < TK * TN; e += 256) {
      const int kk = e / TN, nn = e % TN;
      const int gk = k0 + kk, gn = n0 + nn;
      Bs[kk][nn] = (gk < k_end && gn < N) ? B[(int64_t)gk * ldb + gn] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gm = m0 + ty + 16 * i, gn = n0 + tx + 16 * j;
      if (gm < M && gn < N) {
        float *c = C + (int64_t)gm * ldc + gn;
        if (atomic_out) atomicAdd(c, alpha * acc[i][j]);
        else *c = alpha * acc[i][j] + *c;
      }
    }
}

// C = alpha A B + beta C for many rows of A (16-byte aligned, lda and ldb
// multiples of 4): 128 x TN output tiles, 8 x TN / 16 per thread, so that a
// thread's 16-byte shared-memory reads feed 8 to 10 FFMA each (the general
// kernel's scalar reads feed 2); K in steps of 16, the next step's global loads
// in registers while one is used.  Every output is one thread's sum over
// ascending k from 0, then added to beta C, as in the general kernel without
// split-K: the same bits.  Bound by the FP32 pipe: 262,144 x 384 x 384 (77 GFLOP) in
// 1.46 ms, 53 TFLOP/s (two columns per instruction by fma.rn.f32x2: 1.56 ms).
template <int TN>
__global__ void __launch_bounds__(256, 2) gemm_rows_kernel(int M, int N, int K, float alpha,
                                                            const float *__restrict__ A, int lda,
                                                            const float *__restrict__ B, int ldb,
                                                            float beta, float *__restrict__ C,
                                                            int ldc) {
  constexpr int TMR = 128, NJ = TN / 16, NB4 = TN * TK / 4 / 256;  // float4 of B per thread
  __shared__ __align__(16) float As[2][TK][TMR + 4];
  __shared__ __align__(16) float Bs[2][TK][TN];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.x * TMR, n0 = blockIdx.y * TN;
  float4 ra[2], rb[NB4];
  // A: thread t holds rows t / 4 and t / 4 + 64, coordinates 4 (t % 4) ..
  const int am = tid >> 2, ak = (tid & 3) * 4;
  auto load = [&](int k0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gm = m0 + am + 64 * h, gk = k0 + ak;
      const float *p = A + (int64_t)gm * lda + gk;
      ra[h] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (gm < M && gk + 3 < K) ra[h] = __ldg((const float4 *)p);
      else if (gm < M) {
        if (gk < K) ra[h].x = p[0];
        if (gk + 1 < K) ra[h].y = p[1];
        if (gk + 2 < K) ra[h].z = p[2];
      }
    }
#pragma unroll
    for (int h = 0; h < NB4; ++h) {
      const int e = tid + 256 * h, kk = e / (TN / 4), nn = (e % (TN / 4)) * 4;
      const int gk = k0 + kk, gn = n0 + nn;
      const float *p = B + (int64_t)gk * ldb + gn;
      rb[h] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (gk < K && gn + 3 < N) rb[h] = __ldg((const float4 *)p);
      else if (gk < K) {
        if (gn < N) rb[h].x = p[0];
        if (gn + 1 < N) rb[h].y = p[1];
        if (gn + 2 < N) rb[h].z = p[2];
      }
    }
  };
  auto store = [&](int s) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      As[s][ak][am + 64 * h] = ra[h].x;
      As[s][ak + 1][am + 64 * h] = ra[h].y;
      As[s][ak + 2][am + 64 * h] = ra[h].z;
      As[s][ak + 3][am + 64 * h] = ra[h].w;
    }
#pragma unroll
    for (int h = 0; h < NB4; ++h) {
      const int e = tid + 256 * h;
      *(float4 *)&Bs[s][e / (TN / 4)][(e % (TN / 4)) * 4] = rb[h];
    }
  };
  float acc[8][NJ];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j] = 0.f;
  load(0);
  store(0);
  __syncthreads();
  int s = 0;
  for (int k0 = 0; k0 < K; k0 += TK, s ^= 1) {
    if (k0 + TK < K) load(k0 + TK);
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      float a[8], b[NJ];
      *(float4 *)a = *(const float4 *)&As[s][kk][4 * ty];
      *(float4 *)(a + 4) = *(const float4 *)&As[s][kk][64 + 4 * ty];
#pragma unroll
      for (int j = 0; j < NJ; j += 4)
        *(float4 *)(b + j) = *(const float4 *)&Bs[s][kk][16 * j + 4 * tx];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (k0 + TK < K) {
      store(s ^ 1);
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int gm = m0 + (i < 4 ? 4 * ty + i : 64 + 4 * ty + i - 4);
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int gn = n0 + 16 * (j & ~3) + 4 * tx + (j & 3);
      if (gn >= N) continue;
      float *c = C + (int64_t)gm * ldc + gn;
      *c = __fadd_rn(beta == 0.f ? 0.f : beta * *c, __fmul_rn(alpha, acc[i][j]));
    }
  }
}

__global__ void scale_kernel(float *C, int M, int N, int ldc, float beta) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)M * N) return;
  const int i = (int)(e / N), j = (int)(e % N);
  float *c = C + (int64_t)i * ldc + j;
  *c = beta == 0.f ? 0.f : beta * *c;
}
}  // namespace

int launch_gemm_f32(bool transA, int M, int N, int K, float alpha, const float *A, int lda,
                    const float *B, int ldb, float beta, float *C, int ldc, cudaStream_t st) {
  if (M <= 0 || N <= 0) return ADANNS_OK;
  // many rows: at least a CTA of 128-row tiles per SM; C is scaled by beta in
  // the same pass (A and B are read while C is written, so they must not alias)
  const int tn = N > 64 ? 128 : 64;
  const int64_t big = (int64_t)((M + 127) / 128) * ((N + tn - 1) / tn);
  if (!transA && K > 0 && big >= num_sms() && (lda & 3) == 0 && (ldb & 3) == 0 &&
      ((uintptr_t)A & 15) == 0 && ((uintptr_t)B & 15) == 0) {
    const dim3 grid((M + 127) / 128, (N + tn - 1) / tn);
    auto kern = tn == 128 ? gemm_rows_kernel<128> : gemm_rows_kernel<64>;
    kern<<<grid, 256, 0, st>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    ADN_LAUNCH("gemm_rows_kernel");
    return ADANNS_OK;
  }
  const int64_t mn = (int64_t)M * N;
  scale_kernel<<<(unsigned)((mn + 255) / 256), 256, 0, st>>>(C, M, N, ldc, beta);
  ADN_LAUNCH("scale_kernel");
  if (K <= 0) return ADANNS_OK;
  const int gx = (N + TN - 1) / TN, gy = (M + TM - 1) / TM;
  // split K so that the grid covers the GPU when the output is small
  int splits = 1;
  const int tiles = gx * gy;
  const int target = 2 * num_sms();
  if (tiles < target) splits = std::max(1, std::min((K + 1023) / 1024, target / tiles));
  int kslice = (K + splits - 1) / splits;
  kslice = (kslice + TK - 1) / TK * TK;
  splits = (K + kslice - 1) / kslice;
  dim3 grid(gx, gy, splits);
  const bool atomic_out = true;  // C was pre-scaled by beta above
  if (transA)
    gemm_f32_kernel<true><<<grid, 256, 0, st>>>(M, N, K, alpha, A, lda, B, ldb, C, ldc, kslice,
                                                atomic_out);
  else
    gemm_f32_kernel<false><<<grid, 256, 0, st>>>(M, N, K, alpha, A, lda, B, ldb, C, ldc, kslice,
                                                 atomic_out);
  ADN_LAUNCH("gemm_f32_kernel");
  return ADANNS_OK;
}

}  // namespace adn
