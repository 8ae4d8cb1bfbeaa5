// IVF-OPQ scores through the certified tensor-core filter (Sec. 4.3; Table
// "formula" IVFOPQ row read as asymmetric lookup).
//
// A member's ADC score sum_m ||z_m - C_m[code_m]||^2 is |z - y|^2 for its decoded
// row y.  Where many queries share a probed list, decoding the list once to
// FP16 rows and taking the products on the tensor cores costs far less than M
// shared-memory lookups per (query, member).  The tensor-core scan (mma_scan.cu)
// gives 16-bit approximate keys, the certified shortlist (select16.cu) keeps
// every member within the rounding-error bound of the k'-th, and those are
// scored exactly by the lookup tables in the order of sums of adc_dist_kernel,
// so scores and ids are that kernel's.  Queries whose certified set overflows
// are left to it.
//
// Measured: 8,000 queries, 32 of 1,024 lists, 5.25 M rows, 32-byte codes of 384
// coordinates, rerank 400: 24.2 -> 7.0 ms (ADC stage and selection 22.0 -> 5.2:
// decode 1.05, tensor cores 1.96, shortlist 1.2 of 494 members per query, exact
// scores 0.8); one list of 1.28 M 16-byte codes, 1,000 queries: 10.9 -> 1.7 ms.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "devutil.cuh"
#include "internal.cuh"

namespace adn {
namespace {

constexpr float AC_Y2MAX = 4.f;  // largest squared norm of a decoded row
constexpr int AC_MAX_M = 96;     // lookup table of one query in shared memory
constexpr int AC_CTAS = 6;       // decode CTAs per SM (their tables: 192 KB)
constexpr int AC_WAVES = 2;

// c2[m][c] = |C_m[c]|^2
__global__ void codeword_norms_kernel(const float *__restrict__ C, int n, int dsub,
                                      float *__restrict__ c2) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  float s = 0.f;
  for (int t = 0; t < dsub; ++t) s = fmaf(C[(int64_t)e * dsub + t], C[(int64_t)e * dsub + t], s);
  c2[e] = s;
}

// y2[p] = sum over m of c2[m][code], and their maximum (bits of non-negative floats)
__global__ void code_norms_kernel(const uint8_t *__restrict__ codes, const float *__restrict__ c2,
                                  int64_t N, int M, float *__restrict__ y2, int *__restrict__ mx) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float s = 0.f;
  if (p < N) {
    for (int m = 0; m < M; ++m) s += c2[m * 256 + codes[p * M + m]];
    y2[p] = s;
  }
  int b = __float_as_int(s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
  if ((threadIdx.x & 31) == 0) atomicMax(mx, b);
}

// FP16 rows of the decoded codes of the probed lists, K-block blockIdx.y (64
// coordinates), in the scan's layout [(off nkb + kb n_l + m)][64].  The block's
// slice of the codebook is staged in shared memory as [16 groups of 4
// coordinates][256 codes] (32 KB), so that a member's row is 16 eight-byte
// lookups; eight lanes write a row's 128 bytes.  The chunk after the next and the
// next one's codes are on their way meanwhile (a CTA has only 8 KB of a chunk to
// write per chain of dependent reads), and a CTA takes as many chunks as make two
// waves of CTAs, since staging the table costs as much as a few dozen of them:
// 5.25 M rows x 384 1.38 -> 1.05 ms (two thirds of the measured copy bandwidth);
// four waves 1.05, one or two of 1.28 M x 128 0.12, four 0.16.  VEC4: the groups do not cross
// sub-vectors (d_s / M a multiple of 4), else each coordinate looks up its own
// code.
template <bool VEC4>
__global__ void __launch_bounds__(256) decode_f16_kernel(
    const uint8_t *__restrict__ codes, int M, int dsub, const float *__restrict__ C,
    const int4 *__restrict__ cmap, int nchunk, int per, const int32_t *__restrict__ lcnt, int nkb,
    uint4 *__restrict__ out) {
  __shared__ __align__(16) __half tab[16 * 256 * 4];
  const int kb = blockIdx.y, d_s = M * dsub;
  for (int e = threadIdx.x; e < 64 * 256; e += 256) {
    const int j = e & 63, c = e >> 6, jj = 64 * kb + j;
    float v = 0.f;
    if (jj < d_s) {
      const int m = jj / dsub;
      v = C[((int64_t)m * 256 + c) * dsub + (jj - m * dsub)];
    }
    tab[(j >> 2) * 1024 + c * 4 + (j & 3)] = __float2half_rn(v);
  }
  __syncthreads();
  const int c8 = threadIdx.x & 7, j0 = 64 * kb + 8 * c8;  // this lane's 8 coordinates
  int ms[8];  // their sub-vectors
#pragma unroll
  for (int u = 0; u < 8; ++u) ms[u] = j0 + u < d_s ? (j0 + u) / dsub : -1;
  const int ch0 = blockIdx.x * per, ch1 = min(nchunk, ch0 + per);
  // a chunk (list, first member, list offset, list size); size 0: nothing to write
  auto head = [&](int ch) {
    int4 cl = make_int4(0, 0, 0, 0);
    if (ch < ch1) {
      cl = cmap[ch];
      if (lcnt && lcnt[cl.x] == 0) cl.w = 0;
    }
    return cl;
  };
  // this lane's codes of the chunk's two members
  constexpr int NC = VEC4 ? 2 : 8;
  auto fetch = [&](const int4 &cl, uint32_t(&r)[2][NC]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = cl.y + 32 * h + (threadIdx.x >> 3);
      const uint8_t *cp = codes + ((int64_t)cl.z + m) * M;
#pragma unroll
      for (int u = 0; u < NC; ++u) {
        const int sv = ms[VEC4 ? 4 * u : u];
        r[h][u] = m < cl.w && sv >= 0 ? cp[sv] : 0u;
      }
    }
  };
  int4 cl = head(ch0), nx = head(ch0 + 1);
  uint32_t cd[2][NC], cn[2][NC];
  fetch(cl, cd);
  for (int ch = ch0; ch < ch1; ++ch) {
    const int4 n2 = head(ch + 2);
    fetch(nx, cn);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = cl.y + 32 * h + (threadIdx.x >> 3);
      if (m >= cl.w) continue;
      uint4 r = make_uint4(0u, 0u, 0u, 0u);
      if (VEC4) {
        if (ms[0] >= 0) {
          const uint2 a = *(const uint2 *)(tab + 2 * c8 * 1024 + cd[h][0] * 4);
          r.x = a.x;
          r.y = a.y;
        }
        if (ms[4] >= 0) {
          const uint2 a = *(const uint2 *)(tab + (2 * c8 + 1) * 1024 + cd[h][1] * 4);
          r.z = a.x;
          r.w = a.y;
        }
      } else {
        unsigned short hv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          hv[u] = ms[u] >= 0 ? __half_as_ushort(tab[(2 * c8 + (u >> 2)) * 1024 +
                                                    cd[h][VEC4 ? 0 : u] * 4 + (u & 3)])
                             : (unsigned short)0;
        r = make_uint4(hv[0] | (uint32_t)hv[1] << 16, hv[2] | (uint32_t)hv[3] << 16,
                       hv[4] | (uint32_t)hv[5] << 16, hv[6] | (uint32_t)hv[7] << 16);
      }
      out[((int64_t)cl.z * nkb + (int64_t)kb * cl.w + m) * 8 + c8] = r;
    }
    cl = nx;
    nx = n2;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int u = 0; u < NC; ++u) cd[h][u] = cn[h][u];
  }
}

// One query per CTA: its lookup table in shared memory (as pq_lut_kernel
// computes it), the exact scores of its shortlist (the sums of
// adc_dist_kernel), sorted; the kr smallest keys leave.
constexpr int AR_THREADS = 256;

__global__ void __launch_bounds__(AR_THREADS) adc_rescore_kernel(
    const int64_t *__restrict__ cids, const int32_t *__restrict__ cnt, int kk,
    const float *__restrict__ z, int M, int dsub, const float *__restrict__ C,
    const uint8_t *__restrict__ codes, const int64_t *__restrict__ list_off,
    const int32_t *__restrict__ list_ids, int kr, uint64_t *__restrict__ keys) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int64_t q = blockIdx.x;
  const int n = cnt[q], tid = threadIdx.x, d_s = M * dsub;
  if (n < 0) return;  // left to the lookup scan
  uint64_t *sk = (uint64_t *)smem;
  float *sz = (float *)(sk + kk), *lut = sz + ((d_s + 3) & ~3);
  for (int t = tid; t < d_s; t += AR_THREADS) sz[t] = z[q * d_s + t];
  __syncthreads();
  for (int e = tid; e < M * 256; e += AR_THREADS) {
    const float *cw = C + (int64_t)e * dsub, *zm = sz + (e >> 8) * dsub;
    float acc = 0.f;
    if ((dsub & 3) == 0) {
      for (int t = 0; t < dsub; t += 4) {
        const float4 c = __ldg((const float4 *)(cw + t));
        float df;
        df = zm[t] - c.x; acc = fmaf(df, df, acc);
        df = zm[t + 1] - c.y; acc = fmaf(df, df, acc);
        df = zm[t + 2] - c.z; acc = fmaf(df, df, acc);
        df = zm[t + 3] - c.w; acc = fmaf(df, df, acc);
      }
    } else {
      for (int t = 0; t < dsub; ++t) {
        const float df = zm[t] - cw[t];
        acc = fmaf(df, df, acc);
      }
    }
    lut[e] = acc;
  }
  __syncthreads();
  for (int i = tid; i < n; i += AR_THREADS) {
    const int64_t v = cids[q * kk + i];
    uint64_t key = KEY_MAX;
    if (v >= 0) {
      const int64_t p = list_off[v >> 32] + (v & 0xffffffffll);
      const uint8_t *cp = codes + p * M;
      float d;
      if ((M & 3) == 0 && M <= 64) {
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        const float *L = lut;
        for (int w = 0; w < M >> 2; ++w, L += 1024) {
          const uint32_t word = ((const uint32_t *)cp)[w];
          s0 += L[word & 0xff];
          s1 += L[256 + ((word >> 8) & 0xff)];
          s2 += L[512 + ((word >> 16) & 0xff)];
          s3 += L[768 + (word >> 24)];
        }
        d = (s0 + s1) + (s2 + s3);
      } else {
        d = 0.f;
        for (int m = 0; m < M; ++m) d += lut[m * 256 + cp[m]];
      }
      key = pack_key(d, (uint32_t)list_ids[p]);
    }
    sk[i] = key;
  }
  __syncthreads();
  block_sort<AR_THREADS>(sk, n);
  for (int r = tid; r < kr; r += AR_THREADS) keys[q * kr + r] = r < n ? sk[r] : KEY_MAX;
}

}  // namespace

int launch_code_norms(const adanns_index *x, float *y2, float *y2max_host, cudaStream_t st) {
  const int M = x->opq_M, dsub = x->opq_ds / M;
  Scratch s(st);
  float *c2;
  int *mx, rc;
  if ((rc = s.get(&c2, (size_t)M * 256)) || (rc = s.get(&mx, 1))) return rc;
  ADN_CUDA(cudaMemsetAsync(mx, 0, sizeof(int), st));
  codeword_norms_kernel<<<M, 256, 0, st>>>(x->opq_C, M * 256, dsub, c2);
  ADN_LAUNCH("codeword_norms_kernel");
  code_norms_kernel<<<(unsigned)((x->N + 255) / 256), 256, 0, st>>>(x->codes, c2, x->N, M, y2, mx);
  ADN_LAUNCH("code_norms_kernel");
  ADN_CUDA(cudaMemcpyAsync(y2max_host, mx, sizeof(float), cudaMemcpyDeviceToHost, st));
  ADN_CUDA(cudaStreamSynchronize(st));
  return ADANNS_OK;
}

// the FP16 rows and each list's part-filled query tile
int64_t adc_filter_fixed_bytes(const adanns_index *idx) {
  const int64_t nkb = (idx->opq_ds + 63) / 64;
  return idx->N * nkb * 128 + idx->nlist * nkb * 128 * 128;
}

// Where the filter pays.  In picoseconds, fitted to both sides measured on
// 50,000 to 3 M rows, one list to 1,024, (d_s, M) from (64, 8) to (768, 64):
// the lookup scan spends 2 + 0.42 M + 900 M / (members per list) per (query,
// member), the last term its staging of tables; the filter 0.8 d_s per member
// to decode, 0.0022 d_s per (query, member) of its 128-query tiles, 40,000 +
// 200 d_s per query to re-score, 500 per member of a query's region while one
// warp selects from it, and about 0.2 ms of launches.  At the line the two are
// level (one list of 1.28 M, M 16: 1.02 against 1.11 ms at 64 queries, 1.54
// against 1.15 at 128; 400,000 rows in 200 lists, M 32: 0.59 against 0.61 ms at
// 32 queries per list, 0.96 against 0.66 at 64); far above it the gap is 3- to
// 12-fold.
// With few queries per list and short rows the tiles of 128 queries are mostly
// empty, and what this line leaves out decides: the filter's cost per member and
// per query, and the lookup scan's tables and codes per tile of its own.  There
// the filter also has to be a tenth ahead by the estimates of both (fitted to 608
// calls): without it, lookups against filter in us, 3 M rows in 1,500 lists, (64,
// 32), 49 probes, 163 queries 557 / 841; 1 M in 1,000, (64, 8), 37, 808 486 / 639; (128,
// 16), 15, 1,397 482 / 550.
bool adc_certified(const adanns_index *idx, int64_t B, int nprobe, int kr) {
  const int M = idx->opq_M, d_s = idx->opq_ds;
  if (idx->metric != ADANNS_METRIC_L2_PREFIXNORM || idx->opq_S || !idx->opq_y2) return false;
  if (!(idx->opq_y2max <= AC_Y2MAX) || kr > CERT_MAX_K || nprobe > 128 || M > AC_MAX_M)
    return false;
  const int64_t nkb = (d_s + 63) / 64;
  if (idx->N * nkb > INT32_MAX - 256 || adc_filter_fixed_bytes(idx) > scratch_budget() / 2)
    return false;
  const double N = (double)idx->N, per = N / idx->nlist, qpl = (double)B * nprobe / idx->nlist;
  if (N * qpl * (2.0 + 0.42 * M + 900.0 * M / per) -
          N * d_s * (0.8 + 0.0022 * std::max(qpl, 128.0)) - B * (4e4 + 200.0 * d_s) -
          500.0 * nprobe * per <=
      2e8)
    return false;
  if (qpl >= 48.0 || d_s > 192) return true;
  const double pairs = (double)B * nprobe, tiles = std::max(1.0, qpl / adc_dist_query_tile(M));
  const double filter = 1.83e8 + N * (73.0 + 2.38 * d_s) + 1.89 * N * qpl +
                        B * (14000.0 + 1260.0 * M) + 635.0 * pairs;
  const double lookup = 1.06e8 + N * (6.3 * qpl + 1.68 * M * tiles) + B * (25500.0 + 1320.0 * M) +
                        357.0 * M * pairs;
  return filter < 0.9 * lookup;
}

int launch_decode_f16(const adanns_index *idx, const int32_t *lcnt, int nkb, void *rows,
                      cudaStream_t st) {
  const int M = idx->opq_M, dsub = idx->opq_ds / M, nch = idx->rr_chunks[0];
  if (nch <= 0) return ADANNS_OK;
  const int64_t ctas = (int64_t)num_sms() * AC_CTAS * AC_WAVES;
  const int per = (int)std::max<int64_t>(16, ((int64_t)nch * nkb + ctas - 1) / ctas);
  const dim3 grid((nch + per - 1) / per, nkb);
  auto kern = dsub % 4 == 0 ? decode_f16_kernel<true> : decode_f16_kernel<false>;
  kern<<<grid, 256, 0, st>>>(idx->codes, M, dsub, idx->opq_C, idx->rr_cmap[0], nch, per, lcnt, nkb,
                             (uint4 *)rows);
  ADN_LAUNCH("decode_f16_kernel");
  return ADANNS_OK;
}

int launch_adc_rescore(const adanns_index *idx, const int64_t *cids, const int32_t *cnt, int kk,
                       const float *z, int64_t B, int kr, uint64_t *keys, cudaStream_t st) {
  if (B <= 0) return ADANNS_OK;
  const int M = idx->opq_M, d_s = idx->opq_ds;
  const size_t sm = (size_t)kk * 8 + (size_t)((d_s + 3) & ~3) * 4 + (size_t)M * 1024;
  ADN_CUDA(ensure_smem((const void *)adc_rescore_kernel, sm));
  adc_rescore_kernel<<<(unsigned)B, AR_THREADS, sm, st>>>(cids, cnt, kk, z, M, d_s / M, idx->opq_C,
                                                          idx->codes, idx->list_off, idx->list_ids,
                                                          kr, keys);
  ADN_LAUNCH("adc_rescore_kernel");
  return ADANNS_OK;
}

}  // namespace adn
