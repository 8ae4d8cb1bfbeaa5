// Exact FP32 AdANNS-IVF search through a certified tensor-core filter, for
// batches whose probed lists are shared by several queries (Algorithm 1
// adannsInference, FP32 tier).
//
// The FFMA scan spends two instructions per (query, member, coordinate); at
// most a few hundred members per query can matter.  Here
//  1. the probed lists' normalised d_s prefixes are converted to FP16 rows in
//     scratch (the tensor-core scan's block layout, 2 bytes per coordinate
//     written once per call);
//  2. the tensor-core list scan (mma_scan.cu) turns every (query, member) pair
//     into a 16-bit approximate distance key;
//  3. the certified shortlist (select16.cu) keeps every member whose key is
//     within the error bound of the query's k-th smallest key, so that it
//     holds the exact k nearest whatever the rounding;
//  4. those members are re-scored in FP32 with the FFMA scan's own arithmetic
//     (t = q_j - s x_j, acc += t t over ascending j), sorted by (distance, id).
// Ids and distance bits are therefore those of the tiled and streaming scans.
// A query whose certified set does not fit its shortlist (many members nearly
// as near as the k-th, a zero query, ...) is left to the tiled FP32 scan, run
// on those queries alone.
//
// Measured (1,281,167 x 2048, 50,000 queries, d_s 512, 16 of 1,024 lists,
// k 100): 83.4 ms by the tiled scan (36% of the FFMA peak), 5.25 ms here: FP16
// rows 0.58, tensor-core scan 1.45, shortlist 1.0, re-score of the 118 members
// per query left by the bound 1.7, the rest 0.5.
//
// The bound.  With u = 2^-11 (FP16 rounding; entries of a unit vector below
// 2^-14 lose at most 2^-25 each), p = P(q), y = P(x) of norm at most 1.005:
// |p.y - p~.y~| <= |p||r_y| + |r_p||y| + |r_p||r_y|, |r_y| <= 1.005 u + d 2^-25
// (member side, a constant), |p| and |r_p| measured per query; the FP32 accumulation
// and re-score terms are those of the mixed-precision pruning (e_rest).
// An index that holds a row whose prefix has no usable norm (NaN, infinite, sums of
// squares in the denormal range; known when it is formed) has its batches at that d_s
// answered by the direct scans; where the filter runs all the same, such a row in a
// probed list leaves every query to the tiled scan.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "devutil.cuh"
#include "internal.cuh"

namespace adn {
namespace {

constexpr int CE_MAX_K = 256;       // the shortlist buffer holds k and the bound's margin
constexpr float CE_NORM2 = 1.01f;   // largest |P(v)|^2 the bound covers
constexpr float CE_UNSURE = 1e3f;   // the bound of a query that has none: it keeps every member

__device__ __forceinline__ uint2 half4(float a, float b, float c, float d) {
  const __half2 lo = __floats2half2_rn(a, b), hi = __floats2half2_rn(c, d);
  return make_uint2(*(const uint32_t *)&lo, *(const uint32_t *)&hi);
}

// FP16 rows of the normalised prefixes, block layout [(off nkb + kb n_l + m)][64],
// and x2[p] = |P(x_p)|^2.  One CTA per 64-member chunk of a probed list, four
// lanes per member: a warp reads 512 contiguous bytes of a prefix-major block
// and writes whole 32-byte sectors, the next K-block's loads in flight while
// one is converted.  Memory-bound: 4 bytes read, 2 written per coordinate.
__global__ void __launch_bounds__(256) f16_rows_kernel(
    const float *__restrict__ xpm, int d_pad, int d_s, int nkb, const int4 *__restrict__ cmap,
    const int32_t *__restrict__ lcnt, const float *__restrict__ nu, uint2 *__restrict__ out,
    float *__restrict__ x2, int *__restrict__ unsure) {
  const int4 cl = cmap[blockIdx.x];  // (list, first member, list offset, list size)
  if (lcnt && lcnt[cl.x] == 0) return;
  const int part = threadIdx.x & 3, m = cl.y + (threadIdx.x >> 2), nl = cl.w;
  if (m >= nl) return;  // whole groups of four lanes
  const int64_t off = cl.z;
  const float s = nu[off + m];
  const float *src = xpm + off * d_pad + (int64_t)m * 16 + 4 * part;
  const int64_t bs = (int64_t)16 * nl;
  uint2 *dst = out + ((off * nkb + m) * 64 >> 2) + part;
  float ss = 0.f;
  float4 v[4], w[4];
  auto load = [&](float4(&r)[4], int kb) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int b = 4 * kb + j;
      r[j] = 16 * b + 4 * part < d_s ? __ldg((const float4 *)(src + b * bs))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto store = [&](const float4(&r)[4], int kb) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float a = r[j].x * s, b = r[j].y * s, c = r[j].z * s, d = r[j].w * s;
      ss = fmaf(a, a, ss);
      ss = fmaf(b, b, ss);
      ss = fmaf(c, c, ss);
      ss = fmaf(d, d, ss);
      dst[(int64_t)kb * nl * 16 + 4 * j] = half4(a, b, c, d);
    }
  };
  load(v, 0);
  for (int kb = 0; kb < nkb; kb += 2) {
    if (kb + 1 < nkb) load(w, kb + 1);
    store(v, kb);
    if (kb + 1 >= nkb) break;
    if (kb + 2 < nkb) load(v, kb + 2);
    store(w, kb + 1);
  }
  const unsigned quad = 0xFu << (threadIdx.x & 28);
  ss += __shfl_xor_sync(quad, ss, 1);
  ss += __shfl_xor_sync(quad, ss, 2);
  if (part == 0) {
    x2[off + m] = ss;
    if (!(ss <= CE_NORM2)) atomicExch(unsure, 1);
  }
}

// Per query (one warp) of rows v: |v|^2, the FP16 row (nkb blocks of 64, zero
// beyond d_s) and a bound of |approximate - exact distance| to any member of
// norm at most yn whose FP16 residual is at most yr (see the file's header).
__global__ void f16_queries_kernel(const float *__restrict__ qs, int ldq, int64_t B, int d_s,
                                   int nkb, const int *__restrict__ unsure, float yn, float yr,
                                   float zmax2, float e_rest, uint2 *__restrict__ out,
                                   float *__restrict__ qn2, float *__restrict__ qerr) {
  const int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (q >= B) return;
  const float4 *src = (const float4 *)(qs + q * ldq);
  uint2 *dst = out + q * nkb * 16;
  float s2 = 0.f, r2 = 0.f;
  for (int c = lane; c < nkb * 16; c += 32) {
    const float4 v = 4 * c < d_s ? src[c] : make_float4(0.f, 0.f, 0.f, 0.f);
    const uint2 h = half4(v.x, v.y, v.z, v.w);
    dst[c] = h;
    const float2 lo = __half22float2(*(const __half2 *)&h.x), hi = __half22float2(*(const __half2 *)&h.y);
    const float e[4] = {v.x, v.y, v.z, v.w}, g[4] = {lo.x, lo.y, hi.x, hi.y};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float r = e[u] - g[u];
      s2 = fmaf(e[u], e[u], s2);
      r2 = fmaf(r, r, r2);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    r2 += __shfl_xor_sync(0xffffffffu, r2, o);
  }
  if (lane == 0) {
    const float zn = sqrtf(s2), rho = sqrtf(r2), h = 0.5f * (zn + yn);
    qn2[q] = s2;
    qerr[q] = (unsure && *unsure) || !(s2 <= zmax2)
                  ? CE_UNSURE
                  : 2.f * (zn * yr + rho * yn + rho * yr) * 1.001f + e_rest * fmaxf(1.f, h * h);
  }
}

// probe slots of the queries already answered (cnt >= 0) -> PROBE_NONE
__global__ void mask_answered_kernel(uint64_t *__restrict__ ckeys, int64_t n, int nprobe,
                                     const int32_t *__restrict__ cnt) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n && cnt[e / nprobe] >= 0) ckeys[e] = PROBE_NONE;
}

// Queries in the order of their nearest list along the index's chain of lists,
// so that the re-scores running at one time share member rows in L2.
__global__ void order_count_kernel(const uint64_t *__restrict__ ckeys, int64_t B, int nprobe,
                                   const int32_t *__restrict__ rank, int32_t *__restrict__ cnt) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < B) atomicAdd(&cnt[rank[probe_list(ckeys[q * nprobe])]], 1);
}
__global__ void order_fill_kernel(const uint64_t *__restrict__ ckeys, int64_t B, int nprobe,
                                  const int32_t *__restrict__ rank, int32_t *__restrict__ cursor,
                                  int32_t *__restrict__ order) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < B) order[atomicAdd(&cursor[rank[probe_list(ckeys[q * nprobe])]], 1)] = (int32_t)q;
}

// Exact re-score and top-k of one query per CTA.  A warp takes 32 members at a
// time, one per lane, so that each distance is accumulated by one thread over
// ascending coordinates (the scans' order).  The members' 64-byte blocks come
// through a per-warp ring of RS_ST stages filled by cp.async, four lanes per
// row (a row per lane would touch 32 lines per load); rows are padded to 80
// bytes, so that the row-per-lane reads are free of bank conflicts.
constexpr int RS_W = 4, RS_ST = 4, RS_ROW = 20;

__global__ void __launch_bounds__(RS_W * 32) rescore_kernel(
    const int64_t *__restrict__ cand, const int32_t *__restrict__ cnt, int kk,
    const int32_t *__restrict__ order, const float *__restrict__ qs, int ldq, int d_s,
    const float *__restrict__ xpm, int d_pad, const int64_t *__restrict__ list_off,
    const int32_t *__restrict__ list_ids, const float *__restrict__ nu, int k,
    int64_t *__restrict__ out_ids, float *__restrict__ out_dist) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int64_t q = order ? order[blockIdx.x] : blockIdx.x;
  const int n = cnt[q];
  if (n < 0) return;  // left to the tiled scan
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nblk = (d_s + 15) >> 4;
  float *sq = (float *)smem;                                    // the query row
  float *ring = sq + nblk * 16 + warp * (RS_ST * 32 * RS_ROW);  // this warp's stages
  uint64_t *keys = (uint64_t *)(sq + nblk * 16 + RS_W * RS_ST * 32 * RS_ROW);
  for (int j = threadIdx.x; j < nblk * 4; j += RS_W * 32)
    ((float4 *)sq)[j] = ((const float4 *)(qs + q * ldq))[j];
  __syncthreads();
  const int part = lane & 3;
  for (int i0 = warp * 32; i0 < n; i0 += RS_W * 32) {
    const int i = i0 + lane;
    const int64_t c = i < n ? cand[q * kk + i] : -1;
    int64_t base = 0, off = 0;
    int nl = 0;
    if (c >= 0) {
      const int l = (int)(c >> 32);
      off = list_off[l];
      nl = (int)(list_off[l + 1] - off);
      base = off * d_pad + (c & 0xffffffffll) * 16;
    }
    // this lane copies part `part` of rows lane / 4 + 8 t
    const float *src[4];
    int64_t bs[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int r = (lane >> 2) + 8 * t;
      const int64_t b = __shfl_sync(0xffffffffu, base, r);
      const int w = __shfl_sync(0xffffffffu, nl, r);
      src[t] = xpm + b + 4 * part;
      bs[t] = (int64_t)16 * w;  // 0: an empty slot, nothing to copy
    }
    auto fill = [&](int b) {
      float *d = ring + (b % RS_ST) * (32 * RS_ROW) + (lane >> 2) * RS_ROW + 4 * part;
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (bs[t]) cp_async16(d + 8 * t * RS_ROW, src[t] + b * bs[t]);
    };
    const float s = c >= 0 && nu ? nu[off + (c & 0xffffffffll)] : 1.f;
    const uint32_t id = c >= 0 ? (uint32_t)list_ids[off + (c & 0xffffffffll)] : 0u;
#pragma unroll
    for (int b = 0; b < RS_ST - 1; ++b) {
      if (b < nblk) fill(b);
      cp_async_commit();
    }
    float acc = 0.f;
    for (int b = 0; b < nblk; ++b) {
      if (b + RS_ST - 1 < nblk) fill(b + RS_ST - 1);
      cp_async_commit();
      cp_async_wait<RS_ST - 1>();
      __syncwarp();
      const float *xr = ring + (b % RS_ST) * (32 * RS_ROW) + lane * RS_ROW;
      const float *qr = sq + 16 * b;
      const int nd4 = min(4, (d_s - 16 * b) >> 2);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (u >= nd4) break;
        const float4 x = *(const float4 *)(xr + 4 * u), p = *(const float4 *)(qr + 4 * u);
        float t;
        t = fmaf(-s, x.x, p.x); acc = fmaf(t, t, acc);
        t = fmaf(-s, x.y, p.y); acc = fmaf(t, t, acc);
        t = fmaf(-s, x.z, p.z); acc = fmaf(t, t, acc);
        t = fmaf(-s, x.w, p.w); acc = fmaf(t, t, acc);
      }
      __syncwarp();  // the stage is refilled next
    }
    if (i < n) keys[i] = c >= 0 ? pack_key(acc, id) : KEY_MAX;
  }
  __syncthreads();
  if (warp != 0) return;
  if (n <= 256) warp_sort_regs<8>(keys, n, k);
  else if (n <= 512) warp_sort_regs<16>(keys, n, k);
  else warp_sort(keys, n);
  for (int r = lane; r < k; r += 32) {
    const uint64_t key = r < n ? keys[r] : KEY_MAX;
    out_ids[q * k + r] = key == KEY_MAX ? -1 : (int64_t)(uint32_t)(key & 0xffffffffu);
    out_dist[q * k + r] = key == KEY_MAX ? __int_as_float(0x7f800000)
                                         : __uint_as_float((uint32_t)(key >> 32));
  }
}

}  // namespace

int launch_f16_queries(const float *v, int ldv, int64_t B, int d_s, int nkb, const int *unsure,
                       float yn, float yr, float zmax2, void *out, float *qn2, float *qerr,
                       cudaStream_t st) {
  if (B <= 0) return ADANNS_OK;
  // FP32 accumulation on the tensor cores, the FP32 norms and the re-score's rounding
  const float e_rest = (float)(2.0 * nkb * 64 * std::ldexp(1.0, -22) +
                               8.0 * (d_s + 2) * std::ldexp(1.0, -24) + 1e-4);
  f16_queries_kernel<<<(unsigned)((B + 7) / 8), 256, 0, st>>>(v, ldv, B, d_s, nkb, unsure, yn, yr,
                                                              zmax2, e_rest, (uint2 *)out, qn2,
                                                              qerr);
  ADN_LAUNCH("f16_queries_kernel");
  return ADANNS_OK;
}

int launch_query_order(const adanns_index *idx, const uint64_t *ckeys, int64_t B, int nprobe,
                       int32_t *order, cudaStream_t st) {
  if (B <= 0) return ADANNS_OK;
  Scratch s(st);
  int32_t *cur;
  int rc;
  if ((rc = s.get(&cur, idx->nlist))) return rc;
  const unsigned g = (unsigned)((B + 255) / 256);
  ADN_CUDA(cudaMemsetAsync(cur, 0, sizeof(int32_t) * idx->nlist, st));
  order_count_kernel<<<g, 256, 0, st>>>(ckeys, B, nprobe, idx->rr_rank, cur);
  ADN_LAUNCH("order_count_kernel");
  if ((rc = launch_scan_i32(cur, idx->nlist, cur, st))) return rc;
  order_fill_kernel<<<g, 256, 0, st>>>(ckeys, B, nprobe, idx->rr_rank, cur, order);
  ADN_LAUNCH("order_fill_kernel");
  return ADANNS_OK;
}

int launch_mask_answered(uint64_t *ckeys, int64_t B, int nprobe, const int32_t *cnt,
                         cudaStream_t st) {
  const int64_t n = B * nprobe;
  if (n <= 0) return ADANNS_OK;
  mask_answered_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ckeys, n, nprobe, cnt);
  ADN_LAUNCH("mask_answered_kernel");
  return ADANNS_OK;
}

namespace {

struct Shape {
  int nkb, kk;
  int64_t seg;    // largest candidate segment of a query
  int64_t fixed;  // scratch whatever the slice: rows, one part-filled tile per list
  int64_t per_q;  // and per query of a slice
  int64_t Bc;     // queries per slice
  TiledScan ts;
};

// the FP16 copy with the members' |x|^2, and each list's part-filled query tile
int64_t filter_fixed_bytes(const adanns_index *idx, int64_t nkb) {
  return idx->N * (nkb * 128 + 4) + 256 + idx->nlist * (nkb * 128 * 128 + 96);
}

Shape shape_of(const adanns_index *idx, int64_t B, int d_c, int d_s, int nprobe, int k) {
  Shape h{};
  h.nkb = (d_s + 63) / 64;
  h.kk = shortlist_cap(k);
  h.fixed = filter_fixed_bytes(idx, h.nkb);
  tiled_scan_shape(idx, B, d_s, nprobe, k, &h.ts);
  h.seg = max_probe_members(idx, nprobe);
  h.per_q = h.seg * 2 + (int64_t)nprobe * ((int64_t)h.nkb * 128 + 60) +
            (int64_t)(pad16(d_c) + pad16(d_s)) * 4 + (int64_t)h.nkb * 128 + (int64_t)h.kk * 8 + 64 +
            (int64_t)nprobe * h.ts.nsplit * k * 8 + coarse_scratch_per_query(idx, d_c);
  h.Bc = std::max<int64_t>(1, std::min<int64_t>(B, (scratch_budget() - h.fixed) / h.per_q));
  return h;
}

}  // namespace

// Where the filter pays: where its estimated time is the smallest (f32_cost).
// Measured, filter / streaming / tiled in us: 1.28 M rows x 512, 16 of 1,024 lists, k
// 10, 8 queries per list 967 / 845 / -, 16: 1058 / 1504 / -; 10,000 x 64 in 64 lists, 2
// probed, k 1, 256 queries per list 276 / - / 115; 20,000 x 64 in 64 lists, 2 probed,
// k 256 (every member of the lists is re-scored), 600 per list 1948 / - / 991.
// Below F32_SMALL rows all routes are bound by launches; there the filter stays
// above 100 queries per list while it is within 80 us of the others (65 at k 1), so
// that its small sizes keep being run.  A row without a usable norm would leave every
// query to the tiled scan: the direct scans from the start.  k and the probes must fit the shortlist's buffers,
// and the FP16 rows with the tiles' padding may take half of the call's scratch budget.  Turning the
// streaming scan off asks for the tiled scan everywhere.
constexpr int64_t F32_SMALL = 8192;

bool f32_certified(const adanns_index *idx, int64_t B, int d_s, int nprobe, int k) {
  if (idx->metric != ADANNS_METRIC_L2_PREFIXNORM || k > CE_MAX_K || nprobe > 128) return false;
  if (!option(ADANNS_OPT_FP32_STREAM) || scan_choice_forced()) return false;
  const int64_t nkb = (d_s + 63) / 64;
  if (idx->N * nkb > INT32_MAX - 256) return false;  // 32-bit row coordinates of the copies
  if (filter_fixed_bytes(idx, nkb) > scratch_budget() / 2) return false;
  const int64_t pairs = B * nprobe;
  double other = f32_cost(F32_STREAM, idx, B, pairs, d_s, k);
  if (k == 1 && pairs > 16ll * idx->nlist)
    other = std::min(other, f32_cost(F32_TILED, idx, B, pairs, d_s, k));
  const double qpl = (double)pairs / idx->nlist;
  if (idx->N >= F32_SMALL && (idx->unsure >> gran_index(d_s) & 1)) return false;
  if (idx->N < F32_SMALL && qpl > 100.0 && (double)idx->N * d_s * qpl > 2e7 &&
      nprobe * idx->N > shortlist_cap(k) * (int64_t)idx->nlist)
    other += k == 1 ? 6.5e7 : 8e7;
  return f32_cost(F32_FILTER, idx, B, pairs, d_s, k) < other;
}

int64_t certified_scratch_bytes(const adanns_index *idx, int64_t B, int d_c, int d_s, int nprobe,
                                int k) {
  const Shape h = shape_of(idx, B, d_c, d_s, nprobe, k);
  return h.fixed + h.Bc * h.per_q + Scratch::SLACK;
}

int search_f32_certified(const adanns_index *idx, const float *queries, int64_t B, int d_c,
                         int d_s, int nprobe, int k, int64_t *out_ids, float *out_dist,
                         int32_t *out_probes, cudaStream_t st) {
  const int nlist = idx->nlist, dcp = pad16(d_c), dsp = pad16(d_s), QT = 128;
  Shape h = shape_of(idx, B, d_c, d_s, nprobe, k);
  const int nkb = h.nkb, kk = h.kk;
  const int64_t Bc = h.Bc;
  const int64_t max_tiles = (Bc * nprobe + QT - 1) / QT + nlist;
  const bool ordered = Bc >= 4096 && nlist > 1;  // fewer queries: their rows fit in L2 anyway
  Scratch s(st);
  float *qc, *qs, *qn2, *qerr, *x2;
  uint64_t *ckeys;
  int32_t *lcnt, *lbeg, *lfill, *tbeg, *pair_q, *pair_out, *tl, *tb, *tc, *cnt, *order = nullptr;
  int *ntiles, *flags;  // flags: [0] cluster mapping, [1] scan, [2] tiled scan counters, [3] unsure
  int64_t *qtot, *qbase, *pbase, *cids;
  unsigned char *qlow, *qtile, *rows;
  uint16_t *cand;
  unsigned long long *stats = nullptr;
  int rc;
  if ((rc = s.get(&rows, (size_t)idx->N * nkb * 128 + 256)) || (rc = s.get(&x2, idx->N)) ||
      (rc = s.get(&qc, (size_t)Bc * dcp)) || (rc = s.get(&qs, (size_t)Bc * dsp)) ||
      (rc = s.get(&qn2, Bc)) || (rc = s.get(&qerr, Bc)) ||
      (rc = s.get(&ckeys, (size_t)Bc * nprobe)) || (rc = s.get(&lcnt, nlist)) ||
      (rc = s.get(&lbeg, nlist)) || (rc = s.get(&lfill, nlist)) || (rc = s.get(&tbeg, nlist)) ||
      (rc = s.get(&pair_q, (size_t)Bc * nprobe)) || (rc = s.get(&pair_out, (size_t)Bc * nprobe)) ||
      (rc = s.get(&tl, max_tiles)) || (rc = s.get(&tb, max_tiles)) ||
      (rc = s.get(&tc, max_tiles)) || (rc = s.get(&cnt, Bc)) || (rc = s.get(&ntiles, 1)) ||
      (rc = s.get(&flags, 4)) || (rc = s.get(&qtot, Bc)) || (rc = s.get(&qbase, Bc)) ||
      (rc = s.get(&pbase, (size_t)Bc * nprobe)) || (rc = s.get(&cids, (size_t)Bc * kk)) ||
      (rc = s.get(&qlow, (size_t)Bc * nkb * 128)) ||
      (rc = s.get(&qtile, (size_t)max_tiles * nkb * QT * 128)) ||
      (rc = s.get(&cand, (size_t)(Bc * h.seg))) ||
      (rc = tiled_scan_scratch(s, idx, Bc, nprobe, k, &h.ts)))
    return rc;
  if (ordered && (rc = s.get(&order, Bc))) return rc;
  if (profiling() && (rc = s.get(&stats, 2))) return rc;
  const float *nu = idx->invn + (int64_t)gran_index(d_s) * idx->N;
  const float yn = sqrtf(CE_NORM2);
  const float yr = (float)(yn * std::ldexp(1.0, -11) + d_s * std::ldexp(1.0, -25));
  const size_t rsm = (size_t)pad16(d_s) * 4 + (size_t)RS_W * RS_ST * 32 * RS_ROW * 4 + (size_t)kk * 8;
  ADN_CUDA(ensure_smem((const void *)rescore_kernel, rsm));
  for (int64_t b0 = 0; b0 < B; b0 += Bc) {
    const int64_t nb = std::min(Bc, B - b0);
    int64_t *oi = out_ids + b0 * k;
    float *od = out_dist + b0 * k;
    {
      StageTimer t(ST_PREP, st);
      if ((rc = launch_prep_queries(queries + b0 * idx->d, nb, idx->d, d_c, d_s, idx->metric, qc,
                                    dcp, qs, dsp, st)))
        return rc;
    }
    // the flag of a slice stays set for the following ones
    ADN_CUDA(cudaMemsetAsync(flags, 0, (b0 == 0 ? 4 : 3) * sizeof(int), st));
    {
      StageTimer t(ST_COARSE, st);
      if ((rc = run_coarse(idx, qc, dcp, nb, d_c, nprobe, ckeys, flags, st))) return rc;
    }
    {
      StageTimer t(ST_INVERT, st);
      ProbePlan plan;
      plan.list_off = idx->list_off;
      plan.qbase = qbase;
      plan.pbase = pbase;
      if ((rc = launch_invert_probes(ckeys, nb, nprobe, nlist, QT, lcnt, lbeg, lfill, tbeg, pair_q,
                                     pair_out, tl, tb, tc, ntiles,
                                     out_probes ? out_probes + b0 * nprobe : nullptr, st, &plan)))
        return rc;
      if (!plan.planned && (rc = launch_cand_segments(ckeys, nb, nprobe, idx->list_off, qtot,
                                                      qbase, pbase, st)))
        return rc;
    }
    {
      StageTimer t(ST_PREP, st);
      if (b0 == 0) {  // every list when the batch is sliced, else the probed ones
        f16_rows_kernel<<<(unsigned)idx->rr_chunks[0], 256, 0, st>>>(
            idx->xpm, idx->d_pad, d_s, nkb, idx->rr_cmap[0], Bc < B ? nullptr : lcnt, nu,
            (uint2 *)rows, x2, flags + 3);
        ADN_LAUNCH("f16_rows_kernel");
      }
      if ((rc = launch_f16_queries(qs, dsp, nb, d_s, nkb, flags + 3, yn, yr, CE_NORM2, qlow, qn2,
                                   qerr, st)))
        return rc;
      if ((rc = launch_gather_qtiles(qlow, nkb, max_tiles, tb, tc, ntiles, pair_q, QT, qtile, st)))
        return rc;
    }
    {
      StageTimer t(ST_MMA, st);
      MmaScanArgs m{};
      m.tile_list = tl;
      m.tile_beg = tb;
      m.tile_cnt = tc;
      m.ntiles_dev = ntiles;
      m.list_off = idx->list_off;
      m.pair_out = pair_out;
      m.pbase = pbase;
      m.qn2 = qn2;
      m.x2 = x2;
      m.nprobe = nprobe;
      m.nkb = nkb;
      m.d_blocks = nkb;
      m.cand = cand;
      m.err = idx->dev_err;
      m.tile_counter = flags + 1;
      m.f16 = 1;
      m.nsplit = mma_scan_nsplit(idx, nb * nprobe);
      if ((rc = launch_mma_scan(qtile, max_tiles * nkb * QT, rows, idx->N * (int64_t)nkb, m, st)))
        return rc;
    }
    {
      StageTimer t(ST_SELECT, st);
      if (stats) ADN_CUDA(cudaMemsetAsync(stats, 0, 2 * sizeof(unsigned long long), st));
      if ((rc = launch_certify16(cand, ckeys, nprobe, qbase, idx->list_off, kk, k, qerr, nb,
                                 cids, cnt, stats, st)))
        return rc;
      if (stats) {
        profile_count(PC_RERANK_PAIRS, (const int64_t *)stats, st);
        profile_count(PC_SELECT_SLOW, (const int64_t *)stats + 1, st);
      }
    }
    {
      StageTimer t(ST_RERANK, st);
      if (ordered && (rc = launch_query_order(idx, ckeys, nb, nprobe, order, st))) return rc;
      rescore_kernel<<<(unsigned)nb, RS_W * 32, rsm, st>>>(
          cids, cnt, kk, order, qs, dsp, d_s, idx->xpm, idx->d_pad, idx->list_off, idx->list_ids,
          nu, k, oi, od);
      ADN_LAUNCH("rescore_kernel");
    }
    // the queries left over (usually none): the tiled scan on them alone
    if ((rc = launch_mask_answered(ckeys, nb, nprobe, cnt, st))) return rc;
    MergeMask mm;
    mm.ckeys = ckeys;
    mm.nsplit = h.ts.nsplit;
    mm.only = cnt;
    if ((rc = run_tiled_scan(idx, h.ts, qs, dsp, nb, d_s, nprobe, k, ckeys, flags + 2, nullptr, oi,
                             od, mm, st)))
      return rc;
  }
  return ADANNS_OK;
}

}  // namespace adn
