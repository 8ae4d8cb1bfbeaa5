// Low-dimensional graph shortlist with a high-dimensional rerank: the
// AdANNS-DiskANN composite of Sec. 4.3 ("AdANNS for Composite Indices") --
// the search graph is formed with a low-d MR and its shortlist is re-ranked
// with a high-d MR.
//
// Build (one pass, DiskANN-style pruned proximity graph at the d_g prefix):
//   1. every row's K nearest other rows: a brute-force sweep of the FP32 list
//      scan over one list holding all rows (fused top-(K+1), the row itself
//      dropped);
//   2. robust prune of each candidate list with factor alpha to at most R
//      out-neighbours (one warp per row);
//   3. every edge p -> c offers p to c (counting sort by target); a row whose
//      own and offered neighbours exceed R is pruned again over their union
//      sorted by (distance, id) (one CTA per row);
//   4. entry point: the row nearest to the FP64 mean of the rows.
// Search (one warp per query): best-first with a bounded candidate list of L
// entries in shared memory -- expand the nearest entry not yet expanded, score
// its neighbours that are not in the list (one lane each), keep the L nearest
// by (distance, id) -- until every entry is expanded; then the rerank_k
// nearest are re-scored with the exact FP32 distance at d_s and the k best
// returned.  All distances are FP32 in difference form.
#include <algorithm>
#include <vector>

#include "devutil.cuh"
#include "internal.cuh"

struct adanns_graph {
  int64_t N = 0;
  int d = 0, d_g = 0, dg_pad = 0, R = 0, metric = 0;
  int64_t entry = 0;
  float *xg = nullptr;     // N x dg_pad: P_dg of every row (id order)
  int32_t *nbr = nullptr;  // N x R neighbours, -1 padding, each row by (distance, id)
  float *rows = nullptr;   // N x d FP32 rows (id order), for the rerank
  int *dev_err = nullptr;
};

namespace adn {
namespace {

constexpr int GR_MAXR = 64;      // out-degree limit
constexpr int GR_MAXK = 256;     // candidate list limit of the build
constexpr int GR_MAXDG = 64;     // graph dimension limit (one lane scores a whole row)
constexpr int GR_MAXL = 512;     // search list limit
constexpr int GR_UCAP = 4096;    // own + offered neighbours of one row in the final prune
constexpr int ERR_HUB = 0x200;   // status bit: a row was offered more than GR_UCAP edges

__device__ __forceinline__ float sqdist(const float *a, const float *b, int m) {
  float acc = 0.f;
  for (int j = 0; j < m; ++j) {
    const float t = a[j] - b[j];
    acc = fmaf(t, t, acc);
  }
  return acc;
}

__device__ __forceinline__ uint64_t gkey(float d, int32_t id) {
  return ((uint64_t)__float_as_uint(d) << 32) | (uint32_t)id;
}

// ---------------------------------------------------------------- build
// knn[p][0:K] from the sweep's sorted (K + 1) keys: the row itself (or, among
// rows at distance 0, the last one) is left out
__global__ void knn_drop_self_kernel(const uint64_t *__restrict__ keys, int64_t N, int K,
                                     int32_t *__restrict__ knn, float *__restrict__ kd) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  const uint64_t *k = keys + p * (K + 1);
  int w = 0;
  bool dropped = false;
  for (int r = 0; r <= K && w < K; ++r) {
    const uint64_t v = k[r];
    const int32_t id = v == KEY_MAX ? -1 : (int32_t)(uint32_t)(v & 0xffffffffu);
    if (!dropped && id == (int32_t)p) {
      dropped = true;
      continue;
    }
    knn[p * K + w] = id;
    kd[p * K + w] = id < 0 ? __int_as_float(0x7f800000) : __uint_as_float((uint32_t)(v >> 32));
    ++w;
  }
  for (; w < K; ++w) {
    knn[p * K + w] = -1;
    kd[p * K + w] = __int_as_float(0x7f800000);
  }
}

// one warp per row: robust prune of its K candidates (sorted by (distance, id))
__global__ void prune_kernel(const float *__restrict__ xg, int ldg, int d_g,
                             const int32_t *__restrict__ knn, const float *__restrict__ kd, int K,
                             int64_t N, float alpha, int R, int32_t *__restrict__ fwd,
                             int32_t *__restrict__ nfwd) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  if (p >= N) return;
  constexpr int PER = GR_MAXK / 32;
  int32_t id[PER];
  float dp[PER];
  bool alive[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int r = u * 32 + lane;
    id[u] = r < K ? knn[p * K + r] : -1;
    dp[u] = r < K ? kd[p * K + r] : 0.f;
    alive[u] = id[u] >= 0 && id[u] != (int32_t)p;
  }
  int nout = 0;
  for (int r0 = 0; r0 < K && nout < R; ++r0) {
    // candidate r0 is the nearest alive one when it is alive (list order)
    const int u0 = r0 >> 5;
    bool al = false;
    int32_t c = -1;
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (u == u0) {
        al = alive[u];
        c = id[u];
      }
    al = __shfl_sync(0xffffffffu, al, r0 & 31);
    c = __shfl_sync(0xffffffffu, c, r0 & 31);
    if (!al) continue;
    if (lane == 0) fwd[p * R + nout] = c;
    ++nout;
    const float *xc = xg + (int64_t)c * ldg;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int r = u * 32 + lane;
      if (r == r0) alive[u] = false;
      if (r > r0 && alive[u]) {
        const float dcv = alpha * sqdist(xc, xg + (int64_t)id[u] * ldg, d_g);
        if (dcv <= dp[u]) alive[u] = false;
      }
    }
  }
  for (int r = nout + lane; r < R; r += 32) fwd[p * R + r] = -1;
  if (lane == 0) nfwd[p] = nout;
}

__global__ void offer_count_kernel(const int32_t *__restrict__ fwd, int64_t n, int32_t *cnt) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int32_t c = fwd[e];
  if (c >= 0) atomicAdd(&cnt[c], 1);
}

__global__ void offer_fill_kernel(const int32_t *__restrict__ fwd, int64_t n, int R,
                                  int32_t *__restrict__ cursor, int32_t *__restrict__ rev) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int32_t c = fwd[e];
  if (c >= 0) rev[atomicAdd(&cursor[c], 1)] = (int32_t)(e / R);
}

// one CTA per row q: union of own and offered neighbours by (distance, id),
// duplicates dropped; kept whole when it fits R, else robust-pruned to R
constexpr int FIN_THREADS = 256;
__global__ void __launch_bounds__(FIN_THREADS) final_prune_kernel(
    const float *__restrict__ xg, int ldg, int d_g, const int32_t *__restrict__ fwd,
    const int32_t *__restrict__ nfwd, const int32_t *__restrict__ roff,
    const int32_t *__restrict__ rev, int64_t N, float alpha, int R, int32_t *__restrict__ out,
    int *__restrict__ err) {
  __shared__ uint64_t u[GR_UCAP];
  __shared__ int s_n;
  const int64_t q = blockIdx.x;
  const int tid = threadIdx.x;
  const int nf = nfwd[q];
  const int r0 = roff[q], nr = roff[q + 1] - r0;
  int nu = nf + nr;
  if (nu > GR_UCAP) {  // a hub beyond the buffer: report, keep its own list
    if (tid == 0) atomicOr(err, ERR_HUB);
    for (int r = tid; r < R; r += FIN_THREADS) out[q * R + r] = fwd[q * R + r];
    return;
  }
  const float *xq = xg + q * ldg;
  for (int i = tid; i < nu; i += FIN_THREADS) {
    const int32_t c = i < nf ? fwd[q * R + i] : rev[r0 + i - nf];
    u[i] = gkey(sqdist(xq, xg + (int64_t)c * ldg, d_g), c);
  }
  int P = 1;
  while (P < nu) P <<= 1;
  for (int i = nu + tid; i < P; i += FIN_THREADS) u[i] = KEY_MAX;
  __syncthreads();
  // bitonic sort of P keys
  for (int size = 2; size <= P; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = tid; i < P; i += FIN_THREADS) {
        const int j = i ^ stride;
        if (j > i) {
          const bool up = (i & size) == 0;
          const uint64_t a = u[i], b = u[j];
          if ((a > b) == up) {
            u[i] = b;
            u[j] = a;
          }
        }
      }
      __syncthreads();
    }
  // drop duplicates (equal keys are adjacent)
  if (tid == 0) {
    int w = 0;
    for (int i = 0; i < nu; ++i)
      if (w == 0 || u[i] != u[w - 1]) u[w++] = u[i];
    s_n = w;
  }
  __syncthreads();
  nu = s_n;
  if (nu <= R) {
    for (int r = tid; r < R; r += FIN_THREADS)
      out[q * R + r] = r < nu ? (int32_t)(uint32_t)(u[r] & 0xffffffffu) : -1;
    return;
  }
  // robust prune over the sorted union: a pruned entry is overwritten with
  // the empty key
  int nout = 0;
  for (int i = 0; i < nu && nout < R; ++i) {
    __syncthreads();
    if (u[i] == KEY_MAX) continue;  // uniform: every thread reads the same slot
    const int32_t c = (int32_t)(uint32_t)(u[i] & 0xffffffffu);
    if (tid == 0) out[q * R + nout] = c;
    ++nout;
    const float *xc = xg + (int64_t)c * ldg;
    __syncthreads();
    for (int j = i + 1 + tid; j < nu; j += FIN_THREADS) {
      const uint64_t v = u[j];
      if (v == KEY_MAX) continue;
      const int32_t vid = (int32_t)(uint32_t)(v & 0xffffffffu);
      const float dpv = __uint_as_float((uint32_t)(v >> 32));
      if (alpha * sqdist(xc, xg + (int64_t)vid * ldg, d_g) <= dpv) u[j] = KEY_MAX;
    }
  }
  __syncthreads();
  for (int r = nout + tid; r < R; r += FIN_THREADS) out[q * R + r] = -1;
}

// FP64 coordinate sums of the rows (one thread per (block of rows, coordinate))
__global__ void row_sum_kernel(const float *__restrict__ xg, int ldg, int d_g, int64_t N,
                               double *__restrict__ sum) {
  const int j = threadIdx.x;
  if (j >= d_g) return;
  double acc = 0.0;
  for (int64_t p = blockIdx.x; p < N; p += gridDim.x) acc += (double)xg[p * ldg + j];
  atomicAdd(&sum[j], acc);
}

__global__ void entry_kernel(const float *__restrict__ xg, int ldg, int d_g, int64_t N,
                             const double *__restrict__ sum, unsigned long long *__restrict__ best) {
  __shared__ float mean[GR_MAXDG];
  if (threadIdx.x < d_g) mean[threadIdx.x] = (float)(sum[threadIdx.x] / (double)N);
  __syncthreads();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  atomicMin(best, (unsigned long long)gkey(sqdist(xg + p * ldg, mean, d_g), (int32_t)p));
}

// ---------------------------------------------------------------- search
constexpr int GS_WARPS = 4;

struct GsArgs {
  const float *xg;
  int ldg, d_g;
  const int32_t *nbr;
  int R;
  int64_t entry, N;
  const float *qg;
  int ldq;
  int64_t B;
  int L, kk;
  int64_t *short_ids;  // [B][kk], -1 padding
  int64_t *nexp;       // optional [B]
};

// One warp per query.  The list lives in registers, 32 LR >= L entries sorted
// ascending, position 32 s + lane in lst[s]: (distance bits, id) << 1 | expanded
// (a distance's sign bit and an id's top bit are 0, so the order is that of
// (distance, id)); empty entries are all ones, which read as expanded.
//
// An expansion loads the row's neighbours, drops those that a small table of
// ids remembers as scored (a scored id is in the list, or was turned away or
// dropped by entries that can only have become nearer since: it would change
// nothing), scores the rest one per lane, and keeps those nearer than the last
// entry of a full list and not in the list (the table forgets).  A few are
// inserted one by one, each by a shift of the entries behind it; many are sorted
// and merged block by block with bitonic half-cleaners.  Nothing of the list
// passes through shared memory.  Bound by the two dependent gathers of an
// expansion and by instruction issue: 10,000 queries, L 64, R 32, d_g 16 over
// 262,144 rows 1.72 ms with the list merged in shared memory, 0.34 here.
constexpr int GS_SEEN = 1024;  // remembered ids per query
__device__ __forceinline__ int gs_slot(int32_t u) {
  return (int)(((uint32_t)u * 2654435761u) >> 22);  // the top 10 bits
}

__device__ __forceinline__ uint64_t bitonic_clean32(uint64_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int stride = 16; stride > 0; stride >>= 1) {
    const uint64_t o = __shfl_xor_sync(0xffffffffu, v, stride);
    const uint64_t lo = o < v ? o : v, hi = o < v ? v : o;
    v = lane & stride ? hi : lo;
  }
  return v;
}

// |q - x|^2 over m coordinates (a multiple of 8, rows 16-byte aligned): the
// sums of sqdist with 16-byte loads
__device__ __forceinline__ float sqdist4(const float *q, const float *x, int m) {
  float acc = 0.f;
#pragma unroll 4
  for (int j = 0; j < m; j += 4) {
    const float4 v = __ldg((const float4 *)(x + j)), p = *(const float4 *)(q + j);
    float t;
    t = p.x - v.x; acc = fmaf(t, t, acc);
    t = p.y - v.y; acc = fmaf(t, t, acc);
    t = p.z - v.z; acc = fmaf(t, t, acc);
    t = p.w - v.w; acc = fmaf(t, t, acc);
  }
  return acc;
}

template <int LR>
__global__ void __launch_bounds__(GS_WARPS * 32) graph_search_kernel(GsArgs a) {
  __shared__ __align__(16) float s_q[GS_WARPS][GR_MAXDG];
  __shared__ int32_t s_seen[GS_WARPS][GS_SEEN];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t qi = (int64_t)blockIdx.x * GS_WARPS + warp;
  if (qi >= a.B) return;
  const int L = a.L;
  float *qv = s_q[warp];
  int32_t *seen = s_seen[warp];
  for (int j = lane; j < a.d_g; j += 32) qv[j] = a.qg[qi * a.ldq + j];
  for (int j = lane; j < GS_SEEN; j += 32) seen[j] = -1;
  __syncwarp();
  constexpr uint64_t NONE = ~0ull;
  uint64_t lst[LR];
#pragma unroll
  for (int s = 0; s < LR; ++s) lst[s] = NONE;
  {
    const uint64_t k = gkey(sqdist4(qv, a.xg + a.entry * a.ldg, a.d_g), (int32_t)a.entry) << 1;
    if (lane == 0) lst[0] = k;
  }
  int64_t nexp = 0;
  for (int64_t it = 0; it < a.N; ++it) {
    // the nearest entry not yet expanded
    uint64_t cur = NONE;
#pragma unroll
    for (int s = 0; s < LR; ++s) {
      const unsigned m = __ballot_sync(0xffffffffu, !(lst[s] & 1));
      if (m && cur == NONE) {
        const int src = __ffs(m) - 1;
        cur = __shfl_sync(0xffffffffu, lst[s], src);
        if (lane == src) lst[s] |= 1;
      }
    }
    if (cur == NONE) break;
    const int32_t v = (int32_t)(uint32_t)(cur >> 1);
    ++nexp;
    // the L-th entry: NONE while the list is not full
    uint64_t worst = lst[0];
#pragma unroll
    for (int s = 1; s < LR; ++s) worst = (L - 1) >> 5 >= s ? lst[s] : worst;
    worst = __shfl_sync(0xffffffffu, worst, (L - 1) & 31);
    uint64_t key[2];
    unsigned keep[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      key[h] = NONE;
      keep[h] = 0;
      if (32 * h < a.R) {
        const int r = 32 * h + lane;
        const int32_t u = r < a.R ? __ldg(a.nbr + (int64_t)v * a.R + r) : -1;
        if (u >= 0 && seen[gs_slot(u)] != u)
          key[h] = gkey(sqdist4(qv, a.xg + (int64_t)u * a.ldg, a.d_g), u) << 1;
        keep[h] = __ballot_sync(0xffffffffu, key[h] < worst);
      }
    }
    __syncwarp();  // both halves are looked up before either is remembered
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (key[h] != NONE) {
        const int32_t u = (int32_t)(uint32_t)(key[h] >> 1);
        seen[gs_slot(u)] = u;
      }
    __syncwarp();
    // not in the list already
#pragma unroll
    for (int h = 0; h < 2; ++h)
      for (unsigned m = keep[h]; m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const uint64_t x = __shfl_sync(0xffffffffu, key[h], src) | 1;
        bool eq = false;
#pragma unroll
        for (int s = 0; s < LR; ++s) eq |= (lst[s] | 1) == x;
        if (__any_sync(0xffffffffu, eq)) keep[h] &= ~(1u << src);
      }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (__popc(keep[h]) > 6) {
        // sorted, then carried through the blocks: each keeps its 32 smallest
        uint64_t c = warp_sort_lane(keep[h] >> lane & 1 ? key[h] : NONE);
#pragma unroll
        for (int s = 0; s < LR; ++s) {
          const uint64_t r = __shfl_sync(0xffffffffu, c, 31 - lane);
          const uint64_t lo = lst[s] < r ? lst[s] : r, hi = lst[s] < r ? r : lst[s];
          lst[s] = bitonic_clean32(lo);
          if (s + 1 < LR) c = bitonic_clean32(hi);
        }
      } else {
        for (unsigned m = keep[h]; m; m &= m - 1) {
          const uint64_t x = __shfl_sync(0xffffffffu, key[h], __ffs(m) - 1);
          int p = 0;  // the position x takes
#pragma unroll
          for (int s = 0; s < LR; ++s) p += __popc(__ballot_sync(0xffffffffu, lst[s] < x));
#pragma unroll
          for (int s = LR - 1; s >= 0; --s) {
            if (32 * s + 31 >= p) {  // the blocks before stay
              const uint64_t up = __shfl_up_sync(0xffffffffu, lst[s], 1);
              const uint64_t before =
                  s > 0 ? __shfl_sync(0xffffffffu, lst[s > 0 ? s - 1 : 0], 31) : NONE;
              const int pos = 32 * s + lane;
              if (pos > p) lst[s] = lane == 0 ? before : up;
              else if (pos == p) lst[s] = x;
            }
          }
        }
      }
    }
    // entries past the L-th are dropped
#pragma unroll
    for (int s = 0; s < LR; ++s)
      if (32 * s + lane >= L) lst[s] = NONE;
  }
#pragma unroll
  for (int s = 0; s < LR; ++s) {
    const int r = 32 * s + lane;
    if (r < a.kk)
      a.short_ids[qi * a.kk + r] = lst[s] == NONE ? -1 : (int64_t)(uint32_t)(lst[s] >> 1);
  }
  if (a.nexp && lane == 0) a.nexp[qi] = nexp;
}

// per query (one CTA): exact FP32 distance at d_s of each shortlisted row
// (difference form against the row's own normalised prefix), the k best.
// Shortlists end at their first -1.  A warp holds U rows of up to 32 T
// coordinates in registers between the norm and the distance, so that their
// loads overlap and nothing is read twice (10,000 queries x 40 rows at d_s 512:
// 0.22 ms with one warp per query, row after row, 0.14 here; 3 queries x 64 rows at
// 768: 86 and 12 us).
constexpr int GRR_WARPS = 4;

template <int T, int U>
__global__ void __launch_bounds__(GRR_WARPS * 32) graph_rerank_kernel(
    const int64_t *__restrict__ cand, int kk, const float *__restrict__ qs, int ldq, int d_s,
    const float *__restrict__ rows, int d, int metric, int k, int64_t *__restrict__ out_ids,
    float *__restrict__ out_dist) {
  extern __shared__ uint64_t buf[];  // [kk]
  __shared__ int s_n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q = blockIdx.x;
  const float *qr = qs + q * ldq;
  // sum over the lanes' shares: distances 16 .. 1 by shuffles
  auto total = [&](float v) -> float {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  if (warp == 0) {  // the rows before the first -1
    int n = 0;
    for (int r0 = 0; r0 < kk; r0 += 32) {
      const unsigned m = __ballot_sync(0xffffffffu, r0 + lane < kk && cand[q * kk + r0 + lane] >= 0);
      n += m == 0xffffffffu ? 32 : __ffs(~m) - 1;
      if (m != 0xffffffffu) break;
    }
    if (lane == 0) s_n = n;
  }
  float qv[T];
#pragma unroll
  for (int t = 0; t < T; ++t) qv[t] = lane + 32 * t < d_s ? qr[lane + 32 * t] : 0.f;
  __syncthreads();
  const int n = s_n;
  for (int r = warp * U; r < n; r += GRR_WARPS * U) {
    int64_t id[U];
    float x[U][T];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      id[u] = cand[q * kk + min(r + u, n - 1)];
      const float *row = rows + id[u] * (int64_t)d;
#pragma unroll
      for (int t = 0; t < T; ++t) x[u][t] = lane + 32 * t < d_s ? __ldg(row + lane + 32 * t) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float s2 = 0.f;
#pragma unroll
      for (int t = 0; t < T; ++t)
        if (lane + 32 * t < d_s) s2 = fmaf(x[u][t], x[u][t], s2);
      s2 = total(s2);
      const float nu =
          metric == ADANNS_METRIC_L2_PREFIXNORM ? (s2 > 0.f ? 1.f / sqrtf(s2) : 0.f) : 1.f;
      float acc = 0.f;
#pragma unroll
      for (int t = 0; t < T; ++t)
        if (lane + 32 * t < d_s) {
          const float w = fmaf(-nu, x[u][t], qv[t]);
          acc = fmaf(w, w, acc);
        }
      acc = total(acc);
      if (lane == 0 && r + u < n) buf[r + u] = gkey(acc, (int32_t)id[u]);
    }
  }
  __syncthreads();
  if (warp != 0) return;
  if (n <= 32) {
    const uint64_t v = warp_sort_lane(lane < n ? buf[lane] : KEY_MAX);
    __syncwarp();
    if (lane < n) buf[lane] = v;
    __syncwarp();
  } else if (n <= 64) {
    warp_sort_regs<2>(buf, n, k);
  } else if (n <= 256) {
    warp_sort_regs<8>(buf, n, k);
  } else {
    warp_sort(buf, n);
  }
  for (int r = lane; r < k; r += 32) {
    const bool ok = r < n;
    out_ids[q * k + r] = ok ? (int64_t)(uint32_t)(buf[r] & 0xffffffffu) : -1;
    out_dist[q * k + r] = ok ? __uint_as_float((uint32_t)(buf[r] >> 32)) : __int_as_float(0x7f800000);
  }
}

// flag (bit 1) any neighbour id outside [-1, N)
__global__ void graph_check_kernel(const int32_t *__restrict__ nbr, int64_t n, int64_t N,
                                   int *__restrict__ bad) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n && (nbr[e] < -1 || (int64_t)nbr[e] >= N)) atomicOr(bad, 1);
}

template <class T>
int gmalloc(T **p, size_t count) {
  if (cudaMalloc((void **)p, std::max<size_t>(count * sizeof(T), 16)) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return fail(ADANNS_ERR_OOM, "graph allocation failed");
  }
  return ADANNS_OK;
}

void free_graph(adanns_graph *g) {
  if (!g) return;
  cudaFree(g->xg);
  cudaFree(g->nbr);
  cudaFree(g->rows);
  cudaFree(g->dev_err);
  delete g;
}

int check_graph_shape(int64_t N, int d, int d_g, int R, int metric) {
  if (N < 2 || N > INT32_MAX || d < 1) return fail(ADANNS_ERR_ARG, "bad sizes");
  if (gran_index(d_g) < 0 || d_g > d || d_g > GR_MAXDG)
    return fail(ADANNS_ERR_DIM, "d_g must be an MR granularity <= min(d, 64)");
  if (R < 1 || R > GR_MAXR) return fail(ADANNS_ERR_ARG, "need 1 <= R <= 64");
  if (metric != ADANNS_METRIC_L2 && metric != ADANNS_METRIC_L2_PREFIXNORM)
    return fail(ADANNS_ERR_ARG, "unknown metric");
  return ADANNS_OK;
}

// a graph shell holding the rows and their d_g prefixes
int make_shell(const float *db, int64_t N, int d, int d_g, int R, int metric, cudaStream_t st,
               adanns_graph **out) {
  adanns_graph *g = new adanns_graph();
  g->N = N;
  g->d = d;
  g->d_g = d_g;
  g->dg_pad = pad16(d_g);
  g->R = R;
  g->metric = metric;
  int rc;
  if ((rc = gmalloc(&g->xg, (size_t)N * g->dg_pad)) || (rc = gmalloc(&g->nbr, (size_t)N * R)) ||
      (rc = gmalloc(&g->rows, (size_t)N * d)) || (rc = gmalloc(&g->dev_err, 1))) {
    free_graph(g);
    return rc;
  }
  if (cudaMemcpyAsync(g->rows, db, sizeof(float) * N * d, cudaMemcpyDeviceToDevice, st) !=
          cudaSuccess ||
      cudaMemsetAsync(g->dev_err, 0, sizeof(int), st) != cudaSuccess) {
    free_graph(g);
    return cuda_fail(cudaGetLastError(), "graph copy");
  }
  if ((rc = launch_gather_normalize(db, N, d, nullptr, d_g, metric, g->xg, g->dg_pad, st))) {
    free_graph(g);
    return rc;
  }
  *out = g;
  return ADANNS_OK;
}

}  // namespace
}  // namespace adn

using namespace adn;

extern "C" {

int adanns_graph_build(const float *db, int64_t N, int d, int d_g, int K, int R, float alpha,
                       int metric, void *cuda_stream, adanns_graph **out) {
  if (!out) return fail(ADANNS_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!db) return fail(ADANNS_ERR_ARG, "db is NULL");
  int rc;
  if ((rc = check_graph_shape(N, d, d_g, R, metric))) return rc;
  if (K < 1 || K > GR_MAXK || K >= N) return fail(ADANNS_ERR_ARG, "need 1 <= K <= 256, K < N");
  if (!(alpha >= 1.f) || !(alpha < 3.0e38f)) return fail(ADANNS_ERR_ARG, "need alpha >= 1");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  adanns_graph *g = nullptr;
  if ((rc = make_shell(db, N, d, d_g, R, metric, st, &g))) return rc;
  auto bail = [&](int code) {
    cudaStreamSynchronize(st);
    free_graph(g);
    return code;
  };
  {
    Scratch s(st);
    float *xpm, *kd;
    int64_t *off;
    uint64_t *keys;
    int32_t *knn, *fwd, *nfwd, *cnt, *roff, *cursor, *rev;
    int *counter;
    double *sum;
    unsigned long long *best;
    if ((rc = s.get(&xpm, (size_t)N * g->dg_pad)) || (rc = s.get(&off, 2)) ||
        (rc = s.get(&keys, (size_t)N * (K + 1))) || (rc = s.get(&knn, (size_t)N * K)) ||
        (rc = s.get(&kd, (size_t)N * K)) || (rc = s.get(&fwd, (size_t)N * R)) ||
        (rc = s.get(&nfwd, (size_t)N)) || (rc = s.get(&cnt, (size_t)N + 1)) ||
        (rc = s.get(&roff, (size_t)N + 1)) || (rc = s.get(&cursor, (size_t)N + 1)) ||
        (rc = s.get(&rev, (size_t)N * R)) || (rc = s.get(&counter, 1)) ||
        (rc = s.get(&sum, GR_MAXDG)) || (rc = s.get(&best, 1)))
      return bail(rc);
    const int64_t h_off[2] = {0, N};
    if (cudaMemcpyAsync(off, h_off, sizeof(h_off), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemsetAsync(counter, 0, sizeof(int), st) != cudaSuccess)
      return bail(cuda_fail(cudaGetLastError(), "graph build"));
    // 1. K nearest other rows: one list of all rows, a dense sweep of every row
    if ((rc = launch_prefix_major(g->xg, g->dg_pad, g->dg_pad, g->dg_pad, nullptr, nullptr, nullptr,
                                  N, xpm, st)))
      return bail(rc);
    ScanArgs a{};
    a.xpm = xpm;
    a.d_pad = g->dg_pad;
    a.dims = d_g;
    a.list_off = off;
    a.qn = g->xg;
    a.ldq = g->dg_pad;
    a.nq = (int)N;
    a.counter = counter;
    a.k = K + 1;
    a.out_keys = keys;
    if ((rc = launch_scan_f32(a, st))) return bail(rc);
    knn_drop_self_kernel<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(keys, N, K, knn, kd);
    ADN_LAUNCH("knn_drop_self_kernel");
    // 2. robust prune of every candidate list
    prune_kernel<<<(unsigned)((N + 7) / 8), 256, 0, st>>>(g->xg, g->dg_pad, d_g, knn, kd, K, N,
                                                         alpha, R, fwd, nfwd);
    ADN_LAUNCH("prune_kernel");
    // 3. offered edges grouped by target (counting sort), then the final prune
    if (cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (N + 1), st) != cudaSuccess)
      return bail(cuda_fail(cudaGetLastError(), "graph build"));
    const int64_t ne = N * R;
    offer_count_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(fwd, ne, cnt);
    ADN_LAUNCH("offer_count_kernel");
    if ((rc = launch_scan_i32(cnt, N + 1, roff, st))) return bail(rc);
    if (cudaMemcpyAsync(cursor, roff, sizeof(int32_t) * (N + 1), cudaMemcpyDeviceToDevice, st) !=
        cudaSuccess)
      return bail(cuda_fail(cudaGetLastError(), "graph build"));
    offer_fill_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(fwd, ne, R, cursor, rev);
    ADN_LAUNCH("offer_fill_kernel");
    final_prune_kernel<<<(unsigned)N, FIN_THREADS, 0, st>>>(g->xg, g->dg_pad, d_g, fwd, nfwd, roff,
                                                            rev, N, alpha, R, g->nbr, g->dev_err);
    ADN_LAUNCH("final_prune_kernel");
    // 4. entry point
    if (cudaMemsetAsync(sum, 0, sizeof(double) * GR_MAXDG, st) != cudaSuccess ||
        cudaMemsetAsync(best, 0xFF, sizeof(unsigned long long), st) != cudaSuccess)
      return bail(cuda_fail(cudaGetLastError(), "graph build"));
    row_sum_kernel<<<1024, 64, 0, st>>>(g->xg, g->dg_pad, d_g, N, sum);
    ADN_LAUNCH("row_sum_kernel");
    entry_kernel<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(g->xg, g->dg_pad, d_g, N, sum, best);
    ADN_LAUNCH("entry_kernel");
    unsigned long long hb = 0;
    int herr = 0;
    if (cudaMemcpyAsync(&hb, best, sizeof(hb), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&herr, g->dev_err, sizeof(int), cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return bail(cuda_fail(cudaGetLastError(), "graph build"));
    if (herr & ERR_HUB)
      return bail(fail(ADANNS_ERR_ARG, "a row was offered more than 4096 edges (lower R or K)"));
    g->entry = (int64_t)(hb & 0xffffffffu);
  }
  *out = g;
  return ADANNS_OK;
}

int adanns_graph_create(const float *db, int64_t N, int d, int d_g, const int32_t *graph, int R,
                        int64_t entry, int metric, void *cuda_stream, adanns_graph **out) {
  if (!out) return fail(ADANNS_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!db || !graph) return fail(ADANNS_ERR_ARG, "NULL argument");
  int rc;
  if ((rc = check_graph_shape(N, d, d_g, R, metric))) return rc;
  if (entry < 0 || entry >= N) return fail(ADANNS_ERR_ARG, "entry out of range");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  adanns_graph *g = nullptr;
  if ((rc = make_shell(db, N, d, d_g, R, metric, st, &g))) return rc;
  g->entry = entry;
  if (cudaMemcpyAsync(g->nbr, graph, sizeof(int32_t) * N * R, cudaMemcpyDeviceToDevice, st) !=
      cudaSuccess) {
    free_graph(g);
    return cuda_fail(cudaGetLastError(), "graph copy");
  }
  graph_check_kernel<<<(unsigned)((N * R + 255) / 256), 256, 0, st>>>(g->nbr, N * R, N, g->dev_err);
  int bad = 0;
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(&bad, g->dev_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    free_graph(g);
    return cuda_fail(cudaGetLastError(), "graph check");
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (bad) {
    free_graph(g);
    return fail(ADANNS_ERR_ARG, "graph holds neighbour ids outside [-1, N)");
  }
  *out = g;
  return ADANNS_OK;
}

int adanns_graph_info(const adanns_graph *g, int64_t *N, int *d, int *d_g, int *R, int64_t *entry) {
  if (!g) return fail(ADANNS_ERR_ARG, "graph is NULL");
  if (N) *N = g->N;
  if (d) *d = g->d;
  if (d_g) *d_g = g->d_g;
  if (R) *R = g->R;
  if (entry) *entry = g->entry;
  return ADANNS_OK;
}

int adanns_graph_get(const adanns_graph *g, int32_t *graph, void *cuda_stream) {
  if (!g || !graph) return fail(ADANNS_ERR_ARG, "NULL argument");
  ADN_CUDA(cudaMemcpyAsync(graph, g->nbr, sizeof(int32_t) * g->N * g->R, cudaMemcpyDeviceToDevice,
                           (cudaStream_t)cuda_stream));
  return ADANNS_OK;
}

int adanns_graph_search(const adanns_graph *g, const float *queries, int64_t B, int L, int d_s,
                        int k, int rerank_k, int64_t *out_ids, float *out_dist,
                        int64_t *out_shortlist, void *cuda_stream) {
  if (!g) return fail(ADANNS_ERR_ARG, "graph is NULL");
  if (B < 0 || B > INT32_MAX) return fail(ADANNS_ERR_ARG, "bad batch size");
  if (B > 0 && (!queries || !out_ids || !out_dist)) return fail(ADANNS_ERR_ARG, "NULL argument");
  if (gran_index(d_s) < 0 || d_s > g->d) return fail(ADANNS_ERR_DIM, "bad d_s");
  if (L < 1 || L > GR_MAXL) return fail(ADANNS_ERR_ARG, "need 1 <= L <= 512");
  if (k < 1 || rerank_k < k || rerank_k > L || rerank_k > 1024)
    return fail(ADANNS_ERR_ARG, "need 1 <= k <= rerank_k <= min(L, 1024)");
  if (B == 0) return ADANNS_OK;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int dsp = pad16(d_s);
  const int64_t Bc = std::max<int64_t>(1, std::min<int64_t>(B, scratch_budget() /
                                                                  (int64_t)(dsp * 4 + 80 +
                                                                            rerank_k * 8)));
  Scratch s(st);
  float *qg, *qs;
  int64_t *sid;
  int rc;
  if ((rc = s.get(&qg, (size_t)Bc * g->dg_pad)) || (rc = s.get(&qs, (size_t)Bc * dsp)) ||
      (rc = s.get(&sid, (size_t)Bc * rerank_k)))
    return rc;
  auto search = L <= 32    ? graph_search_kernel<1>
                : L <= 64  ? graph_search_kernel<2>
                : L <= 128 ? graph_search_kernel<4>
                : L <= 256 ? graph_search_kernel<8>
                           : graph_search_kernel<16>;
  const size_t rsm = (size_t)rerank_k * 8;
  auto rerank = d_s <= 512    ? graph_rerank_kernel<16, 2>
                : d_s <= 1024 ? graph_rerank_kernel<32, 2>
                              : graph_rerank_kernel<64, 1>;
  for (int64_t b0 = 0; b0 < B; b0 += Bc) {
    const int64_t nb = std::min(Bc, B - b0);
    {
      StageTimer t(ST_PREP, st);
      if ((rc = launch_prep_queries(queries + b0 * g->d, nb, g->d, g->d_g, d_s, g->metric, qg,
                                    g->dg_pad, qs, dsp, st)))
        return rc;
    }
    {
      StageTimer t(ST_SCAN, st);
      GsArgs a{};
      a.xg = g->xg;
      a.ldg = g->dg_pad;
      a.d_g = g->d_g;
      a.nbr = g->nbr;
      a.R = g->R;
      a.entry = g->entry;
      a.N = g->N;
      a.qg = qg;
      a.ldq = g->dg_pad;
      a.B = nb;
      a.L = L;
      a.kk = rerank_k;
      a.short_ids = out_shortlist ? out_shortlist + b0 * rerank_k : sid;
      search<<<(unsigned)((nb + GS_WARPS - 1) / GS_WARPS), GS_WARPS * 32, 0, st>>>(a);
      ADN_LAUNCH("graph_search_kernel");
    }
    {
      StageTimer t(ST_RERANK, st);
      rerank<<<(unsigned)nb, GRR_WARPS * 32, rsm, st>>>(
          out_shortlist ? out_shortlist + b0 * rerank_k : sid, rerank_k, qs, dsp, d_s, g->rows,
          g->d, g->metric, k, out_ids + b0 * k, out_dist + b0 * k);
      ADN_LAUNCH("graph_rerank_kernel");
    }
  }
  return ADANNS_OK;
}

void adanns_graph_free(adanns_graph *g) {
  if (!g) return;
  cudaDeviceSynchronize();
  free_graph(g);
}

}  // extern "C"
