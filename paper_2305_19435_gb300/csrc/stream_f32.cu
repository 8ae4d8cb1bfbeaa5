// Exact FP32 list scan for the memory-bound regime: few queries probe each
// list (Algorithm 1 linear scan when the batch is small against nlist), so a
// member row is used by a handful of queries and the scan is a stream of the
// probed lists' d_s prefixes.
//
// Work unit = (probe tile, chunk of 128 members, group of up to 8 of the
// tile's queries): units cost about the same whatever the list's popularity,
// and are enumerated by an exclusive scan of each tile's unit count.  One
// thread per member: the member's 16-coordinate prefix blocks are read with
// 16-byte loads straight into registers (a warp covers 32 consecutive
// members, 2 KB contiguous per block in the prefix-major layout), the next
// two blocks in flight, and the distances to the group's queries accumulate
// in registers; no barrier inside the stream.  The group's rows are staged in
// shared memory: a query operand is then one broadcast read a few tens of
// cycles away, also while the member stream evicts whatever L1 holds.  The
// arithmetic is the FP32 scan's (t = q_j - s_x x_j, acc += t * t over j
// ascending), so the distances are bit-identical to it; each one is written
// as FP32 bits into the query's candidate segment, and select32_kernel then
// keeps the k best by (distance, id).
//
// A batch of queries with their own budgets (d_s, nprobe, k per query) runs
// as one launch of each kernel: masked probe slots make no pairs, a unit
// streams its member rows up to the largest d_s of its queries while each
// query stops accumulating at its own d_s (with its own per-member scale at
// that prefix), and the selection keeps the batch's largest k, of which a
// query's own k results are the prefix.  A tile's queries are grouped by
// descending d_s: the queries still active in a block are a prefix of the group,
// and the second group of a full tile streams short prefixes only.
//
// Bound by the broadcast reads and the latency of the member stream (six CTAs of
// 128 threads per SM; 256 x 3 and 64 x 12 were 10% and 5% slower, groups of 4 and
// 16 18% and 10%).  Measured on 1,281,167 x 2048 (1,024 lists), 1,021 queries with
// d_s 64 to 512, 1 to 16 probes: 1.33 ms with groups of 4 in arrival order and
// operands from L1, 0.61 ms here (4.3 TB/s of the rows); one d_s for all, 300,000 x
// 1024 (300 lists), 300 queries x 8 lists at 256: 220 -> 147 us.
#include <algorithm>

#include "devutil.cuh"
#include "internal.cuh"

namespace adn {
namespace {

constexpr int SF_THREADS = 128;  // one chunk of members per work unit
constexpr int SF_CTAS = 6;       // resident per SM
constexpr int SF_QT = 16;        // queries per probe tile
constexpr int SF_QG = 8;         // queries per work unit, as far as
constexpr int SF_SMEM = 32768;   // their staged rows fit (six CTAs: 192 KB)
constexpr int SFF_QG = 4;        // the same in dist_f32_few_kernel

struct StreamArgs {
  const float *xpm;  // prefix-major FP32 lists
  int d_pad, dims;
  const int64_t *list_off;
  const float *mscale;  // per-member scale (inverse prefix norm), or null
  const float *qn;      // prepared query rows
  int ldq;
  // per-query prefixes (or null: every query scans a.dims): d_s of each query
  // and the index's inverse prefix norms [granularity][N] with each query's
  // granularity index (null with the raw metric)
  const int32_t *qds, *qgi;
  const float *invn;
  int64_t N;
  int qg;  // queries per unit
  const int32_t *tile_list, *tile_beg, *tile_cnt;
  const int *ntiles_dev;
  const int64_t *uoff;  // first work unit of each tile (exclusive scan of its units)
  const int64_t *nunits;
  const int4 *unit;     // dist_f32_few_kernel: the units themselves
  const int32_t *pair_q, *pair_out;
  const int64_t *pbase;  // candidate segment start of each (query, probe) pair
  uint32_t *cand;
  int *counter;
};

__device__ __forceinline__ float4 ldg4(const float *p) { return __ldg((const float4 *)p); }

// units of a tile: member chunks x query groups (0 past the tile count)
__global__ void stream_units_kernel(const int32_t *__restrict__ tl, const int32_t *__restrict__ tc,
                                    const int *__restrict__ ntiles, const int64_t *__restrict__ list_off,
                                    int64_t max_tiles, int um, int qg, int64_t *__restrict__ units) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= max_tiles) return;
  int64_t u = 0;
  if (t < *ntiles) {
    const int l = tl[t];
    const int64_t npad = (list_off[l + 1] - list_off[l] + 7) & ~7ll;
    u = ((npad + um - 1) / um) * ((tc[t] + qg - 1) / qg);
  }
  units[t] = u;
}

// One block of one query: nd4 groups of 4 coordinates of a row in shared memory.
template <bool FULL>
__device__ __forceinline__ void row_step(float &acc, const float4 (&x)[4], float sc,
                                         const float4 *qb, int nd4) {
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (!FULL && s >= nd4) break;
    const float4 q = qb[s];
    float t;
    t = fmaf(-sc, x[s].x, q.x);
    acc = fmaf(t, t, acc);
    t = fmaf(-sc, x[s].y, q.y);
    acc = fmaf(t, t, acc);
    t = fmaf(-sc, x[s].z, q.z);
    acc = fmaf(t, t, acc);
    t = fmaf(-sc, x[s].w, q.w);
    acc = fmaf(t, t, acc);
  }
}

// The last tile whose first unit is <= item, found by a warp 32 tiles at a time.
__device__ __forceinline__ int unit_tile(const int64_t *__restrict__ uoff, int ntiles,
                                         int64_t item) {
  int lo = 0, n = ntiles;  // it lies in [lo, lo + n)
  while (n > 1) {
    const int step = (n + 31) >> 5, i = lo + (int)(threadIdx.x & 31) * step;
    const unsigned le = __ballot_sync(0xffffffffu, i < lo + n && uoff[i] <= item);
    const int at = 31 - __clz(le);  // uoff[lo] <= item: lane 0 always votes
    n = min(step, n - at * step);
    lo += at * step;
  }
  return lo;
}

// VAR: every query its own d_s (see the file's header).
template <bool VAR>
__global__ void __launch_bounds__(SF_THREADS, SF_CTAS) dist_f32_kernel(StreamArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  __shared__ const float *s_qp[SF_QG];  // the unit's query rows
  __shared__ const float *s_sp[SF_QG];  // each query's per-member scales (or null)
  __shared__ int64_t s_pb[SF_QG];
  __shared__ int s_ds[SF_QG];
  float4 *s_q = (float4 *)smem;  // [qg][a.dims / 4]
  const int nq4 = a.dims >> 2, qg = a.qg, tid = threadIdx.x;
  const int64_t nunits = *a.nunits;
  const int ntiles = *a.ntiles_dev;
  for (;;) {
    if (tid == 0) s_item = atomicAdd(a.counter, 1);
    __syncthreads();
    const int64_t item = s_item;
    if (item >= nunits) break;
    const int tile = unit_tile(a.uoff, ntiles, item);
    const int list = a.tile_list[tile], beg = a.tile_beg[tile], tcnt = a.tile_cnt[tile];
    const int ngrp = (tcnt + qg - 1) / qg;
    const int u = (int)(item - a.uoff[tile]);
    const int chunk = u / ngrp, g = u - chunk * ngrp;
    const int q0 = g * qg, cnt = min(qg, tcnt - q0);
    if (tid < 32) {  // rank of each of the tile's pairs by descending d_s
      const int q = tid < tcnt ? a.pair_q[beg + tid] : 0;
      const int ds = tid >= tcnt ? -1 : VAR ? a.qds[q] : a.dims;
      int r = VAR ? 0 : tid;
      if (VAR) {
#pragma unroll
        for (int i = 0; i < SF_QT; ++i) {
          const int o = __shfl_sync(0xffffffffu, ds, i);
          r += o > ds || (o == ds && i < tid);
        }
      }
      const int j = r - q0;
      if (tid < tcnt && j >= 0 && j < cnt) {
        s_qp[j] = a.qn + (int64_t)q * a.ldq;
        s_pb[j] = a.pbase[a.pair_out[beg + tid]];
        if (VAR) {
          s_ds[j] = ds;
          s_sp[j] = a.invn ? a.invn + (int64_t)a.qgi[q] * a.N : nullptr;
        }
      }
    }
    __syncthreads();
    for (int j = tid >> 5; j < cnt; j += SF_THREADS / 32) {
      const int n4 = (VAR ? s_ds[j] : a.dims) >> 2;
      for (int t = tid & 31; t < n4; t += 32) cp_async16(s_q + j * nq4 + t, s_qp[j] + 4 * t);
    }
    cp_async_commit();
    const int64_t moff = a.list_off[list];
    const int nl = (int)(a.list_off[list + 1] - moff), npad = (nl + 7) & ~7;
    const int m = chunk * SF_THREADS + tid;
    const bool live = m < nl;
    const int nblk = ((VAR ? s_ds[0] : a.dims) + 15) >> 4;
    const float *xr = a.xpm + moff * (int64_t)a.d_pad + (int64_t)m * 16;
    const int64_t bstride = (int64_t)16 * nl;
    float4 x[2][4];
    float sc[VAR ? SF_QG : 1], acc[SF_QG];
    if (!VAR) sc[0] = live && a.mscale ? __ldg(a.mscale + moff + m) : 1.f;
#pragma unroll
    for (int b = 0; b < 2; ++b)
      if (live && b < nblk) {
#pragma unroll
        for (int s = 0; s < 4; ++s) x[b][s] = ldg4(xr + b * bstride + 4 * s);
      }
#pragma unroll
    for (int j = 0; j < SF_QG; ++j) {
      if (VAR) sc[j] = live && j < cnt && s_sp[j] ? __ldg(s_sp[j] + moff + m) : 1.f;
      acc[j] = 0.f;
    }
    cp_async_wait<0>();
    __syncthreads();  // the queries are staged
    if (live) {
      int na = cnt;  // queries that reach the current block
      for (int b0 = 0; b0 < nblk; b0 += 2) {
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          if (b0 + b >= nblk) break;
          const int off = 16 * (b0 + b);
          if (VAR)
            while (s_ds[na - 1] <= off) --na;  // the first one does
          const float4 *qb = s_q + (off >> 2);
          if ((VAR ? s_ds[na - 1] : a.dims) >= off + 16) {
#pragma unroll
            for (int j = 0; j < SF_QG; ++j) {
              if (j >= na) break;
              row_step<true>(acc[j], x[b], sc[VAR ? j : 0], qb + j * nq4, 4);
            }
          } else {
#pragma unroll
            for (int j = 0; j < SF_QG; ++j) {
              if (j >= na) break;
              row_step<false>(acc[j], x[b], sc[VAR ? j : 0], qb + j * nq4, ((VAR ? s_ds[j] : a.dims) - off) >> 2);
            }
          }
          if (b0 + b + 2 < nblk) {
#pragma unroll
            for (int s = 0; s < 4; ++s) x[b][s] = ldg4(xr + (b0 + b + 2) * bstride + 4 * s);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < SF_QG; ++j)
        if (j < cnt) a.cand[s_pb[j] + m] = __float_as_uint(acc[j]);
    } else if (m < npad) {
      for (int j = 0; j < cnt; ++j) a.cand[s_pb[j] + m] = 0xFFFFFFFFu;
    }
    __syncthreads();
  }
}

// Small batches, whose members in flight would not fill the GPU one 64-byte
// block ahead (80 CTAs of one query over 16 lists): units of 64 members and
// SFF_PF blocks of a row in flight per thread, from the plan's unit table (no
// search for the tile), the unit's query rows staged in shared memory beside
// the first blocks.  The sums are those above.  One query, 16 lists of
// about 1,250 at d_s 512: 59 us with its units' two kernels before, 18 here.
constexpr int SFF_THREADS = 64, SFF_PF = 6;

template <bool VAR>
__global__ void __launch_bounds__(SFF_THREADS) dist_f32_few_kernel(StreamArgs a) {
  extern __shared__ __align__(16) float s_q[];  // [SFF_QG][dims]
  const int64_t nunits = *a.nunits;
  for (int64_t item = blockIdx.x; item < nunits; item += gridDim.x) {
    const int4 un = a.unit[item];  // (list, first pair, pairs, first member)
    const int cnt = un.z, m = un.w + threadIdx.x, nq4 = a.dims >> 2;
    const float *sp[SFF_QG];
    int64_t pb[SFF_QG];
    int ds[SFF_QG], dmax = VAR ? 0 : a.dims;
    __syncthreads();  // the previous unit's queries are no longer read
#pragma unroll
    for (int j = 0; j < SFF_QG; ++j) {
      const int pr = un.y + min(j, cnt - 1), q = a.pair_q[pr];
      if (j < cnt) {
        const float4 *src = (const float4 *)(a.qn + (int64_t)q * a.ldq);
        for (int t = threadIdx.x; t < nq4; t += SFF_THREADS)
          cp_async16(s_q + 4 * (j * nq4 + t), src + t);
      }
      pb[j] = a.pbase[a.pair_out[pr]];
      ds[j] = VAR ? a.qds[q] : a.dims;
      sp[j] = VAR ? (a.invn ? a.invn + (int64_t)a.qgi[q] * a.N : nullptr) : a.mscale;
      if (VAR) dmax = max(dmax, ds[j]);
    }
    cp_async_commit();
    const int64_t moff = a.list_off[un.x];
    const int nl = (int)(a.list_off[un.x + 1] - moff), npad = (nl + 7) & ~7;
    const int nblk = (dmax + 15) >> 4;
    const float *xr = a.xpm + moff * (int64_t)a.d_pad + (int64_t)m * 16;
    const int64_t bstride = (int64_t)16 * nl;
    float4 x[SFF_PF][4];
#pragma unroll
    for (int b = 0; b < SFF_PF; ++b)
      if (m < nl && b < nblk) {
#pragma unroll
        for (int s = 0; s < 4; ++s) x[b][s] = ldg4(xr + b * bstride + 4 * s);
      }
    float sc[SFF_QG], acc[SFF_QG];
#pragma unroll
    for (int j = 0; j < SFF_QG; ++j) {
      sc[j] = m < nl && sp[j] ? __ldg(sp[j] + moff + m) : 1.f;
      acc[j] = 0.f;
    }
    cp_async_wait<0>();
    __syncthreads();  // the queries are staged
    if (m < nl) {
      for (int b0 = 0; b0 < nblk; b0 += SFF_PF) {
#pragma unroll
        for (int b = 0; b < SFF_PF; ++b) {
          if (b0 + b >= nblk) break;
          const int off = 16 * (b0 + b);
#pragma unroll
          for (int j = 0; j < SFF_QG; ++j) {
            if (j >= cnt) break;
            const int nd4 = (ds[j] - off) >> 2;
            const float4 *qb = (const float4 *)s_q + j * nq4 + (off >> 2);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
              if (s >= nd4) break;
              const float4 q = qb[s];
              float t;
              t = fmaf(-sc[j], x[b][s].x, q.x);
              acc[j] = fmaf(t, t, acc[j]);
              t = fmaf(-sc[j], x[b][s].y, q.y);
              acc[j] = fmaf(t, t, acc[j]);
              t = fmaf(-sc[j], x[b][s].z, q.z);
              acc[j] = fmaf(t, t, acc[j]);
              t = fmaf(-sc[j], x[b][s].w, q.w);
              acc[j] = fmaf(t, t, acc[j]);
            }
          }
          if (b0 + b + SFF_PF < nblk) {
#pragma unroll
            for (int s = 0; s < 4; ++s) x[b][s] = ldg4(xr + (b0 + b + SFF_PF) * bstride + 4 * s);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < SFF_QG; ++j)
        if (j < cnt) a.cand[pb[j] + m] = __float_as_uint(acc[j]);
    } else if (m < npad) {
#pragma unroll
      for (int j = 0; j < SFF_QG; ++j)
        if (j < cnt) a.cand[pb[j] + m] = 0xFFFFFFFFu;
    }
  }
}

}  // namespace

static int64_t stream_per_query(const adanns_index *idx, int d_c, int d_s, int nprobe, int k) {
  return max_probe_members(idx, nprobe) * 4 + (int64_t)(pad16(d_c) + pad16(d_s)) * 4 +
         (int64_t)k * 8 + (int64_t)nprobe * 40 + 16;
}

// few members in all: small units from a table (the whole batch is then one slice),
// a unit per 64 members of each probed list and group of queries at most; 0: not so
static int64_t few_units(const adanns_index *idx, int64_t B, int64_t Bc, int nprobe) {
  const int64_t n = B * nprobe * (((int64_t)idx->max_list + 7 + SFF_THREADS) / SFF_THREADS);
  const bool few = Bc >= B && probe_plan_small(B * nprobe, idx->nlist) && n <= 1 << 20 &&
                   (double)B * nprobe * idx->N / idx->nlist <= (double)num_sms() * 1024;
  return few ? n : 0;
}

int64_t stream_scratch_bytes(const adanns_index *idx, int64_t B, int d_c, int d_s, int nprobe,
                             int k) {
  const int64_t per_q = stream_per_query(idx, d_c, d_s, nprobe, k);
  const int64_t Bc = std::max<int64_t>(1, std::min<int64_t>(B, scratch_budget() / per_q));
  return Bc * (per_q + coarse_scratch_per_query(idx, d_c)) + (int64_t)idx->nlist * 64 +
         16 * few_units(idx, B, Bc, nprobe) + Scratch::SLACK;
}

// Where the streaming scan is taken (ADANNS_OPT_FP32_STREAM = 0 keeps the
// shared-memory tiled scan everywhere).  Up to 16 queries per probed list it
// always is.  Above, per (query, member) in picoseconds, it spends 6 + 0.122 per
// coordinate (0.166 beyond 1,024, where fewer staged rows fit) and the tiled scan
// 9 + 0.27 k + 0.104 per coordinate, more while its tiles are not full: tiled
// against streaming, 400,000 rows in 400 lists, 500 queries per list, k 10: d_s 64
// 3.65 / 2.85 ms, 512 12.9 / 13.8, 1024 23.5 / 26.3; k 100: 8.4 / 3.0, 17.6 / 13.9,
// 28.0 / 26.5; 100,000 x 2048, k 10, 32 and 64 queries per list: 1.39 / 1.19 and
// 2.05 / 2.23.  At k = 1, where the tiled scan keeps no buffer and the selection's CTA
// per query is most of the call, by their estimated times (f32_cost): 200,000 rows in
// 256 lists, d_s 16, 2 probes, 90 queries per list 197 / 323 us; 640,000 in 700, d_s 64, 1
// probe, 47 per list 529 / 759; 60,000 in 60, d_s 64, 4 probes, 68 per list 109 / 100.
// A batch with a d_s per query goes by their mean (6,000 queries with
// d_s 64 to 2048, 20,000 rows in 16 lists, k 100: 9.98 / 9.25; 2,000 with 64 to 512, 1
// M rows, k 10: 2.45 / 1.08).  The distances must fit the scratch at once, or in slices of at
// least 64 queries per list, which still share their rows.
bool fp32_stream_enabled(const adanns_index *idx, int64_t B, int64_t pairs, int d_c, int d_s,
                         int nprobe, int k, int mean_ds) {
  if (!option(ADANNS_OPT_FP32_STREAM) || nprobe > 256) return false;
  const double qpl = (double)pairs / idx->nlist;
  const int t = mean_ds ? 0 : tuned_scan_tq(k, d_s, qpl);
  if (t != 0) return t == TUNE_STREAM;
  if (qpl <= 16.0) return true;
  const int ds = mean_ds ? mean_ds : d_s;
  if (k == 1 && !mean_ds) {
    if (f32_cost(F32_TILED, idx, B, pairs, d_s, k) < f32_cost(F32_STREAM, idx, B, pairs, d_s, k))
      return false;
  } else if (qpl * ds > 65536.0 && k < (ds <= 1024 ? (ds - 256) / 14 : ds / 4)) {
    return false;
  }
  const int64_t fit = scratch_budget() / stream_per_query(idx, d_c, d_s, nprobe, k);
  return fit >= B || (double)fit * pairs / B >= 64.0 * idx->nlist;
}

int search_f32_stream(const adanns_index *idx, const float *queries, int64_t B, int d_c, int d_s,
                      int nprobe, int k, int64_t *out_ids, float *out_dist, int32_t *out_probes,
                      cudaStream_t st, const QueryBudgets *qb) {
  const int nlist = idx->nlist;
  const int dcp = pad16(d_c), dsp = pad16(d_s);
  const int64_t seg_q = max_probe_members(idx, nprobe);
  const int64_t per_q = stream_per_query(idx, d_c, d_s, nprobe, k);
  const int64_t Bc = std::max<int64_t>(1, std::min<int64_t>(B, scratch_budget() / per_q));
  const int64_t max_tiles = (Bc * nprobe + SF_QT - 1) / SF_QT + nlist;
  const int64_t max_units = few_units(idx, B, Bc, nprobe);
  const bool few = max_units > 0;
  const bool var = qb && qb->ds;
  const int um = few ? SFF_THREADS : SF_THREADS;
  const int qg = few ? SFF_QG : std::max(1, std::min(SF_QG, SF_SMEM / (d_s * 4)));
  Scratch s(st);
  float *qc, *qs;
  uint64_t *ckeys;
  int4 *unit = nullptr;
  uint32_t *cand;
  int64_t *qtot, *qbase, *pbase, *units, *uoff, *nunits;
  int32_t *lcnt, *lbeg, *lfill, *tbeg, *pair_q, *pair_out, *tl, *tb, *tc;
  int *ntiles, *counter;
  int rc;
  if ((rc = s.get(&qc, (size_t)Bc * dcp)) || (rc = s.get(&qs, (size_t)Bc * dsp)) ||
      (rc = s.get(&ckeys, (size_t)Bc * nprobe)) || (rc = s.get(&cand, (size_t)(Bc * seg_q))) ||
      (rc = s.get(&qtot, (size_t)Bc)) ||
      (rc = s.get(&qbase, (size_t)Bc)) || (rc = s.get(&pbase, (size_t)Bc * nprobe)) ||
      (rc = s.get(&lcnt, nlist)) || (rc = s.get(&lbeg, nlist)) || (rc = s.get(&lfill, nlist)) ||
      (rc = s.get(&tbeg, nlist)) || (rc = s.get(&pair_q, (size_t)Bc * nprobe)) ||
      (rc = s.get(&pair_out, (size_t)Bc * nprobe)) || (rc = s.get(&tl, max_tiles)) ||
      (rc = s.get(&tb, max_tiles)) || (rc = s.get(&tc, max_tiles)) || (rc = s.get(&ntiles, 1)) ||
      (rc = s.get(&counter, 2)) || (rc = s.get(&units, max_tiles)) ||
      (rc = s.get(&uoff, max_tiles)) || (rc = s.get(&nunits, 1)) ||
      (few && (rc = s.get(&unit, (size_t)max_units))))
    return rc;
  const float *mscale = idx->metric == ADANNS_METRIC_L2_PREFIXNORM
                            ? idx->invn + (int64_t)gran_index(d_s) * idx->N
                            : nullptr;
  for (int64_t b0 = 0; b0 < B; b0 += Bc) {
    const int64_t nb = std::min(Bc, B - b0);
    const QueryBudgets bq = qb ? qb->at(b0) : QueryBudgets{};
    {
      StageTimer t(ST_PREP, st);
      if ((rc = launch_prep_queries(queries + b0 * idx->d, nb, idx->d, d_c, d_s, idx->metric, qc,
                                    dcp, qs, dsp, st, bq.ds)))
        return rc;
    }
    {
      StageTimer t(ST_COARSE, st);
      if ((rc = run_coarse(idx, qc, dcp, nb, d_c, nprobe, ckeys, counter, st))) return rc;
      if ((rc = launch_mask_probes(ckeys, nb, nprobe, bq.np, st))) return rc;
    }
    ProbePlan plan;
    {
      StageTimer t(ST_INVERT, st);
      plan.zero = counter + 1;
      plan.nzero = 1;
      plan.list_off = idx->list_off;
      plan.qbase = qbase;
      plan.pbase = pbase;
      plan.unit_members = um;
      plan.unit_queries = qg;
      plan.uoff = uoff;
      plan.nunits = nunits;
      plan.unit = unit;
      if ((rc = launch_invert_probes(ckeys, nb, nprobe, nlist, SF_QT, lcnt, lbeg, lfill, tbeg,
                                     pair_q, pair_out, tl, tb, tc, ntiles,
                                     out_probes ? out_probes + b0 * nprobe : nullptr, st, &plan)))
        return rc;
      if (!plan.planned && (rc = launch_cand_segments(ckeys, nb, nprobe, idx->list_off, qtot,
                                                      qbase, pbase, st)))
        return rc;
    }
    {
      StageTimer t(ST_SCAN, st);
      if (!plan.planned) {
        stream_units_kernel<<<(unsigned)((max_tiles + 255) / 256), 256, 0, st>>>(
            tl, tc, ntiles, idx->list_off, max_tiles, um, qg, units);
        ADN_LAUNCH("stream_units_kernel");
        if ((rc = launch_scan64(units, max_tiles, uoff, nunits, st))) return rc;
      }
      StreamArgs a{};
      a.xpm = idx->xpm;
      a.d_pad = idx->d_pad;
      a.dims = d_s;
      a.list_off = idx->list_off;
      a.mscale = mscale;
      a.qn = qs;
      a.ldq = dsp;
      a.tile_list = tl;
      a.tile_beg = tb;
      a.tile_cnt = tc;
      a.ntiles_dev = ntiles;
      a.uoff = uoff;
      a.nunits = nunits;
      a.unit = unit;
      a.pair_q = pair_q;
      a.pair_out = pair_out;
      a.pbase = pbase;
      a.cand = cand;
      a.counter = counter + 1;
      a.qds = bq.ds;
      a.qgi = bq.gi;
      a.invn = idx->metric == ADANNS_METRIC_L2_PREFIXNORM ? idx->invn : nullptr;
      a.N = idx->N;
      a.qg = qg;
      if (few) {
        // about as many CTAs as units if no query shared a list
        const int64_t est = nb * nprobe * (idx->N / nlist / SFF_THREADS + 1);
        const unsigned grid =
            (unsigned)std::min<int64_t>(std::min(max_units, est), (int64_t)num_sms() * 16);
        const size_t sm = (size_t)SFF_QG * d_s * 4;
        auto kern = bq.ds ? dist_f32_few_kernel<true> : dist_f32_few_kernel<false>;
        ADN_CUDA(ensure_smem((const void *)kern, sm));
        kern<<<grid, SFF_THREADS, sm, st>>>(a);
        ADN_LAUNCH("dist_f32_few_kernel");
      } else {
        auto kern = var ? dist_f32_kernel<true> : dist_f32_kernel<false>;
        const size_t sm = (size_t)qg * d_s * 4;
        ADN_CUDA(ensure_smem((const void *)kern, sm));
        int per_sm = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, um, sm) !=
                cudaSuccess ||
            per_sm < 1) {
          cudaGetLastError();
          per_sm = 1;
        }
        kern<<<num_sms() * per_sm, um, sm, st>>>(a);
        ADN_LAUNCH("dist_f32_kernel");
      }
    }
    {
      StageTimer t(ST_MERGE, st);
      if ((rc = launch_select32_results(cand, ckeys, nprobe, qbase, idx->list_off, idx->list_ids,
                                        nb, k, bq.k, out_ids + b0 * k, out_dist + b0 * k, st)))
        return rc;
    }
  }
  return ADANNS_OK;
}

}  // namespace adn
