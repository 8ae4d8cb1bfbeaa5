// Query-major exact rerank of the shortlists (Sec. 4.3 shortlist-rerank): a CTA
// re-scores (a part of) one query's shortlist with the exact FP32 difference-
// form distance on the d_s prefix, reading each shortlisted member's row from
// the prefix-major storage.  Nothing is sorted or counted first and only the
// shortlisted rows are read, so its cost follows the pairs alone; the
// member-major rerank (rerank_lists.cu) reads every row of every chunk that
// holds a pair, once for all queries.  Measured against it (rerank stage,
// 1.28 M rows): 10,007 queries x 40 slots at d_s 1024 1.20 -> 0.43 ms, 2,048 x 40
// at d_s 2048 0.90 -> 0.20; against one warp per query with a shared-memory sort
// (IVF-OPQ, 8,000 x 400 at d_s 384) 2.39 -> 1.10 ms.  It is bound by the gathered
// 64-byte blocks: 3.4 TB/s in query order, about 7 where the list order keeps
// rows in L2.
#include <algorithm>

#include "devutil.cuh"
#include "internal.cuh"

namespace adn {
namespace {

constexpr int RQ_THREADS = 128;

// |q - nu x|^2 of one row by GL lanes (this one is lane s): lane s takes the 16-byte
// groups s, s + GL, ... of the row in ascending order, up to eight of them requested
// before the first is used, and the lanes' sums are added by shuffles (distances
// GL / 2 .. 1 for 16 lanes, 1 .. GL / 2 for 8)
template <int GL>
__device__ __forceinline__ float row_dist(const float *x0, int nl, float nu, const float *sq, int s,
                                          int nseg, unsigned gmask) {
  const int64_t bs = (int64_t)16 * nl;  // floats between a row's blocks
  const float *row = x0 + (s >> 2) * bs + (s & 3) * 4;
  float acc = 0.f;
  for (int e0 = s; e0 < nseg; e0 += 8 * GL, row += 2 * GL * bs) {
    float4 x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + GL * u < nseg) x[u] = __ldg((const float4 *)(row + u * (GL / 4) * bs));
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (e0 + GL * u >= nseg) break;
      const float4 p = *(const float4 *)(sq + 4 * (e0 + GL * u));
      float d;
      d = fmaf(-nu, x[u].x, p.x); acc = fmaf(d, d, acc);
      d = fmaf(-nu, x[u].y, p.y); acc = fmaf(d, d, acc);
      d = fmaf(-nu, x[u].z, p.z); acc = fmaf(d, d, acc);
      d = fmaf(-nu, x[u].w, p.w); acc = fmaf(d, d, acc);
    }
  }
  if (GL == 16) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(gmask, acc, o);
  } else {
#pragma unroll
    for (int o = 1; o < GL; o <<= 1) acc += __shfl_xor_sync(gmask, acc, o);
  }
  return acc;
}

// GL lanes per candidate (row_dist): the sums of the member-major rerank (16) and
// of the IVF-OPQ rerank (8), bit for bit.  A row's four consecutive lanes read 64
// contiguous bytes.  IDS: cand holds database ids, else (list << 32 | member); -1
// is padding.  A CTA takes `per` slots of its query, 128 at a time: their addresses
// are looked up by one thread each, empty slots dropped.
template <int GL, bool IDS>
__global__ void __launch_bounds__(RQ_THREADS, 7) rerank_query_kernel(
    const int64_t *__restrict__ cand, int kr, int per, const int32_t *__restrict__ order,
    const float *__restrict__ qs, int ldq, int d_s, const float *__restrict__ xpm, int d_pad,
    const int64_t *__restrict__ list_off, const int32_t *__restrict__ list_ids,
    const int32_t *__restrict__ assign, const int32_t *__restrict__ pos,
    const float *__restrict__ mscale, uint64_t *__restrict__ keys,
    unsigned long long *__restrict__ npairs) {
  extern __shared__ __align__(16) float sq[];  // the query row
  __shared__ int64_t s_base[RQ_THREADS];       // float offset of the member's first block
  __shared__ int s_nl[RQ_THREADS], s_slot[RQ_THREADS], s_n;
  __shared__ float s_nu[RQ_THREADS];
  __shared__ uint32_t s_id[RQ_THREADS];
  const int parts = (kr + per - 1) / per;
  const int64_t qi = blockIdx.x / parts, q = order ? order[qi] : qi;
  const int tid = threadIdx.x;
  const int r0 = (int)(blockIdx.x - qi * parts) * per, r1 = min(kr, r0 + per);
  const int nseg = d_s >> 2;  // 16-byte groups (d_s is a multiple of 8)
  for (int j = tid; j < nseg; j += RQ_THREADS)
    ((float4 *)sq)[j] = ((const float4 *)(qs + q * ldq))[j];
  const int s = tid & (GL - 1), grp = tid / GL;
  const unsigned gmask = (GL == 16 ? 0xFFFFu : 0xFFu) << (threadIdx.x & 31 & ~(GL - 1));
  for (int base = r0; base < r1; base += RQ_THREADS) {
    if (tid == 0) s_n = 0;
    __syncthreads();
    if (base + tid < r1) {
      const int64_t v = cand[q * kr + base + tid];
      if (v < 0) {
        keys[q * kr + base + tid] = KEY_MAX;
      } else {
        const int l = IDS ? assign[v] : (int)(v >> 32);
        const int64_t off = list_off[l], p = IDS ? (int64_t)pos[v] : off + (v & 0xffffffffll);
        const int t = atomicAdd(&s_n, 1);
        s_base[t] = off * d_pad + (p - off) * 16;
        s_nl[t] = (int)(list_off[l + 1] - off);
        s_nu[t] = mscale ? mscale[p] : 1.f;
        s_id[t] = IDS ? (uint32_t)v : (uint32_t)list_ids[p];
        s_slot[t] = base + tid;
      }
    }
    __syncthreads();
    const int n = s_n;
    if (npairs && tid == 0) atomicAdd(npairs, (unsigned long long)n);
    for (int t = grp; t < n; t += RQ_THREADS / GL) {
      const float acc = row_dist<GL>(xpm + s_base[t], s_nl[t], s_nu[t], sq, s, nseg, gmask);
      if (s == 0) keys[q * kr + s_slot[t]] = pack_key(acc, s_id[t]);
    }
    __syncthreads();  // the slots' data are rewritten
  }
}

// Short shortlists: a CTA takes nq whole queries, at most 128 slots in all, and a warp
// sorts a query's distances in registers and writes its results, so that the slots'
// dependent lookups (list, offset, scale, id) and the barriers are paid once for nq
// queries and no second kernel reads the keys.  With a CTA per query and a kernel for
// the sort these cost more than the rows: rerank stage of 12,000 queries x 4 slots at
// d_s 64 (IVF-OPQ) 93 us, 26 here; x 64 slots 116 and 76; 50,000 x 4 at d_s 1,024 (FP8)
// 446 and 215.
template <int GL, bool IDS, int J>  // up to 32 J slots per query
__global__ void __launch_bounds__(RQ_THREADS, 7) rerank_few_kernel(
    const int64_t *__restrict__ cand, int kr, int nq, int64_t B, const int32_t *__restrict__ order,
    const float *__restrict__ qs, int ldq, int d_s, const float *__restrict__ xpm, int d_pad,
    const int64_t *__restrict__ list_off, const int32_t *__restrict__ list_ids,
    const int32_t *__restrict__ assign, const int32_t *__restrict__ pos,
    const float *__restrict__ mscale, int k, int64_t *__restrict__ out_ids,
    float *__restrict__ out_dist, unsigned long long *__restrict__ npairs) {
  extern __shared__ __align__(16) float sq[];  // [nq][d_s] the query rows
  __shared__ int64_t s_base[RQ_THREADS];       // float offset of the member's first block
  __shared__ int s_nl[RQ_THREADS], s_slot[RQ_THREADS], s_n;
  __shared__ int64_t s_qid[RQ_THREADS];
  __shared__ float s_nu[RQ_THREADS];
  __shared__ uint32_t s_id[RQ_THREADS];
  __shared__ uint64_t s_key[RQ_THREADS];
  const int64_t q0 = (int64_t)blockIdx.x * nq;
  const int tid = threadIdx.x, n_q = (int)min((int64_t)nq, B - q0);
  const int nseg = d_s >> 2;  // 16-byte groups (d_s is a multiple of 8)
  if (tid < n_q) s_qid[tid] = order ? order[q0 + tid] : q0 + tid;
  if (tid == 0) s_n = 0;
  __syncthreads();
  for (int e = tid; e < n_q * nseg; e += RQ_THREADS) {
    const int ql = e / nseg;
    cp_async16((float4 *)sq + e, (const float4 *)(qs + s_qid[ql] * ldq) + (e - ql * nseg));
  }
  cp_async_commit();
  if (tid < n_q * kr) {
    const int ql = tid / kr;
    const int64_t v = cand[s_qid[ql] * kr + (tid - ql * kr)];
    s_key[tid] = KEY_MAX;
    if (v >= 0) {
      const int l = IDS ? assign[v] : (int)(v >> 32);
      const int64_t off = list_off[l], p = IDS ? (int64_t)pos[v] : off + (v & 0xffffffffll);
      const int t = atomicAdd(&s_n, 1);
      s_base[t] = off * d_pad + (p - off) * 16;
      s_nl[t] = (int)(list_off[l + 1] - off);
      s_nu[t] = mscale ? mscale[p] : 1.f;
      s_id[t] = IDS ? (uint32_t)v : (uint32_t)list_ids[p];
      s_slot[t] = tid;
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  const int n = s_n;
  if (npairs && tid == 0) atomicAdd(npairs, (unsigned long long)n);
  const int s = tid & (GL - 1);
  const unsigned gmask = (GL == 16 ? 0xFFFFu : 0xFFu) << (threadIdx.x & 31 & ~(GL - 1));
  for (int t = tid / GL; t < n; t += RQ_THREADS / GL) {
    const float acc = row_dist<GL>(xpm + s_base[t], s_nl[t], s_nu[t], sq + s_slot[t] / kr * d_s, s,
                                   nseg, gmask);
    if (s == 0) s_key[s_slot[t]] = pack_key(acc, s_id[t]);
  }
  __syncthreads();
  const int lane = tid & 31;
  for (int ql = tid >> 5; ql < n_q; ql += RQ_THREADS / 32) {
    uint64_t key[J];  // positions J lane ..
#pragma unroll
    for (int j = 0; j < J; ++j)
      key[j] = J * lane + j < kr ? s_key[ql * kr + J * lane + j] : KEY_MAX;
    if (J == 1) key[0] = warp_sort_lane(key[0]);
    else warp_sort_lanes<J>(key);
#pragma unroll
    for (int j = 0; j < J; ++j) {
      if (J * lane + j >= k) continue;
      const int64_t o = s_qid[ql] * k + J * lane + j;
      out_ids[o] = key[j] == KEY_MAX ? -1 : (int64_t)(uint32_t)(key[j] & 0xffffffffu);
      out_dist[o] = key[j] == KEY_MAX ? __int_as_float(0x7f800000)
                                      : __uint_as_float((uint32_t)(key[j] >> 32));
    }
  }
}

}  // namespace

// Whether taking the queries in the order of their nearest list pays: the
// ordering is six small launches, and rows that all fit in L2 need none
// (2,048 queries, 40 slots, d_s 2048, 0.67 GB: 0.23 ms without, 0.24 with; 8,192
// queries, 2.7 GB: 0.79 and 0.67; 50,000 queries, 400 slots, d_s 512: 5.3 and
// 2.0).
bool rerank_order_pays(const adanns_index *idx, int64_t slots, int d_s) {
  return idx->nlist > 1 && (double)slots * d_s * 4 > 1e9;
}

// Rerank and results of short shortlists in one launch; returns 1 (nothing launched)
// for longer ones: above 32 slots, above 64 of rows of at most 128 coordinates (whose
// reads cost less than what is saved).  As many queries per CTA as leave the GPU two
// waves of CTAs, but 64 KB of member rows at most: more queries in flight at a time
// share less of their rows in L2 (150,000 x 2,048, 16,400 queries x 32 slots: rerank
// stage 1,230 us with three queries per CTA, 379 with one).
int launch_rerank_few(const int64_t *cand, int kr, int64_t B, const int32_t *order, const float *qs,
                      int ldq, int d_s, const adanns_index *idx, const float *mscale, int lanes,
                      int k, int64_t *out_ids, float *out_dist, cudaStream_t st, int64_t *npairs) {
  if (kr > 64 || (kr > 32 && d_s > 128)) return 1;
  if (B <= 0) return ADANNS_OK;
  const int64_t fill = B / ((int64_t)num_sms() * 14);
  // (their query rows 24 KB at most)
  const int cap = std::min({RQ_THREADS / kr, 65536 / (kr * d_s * 4), 24576 / (d_s * 4)});
  const int nq = (int)std::max<int64_t>(1, std::min<int64_t>(fill, cap));
  const unsigned grid = (unsigned)((B + nq - 1) / nq);
  auto kern = lanes == 16 ? (kr > 32 ? rerank_few_kernel<16, false, 2> : rerank_few_kernel<16, false, 1>)
                          : (kr > 32 ? rerank_few_kernel<8, true, 2> : rerank_few_kernel<8, true, 1>);
  kern<<<grid, RQ_THREADS, (size_t)nq * d_s * 4, st>>>(
      cand, kr, nq, B, order, qs, ldq, d_s, idx->xpm, idx->d_pad, idx->list_off, idx->list_ids,
      idx->assign, idx->pos_of_id, mscale, k, out_ids, out_dist, (unsigned long long *)npairs);
  ADN_LAUNCH("rerank_few_kernel");
  return ADANNS_OK;
}

// lanes: 16 (the low-precision tiers' rerank) or 8 (IVF-OPQ's, cand = ids)
int launch_rerank_query(const int64_t *cand, int kr, int64_t B, const int32_t *order,
                        const float *qs, int ldq, int d_s, const adanns_index *idx,
                        const float *mscale, int lanes, uint64_t *keys, cudaStream_t st,
                        int64_t *npairs) {
  if (B <= 0) return ADANNS_OK;
  // A shortlist is split over consecutive CTAs: into at least 16 slots each so
  // that few queries fill the GPU, and with an order into pieces of 256 KB of
  // rows (at least 32), so that the queries in flight are few and their common
  // rows still in L2 (50,000 queries, 400 slots, d_s 2048: 11.6 ms whole, 7.5 in
  // pieces of 32; d_s 512: 1.94 whole, 2.05 of 128, 2.75 of 32).
  const int64_t want = (int64_t)num_sms() * 8;
  int parts = (int)std::max<int64_t>(1, std::min<int64_t>((want + B - 1) / B, (kr + 15) / 16));
  if (order) {
    const int piece = std::max(32, 65536 / d_s);
    parts = std::max(parts, (kr + piece - 1) / piece);
  }
  const int per = (kr + parts - 1) / parts;
  parts = (kr + per - 1) / per;
  if (B * parts > INT32_MAX) return fail(ADANNS_ERR_ARG, "rerank slice too large");
  const unsigned grid = (unsigned)(B * parts);
  const size_t sm = (size_t)d_s * 4;
  auto go = [&](auto kern) {
    kern<<<grid, RQ_THREADS, sm, st>>>(cand, kr, per, order, qs, ldq, d_s, idx->xpm, idx->d_pad,
                                       idx->list_off, idx->list_ids, idx->assign, idx->pos_of_id,
                                       mscale, keys,
                                       (unsigned long long *)npairs);
  };
  if (lanes == 16) go(rerank_query_kernel<16, false>);
  else go(rerank_query_kernel<8, true>);
  ADN_LAUNCH("rerank_query_kernel");
  return ADANNS_OK;
}

}  // namespace adn
