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

// GL lanes per candidate: lane s takes the 16-byte groups s, s + GL, ... of the
// row in ascending order, and the lanes' sums are added by shuffles (distances
// GL / 2 .. 1 for 16 lanes, 1 .. GL / 2 for 8): the sums of the member-major
// rerank (16) and of the IVF-OPQ rerank (8), bit for bit.  Up to eight groups
// per lane are requested before the first is used: a row's four consecutive
// lanes read 64 contiguous bytes.  IDS: cand holds database ids, else (list <<
// 32 | member); -1 is padding.  A CTA takes `per` slots of its query, 128 at a
// time: their addresses are looked up by one thread each, empty slots dropped.
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
      const int64_t bs = (int64_t)16 * s_nl[t];  // floats between a row's blocks
      const float *row = xpm + s_base[t] + (s >> 2) * bs + (s & 3) * 4;
      const float nu = s_nu[t];
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
      if (s == 0) keys[q * kr + s_slot[t]] = pack_key(acc, s_id[t]);
    }
    __syncthreads();  // the slots' data are rewritten
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
