// Per-query selection of the kk smallest 32-bit keys over the query's
// candidate segments (the ADC distances of the probed lists, one FP32
// distance per member, whose bits order like the distances).  One CTA per
// query:
//  1. a sample of up to 8,192 keys (2,048 evenly spaced 16-byte runs) gives a
//     threshold T with about (kk + 4,096) / 2 smaller keys (a histogram of the
//     sample);
//  2. one pass compacts every key < T, with its position, into a shared buffer;
//  3. if the buffer holds between kk and S32_BUF keys, an exact radix select
//     (four 8-bit digits) on the buffer fixes the cut, otherwise the same
//     select runs over the whole region.
// Ties at the cut go to the smallest database ids, so the kk keys are the kk
// smallest (distance, id) pairs, as a sort of the packed keys would give.
#include "devutil.cuh"
#include "internal.cuh"

namespace adn {
namespace {

constexpr int S32_SAMPLE = 8192;  // keys sampled (2,048 runs of 4)
constexpr int S32_BUF = 4096;     // keys compacted below the threshold (same shared space)
constexpr int S32_TIE = 512;
constexpr int S32_UNROLL = 4;     // 16-byte loads in flight per thread in the compaction
constexpr int S32_MAXP = 256;  // probed lists per query

struct S32State {
  int hist[256];
  int sh[2], lt, eq;
  uint64_t ties[S32_TIE];  // (id << 32 | index) of the keys equal to the cut
};

// the kth smallest (1-based) of n keys; below = keys below it, neq = keys equal
template <int NT, class KeyF>
__device__ uint32_t radix_kth32(int n, int kth, KeyF key, S32State &st, int &below, int &neq) {
  return block_radix_kth<NT, 4>(n, kth, key, st.hist, st.sh, &below, &neq);
}

// the kk smallest of n keys in (key, id) order: key(i), database id id(i)
// (distinct over the n keys, below 0xFFFFFFFF), output value val(i)
// (key << 32 | id), written to o[0, kk) in no particular order.  The keys equal
// to the cut go by ascending id: a warp sort when at most S32_TIE of them
// tie, else a second radix select on their ids.
template <int NT, class KeyF, class IdF, class ValF>
__device__ void select_into(int n, int kk, KeyF key, IdF id, ValF val, uint64_t *o, S32State &st) {
  const int tid = threadIdx.x;
  int below, neq;
  const uint32_t T = radix_kth32<NT>(n, kk, key, st, below, neq);
  const int need_eq = kk - below;
  if (tid == 0) st.lt = st.eq = 0;
  __syncthreads();
  for (int i = tid; i < n; i += NT) {
    const uint32_t k = key(i);
    if (k < T) {
      o[atomicAdd(&st.lt, 1)] = val(i);
    } else if (k == T && neq <= S32_TIE) {
      const int p = atomicAdd(&st.eq, 1);
      if (p < S32_TIE) st.ties[p] = ((uint64_t)id(i) << 32) | (uint32_t)i;
    }
  }
  __syncthreads();
  if (neq <= S32_TIE) {
    if (tid < 32) {
      warp_sort(st.ties, neq);
      for (int j = tid; j < need_eq; j += 32) o[below + j] = val((int)(uint32_t)st.ties[j]);
    }
  } else {
    int b2, n2;
    const uint32_t idT = radix_kth32<NT>(
        n, need_eq, [&](int i) -> uint32_t { return key(i) == T ? id(i) : 0xFFFFFFFFu; }, st, b2,
        n2);
    if (tid == 0) st.eq = 0;
    __syncthreads();
    for (int i = tid; i < n; i += NT)
      if (key(i) == T && id(i) <= idT) {
        const int p = atomicAdd(&st.eq, 1);
        if (p < need_eq) o[below + p] = val(i);
      }
  }
  __syncthreads();
}

// n distinct keys v into sorted order, the kk smallest of them in o: every key's
// rank by comparison with all (no barrier per step, unlike a block-wide sorting
// network, whose 55 steps for 1,024 keys take 14 us)
template <int NT>
__device__ __forceinline__ void rank_sort(const uint64_t *v, int n, int kk, uint64_t *o) {
  for (int i = threadIdx.x; i < n; i += NT) {
    const uint64_t key = v[i];
    int r = 0;
#pragma unroll 4
    for (int j = 0; j < n; ++j) r += v[j] < key ? 1 : 0;
    if (r < kk) o[r] = key;
  }
  __syncthreads();
}

// the kk smallest keys of query blockIdx.x into o[0, kk), by NT threads.
// SORTED: o is shared and ends up sorted (kk <= S32_SORT); the threshold then
// aims at little more than kk keys.
constexpr int S32_SORT = 1024;

template <int NT, bool SORTED>
__device__ __forceinline__ void select32_query(const uint32_t *cand, const uint64_t *ckeys,
                                               int nprobe, const int64_t *qbase,
                                               const int64_t *list_off, const int32_t *list_ids,
                                               int kk, uint64_t *o) {
  __shared__ S32State st;
  // the sample, then (once the threshold is known) the compacted keys and positions
  __shared__ __align__(16) uint32_t space[S32_SAMPLE];
  uint32_t *samp = space, *bkey = space, *bidx = space + S32_BUF;
  // up to S32_SORT keys to be sorted, in the part of the buffer that as many
  // compacted keys leave free
  uint64_t *sv = (uint64_t *)(space + S32_SORT);
  __shared__ int s_n, s_total;
  __shared__ uint32_t s_lo, s_hi;
  __shared__ int64_t s_off[S32_MAXP];
  __shared__ int s_nl[S32_MAXP], s_pst[S32_MAXP + 1];
  const int64_t q = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31;
  for (int s = tid; s < nprobe; s += NT) {
    const int l = probe_list(ckeys[q * nprobe + s]);
    s_off[s] = l >= 0 ? list_off[l] : 0;
    s_nl[s] = l >= 0 ? (int)(list_off[l + 1] - list_off[l]) : 0;
  }
  for (int i = tid; i < 256; i += NT) st.hist[i] = 0;
  if (tid == 0) {
    s_n = 0;
    s_lo = 0xFFFFFFFFu;
    s_hi = 0;
  }
  __syncthreads();
  if (tid < 32) {  // padded starts and the members in all: 8 slots per lane
    int pad[8], sum = 0, mem = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int sl = lane * 8 + j, nl = sl < nprobe ? s_nl[sl] : 0;
      pad[j] = (nl + 7) & ~7;
      sum += pad[j];
      mem += nl;
    }
    int inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += y;
      mem += __shfl_xor_sync(0xffffffffu, mem, d);
    }
    int run = inc - sum;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (lane * 8 + j <= nprobe) s_pst[lane * 8 + j] = run;
      run += pad[j];
    }
    if (lane == 31 && nprobe == 256) s_pst[256] = run;
    if (lane == 0) s_total = mem;
  }
  __syncthreads();
  const int ptotal = s_pst[nprobe], total = s_total;
  const uint32_t *src = cand + qbase[q];
  // value of candidate position i: (key << 32 | database id), KEY_MAX for padding
  auto val_at = [&](int i) -> uint64_t {
    int lo = 0, hi = nprobe - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_pst[mid] <= i) lo = mid; else hi = mid - 1;
    }
    const int m = i - s_pst[lo];
    return m < s_nl[lo] ? (((uint64_t)src[i] << 32) | (uint32_t)list_ids[s_off[lo] + m]) : KEY_MAX;
  };
  auto id_at = [&](int i) -> uint32_t { return (uint32_t)(val_at(i) & 0xffffffffu); };
  auto sort_out = [&]() {
    for (int i = tid; i < kk; i += NT) sv[i] = o[i];
    __syncthreads();
    rank_sort<NT>(sv, kk, kk, o);
  };
  if (total <= kk) {
    uint64_t *d = SORTED ? sv : o;
    for (int s = 0; s < nprobe; ++s) {
      int p0 = 0;
      for (int s2 = 0; s2 < s; ++s2) p0 += s_nl[s2];
      for (int m = tid; m < s_nl[s]; m += NT)
        d[p0 + m] = ((uint64_t)src[s_pst[s] + m] << 32) | (uint32_t)list_ids[s_off[s] + m];
    }
    for (int r = total + tid; r < kk; r += NT) o[r] = KEY_MAX;
    __syncthreads();
    if (SORTED) rank_sort<NT>(sv, total, total, o);
    return;
  }
  if (SORTED || ptotal > 2 * S32_BUF) {
    // 1. threshold from a sample of up to S32_SAMPLE / 4 evenly spaced 16-byte
    //    runs, aimed at (kk + S32_BUF) / 2 keys below it (at kk, and four standard
    //    deviations of the sample's rank, when they are to be sorted): the end
    //    of the bucket, of 256 equal ones between the
    //    sample's extremes, that holds the wanted rank.  (Equal buckets spread
    //    the counts over the histogram; the keys' leading bits are nearly all
    //    alike and would queue at a few of its entries.)
    const uint4 *g = (const uint4 *)src;
    const int nvec = ptotal >> 2;
    const int nrun = min(S32_SAMPLE / 4, nvec), ns = 4 * nrun;
    const uint64_t step = ((uint64_t)nvec << 20) / (uint64_t)nrun;  // 2^-20 units
    uint32_t lo = 0xFFFFFFFFu, hi = 0;
    for (int j = tid; j < nrun; j += NT) {
      const uint4 v = g[(int)(((uint64_t)j * step) >> 20)];
      *(uint4 *)&samp[4 * j] = v;
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (w[e] != 0xFFFFFFFFu) {
          lo = min(lo, w[e]);
          hi = max(hi, w[e]);
        }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      atomicMin(&s_lo, lo);
      atomicMax(&s_hi, hi);
    }
    __syncthreads();
    lo = s_lo;
    hi = max(s_hi, lo);
    int shift = 0;
    while (((hi - lo) >> shift) > 255u) ++shift;
    for (int i = tid; i < ns; i += NT) {
      const uint32_t kv = samp[i];
      atomicAdd(&st.hist[kv == 0xFFFFFFFFu ? 255u : min((kv - lo) >> shift, 255u)], 1);
    }
    __syncthreads();
    int r;
    if (SORTED) {
      const float rf = (float)kk * ns / ptotal;
      r = ns < ptotal ? (int)(rf + 4.f * sqrtf(rf)) + 4 : kk - 1;
    } else {
      r = (int)(0.5 * (kk + S32_BUF) * ns / ptotal);
    }
    r = max(0, min(r, ns - 1));
    if (tid < 32) warp_find_bucket(st.hist, 0, r + 1, &st.sh[0], &st.sh[1]);
    __syncthreads();
    const uint64_t end = (uint64_t)lo + ((uint64_t)(st.sh[0] + 1) << shift);
    const uint32_t T = (uint32_t)min(end, (uint64_t)0xFFFFFFFFu);  // keys strictly below T survive
    __syncthreads();  // the sample's space is reused by the compaction
    // 2. compact the keys below T: S32_UNROLL 16-byte loads in flight per
    //    thread; a warp votes once per load and skips the word-by-word
    //    ranking when none of its 128 keys survives (the common case)
    for (int c0 = 0; c0 < nvec; c0 += NT * S32_UNROLL) {
      uint4 v[S32_UNROLL];
#pragma unroll
      for (int u = 0; u < S32_UNROLL; ++u) {
        const int c = c0 + u * NT + tid;
        v[u] = c < nvec ? g[c] : make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
      }
#pragma unroll
      for (int u = 0; u < S32_UNROLL; ++u) {
        const int c = c0 + u * NT + tid;
        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
        const uint32_t mn = min(min(w[0], w[1]), min(w[2], w[3]));
        if (!__any_sync(0xffffffffu, mn < T)) continue;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const bool take = w[e] < T;
          const unsigned m = __ballot_sync(0xffffffffu, take);
          int base = 0;
          if (lane == 0 && m) base = atomicAdd(&s_n, __popc(m));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (take) {
            const int p = base + __popc(m & lanemask_lt());
            if (p < S32_BUF) {
              bkey[p] = w[e];
              bidx[p] = (uint32_t)(4 * c + e);
            }
          }
        }
      }
    }
    __syncthreads();
    const int n = s_n;
    if (SORTED && n >= kk && n <= S32_SORT) {
      for (int i = tid; i < n; i += NT) sv[i] = val_at((int)bidx[i]);
      __syncthreads();
      rank_sort<NT>(sv, n, kk, o);
      return;
    }
    if (n >= kk && n <= S32_BUF) {
      select_into<NT>(n, kk, [&](int i) -> uint32_t { return bkey[i]; },
                      [&](int i) -> uint32_t { return id_at((int)bidx[i]); },
                      [&](int i) -> uint64_t { return val_at((int)bidx[i]); }, o, st);
      if (SORTED) sort_out();
      return;
    }
  }
  // 3. exact select over the whole region (index = candidate position)
  select_into<NT>(ptotal, kk, [&](int i) -> uint32_t { return src[i]; }, id_at,
                  [&](int i) -> uint64_t { return val_at(i); }, o, st);
  if (SORTED) sort_out();
}

constexpr int S32_NT = 256, S32_NT_FEW = 1024;

__global__ void __launch_bounds__(S32_NT) select32_kernel(
    const uint32_t *__restrict__ cand, const uint64_t *__restrict__ ckeys, int nprobe,
    const int64_t *__restrict__ qbase, const int64_t *__restrict__ list_off,
    const int32_t *__restrict__ list_ids, int kk, uint64_t *__restrict__ out,
    const int32_t *__restrict__ only) {
  if (only && only[blockIdx.x] >= 0) return;
  select32_query<S32_NT, false>(cand, ckeys, nprobe, qbase, list_off, list_ids, kk,
                                out + (int64_t)blockIdx.x * kk);
}

// selection, sort and results in one launch; few queries get 1,024 threads each
// (one query over 22,000 candidates, k 100: 31 + 6 us in two launches, 13 here;
// 200 queries over 800, k 10: 9 + 6 and 7)
template <int NT>
__global__ void __launch_bounds__(NT) select32_results_kernel(
    const uint32_t *__restrict__ cand, const uint64_t *__restrict__ ckeys, int nprobe,
    const int64_t *__restrict__ qbase, const int64_t *__restrict__ list_off,
    const int32_t *__restrict__ list_ids, int k, const int32_t *__restrict__ kq,
    int64_t *__restrict__ out_ids, float *__restrict__ out_dist) {
  extern __shared__ __align__(16) uint64_t o[];  // [k]
  select32_query<NT, true>(cand, ckeys, nprobe, qbase, list_off, list_ids, k, o);
  const int64_t q = blockIdx.x;
  const int kn = kq ? min(k, kq[q]) : k;
  for (int r = threadIdx.x; r < k; r += NT) {
    const uint64_t key = r < kn ? o[r] : KEY_MAX;
    out_ids[q * k + r] = key == KEY_MAX ? -1 : (int64_t)(uint32_t)(key & 0xffffffffu);
    out_dist[q * k + r] = key == KEY_MAX ? __int_as_float(0x7f800000)
                                         : __uint_as_float((uint32_t)(key >> 32));
  }
}

}  // namespace

namespace {
__global__ void keys_to_ids_kernel(const uint64_t *__restrict__ keys, int64_t n,
                                   int64_t *__restrict__ ids) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) ids[i] = keys[i] == KEY_MAX ? -1 : (int64_t)(uint32_t)(keys[i] & 0xffffffffu);
}
}  // namespace

int launch_keys_to_ids(const uint64_t *keys, int64_t n, int64_t *ids, cudaStream_t st) {
  if (n <= 0) return ADANNS_OK;
  keys_to_ids_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(keys, n, ids);
  ADN_LAUNCH("keys_to_ids_kernel");
  return ADANNS_OK;
}

int launch_select32(const uint32_t *cand, const uint64_t *ckeys, int nprobe, const int64_t *qbase,
                    const int64_t *list_off, const int32_t *list_ids, int64_t B, int kk,
                    uint64_t *out, cudaStream_t st, const int32_t *only) {
  if (nprobe > S32_MAXP) return fail(ADANNS_ERR_ARG, "select32: nprobe above 256");
  if (B <= 0) return ADANNS_OK;
  select32_kernel<<<(unsigned)B, S32_NT, 0, st>>>(cand, ckeys, nprobe, qbase, list_off,
                                                       list_ids, kk, out, only);
  ADN_LAUNCH("select32_kernel");
  return ADANNS_OK;
}

int launch_select32_results(const uint32_t *cand, const uint64_t *ckeys, int nprobe,
                            const int64_t *qbase, const int64_t *list_off, const int32_t *list_ids,
                            int64_t B, int k, const int32_t *kq, int64_t *out_ids, float *out_dist,
                            cudaStream_t st) {
  if (nprobe > S32_MAXP) return fail(ADANNS_ERR_ARG, "select32: nprobe above 256");
  if (B <= 0) return ADANNS_OK;
  if (k > S32_SORT) return fail(ADANNS_ERR_ARG, "select32: k above 1024");
  const size_t sm = (size_t)k * 8;
  auto go = [&](auto kern, int nt) -> int {
    ADN_CUDA(ensure_smem((const void *)kern, sm));
    kern<<<(unsigned)B, nt, sm, st>>>(cand, ckeys, nprobe, qbase, list_off, list_ids, k, kq,
                                      out_ids, out_dist);
    ADN_LAUNCH("select32_results_kernel");
    return ADANNS_OK;
  };
  return B <= num_sms() ? go(select32_results_kernel<S32_NT_FEW>, S32_NT_FEW)
                        : go(select32_results_kernel<S32_NT>, S32_NT);
}

}  // namespace adn
