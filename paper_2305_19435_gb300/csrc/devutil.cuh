// Device helpers: async copies, warp sorting of packed (distance, id) keys.
#pragma once
#include <stdint.h>

namespace adn {

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// L2 eviction-priority policies (per-access hints; no device state changes)
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void cp_async16_hint(void *smem, const void *gmem, uint64_t pol) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem),
               "l"(pol)
               : "memory");
}
__device__ __forceinline__ float4 ldg_f4_hint(const float4 *p, uint64_t pol) {
  float4 v;
  asm volatile("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(pol));
  return v;
}

// Two FP32 operations per instruction (each half rounds as the scalar one)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// One full warp: the smallest bucket b of a 256-bucket histogram h with
// base + h[0] + ... + h[b] >= target, and the count below it
// (base + h[0] + ... + h[b-1]).  Needs target <= base + sum(h).
__device__ __forceinline__ void warp_find_bucket(const int *h, int base, int target, int *b_out,
                                                 int *below_out) {
  const int lane = threadIdx.x & 31;
  int v[8], sum = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    v[j] = h[lane * 8 + j];
    sum += v[j];
  }
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  const unsigned m = __ballot_sync(0xffffffffu, base + inc >= target);
  const int L = m ? __ffs(m) - 1 : 31;
  if (lane == L) {
    // first bucket j of the lane's 8 whose running count reaches target
    int c = base + inc - sum, jb = 7;
    bool found = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (!found) {
        if (j == 7 || c + v[j] >= target) {
          jb = j;
          found = true;
        } else {
          c += v[j];
        }
      }
    }
    *b_out = L * 8 + jb;
    *below_out = c;
  }
}

// One warp: the kth smallest (1-based, 1 <= kth <= n) of n keys key(i) of
// NPASS * 8 bits, by NPASS passes of 8-bit digits over the warp's 256-int
// shared histogram hist (sh: 2 shared ints).  below = keys smaller than the
// result, neq = keys equal to it.
template <int NPASS, class KeyF>
__device__ __forceinline__ uint32_t warp_radix_kth(int n, int kth, KeyF key, int *hist, int *sh,
                                                   int &below, int &neq) {
  const int lane = threadIdx.x & 31;
  uint32_t prefix = 0, mask = 0;
  int bl = 0;
#pragma unroll 1
  for (int pass = 0; pass < NPASS; ++pass) {
    const int shift = 8 * (NPASS - 1 - pass);
    for (int i = lane; i < 256; i += 32) hist[i] = 0;
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
      const uint32_t k = key(i);
      if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1);
    }
    __syncwarp();
    warp_find_bucket(hist, bl, kth, sh, sh + 1);
    __syncwarp();
    const int digit = sh[0];
    prefix |= (uint32_t)digit << shift;
    mask |= 255u << shift;
    bl = sh[1];
    if (pass == NPASS - 1) neq = hist[digit];
    __syncwarp();
  }
  below = bl;
  return prefix;
}

// Block-wide radix select over n keys key(i) of NPASS * 8 bits: the kth
// smallest (1-based, 1 <= kth <= n) by NPASS passes of 8-bit digits, most
// significant first, over the 256-int shared histogram hist.  *below = keys
// smaller than the result, *neq = keys equal to it.  All NT threads of the
// block call it; sh is 2 shared ints; it ends with the block synchronised.
template <int NT, int NPASS, class KeyF>
__device__ uint32_t block_radix_kth(int n, int kth, KeyF key, int *hist, int *sh, int *below_out,
                                    int *neq_out) {
  const int tid = threadIdx.x;
  uint32_t prefix = 0, mask = 0;
  int below = 0, neq = 0;
  for (int pass = 0; pass < NPASS; ++pass) {
    const int shift = 8 * (NPASS - 1 - pass);
    for (int i = tid; i < 256; i += NT) hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += NT) {
      const uint32_t k = key(i);
      if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1);
    }
    __syncthreads();
    if (tid < 32) warp_find_bucket(hist, below, kth, sh, sh + 1);
    __syncthreads();
    const int digit = sh[0];
    prefix |= (uint32_t)digit << shift;
    mask |= 255u << shift;
    below = sh[1];
    if (pass == NPASS - 1) neq = hist[digit];
    __syncthreads();  // hist and sh are rewritten by the next pass or the caller
  }
  *below_out = below;
  *neq_out = neq;
  return prefix;
}

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    uint64_t w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w < v ? w : v;
  }
  return v;
}

// Ascending sort of a[0:n) in shared memory by one warp.  Bitonic network in
// its "flip" form over the next power of two P >= n: every compare-exchange
// puts the smaller key at the lower index, so the missing elements [n, P)
// behave as +inf and are simply skipped.
__device__ __forceinline__ void warp_sort(uint64_t *a, int n) {
  const int lane = threadIdx.x & 31;
  int P = 1;
  while (P < n) P <<= 1;
  const int pairs = P >> 1;
  for (int size = 2; size <= P; size <<= 1) {
    const int half = size >> 1;
    const int lh = __ffs(half) - 1;
    for (int p = lane; p < pairs; p += 32) {
      const int blk = p >> lh, off = p & (half - 1);
      const int i = blk * size + off, j = blk * size + size - 1 - off;
      if (j < n) {
        uint64_t x = a[i], y = a[j];
        if (y < x) { a[i] = y; a[j] = x; }
      }
    }
    __syncwarp();
    for (int stride = half >> 1; stride > 0; stride >>= 1) {
      const int ls = __ffs(stride) - 1;
      for (int p = lane; p < pairs; p += 32) {
        const int i = ((p >> ls) << (ls + 1)) + (p & (stride - 1)), j = i + stride;
        if (j < n) {
          uint64_t x = a[i], y = a[j];
          if (y < x) { a[i] = y; a[j] = x; }
        }
      }
      __syncwarp();
    }
  }
}

// ascending bitonic sort of one key per lane across the warp (shuffles only)
__device__ __forceinline__ uint64_t warp_sort_lane(uint64_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const uint64_t o = __shfl_xor_sync(0xffffffffu, v, stride);
      const bool up = (lane & size) == 0;        // direction of this lane's sequence
      const bool lower = (lane & stride) == 0;   // this lane holds the smaller position
      v = (lower == up) == (o < v) ? o : v;  // the smaller where lower == up, else the larger
    }
  }
  return v;
}

// Ascending bitonic sort of 32 J keys held J per lane (lane l holds positions
// J l .. J l + J - 1): strides below J compare within a lane, larger ones across
// lanes by shuffles; the direction of each compare-exchange is that of the
// block of `size` positions holding it (ascending for even blocks).
template <int J>
__device__ __forceinline__ void warp_sort_lanes(uint64_t (&v)[J]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32 * J; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= J) {
        const int ls = stride / J;
        const bool lower = (lane & ls) == 0;
        const bool asc = ((lane * J) & size) == 0;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const uint64_t o = __shfl_xor_sync(0xffffffffu, v[j], ls);
          const uint64_t lo = o < v[j] ? o : v[j], hi = o < v[j] ? v[j] : o;
          v[j] = lower == asc ? lo : hi;
        }
      } else {
#pragma unroll
        for (int j = 0; j < J; ++j) {
          if (j & stride) continue;
          const bool asc = ((lane * J + j) & size) == 0;
          const uint64_t a = v[j], b = v[j | stride];
          const uint64_t lo = a < b ? a : b, hi = a < b ? b : a;
          v[j] = asc ? lo : hi;
          v[j | stride] = asc ? hi : lo;
        }
      }
    }
  }
}

// One warp: ascending sort of a[0:n), n <= 32 J, in shared memory through
// registers; only the first `keep` are put back.
template <int J>
__device__ __forceinline__ void warp_sort_regs(uint64_t *a, int n, int keep) {
  const int lane = threadIdx.x & 31;
  uint64_t v[J];
#pragma unroll
  for (int j = 0; j < J; ++j) v[j] = lane * J + j < n ? a[lane * J + j] : ~0ull;
  __syncwarp();
  warp_sort_lanes<J>(v);
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (lane * J + j < min(n, keep)) a[lane * J + j] = v[j];
  __syncwarp();
}

// Ascending sort of a[0:n) in shared memory by the NT threads of a block (the
// flip form of the bitonic network, as warp_sort); ends synchronised.
template <int NT>
__device__ __forceinline__ void block_sort(uint64_t *a, int n) {
  int P = 1;
  while (P < n) P <<= 1;
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const bool flip = stride == size >> 1;
      const int ls = __ffs(stride) - 1;
      for (int p = threadIdx.x; p < P >> 1; p += NT) {
        const int off = p & (stride - 1), base = (p >> ls) << (ls + 1);
        const int i = base + off, j = flip ? base + 2 * stride - 1 - off : i + stride;
        if (j < n) {
          const uint64_t x = a[i], y = a[j];
          if (y < x) { a[i] = y; a[j] = x; }
        }
      }
      __syncthreads();
    }
  }
}

}  // namespace adn
