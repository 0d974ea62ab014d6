// Device-side building blocks of single-pass scans: block scans of small
// packed counts and the decoupled look-back over tiles for several sums at
// once, and the write of a kernel's result into the host's mapped page.
#pragma once
#include "common.cuh"

// Exclusive scan of one value per thread over a block of NT threads; several
// counts may be packed into the word as long as none overflows its field.
template <int NT>
__device__ inline u64 block_scan(u64 v, u64* total) {
  __shared__ u64 wsum[NT / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  u64 x = v;
  for (int d = 1; d < 32; d <<= 1) {
    const u64 y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  if (wid == 0) {
    u64 s = lane < NT / 32 ? wsum[lane] : 0;
    for (int d = 1; d < 32; d <<= 1) {
      const u64 y = __shfl_up_sync(0xffffffffu, s, d);
      if (lane >= d) s += y;
    }
    if (lane < NT / 32) wsum[lane] = s;
  }
  __syncthreads();
  const u64 before = wid ? wsum[wid - 1] : 0;
  *total = wsum[NT / 32 - 1];
  __syncthreads();
  return before + x - v;
}

// Last i in [lo, n) with pre[i] <= c, by the whole warp (c the same in every
// lane, pre[lo] <= c): 32 pivots a step, so three dependent loads for 10^4 nodes instead of
// fourteen.
template <class T>
__device__ inline int64_t warp_find(const T* pre, int64_t n, int64_t c, int64_t lo = 0) {
  const int lane = threadIdx.x & 31;
  int64_t hi = n;
  __syncwarp();
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) >> 5, at = lo + (lane + 1) * step;
    const int k = __popc(__ballot_sync(0xffffffffu, at < hi && pre[at] <= c));
    lo += k * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// Decoupled look-back over tiles for NC sums at once (see k_scan_lb for the
// scheme and why the waits end): tile t's words are st[t * NC ..], each
// (value << 10 | epoch << 2 | status) with status 1 = the tile's own sum and
// 2 = the inclusive prefix; a tile whose words differ in status is being
// rewritten and read again.  Run by warp 0 with the tile's sums in every lane;
// returns the exclusive prefixes in every lane.  Past LB_SPINS polls it sets
// *err and carries on.
constexpr uint32_t LB_SPINS = 1u << 20;

template <int NC>
__device__ inline void look_back(u64* st, int64_t tile, const int64_t (&agg)[NC], int64_t (&pre)[NC], uint32_t ep,
                                 int32_t* err) {
  const int lane = threadIdx.x & 31;
  const u64 tag = (u64)(ep & 255u) << 2;
#pragma unroll
  for (int k = 0; k < NC; ++k) pre[k] = 0;
  if (tile > 0) {
#pragma unroll
    for (int k = 0; k < NC; ++k)
      if (lane == k) atomicExch((unsigned long long*)&st[tile * NC + k], ((u64)agg[k] << 10) | tag | 1u);
    uint32_t spins = 0;
    for (int64_t j0 = tile - 1;;) {
      const int64_t j = j0 - lane;
      u64 x[NC];
      u64 all = 3, any = 0;
      bool fresh = true;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        x[k] = j >= 0 ? *(volatile const u64*)&st[j * NC + k] : 0;
        fresh = fresh && ((x[k] >> 2) & 255u) == (ep & 255u);
        all &= x[k];
        any |= x[k] & 3u;
      }
      const bool ready = j < 0 || (fresh && all != 0 && any == all);
      const unsigned rmask = __ballot_sync(0xffffffffu, ready);
      const unsigned pmask = __ballot_sync(0xffffffffu, j >= 0 && ready && any == 2u);
      const int nr = rmask == 0xffffffffu ? 32 : __ffs(~rmask) - 1;  // nearest tile not ready
      const int fp = pmask ? __ffs(pmask) - 1 : 32;                  // nearest inclusive prefix
      if (fp < nr || nr == 32) {
        const int upto = fp < 32 ? fp : 31;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          int64_t v = j >= 0 && lane <= upto ? (int64_t)(x[k] >> 10) : 0;
          for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
          pre[k] += v;
        }
        if (fp < 32 || j0 < 32) break;  // a prefix, or every tile before this one, was summed
        j0 -= 32;
        continue;
      }
      if (++spins > LB_SPINS) {
        if (lane == 0) atomicExch(err, 1);
        break;
      }
      __nanosleep(32);
    }
  }
#pragma unroll
  for (int k = 0; k < NC; ++k)
    if (lane == k) atomicExch((unsigned long long*)&st[tile * NC + k], ((u64)(pre[k] + agg[k]) << 10) | tag | 2u);
}

// A kernel's result for the host: each 32-bit word goes into the mapped page
// as one 64-bit store of (sequence number << 32 | word), so that a word tells
// by itself whether it belongs to this read.  The host waits for every word;
// nothing has to order them (a fence to the host between the payload and a
// sequence number cost 1.5 us a read).
__device__ inline void put_word(u64* page, uint32_t seq, int w, uint32_t v) {
  *(volatile u64*)(page + w) = ((u64)seq << 32) | v;
}

// Values that a kernel hands to the host when its last block is done: device
// words (4-byte multiples).  The ticket counts the blocks that are through
// (zero before the launch).  seq = 0: nothing to hand over.
constexpr int TAIL_MAX = 8;
struct Tail {
  const uint32_t* src[TAIL_MAX];
  int32_t off[TAIL_MAX], words[TAIL_MAX];  // in 4-byte words of the payload
  int32_t n;
  u64* page;
  uint32_t seq;
  int32_t* ticket;
};

// (except values whose source is `skip`: the kernel puts those itself)
__device__ inline void put_tail(const Tail& t, const void* skip = nullptr) {
  for (int i = 0; i < t.n; ++i) {
    if (skip && t.src[i] == skip) continue;
    for (int w = threadIdx.x; w < t.words[i]; w += blockDim.x)
      put_word(t.page, t.seq, t.off[i] + w, __ldcg(t.src[i] + w));
  }
}

// Entry `src` of the tail from N values of the calling thread.
template <int N>
__device__ inline void put_values(const Tail& t, const void* src, const int64_t (&v)[N]) {
  for (int i = 0; i < t.n; ++i) {
    if (t.src[i] != src) continue;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      put_word(t.page, t.seq, t.off[i] + 2 * k, (uint32_t)(u64)v[k]);
      put_word(t.page, t.seq, t.off[i] + 2 * k + 1, (uint32_t)((u64)v[k] >> 32));
    }
  }
}

// Called by every thread of every block as the kernel's last step: a separate
// one-block kernel for the copy costs 2.6 us and the gap in front of it.
__device__ inline void pub_tail(const Tail& t) {
  if (t.seq == 0) return;
  __threadfence();  // this thread's writes, before its block's ticket
  __syncthreads();
  if (gridDim.x > 1) {
    __shared__ int s_last;
    if (threadIdx.x == 0) s_last = atomicAdd(t.ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
  }
  put_tail(t);
}
