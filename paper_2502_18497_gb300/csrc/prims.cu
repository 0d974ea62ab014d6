// Device primitives: exclusive scan, stable LSD radix sort of (key, value)
// pairs, and reduce-by-key of sorted pairs.  Hand-written; no library sort.
#include <cooperative_groups.h>

#include <algorithm>

#include "prims.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int SC_THREADS = 256;
constexpr int SC_ITEMS = 4;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;

__device__ inline int64_t block_excl_scan_i64(int64_t v, int64_t* total) {
  __shared__ int64_t wsum[SC_THREADS / WARP];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t x = v;
  for (int d = 1; d < 32; d <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int64_t s = lane < SC_THREADS / WARP ? wsum[lane] : 0;
    for (int d = 1; d < 32; d <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, s, d);
      if (lane >= d) s += y;
    }
    if (lane < SC_THREADS / WARP) wsum[lane] = s;
  }
  __syncthreads();
  int64_t before = wid ? wsum[wid - 1] : 0;
  *total = wsum[SC_THREADS / WARP - 1];
  __syncthreads();
  return before + x - v;
}

// Scan input: an array.
template <class T>
struct ArrayIn {
  const T* p;
  __device__ int64_t operator()(int64_t i) const { return (int64_t)p[i]; }
};

// whole input in one tile: scan and total in one launch
template <class In>
__global__ void k_scan_one(In in, int64_t* out, int64_t n, int64_t* total) {
  pdl_enter();
  const int64_t base = (int64_t)threadIdx.x * SC_ITEMS;
  int64_t loc[SC_ITEMS];
  int64_t s = 0;
  for (int k = 0; k < SC_ITEMS; ++k) {
    int64_t i = base + k;
    loc[k] = i < n ? in(i) : 0;
    s += loc[k];
  }
  int64_t tot;
  int64_t pre = block_excl_scan_i64(s, &tot);
  for (int k = 0; k < SC_ITEMS; ++k) {
    int64_t i = base + k;
    if (i < n) out[i] = pre;
    pre += loc[k];
  }
  if (threadIdx.x == 0 && total) *total = tot;
}

// Single-pass scan with decoupled look-back.  Tiles are claimed in order
// from a counter, so a tile only waits on tiles claimed before it, and every
// tile publishes its own aggregate before it waits: the waits always end.
// A tile's state word packs (value << 10 | epoch << 2 | status) with status
// 1 = tile aggregate, 2 = inclusive prefix; words of another epoch (an
// earlier scan) read as not ready.  Inputs are non-negative counts below
// 2^53.  The wait is bounded all the same: past LB_SPINS polls the tile sets
// *err and carries on (the host turns the flag into LDL_E_TIMEOUT).
constexpr int LB_ITEMS = 8;
constexpr int LB_TILE = SC_THREADS * LB_ITEMS;

template <class In>
__global__ void __launch_bounds__(SC_THREADS) k_scan_lb(In in, int64_t* out, int64_t n, u64* st, int32_t* ctr,
                                                        uint32_t ep, int64_t* total, int32_t* err) {
  pdl_enter();
  __shared__ int64_t s_tile, s_pre;
  if (threadIdx.x == 0) s_tile = atomicAdd(ctr, 1);
  __syncthreads();
  const int64_t tile = s_tile;
  if (tile * LB_TILE >= n && tile > 0) return;
  const int64_t base = tile * LB_TILE + (int64_t)threadIdx.x * LB_ITEMS;
  int64_t loc[LB_ITEMS];
  int64_t sum = 0;
  for (int k = 0; k < LB_ITEMS; ++k) {
    const int64_t i = base + k;
    loc[k] = i < n ? in(i) : 0;
    sum += loc[k];
  }
  int64_t agg;
  const int64_t pre = block_excl_scan_i64(sum, &agg);
  if (threadIdx.x < 32) {
    // warp 0 looks back over 32 predecessors at a time: it sums aggregates
    // until the nearest inclusive prefix, waiting only for tiles before it
    const int lane = threadIdx.x;
    const u64 tag = (u64)(ep & 255u) << 2;
    int64_t acc = 0;
    if (tile > 0) {
      if (lane == 0) atomicExch((unsigned long long*)&st[tile], ((u64)agg << 10) | tag | 1u);
      uint32_t spins = 0;
      for (int64_t j0 = tile - 1;;) {
        const int64_t j = j0 - lane;
        u64 x = 0;
        if (j >= 0) x = *(volatile const u64*)&st[j];
        const bool ready = j < 0 || (((x >> 2) & 255u) == (ep & 255u) && (x & 3u) != 0);
        const unsigned rmask = __ballot_sync(0xffffffffu, ready);
        const unsigned pmask = __ballot_sync(0xffffffffu, j >= 0 && ready && (x & 3u) == 2u);
        const int nr = rmask == 0xffffffffu ? 32 : __ffs(~rmask) - 1;  // nearest tile not ready
        const int fp = pmask ? __ffs(pmask) - 1 : 32;                  // nearest inclusive prefix
        if (fp < nr || nr == 32) {
          const int upto = fp < 32 ? fp : 31;
          const int64_t v = (j >= 0 && lane <= upto) ? (int64_t)(x >> 10) : 0;
          acc += warp_sum_i64(v);
          acc = __shfl_sync(0xffffffffu, acc, 0);
          if (fp < 32) break;
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
    if (lane == 0) {
      atomicExch((unsigned long long*)&st[tile], ((u64)(acc + agg) << 10) | tag | 2u);
      s_pre = acc;
      if ((tile + 1) * LB_TILE >= n && total) *total = acc + agg;
    }
  }
  __syncthreads();
  int64_t p = s_pre + pre;
  for (int k = 0; k < LB_ITEMS; ++k) {
    const int64_t i = base + k;
    if (i < n) out[i] = p;
    p += loc[k];
  }
}

// Scan of the chunk counts of a node list (chunks.cuh: ceil(len / chunk) per
// row, at least 1 per listed node, 0 past the list's device-side count).  One
// node per thread: the counts hang on two dependent loads each (5 us for some
// 10^4 nodes; 10 with eight nodes per thread).
constexpr int CC_TPB = 512;
__global__ void __launch_bounds__(CC_TPB) k_scan_chunks(const int32_t* list, const int32_t* nlist, int64_t n_hint,
                                                        const int32_t* la, const int32_t* lb, int32_t chunk,
                                                        int64_t* out, LookBack q) {
  pdl_enter();
  __shared__ int64_t s_tile, s_pre;
  if (threadIdx.x == 0) s_tile = atomicAdd(q.ctr, 1);
  __syncthreads();
  const int64_t tile = s_tile, i = tile * CC_TPB + threadIdx.x;
  int64_t c = 0;
  if (i < n_hint && i < *nlist) {
    const int32_t v = list[i];
    c = (la[v] + chunk - 1) / chunk + (lb ? (lb[v] + chunk - 1) / chunk : 0);
    if (c == 0) c = 1;
  }
  u64 tot;
  const u64 ex = block_scan<CC_TPB>((u64)c, &tot);
  if (threadIdx.x < 32) {
    const int64_t agg[1] = {(int64_t)tot};
    int64_t pre[1];
    look_back<1>(q.st, tile, agg, pre, q.ep, q.err);
    if (threadIdx.x == 0) s_pre = pre[0];
  }
  __syncthreads();
  if (i <= n_hint) out[i] = s_pre + (int64_t)ex;
}

// ---------------------------------------------------------------- radix sort
constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
// A sort's extras: the device count of its pairs (else the host's n), and,
// with tbits > 0, the read transposes each key ((row, col) -> (col + row_off,
// row) with tbits per half) and the result goes behind the n input pairs.
struct RsExt {
  const int32_t* n_dev;
  int tbits;
  int64_t row_off;
  int64_t* zero;  // n words cleared on the way (null: none)
};
__device__ inline u64 transposed(u64 key, int bits, int64_t row_off) {
  return (((key & ((((u64)1) << bits) - 1)) + (u64)row_off) << bits) | (key >> bits);
}
static_assert(RS_THREADS == 256 && SC_THREADS == 256, "one thread per digit");

// Digit histogram of tile b (RS_TILE keys from b * RS_TILE) into column b
// of ghist (digit-major: ghist[d * nb + b]).
__device__ inline void rs_hist_tile(const u64* keys, int64_t n, int shift, int64_t nb, int64_t* ghist, int64_t b,
                                    int tbits = 0, int64_t row_off = 0) {
  __shared__ uint32_t h[256];
  for (int i = threadIdx.x; i < 256; i += RS_THREADS) h[i] = 0;
  const int lane = threadIdx.x & 31;
  const int64_t base = b * RS_TILE;
  int d[RS_ITEMS];
  for (int k = 0; k < RS_ITEMS; ++k) {  // all loads in flight before any shuffle
    const int64_t i = base + (int64_t)k * RS_THREADS + threadIdx.x;
    u64 x = i < n ? keys[i] : 0;
    if (tbits) x = transposed(x, tbits, row_off);
    d[k] = i < n ? (int)((x >> shift) & 255) : 256;
  }
  __syncthreads();
  for (int k = 0; k < RS_ITEMS; ++k) {
    // one shared atomic per distinct digit of the warp (skewed digits collide)
    const unsigned peers = __match_any_sync(0xffffffffu, d[k]);
    if (d[k] < 256 && lane == __ffs(peers) - 1) atomicAdd(&h[d[k]], (uint32_t)__popc(peers));
  }
  __syncthreads();
  for (int x = threadIdx.x; x < 256; x += RS_THREADS) ghist[(int64_t)x * nb + b] = h[x];
  __syncthreads();  // h is reset by the block's next tile
}

__global__ void k_rs_hist(const u64* keys, int64_t n, int shift, int64_t nb, int64_t* ghist, RsExt x, int first,
                          int in_off) {
  pdl_enter();
  if (x.n_dev) n = min(n, (int64_t)*x.n_dev);
  if (x.zero && first)
    for (int64_t i = (int64_t)blockIdx.x * RS_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * RS_THREADS)
      x.zero[i] = 0;
  rs_hist_tile(in_off ? keys + n : keys, n, shift, nb, ghist, blockIdx.x, first ? x.tbits : 0, x.row_off);
}

// One block per digit: exclusive scan of the digit's tile counts in place
// (8 consecutive counts per thread per step), and the digit's total.
__device__ inline void rs_dscan_digit(int64_t* ghist, int64_t nb, int64_t* dtot, int d) {
  constexpr int IT = 8;
  int64_t* row = ghist + (int64_t)d * nb;
  int64_t carry = 0;
  for (int64_t b0 = 0; b0 < nb; b0 += SC_THREADS * IT) {
    const int64_t base = b0 + (int64_t)threadIdx.x * IT;
    int64_t v[IT];
    int64_t sum = 0;
    for (int k = 0; k < IT; ++k) {
      v[k] = base + k < nb ? row[base + k] : 0;
      sum += v[k];
    }
    int64_t total;
    int64_t ex = carry + block_excl_scan_i64(sum, &total);
    for (int k = 0; k < IT; ++k) {
      if (base + k < nb) row[base + k] = ex;
      ex += v[k];
    }
    carry += total;
  }
  if (threadIdx.x == 0) dtot[d] = carry;
}

__global__ void __launch_bounds__(SC_THREADS) k_rs_dscan(int64_t* ghist, int64_t nb, int64_t* dtot) {
  pdl_enter();
  rs_dscan_digit(ghist, nb, dtot, blockIdx.x);
}

// One tile of RS_TILE pairs per block.  Each warp ranks a contiguous sub-tile
// of RS_ITEMS * 32 pairs (rounds of 32, stable), the block turns the warp
// counts into digit-sorted positions inside the tile, the tile is staged in
// shared memory in digit order, and consecutive threads then write
// consecutive output slots of each digit.  The global start of (digit d,
// tile b) is the exclusive prefix of the digit totals dtot at d plus the
// per-digit scanned tile count goff[d * nb + b].
__device__ inline void rs_scatter_tile(const u64* keys, const u64* vals, u64* okeys, u64* ovals, int64_t n, int shift,
                                       int64_t nb, const int64_t* goff, const int64_t* dtot, int64_t b, int tbits = 0,
                                       int64_t row_off = 0) {
  constexpr int NW = RS_THREADS / WARP;
  __shared__ int32_t whist[NW][256];  // per-warp digit counts, then per-warp exclusive bases
  __shared__ int32_t tstart[256];     // tile-local start of each digit
  __shared__ int64_t gstart[256];     // global start of each digit for this tile
  __shared__ u64 sk[RS_TILE];
  __shared__ u64 sv[RS_TILE];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t base = b * RS_TILE;
  const int tile_n = (int)max((int64_t)0, min((int64_t)RS_TILE, n - base));
  for (int d = lane; d < 256; d += 32) whist[wid][d] = 0;
  {
    int64_t total;
    const int64_t dbase = block_excl_scan_i64(dtot[tid], &total);  // RS_THREADS == 256 digits
    gstart[tid] = dbase + goff[(int64_t)tid * nb + b];
  }
  u64 key[RS_ITEMS], val[RS_ITEMS];
  int rk[RS_ITEMS];
  for (int k = 0; k < RS_ITEMS; ++k) {
    const int li = wid * (RS_ITEMS * 32) + k * 32 + lane;
    const bool valid = li < tile_n;
    key[k] = valid ? keys[base + li] : 0;
    val[k] = valid ? vals[base + li] : 0;
    if (tbits) key[k] = transposed(key[k], tbits, row_off);
  }
  for (int k = 0; k < RS_ITEMS; ++k) {
    const int li = wid * (RS_ITEMS * 32) + k * 32 + lane;
    const int d = li < tile_n ? (int)((key[k] >> shift) & 255) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int before = d < 256 ? whist[wid][d] : 0;
    rk[k] = before + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
    if (d < 256 && lane == __ffs(peers) - 1) whist[wid][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // thread d: exclusive scan of digit d over the warps, then over the digits
  int cnt = 0;
  {
    const int d = tid;  // RS_THREADS == 256
    for (int w = 0; w < NW; ++w) {
      const int c = whist[w][d];
      whist[w][d] = cnt;
      cnt += c;
    }
  }
  int64_t total;
  const int64_t ds = block_excl_scan_i64(cnt, &total);
  tstart[tid] = (int32_t)ds;
  __syncthreads();
  for (int k = 0; k < RS_ITEMS; ++k) {
    const int li = wid * (RS_ITEMS * 32) + k * 32 + lane;
    if (li < tile_n) {
      const int d = (int)((key[k] >> shift) & 255);
      const int p = tstart[d] + whist[wid][d] + rk[k];
      sk[p] = key[k];
      sv[p] = val[k];
    }
  }
  __syncthreads();
  for (int j = tid; j < tile_n; j += RS_THREADS) {
    const u64 k = sk[j];
    const int d = (int)((k >> shift) & 255);
    const int64_t p = gstart[d] + (j - tstart[d]);
    okeys[p] = k;
    ovals[p] = sv[j];
  }
  __syncthreads();  // the tile buffers are reused by the caller's next tile
}

__global__ void __launch_bounds__(RS_THREADS, 4) k_rs_scatter(const u64* keys, const u64* vals, u64* okeys,
                                                              u64* ovals, int64_t n, int shift, int64_t nb,
                                                              const int64_t* goff, const int64_t* dtot, RsExt x,
                                                              int first, int in_off, int out_off) {
  pdl_enter();
  if (x.n_dev) n = min(n, (int64_t)*x.n_dev);
  rs_scatter_tile(in_off ? keys + n : keys, in_off ? vals + n : vals, out_off ? okeys + n : okeys,
                  out_off ? ovals + n : ovals, n, shift, nb, goff, dtot, blockIdx.x, first ? x.tbits : 0, x.row_off);
}

// The whole multi-tile sort in one cooperative launch, one block per SM and one
// tile per block: the tiles are T pairs, a multiple of the block's threads, so
// that any list up to CO_ITEMS pairs per thread is one wave.  Per 8-bit pass a
// block loads its tile into registers once, ranks it per warp (stable) and
// publishes its digit counts; warps scan the digits over the tiles; the tile
// goes through shared memory in digit order to its global places.  A grid
// barrier after each.  Bound by the barriers and the passes' latency: 82 us for
// six passes over some 10^5 pairs (2M-vertex power-law graph), 113 with four
// small blocks per SM, a second load and a scan block per digit.  A transposing
// sort ping-pongs between the place behind its input and (tk, tv) such that the
// last pass ends there.
constexpr int CO_THREADS = 512;
constexpr int CO_ITEMS = 16;
constexpr int CO_TILE = CO_THREADS * CO_ITEMS;
constexpr int CO_NW = CO_THREADS / WARP;
struct CoShared {
  int32_t whist[CO_NW][256];
  int32_t tstart[256];
  int64_t gstart[256];
  u64 sk[CO_TILE];
  u64 sv[CO_TILE];
};

__global__ void __launch_bounds__(CO_THREADS, 1) k_rs_coop(u64* keys, u64* vals, u64* tk, u64* tv, int64_t n,
                                                           int lo_bit, int bits, int32_t* ghist, int32_t* dtot,
                                                           RsExt x) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char co_smem[];
  CoShared& m = *(CoShared*)co_smem;
  cg::grid_group grid = cg::this_grid();
  if (x.n_dev) n = min(n, (int64_t)*x.n_dev);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int items = (int)max((int64_t)1, (n + (int64_t)gridDim.x * CO_THREADS - 1) / ((int64_t)gridDim.x * CO_THREADS));
  const int T = items * CO_THREADS;
  const int nb = (int)((n + T - 1) / T), b = blockIdx.x;  // nb <= gridDim.x
  const int64_t base = (int64_t)b * T;
  const int tile_n = (int)max((int64_t)0, min((int64_t)T, n - base));
  if (x.zero)
    for (int64_t i = (int64_t)b * CO_THREADS + tid; i < n; i += (int64_t)gridDim.x * CO_THREADS) x.zero[i] = 0;
  u64 *ik = keys, *iv = vals, *ok = tk, *ov = tv;
  u64 *nk = keys, *nv = vals;  // written by the pass after the first
  if (x.tbits) {
    nk = keys + n;
    nv = vals + n;
    if (((bits - lo_bit + 7) / 8) & 1) {
      ok = nk; ov = nv;
      nk = tk; nv = tv;
    }
  }
  for (int shift = lo_bit; shift < bits; shift += 8) {
    u64 key[CO_ITEMS], val[CO_ITEMS];
    int rk[CO_ITEMS];
#pragma unroll
    for (int k = 0; k < CO_ITEMS; ++k) {
      const int li = wid * (items * 32) + k * 32 + lane;
      const bool on = k < items && li < tile_n;
      key[k] = on ? ik[base + li] : 0;
      val[k] = on ? iv[base + li] : 0;
      if (x.tbits && shift == lo_bit) key[k] = transposed(key[k], x.tbits, x.row_off);
    }
    for (int d = lane; d < 256; d += 32) m.whist[wid][d] = 0;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < CO_ITEMS; ++k) {
      if (k >= items) break;  // the same in every thread
      const int li = wid * (items * 32) + k * 32 + lane;
      const int d = li < tile_n ? (int)((key[k] >> shift) & 255) : 256;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const int before = d < 256 ? m.whist[wid][d] : 0;
      rk[k] = before + __popc(peers & ((1u << lane) - 1u));
      __syncwarp();
      if (d < 256 && lane == __ffs(peers) - 1) m.whist[wid][d] = before + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    int cnt = 0;
    if (tid < 256) {
      for (int w = 0; w < CO_NW; ++w) {  // thread = digit
        const int c = m.whist[w][tid];
        m.whist[w][tid] = cnt;
        cnt += c;
      }
      if (b < nb) ghist[tid * nb + b] = cnt;
    }
    u64 total;
    const u64 ts = block_scan<CO_THREADS>((u64)cnt, &total);
    if (tid < 256) m.tstart[tid] = (int32_t)ts;
    grid.sync();
    for (int d = b * CO_NW + wid; d < 256; d += gridDim.x * CO_NW) {  // a warp per digit
      int32_t* row = ghist + (int64_t)d * nb;
      int carry = 0;
      for (int c0 = 0; c0 < nb; c0 += 32) {
        const int v = c0 + lane < nb ? row[c0 + lane] : 0;
        int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        if (c0 + lane < nb) row[c0 + lane] = carry + incl - v;
        carry += __shfl_sync(0xffffffffu, incl, 31);
      }
      if (lane == 0) dtot[d] = carry;
    }
    grid.sync();
    const u64 dbase = block_scan<CO_THREADS>(tid < 256 ? (u64)dtot[tid] : 0, &total);
    if (tid < 256 && b < nb) m.gstart[tid] = (int64_t)dbase + ghist[tid * nb + b];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < CO_ITEMS; ++k) {
      const int li = wid * (items * 32) + k * 32 + lane;
      if (k < items && li < tile_n) {
        const int d = (int)((key[k] >> shift) & 255);
        const int p = m.tstart[d] + m.whist[wid][d] + rk[k];
        m.sk[p] = key[k];
        m.sv[p] = val[k];
      }
    }
    __syncthreads();
    for (int j = tid; j < tile_n; j += CO_THREADS) {
      const u64 k = m.sk[j];
      const int d = (int)((k >> shift) & 255);
      const int64_t p = m.gstart[d] + (j - m.tstart[d]);
      ok[p] = k;
      ov[p] = m.sv[j];
    }
    grid.sync();
    ik = ok; iv = ov;
    u64* t = ok; ok = nk; nk = t;
    t = ov; ov = nv; nv = t;
  }
}

// Whole sort in one block (n <= RS_TILE).  Each thread holds RS_ITEMS pairs
// in registers across the passes: per 8-bit pass every warp ranks its
// contiguous sub-tile (rounds of 32, stable), the block turns the per-warp
// digit counts into positions, the pairs are placed in shared memory in
// digit order and read back in the same warp-contiguous layout.
// Up to RK_MAX pairs are placed by counting instead: a thread compares its key
// with all others (a few pairs: 2.1 us instead of 5.4, with sums 4.3 instead
// of 7.9; some hundred 3.3 instead of 6.4).
constexpr int SM_THREADS = 512;
constexpr int SM_ITEMS = RS_TILE / SM_THREADS;
constexpr int SM_WARPS = SM_THREADS / WARP;
constexpr int RK_MAX = 256;
struct RsSmall {
  int32_t whist[SM_WARPS][256];
  int32_t tstart[256];
  u64 sk[RS_TILE];
  u64 sv[RS_TILE];
};

// place of pair k of this thread: contiguous per warp
__device__ inline int sm_at(int k) { return (threadIdx.x >> 5) * (SM_ITEMS * 32) + k * 32 + (threadIdx.x & 31); }

__device__ inline void rs_small_sort(RsSmall& m, u64 (&key)[SM_ITEMS], u64 (&val)[SM_ITEMS], int n, int lo_bit,
                                     int bits) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (n <= RK_MAX) {
    // the pairs are in the first warps: pair i belongs to warp i / (SM_ITEMS * 32)
    const u64 mask = bits >= 64 ? ~(u64)0 : (((u64)1) << bits) - 1;
    for (int k = 0; k < SM_ITEMS; ++k)
      if (sm_at(k) < n) {
        m.sk[sm_at(k)] = key[k];
        m.sv[sm_at(k)] = val[k];
      }
    __syncthreads();
    u64 mk = 0, mv = 0;
    int rank = 0;
    if (tid < n) {
      mk = m.sk[tid];
      mv = m.sv[tid];
      const u64 x = (mk & mask) >> lo_bit;
#pragma unroll 4
      for (int j = 0; j < n; ++j) {
        const u64 y = (m.sk[j] & mask) >> lo_bit;
        rank += y < x || (y == x && j < tid);
      }
    }
    __syncthreads();
    if (tid < n) {
      m.sk[rank] = mk;
      m.sv[rank] = mv;
    }
    __syncthreads();
    for (int k = 0; k < SM_ITEMS; ++k)
      if (sm_at(k) < n) {
        key[k] = m.sk[sm_at(k)];
        val[k] = m.sv[sm_at(k)];
      }
    __syncthreads();
    return;
  }
  for (int shift = lo_bit; shift < bits; shift += 8) {
    for (int d = lane; d < 256; d += 32) m.whist[wid][d] = 0;
    __syncwarp();
    int rk[SM_ITEMS];
    for (int k = 0; k < SM_ITEMS; ++k) {
      const int d = sm_at(k) < n ? (int)((key[k] >> shift) & 255) : 256;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const int before = d < 256 ? m.whist[wid][d] : 0;
      rk[k] = before + __popc(peers & ((1u << lane) - 1u));
      __syncwarp();
      if (d < 256 && lane == __ffs(peers) - 1) m.whist[wid][d] = before + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    int cnt = 0;
    if (tid < 256)
      for (int w = 0; w < SM_WARPS; ++w) {  // thread = digit
        const int c = m.whist[w][tid];
        m.whist[w][tid] = cnt;
        cnt += c;
      }
    u64 total;
    const u64 start = block_scan<SM_THREADS>((u64)cnt, &total);
    if (tid < 256) m.tstart[tid] = (int32_t)start;
    __syncthreads();
    for (int k = 0; k < SM_ITEMS; ++k) {
      if (sm_at(k) < n) {
        const int d = (int)((key[k] >> shift) & 255);
        const int p = m.tstart[d] + m.whist[wid][d] + rk[k];
        m.sk[p] = key[k];
        m.sv[p] = val[k];
      }
    }
    __syncthreads();
    for (int k = 0; k < SM_ITEMS; ++k) {
      if (sm_at(k) < n) {
        key[k] = m.sk[sm_at(k)];
        val[k] = m.sv[sm_at(k)];
      }
    }
    __syncthreads();  // whist, tstart and the staging buffers are rewritten next pass
  }
}

extern __shared__ __align__(16) unsigned char small_smem[];

__global__ void __launch_bounds__(SM_THREADS) k_rs_small(u64* keys, u64* vals, int n, const int32_t* n_dev, int lo_bit,
                                                         int bits) {
  pdl_enter();
  RsSmall& m = *(RsSmall*)small_smem;
  if (n_dev) n = min(n, *n_dev);
  u64 key[SM_ITEMS], val[SM_ITEMS];
  for (int k = 0; k < SM_ITEMS; ++k) {
    key[k] = sm_at(k) < n ? keys[sm_at(k)] : 0;
    val[k] = sm_at(k) < n ? vals[sm_at(k)] : 0;
  }
  rs_small_sort(m, key, val, n, lo_bit, bits);
  for (int k = 0; k < SM_ITEMS; ++k)
    if (sm_at(k) < n) {
      keys[sm_at(k)] = key[k];
      vals[sm_at(k)] = val[k];
    }
}

// Sort by the low 2 * bits key bits, sum per key with zero sums dropped, and
// with `both` the same records transposed behind them, in (row, col) order
// (rows from row_off): sort_reduce() for n <= RS_TILE in one launch.
__global__ void __launch_bounds__(SM_THREADS) k_rs_small_reduce(const u64* keys, const u64* vals, int n,
                                                                const int32_t* n_dev, int bits, int both,
                                                                int64_t row_off, u64* okeys, int64_t* ovals,
                                                                int32_t* nr) {
  pdl_enter();
  RsSmall& m = *(RsSmall*)small_smem;
  if (n_dev) n = min(n, *n_dev);
  const int tid = threadIdx.x;
  u64 key[SM_ITEMS], val[SM_ITEMS];
  for (int k = 0; k < SM_ITEMS; ++k) {
    const int li = sm_at(k);
    key[k] = li < n ? keys[li] : 0;
    val[k] = li < n ? vals[li] : 0;
  }
  rs_small_sort(m, key, val, n, 0, 2 * bits);
  // sorted pairs into shared memory, SM_ITEMS consecutive ones per thread
  for (int k = 0; k < SM_ITEMS; ++k) {
    const int li = sm_at(k);
    m.sk[li] = key[k];
    m.sv[li] = val[k];
  }
  __syncthreads();
  const int i0 = tid * SM_ITEMS;
  int heads = 0;
  int64_t sum = 0;
  for (int k = 0; k < SM_ITEMS; ++k) {
    const int i = i0 + k;
    key[k] = m.sk[i];
    heads += i < n && (i == 0 || key[k] != m.sk[i - 1]);
    sum += i < n ? (int64_t)m.sv[i] : 0;
  }
  // segment numbers, and running sums whose differences at the segments' ends
  // are the segment sums (both modulo 2^64)
  u64 nseg64, all64;
  int seg = (int)block_scan<SM_THREADS>((u64)heads, &nseg64);
  int64_t run = (int64_t)block_scan<SM_THREADS>((u64)sum, &all64);
  const int nseg = (int)nseg64;
  const int64_t all = (int64_t)all64;
  u64 hk[SM_ITEMS];
  int64_t hr[SM_ITEMS];
  int hs = 0;
  for (int k = 0; k < SM_ITEMS; ++k) {
    const int i = i0 + k;
    if (i < n && (i == 0 || key[k] != m.sk[i - 1])) {
      hk[hs] = key[k];
      hr[hs] = run;
      ++hs;
    }
    run += i < n ? (int64_t)m.sv[i] : 0;
  }
  __syncthreads();
  for (int k = 0; k < hs; ++k) {
    m.sk[seg + k] = hk[k];
    m.sv[seg + k] = (u64)hr[k];
  }
  __syncthreads();
  int live = 0;
  for (int k = 0; k < SM_ITEMS; ++k) {
    const int s = i0 + k;
    hk[k] = s < nseg ? m.sk[s] : 0;
    hr[k] = s < nseg ? (s + 1 < nseg ? (int64_t)m.sv[s + 1] : all) - (int64_t)m.sv[s] : 0;
    live += hr[k] != 0;
  }
  u64 nlive;
  int p = (int)block_scan<SM_THREADS>((u64)live, &nlive);  // its barriers also end the reads above
  for (int k = 0; k < SM_ITEMS; ++k)
    if (hr[k] != 0) {
      okeys[p] = hk[k];
      ovals[p] = hr[k];
      m.sk[p] = transposed(hk[k], bits, row_off);
      m.sv[p] = (u64)hr[k];
      ++p;
    }
  if (tid == 0) *nr = (int32_t)nlive;
  if (!both) return;
  __syncthreads();
  n = (int)nlive;
  for (int k = 0; k < SM_ITEMS; ++k) {
    const int li = sm_at(k);
    key[k] = li < n ? m.sk[li] : 0;
    val[k] = li < n ? m.sv[li] : 0;
  }
  __syncthreads();
  // the records are in (row, col) order: a stable sort on the new row alone
  rs_small_sort(m, key, val, n, bits, 2 * bits + 1);
  for (int k = 0; k < SM_ITEMS; ++k) {
    const int li = sm_at(k);
    if (li < n) {
      okeys[n + li] = key[k];
      ovals[n + li] = (int64_t)val[k];
    }
  }
}

// Whole sort in one thread-block cluster of CL blocks (n <= CL * CS_TILE):
// the pairs are cut into CL tiles of T (a multiple of the block's threads, so
// that short lists spread over the cluster too), block c holds the pairs at
// positions [c * T, (c+1) * T), up to CS_ITEMS per thread in registers.  Per
// 8-bit pass every warp ranks its contiguous sub-tile (stable), each block
// publishes its digit counts in shared memory, and after a cluster barrier
// every block reads all blocks' counts (distributed shared memory) to place
// each of its pairs at its global position: digit start + counts of lower
// blocks + counts of lower warps + rank.  The pair is stored into the shared
// memory of the block that owns that position; after a second barrier each
// block reloads its slice.  The pairs never leave the chip between passes.
constexpr int CS_THREADS = 512;
constexpr int CS_ITEMS = 12;
constexpr int CS_TILE = CS_THREADS * CS_ITEMS;  // 6144 pairs, 96 KB per block
constexpr int CS_NW = CS_THREADS / WARP;

template <int CL>
__global__ void __launch_bounds__(CS_THREADS, 1) k_rs_cluster(u64* keys, u64* vals, int n, int lo_bit, int bits,
                                                              RsExt x) {
  pdl_enter();
  extern __shared__ u64 cs_smem[];
  u64* sk = cs_smem;
  u64* sv = cs_smem + CS_TILE;
  __shared__ int32_t whist[CS_NW][256];
  __shared__ int32_t hist[256];   // this block's digit counts, read by the whole cluster
  __shared__ int32_t s_tot[256];  // cluster-wide digit counts
  __shared__ int32_t tpos[256];   // global start of (digit, this block)
  cg::cluster_group cl = cg::this_cluster();
  const int c = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (x.n_dev) n = min(n, *x.n_dev);
  const int items = max(1, (n + CL * CS_THREADS - 1) / (CL * CS_THREADS));  // per thread
  const int T = items * CS_THREADS, base = c * T;
  const int tile_n = max(0, min(T, n - base));
  const uint32_t magic = (uint32_t)((((u64)1 << 32) + T - 1) / T);  // p / T = p * magic >> 32 for p < 2^17
  u64 key[CS_ITEMS], val[CS_ITEMS];
  for (int k = 0; k < CS_ITEMS; ++k) {
    const int li = wid * (items * 32) + k * 32 + lane;
    const bool on = k < items && li < tile_n;
    key[k] = on ? keys[base + li] : 0;
    val[k] = on ? vals[base + li] : 0;
    if (x.tbits) key[k] = transposed(key[k], x.tbits, x.row_off);
    if (x.zero && on) x.zero[base + li] = 0;
  }
  if (x.tbits) {  // the result goes behind the input
    keys += n;
    vals += n;
  }
  for (int shift = lo_bit; shift < bits; shift += 8) {
    for (int d = lane; d < 256; d += 32) whist[wid][d] = 0;
    __syncwarp();
    int rk[CS_ITEMS];
#pragma unroll
    for (int k = 0; k < CS_ITEMS; ++k) {
      if (k >= items) break;  // the same in every thread
      const int li = wid * (items * 32) + k * 32 + lane;
      const int d = li < tile_n ? (int)((key[k] >> shift) & 255) : 256;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const int before = d < 256 ? whist[wid][d] : 0;
      rk[k] = before + __popc(peers & ((1u << lane) - 1u));
      __syncwarp();
      if (d < 256 && lane == __ffs(peers) - 1) whist[wid][d] = before + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    if (tid < 256) {  // thread = digit: exclusive prefix over the warps
      int cnt = 0;
      for (int w = 0; w < CS_NW; ++w) {
        const int x = whist[w][tid];
        whist[w][tid] = cnt;
        cnt += x;
      }
      hist[tid] = cnt;
    }
    cl.sync();  // every block's counts are published
    if (tid < 256) {
      int tot = 0, lower = 0;
      for (int b = 0; b < CL; ++b) {
        const int x = cl.map_shared_rank(hist, b)[tid];
        tot += x;
        if (b < c) lower += x;
      }
      s_tot[tid] = tot;
      tpos[tid] = lower;
    }
    __syncthreads();
    if (wid == 0) {  // digit starts: exclusive scan of the totals, 8 digits per lane
      int v[8], sum = 0;
      for (int j = 0; j < 8; ++j) {
        v[j] = s_tot[lane * 8 + j];
        sum += v[j];
      }
      int incl = sum;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      int run = incl - sum;
      for (int j = 0; j < 8; ++j) {
        tpos[lane * 8 + j] += run;
        run += v[j];
      }
    }
    __syncthreads();
    for (int k = 0; k < CS_ITEMS; ++k) {
      const int li = wid * (items * 32) + k * 32 + lane;
      if (k < items && li < tile_n) {
        const int d = (int)((key[k] >> shift) & 255);
        const int p = tpos[d] + whist[wid][d] + rk[k];
        const int owner = (int)__umulhi((uint32_t)p, magic), slot = p - owner * T;
        cl.map_shared_rank(sk, owner)[slot] = key[k];
        cl.map_shared_rank(sv, owner)[slot] = val[k];
      }
    }
    cl.sync();  // every pair is in place; counts and staging are reused next pass
    for (int k = 0; k < CS_ITEMS; ++k) {
      const int li = wid * (items * 32) + k * 32 + lane;
      if (k < items && li < tile_n) {
        key[k] = sk[li];
        val[k] = sv[li];
      }
    }
  }
  for (int k = 0; k < CS_ITEMS; ++k) {
    const int li = wid * (items * 32) + k * 32 + lane;
    if (k < items && li < tile_n) {
      keys[base + li] = key[k];
      vals[base + li] = val[k];
    }
  }
}

// ---------------------------------------------------------------- reduce by key
// Segment sums of sorted keys: each thread takes RBK_RUN consecutive pairs.
// A segment that starts and ends inside the run is stored; a segment that
// crosses a run boundary is added atomically at its head (usum is zeroed
// first).  The head of a run's leading partial segment is found by a binary
// search for the first equal key.
constexpr int RBK_RUN = 8;
__global__ void k_segsum(const u64* keys, const u64* vals, int64_t n, const int32_t* n_dev, int64_t* usum) {
  pdl_enter();
  if (n_dev) n = min(n, (int64_t)*n_dev);
  const int64_t nt = (n + RBK_RUN - 1) / RBK_RUN;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nt; r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i0 = r * RBK_RUN, i1 = min(i0 + RBK_RUN, n);
    int64_t head = i0;
    if (i0 > 0 && keys[i0 - 1] == keys[i0]) {
      int64_t lo = 0, hi = i0;
      const u64 k = keys[i0];
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (keys[mid] < k) lo = mid + 1; else hi = mid;
      }
      head = lo;
    }
    int64_t acc = 0;
    for (int64_t i = i0; i < i1; ++i) {
      if (i > i0 && keys[i] != keys[i - 1]) {
        if (head < i0) atomic_add_i64(&usum[head], acc);
        else usum[head] = acc;
        head = i;
        acc = 0;
      }
      acc += (int64_t)vals[i];
    }
    const bool open_end = i1 < n && keys[i1] == keys[i1 - 1];
    if (head < i0 || open_end) atomic_add_i64(&usum[head], acc);
    else usum[head] = acc;
  }
}

// Compacts the segment heads with nonzero sums (keys, sums) in one pass with
// look-back; the last tile writes their number.
__global__ void __launch_bounds__(SC_THREADS) k_reduce_out(const u64* keys, const int64_t* usum, int64_t n,
                                                           const int32_t* n_dev, u64* okeys, int64_t* ovals,
                                                           int32_t* nr, int64_t* nr64, LookBack q) {
  pdl_enter();
  __shared__ int64_t s_tile, s_pre;
  if (n_dev) n = min(n, (int64_t)*n_dev);
  if (threadIdx.x == 0) s_tile = atomicAdd(q.ctr, 1);
  __syncthreads();
  const int64_t tile = s_tile;
  if (tile * LB_TILE >= n && tile > 0) return;
  // warp-contiguous rounds, so that a warp's loads are whole lines
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t base = tile * LB_TILE + wid * (LB_ITEMS * 32);
  u64 key[LB_ITEMS];
  int64_t sum[LB_ITEMS];
  unsigned live = 0, mask[LB_ITEMS];
  int cnt = 0;
  for (int k = 0; k < LB_ITEMS; ++k) {
    const int64_t i = base + k * 32 + lane;
    key[k] = i < n ? keys[i] : 0;
    sum[k] = i < n && (i == 0 || key[k] != keys[i - 1]) ? usum[i] : 0;
    mask[k] = __ballot_sync(0xffffffffu, sum[k] != 0);
    live |= (sum[k] != 0 ? 1u : 0u) << k;
    cnt += __popc(mask[k]);
  }
  // exclusive offset of the warp: only lane 0 contributes its count
  u64 tot;
  u64 ex = block_scan<SC_THREADS>(lane == 0 ? (u64)cnt : 0, &tot);
  ex = __shfl_sync(0xffffffffu, ex, 0);
  if (threadIdx.x < 32) {
    const int64_t agg[1] = {(int64_t)tot};
    int64_t pre[1];
    look_back<1>(q.st, tile, agg, pre, q.ep, q.err);
    if (threadIdx.x == 0) {
      s_pre = pre[0];
      if ((tile + 1) * LB_TILE >= n) {
        if (nr) *nr = (int32_t)(pre[0] + agg[0]);
        if (nr64) *nr64 = pre[0] + agg[0];
      }
    }
  }
  __syncthreads();
  int64_t p = s_pre + (int64_t)ex;
  for (int k = 0; k < LB_ITEMS; ++k) {
    if ((live >> k) & 1u) {
      const int64_t at = p + __popc(mask[k] & ((1u << lane) - 1u));
      okeys[at] = key[k];
      ovals[at] = sum[k];
    }
    p += __popc(mask[k]);
  }
}

}  // namespace

// ---------------------------------------------------------------- host wrappers
// Look-back state for the next multi-tile scan of n items: the tile words,
// this scan's epoch (1..255) and its tile counter.  When the epoch wraps, or
// the state grows, everything is cleared so that no stale word matches.
static uint32_t lb_begin(Prims& P, int64_t n, cudaStream_t s) {
  const int64_t tiles = (n + LB_TILE - 1) / LB_TILE;
  if (P.lb_ctl.cap == 0) {
    P.lb_ctl.exact(257);  // 256 epoch counters + the error flag
    CK(cudaMemsetAsync(P.lb_ctl.p, 0, sizeof(int32_t) * 257, s));
    P.lb_ep = 0;
  }
  bool clear = false;
  if (tiles > P.lb_st.cap) {
    P.lb_st.reserve(tiles, s);
    clear = true;
  }
  if (++P.lb_ep > 255) clear = true;
  if (clear) {
    CK(cudaMemsetAsync(P.lb_st.p, 0, sizeof(u64) * (size_t)P.lb_st.cap, s));
    CK(cudaMemsetAsync(P.lb_ctl.p, 0, sizeof(int32_t) * 256, s));
    P.lb_ep = 1;
  }
  return P.lb_ep;
}

LookBack look_back_begin(Prims& P, int64_t words, cudaStream_t s) {
  const uint32_t ep = lb_begin(P, words * LB_TILE, s);
  return LookBack{P.lb_st.p, P.lb_ctl.p + ep, ep, P.lb_ctl.p + 256};
}

// n items; the total goes to total_dev (device) when given.
template <class In>
static void scan_launch(In in, int64_t* out, int64_t n, int64_t* total_dev, Prims& P, cudaStream_t s) {
  if (n <= SC_TILE) {
    launch(k_scan_one<In>, 1, SC_THREADS, 0, s, in, out, n, total_dev);
    CKL("k_scan_one");
  } else {
    const uint32_t ep = lb_begin(P, n, s);
    const int64_t tiles = (n + LB_TILE - 1) / LB_TILE;
    launch(k_scan_lb<In>, (unsigned)tiles, SC_THREADS, 0, s, in, out, n, P.lb_st.p, P.lb_ctl.p + ep, ep, total_dev,
                                                         P.lb_ctl.p + 256);
    CKL("k_scan_lb");
  }
}

template <class T>
static int64_t scan_t(const T* in, int64_t* out, int64_t n, Prims& P, cudaStream_t s, bool want_total) {
  if (n <= 0) return 0;
  P.bsum.reserve(2, s);
  scan_launch(ArrayIn<T>{in}, out, n, P.bsum.p + 1, P, s);
  if (!want_total) return -1;
  int64_t tot = 0;
  const HostRead r{P.bsum.p + 1, &tot, sizeof(int64_t)};
  P.read(&r, 1, s);
  return tot;
}

int64_t scan_exclusive(const int64_t* in, int64_t* out, int64_t n, Prims& P, cudaStream_t s, bool want_total) {
  return scan_t<int64_t>(in, out, n, P, s, want_total);
}

int64_t scan_exclusive_i32(const int32_t* in, int64_t* out, int64_t n, Prims& P, cudaStream_t s, bool want_total) {
  return scan_t<int32_t>(in, out, n, P, s, want_total);
}

void scan_chunk_counts(const int32_t* list, const int32_t* nlist, int64_t n_hint, const int32_t* la,
                       const int32_t* lb, int32_t chunk, int64_t* out, Prims& P, cudaStream_t s) {
  const int tiles = div_up(n_hint + 1, CC_TPB);
  const LookBack q = look_back_begin(P, tiles, s);
  launch(k_scan_chunks, tiles, CC_TPB, 0, s, list, nlist, n_hint, la, lb, chunk, out, q);
  CKL("k_scan_chunks");
}

int32_t* scan_error_flag(Prims& P) { return P.lb_ctl.cap ? P.lb_ctl.p + 256 : nullptr; }

bool scan_wait_gives_up(cudaStream_t s) {
  // Two tiles; the tile counter starts at 1 and one block runs, so tile 1
  // waits on tile 0, which nothing publishes: the bounded wait must give up.
  Prims P;
  const int64_t n = 2 * LB_TILE;
  int32_t bad = 0;
  int64_t *in = nullptr, *out = nullptr;
  try {
    in = (int64_t*)dalloc(sizeof(int64_t) * (size_t)n);
    out = (int64_t*)dalloc(sizeof(int64_t) * (size_t)(n + 1));
    CK(cudaMemsetAsync(in, 0, sizeof(int64_t) * (size_t)n, s));
    const uint32_t ep = lb_begin(P, n, s);
    const int32_t one = 1;
    CK(cudaMemcpyAsync(P.lb_ctl.p + ep, &one, sizeof(int32_t), cudaMemcpyHostToDevice, s));
    launch(k_scan_lb<ArrayIn<int64_t>>, 1, SC_THREADS, 0, s, ArrayIn<int64_t>{in}, out, n, P.lb_st.p, P.lb_ctl.p + ep, ep,
                                                          out + n, P.lb_ctl.p + 256);
    CKL("k_scan_lb");
    CK(cudaMemcpyAsync(&bad, P.lb_ctl.p + 256, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
  } catch (...) {
    if (in) dfree(in);
    if (out) dfree(out);
    P.release();
    throw;
  }
  dfree(in);
  dfree(out);
  P.release();
  return bad != 0;
}

// The one-block sorts use 49 KB of shared memory: opted in once per device,
// thread and kernel.
static void small_smem_opt_in(const void* f) {
  static thread_local const void* done[2] = {nullptr, nullptr};
  static thread_local int done_dev = -1;
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (done_dev != dev) done[0] = done[1] = nullptr;
  done_dev = dev;
  if (done[0] == f || done[1] == f) return;
  CK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RsSmall)));
  done[done[0] ? 1 : 0] = f;
}

// Blocks of a sorting cluster: 16 where the device can place such a cluster
// (it is beyond the portable size), else 8.  Asked once per device and thread.
constexpr int CS_SMEM = 2 * CS_TILE * (int)sizeof(u64);
static int cluster_size() {
  static thread_local int size = 0, at_dev = -1;
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (at_dev == dev) return size;
  CK(cudaFuncSetAttribute(k_rs_cluster<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, CS_SMEM));
  CK(cudaFuncSetAttribute(k_rs_cluster<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, CS_SMEM));
  CK(cudaFuncSetAttribute(k_rs_cluster<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(CS_THREADS);
  cfg.dynamicSmemBytes = CS_SMEM;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 16;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k_rs_cluster<16>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    clusters = 0;
  }
  size = clusters > 0 ? 16 : 8;
  at_dev = dev;
  return size;
}

// Launches the sort of n pairs (an upper bound with x.n_dev).  A plain sort's
// result is in (keys, vals) afterwards, which may have been swapped with (tk,
// tv); a transposing one's lies behind its input.
static void sort_launch(u64*& keys, u64*& vals, u64*& tk, u64*& tv, int64_t n, int bits, Prims& P, cudaStream_t s,
                        int lo_bit, const RsExt& x) {
  const int cl = cluster_size();
  if (n <= (int64_t)cl * CS_TILE) {  // one cluster, the pairs kept on chip
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cl);
    cfg.blockDim = dim3(CS_THREADS);
    cfg.dynamicSmemBytes = CS_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    CK(cudaLaunchKernelEx(&cfg, cl == 16 ? k_rs_cluster<16> : k_rs_cluster<8>, keys, vals, (int)n, lo_bit, bits, x));
    CKL("k_rs_cluster");
    return;
  }
  const int64_t nb = (n + RS_TILE - 1) / RS_TILE;
  P.hist.reserve(std::max<int64_t>(256 * nb + 1, 128 * (int64_t)device_sms() + 1), s);
  P.bsum.reserve(256, s);
  // up to one tile per SM: one cooperative launch for all passes
  if (n <= (int64_t)device_sms() * CO_TILE) {
    static thread_local int co_attr_dev = -1;
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (co_attr_dev != dev) {
      CK(cudaFuncSetAttribute(k_rs_coop, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CoShared)));
      co_attr_dev = dev;
    }
    int64_t n_ = n;
    int lo_ = lo_bit, bits_ = bits;
    int32_t *gh = (int32_t*)P.hist.p, *dt = (int32_t*)P.bsum.p;
    RsExt x_ = x;
    void* args[] = {&keys, &vals, &tk, &tv, &n_, &lo_, &bits_, &gh, &dt, &x_};
    CK(cudaLaunchCooperativeKernel((const void*)k_rs_coop, dim3(device_sms()), dim3(CO_THREADS), args, sizeof(CoShared),
                                   s));
    CKL("k_rs_coop");
    if (!x.tbits)
      for (int shift = lo_bit; shift < bits; shift += 8) {  // where the result ended up
        u64* t = keys; keys = tk; tk = t;
        t = vals; vals = tv; tv = t;
      }
    return;
  }
  // three launches per pass; (place, behind its n pairs?) as in k_rs_coop
  struct Place {
    u64 *k, *v;
    int off;
  };
  Place in{keys, vals, 0}, out{tk, tv, 0}, nxt{keys, vals, 0};
  if (x.tbits) {
    nxt.off = 1;
    if (((bits - lo_bit + 7) / 8) & 1) std::swap(out, nxt);
  }
  for (int shift = lo_bit; shift < bits; shift += 8) {
    const int first = shift == lo_bit;
    launch(k_rs_hist, (unsigned)nb, RS_THREADS, 0, s, in.k, n, shift, nb, P.hist.p, x, first, in.off);
    CKL("k_rs_hist");
    launch(k_rs_dscan, 256, SC_THREADS, 0, s, P.hist.p, nb, P.bsum.p);
    CKL("k_rs_dscan");
    launch(k_rs_scatter, (unsigned)nb, RS_THREADS, 0, s, in.k, in.v, out.k, out.v, n, shift, nb, P.hist.p, P.bsum.p, x,
                                                     first, in.off, out.off);
    CKL("k_rs_scatter");
    in = out;
    std::swap(out, nxt);
    if (!x.tbits) {
      u64* t = keys; keys = tk; tk = t;
      t = vals; vals = tv; tv = t;
    }
  }
}

void radix_sort_pairs(u64*& keys, u64*& vals, u64*& tk, u64*& tv, int64_t n, int bits, Prims& P, cudaStream_t s,
                      int lo_bit, const int32_t* n_dev) {
  if (n <= 1 || bits <= lo_bit) return;
  if (n <= RS_TILE) {
    small_smem_opt_in((const void*)k_rs_small);
    launch(k_rs_small, 1, SM_THREADS, sizeof(RsSmall), s, keys, vals, (int)n, n_dev, lo_bit, bits);
    CKL("k_rs_small");
    return;
  }
  sort_launch(keys, vals, tk, tv, n, bits, P, s, lo_bit, RsExt{n_dev, 0, 0, nullptr});
}

void sort_reduce(DBuf<u64>& k, DBuf<u64>& v, DBuf<u64>& tk, DBuf<u64>& tv, int64_t n, const int32_t* n_dev, int bits,
                 bool both, int64_t row_off, u64* okeys, int64_t* ovals, int32_t* nr, Prims& P, cudaStream_t s) {
  if (n <= RS_TILE) {
    // one block sorts, sums and transposes: 4.3 us for a few records and 8.8
    // for some hundred, where the launches of the larger sizes take 16.4 and
    // 23.5 and the gaps between them
    small_smem_opt_in((const void*)k_rs_small_reduce);
    launch(k_rs_small_reduce, 1, SM_THREADS, sizeof(RsSmall), s, k.p, v.p, (int)n, n_dev, bits, both ? 1 : 0, row_off, okeys, ovals, nr);
    CKL("k_rs_small_reduce");
    return;
  }
  tk.reserve(n, s);
  tv.reserve(n, s);
  P.usum.reserve(n + 1, s);
  u64 *kp = k.p, *vp = v.p, *tkp = tk.p, *tvp = tv.p;
  // a segment crossing a run boundary is summed atomically into a slot the sort zeroes
  sort_launch(kp, vp, tkp, tvp, n, 2 * bits, P, s, 0, RsExt{n_dev, 0, 0, P.usum.p});
  if (kp != k.p) {
    swap_buf(k, tk);
    swap_buf(v, tv);
  }
  launch(k_segsum, grid_for((n + RBK_RUN - 1) / RBK_RUN, 256), 256, 0, s, k.p, v.p, n, n_dev, P.usum.p);
  CKL("k_segsum");
  const int tiles = div_up(n, LB_TILE);
  const LookBack q = look_back_begin(P, tiles, s);
  launch(k_reduce_out, tiles, SC_THREADS, 0, s, k.p, P.usum.p, n, n_dev, okeys, ovals, nr, nullptr, q);
  CKL("k_reduce_out");
  if (both) {
    // in (row, col) order already: a stable sort on the new row alone
    u64 *ok = okeys, *ov = (u64*)ovals, *t1 = tk.p, *t2 = tv.p;
    sort_launch(ok, ov, t1, t2, n, 2 * bits + 1, P, s, bits, RsExt{nr, bits, row_off, nullptr});
  }
}

int64_t reduce_by_key(const u64* keys, const u64* vals, int64_t n, u64* okeys, int64_t* ovals, Prims& P,
                      cudaStream_t s) {
  if (n <= 0) return 0;
  P.usum.reserve(n + 1, s);
  // a segment crossing a run boundary is summed atomically into a zeroed slot
  CK(cudaMemsetAsync(P.usum.p, 0, sizeof(int64_t) * (size_t)n, s));
  launch(k_segsum, grid_for((n + RBK_RUN - 1) / RBK_RUN, 256), 256, 0, s, keys, vals, n, nullptr, P.usum.p);
  CKL("k_segsum");
  const int tiles = div_up(n, LB_TILE);
  const LookBack q = look_back_begin(P, tiles, s);
  P.bsum.reserve(2, s);
  launch(k_reduce_out, tiles, SC_THREADS, 0, s, keys, P.usum.p, n, nullptr, okeys, ovals, nullptr, P.bsum.p, q);
  CKL("k_reduce_out");
  int64_t nz = 0;
  const HostRead r{P.bsum.p, &nz, sizeof(int64_t)};
  P.read(&r, 1, s);
  return nz;
}

