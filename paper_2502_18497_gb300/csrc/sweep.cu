// Frontier sweeps of Algorithm 1: candidate-set expansion (Expand, SPExpand),
// BestMove / BestRef with the exact Eq. 2 gain, the decoupling
// filter of Sec. III-E as deterministic parallel rounds, and the commit of an
// accepted mini-batch with the additive repair of the community totals and
// the exact modularity change dQ(B) with its rollback test.
#include <atomic>
#include <type_traits>
#include <cooperative_groups.h>

#include "chunks.cuh"
#include "kern.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int TPB = 256;
constexpr int HG8 = 64;      // hash slots per 8-lane group (lowest bin)
constexpr int HG32 = 256;    // hash slots per warp (second bin)
constexpr int HB = 4096;     // per-block hash slots (upper mid bin)
constexpr int MID_DEG = 2048;   // rows above it: clusters (optional) or the hub path
constexpr int CL = 8;             // blocks per cluster (hub rows up to CLUSTER_DEG entries)
constexpr int CL_SLOTS = 8192;    // hash slots per block of a cluster (96 KB of shared memory)
constexpr int CLUSTER_DEG = CL * CL_SLOTS / 2;  // upper limit of cluster_max_deg
constexpr int64_t HUB_TABLE_SLOTS = (int64_t)1 << 28;  // hub hash slots held at once (3 GB)
// the bound in force (a test hook lowers it)
std::atomic<int64_t> g_hub_table_slots{HUB_TABLE_SLOTS};
// the bin bounds a context may use keep every table at most half full
static_assert(BIN_MAX[0] == HG8 / 2 && BIN_MAX[1] == HG32 / 2 && BIN_MAX[2] == 2048 / 2 &&
                  BIN_MAX[3] == HB / 2 && BIN_MAX[3] == MID_DEG,
              "bin bounds and table sizes");
// Bound of the list up to which a sweep uses one kernel for all degrees (the
// bound the host has when it launches: in a level's first round the frontier and
// its row entries, later the number of vertices).  One edge on 10k vertices took
// 621 us a batch with a launch per bin, 531 with one; with 4096 here, batches of
// 100 to 1000 measure the same as with 1024 (within 1%).  The last bin bound
// still says which rows go to clusters or the hub path.
constexpr int SWEEP_FEW = 1024;
// The same bound up to which a sweep runs all four bins in one launch
// (k_sweep_bins), so that short bins fill one another's idle blocks instead of
// waiting for one another; with long bins the groups' own kernel pays with its 6
// blocks an SM to 4.  As later rounds are bounded by the vertex count, the line
// mostly tells graphs apart.  One launch for every sweep against a launch per
// bin, in batches of 10^2, 10^3 and 10^4:
//   vertices    R-MAT, 16 arcs a vertex    power law, 32 neighbours
//   150k        0.990 .. 0.993             0.944 .. 0.958
//   250k        0.989 .. 0.996             0.946 .. 0.972
//   400k        1.004 .. 1.020             0.956 .. 0.975
//   600k        1.036 .. 1.042             0.953 .. 0.986
//   900k        1.025 .. 1.036             0.976 .. 1.002
// (times as a share of the launch per bin's, 0.9 to 5.2 ms a batch, two runs of
// one side within 0.5% but for one pair of 2.4%); at 200k and 262k vertices, 20
// and 10^3 updates, planted graphs 0.957 .. 0.986, R-MATs of 8 and 32 neighbours
// 0.970 .. 0.998.  Below the line no graph loses.
constexpr int64_t SWEEP_FUSE = 262144;
// Hub entries per block of the accumulation (four chunks for its eight warps).
// The grid follows the tables' size, which is 2..4 slots an entry; with eight
// blocks per hub a few rows of 10^5 entries were walked by 64 warps each, one
// chunk after the other (batches on the 2M-vertex power-law graph: 10^5 updates
// 4473 -> 4417 us, 100 updates 1571 -> 1563 us; 2 * TPB here measures the same).
constexpr int HUB_ACC = 4 * TPB;
constexpr int EVAL_CH = 1024;  // hub table slots evaluated per block (4096: one block a hub, 17 us where this takes 16)

// ---------------------------------------------------------------- expand
// out = U plus every out- and in-neighbour of U (dedup by stamp).  A lane holds
// all its entries of a chunk: their ids, stamps and claims are in flight
// together, and one counter atomic appends the chunk's new nodes.  Bound by
// the latency of those three and the counter's atomics: one step of 32 entries
// after the other, each with its own atomic, took 148 us for a level-0
// expansion of a 10^4 batch on the R-MAT of 2^20, this form takes 77.
template <class WT>
__global__ void k_expand(Adj<WT> out, Adj<WT> in, ChunkMap m, int32_t* stamp, int32_t ep, int32_t* olist,
                         int32_t* nout, Tail tail) {
  pdl_enter();
  constexpr int PL = CH / 32;  // entries per lane
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    // both directions' rows lie in one pool
    const int64_t o = ch.row < 0 ? 0 : (ch.row ? in.off[ch.v] : out.off[ch.v]) + ch.k0;
    const int len = ch.k1 - ch.k0;
    int32_t u[PL];
    bool want[PL];
    bool self = ch.first && lane == 0 && stamp[ch.v] != ep;
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      want[j] = j * 32 + lane < len;
      u[j] = want[j] ? out.col[o + j * 32 + lane] : 0;
    }
#pragma unroll
    for (int j = 0; j < PL; ++j)
      if (want[j]) want[j] = stamp[u[j]] != ep;
#pragma unroll
    for (int j = 0; j < PL; ++j)
      if (want[j]) want[j] = atomicExch(&stamp[u[j]], ep) != ep;
    if (self) self = atomicExch(&stamp[ch.v], ep) != ep;
    unsigned mask[PL];
    int cnt = 0;
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      mask[j] = __ballot_sync(0xffffffffu, want[j]);
      cnt += __popc(mask[j]);
    }
    int32_t base = 0;
    if (lane == 0 && cnt + self) base = atomicAdd(nout, cnt + self);
    if (self) olist[base + cnt] = ch.v;
    base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      if (want[j]) olist[base + __popc(mask[j] & ((1u << lane) - 1u))] = u[j];
      base += __popc(mask[j]);
    }
  }
  pub_tail(tail);
}

// U = U* = the existing nodes of a frontier list (each listed once), and the
// entries of their rows (which bound the first candidate set).
__global__ void k_frontier(const int32_t* list, const int32_t* nlist, const uint8_t* alive, int32_t* lU, int32_t* nU,
                           int32_t* stU, int32_t epU, int32_t* lUs, int32_t* nUs, const int32_t* len_out,
                           const int32_t* len_in, int64_t* deg, Tail tail) {
  pdl_enter();
  const int32_t nl = *nlist;
  int64_t sum = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // warp-uniform trip counts, so that appends aggregate over the warp
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < nl; base += stride) {
    const int64_t t = base + (threadIdx.x & 31);
    const int32_t v = t < nl ? list[t] : 0;
    const bool on = t < nl && (!alive || alive[v]);
    if (on) {
      stU[v] = epU;
      sum += (int64_t)len_out[v] + (len_in ? len_in[v] : 0);
    }
    warp_append(on, v, lU, nU);
    warp_append(on, v, lUs, nUs);
  }
  sum = warp_sum_i64(sum);
  if ((threadIdx.x & 31) == 0 && sum) atomic_add_i64(deg, sum);
  pub_tail(tail);
}

__global__ void k_union(const int32_t* list, const int32_t* nlist, int32_t* stamp, int32_t ep, int32_t* olist,
                        int32_t* nout) {
  pdl_enter();
  const int32_t nl = *nlist;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nl; t += (int64_t)gridDim.x * blockDim.x)
    stamp_add(stamp, ep, list[t], olist, nout);
}

// ---------------------------------------------------------------- sweep
// MODE 0: BestMove over community labels.  MODE 1: BestRef over refined ids
// (level-r parents) restricted to neighbours of the same community.
template <class WT>
struct SweepArgs {
  Adj<WT> out, in;  // both directions' rows lie in one pool: out.col == in.col, out.w == in.w
  int directed;
  const int32_t* lab;
  const int32_t* par;
  const int64_t* kout;
  const int64_t* kin;
  const int64_t* Tout;  // MODE 0: community K_out; MODE 1: level r+1 k_out
  const int64_t* Tin;
  int64_t m, gn, gd;
  int32_t* cv;
  int32_t* csrc;
  int32_t* cdst;
  int64_t* cghi;
  uint64_t* cglo;
  int32_t* ncand;
  int64_t* scanned;
  DevScalars* stats;
};

// A node's shared-memory table: keys and the sums of their weights.  Shared
// memory has no native 64-bit add (it becomes a compare-and-swap loop that
// lanes with one key run through one after the other), so sums are kept in
// 32-bit words: one word when the gains fit int64 (then m < 2^30 and no sum
// of a node's in- and out-weights reaches 2^31), else a low and a high word
// with the carry passed on.  Both are exact.  Measured per level-0 sweep of a
// batch of 10^5 on the 2M-vertex power-law graph, 64-bit sums before: 128-
// thread blocks 873 -> 263 us, warps 781 -> 456 us, 8-lane groups 398 -> 198.
template <bool WIDE>
struct Tab {
  int32_t* K;
  uint32_t* lo;
  uint32_t* hi;  // WIDE only
  __device__ void clear4(uint32_t k) const {  // slots k .. k + 3, k a multiple of 4
    *(int4*)(K + k) = make_int4(-1, -1, -1, -1);
    *(uint4*)(lo + k) = make_uint4(0, 0, 0, 0);
    if (WIDE) *(uint4*)(hi + k) = make_uint4(0, 0, 0, 0);
  }
  __device__ void add(uint32_t mask, int32_t key, int64_t w) const {
    // the upper bits of a multiplicative hash (H = mask + 1 slots)
    uint32_t h = __umulhi((uint32_t)key * 0x9E3779B1u, mask + 1);
    while (true) {
      const int32_t prev = atomicCAS(&K[h], -1, key);
      if (prev == -1 || prev == key) break;
      h = (h + 1) & mask;
    }
    const uint32_t wl = (uint32_t)w;
    if (!WIDE) {
      atomicAdd(&lo[h], wl);
    } else {
      const uint32_t old = atomicAdd(&lo[h], wl);
      const uint32_t up = (uint32_t)((uint64_t)w >> 32) + (old + wl < old ? 1u : 0u);
      if (up) atomicAdd(&hi[h], up);
    }
  }
  __device__ int64_t sum(uint32_t h) const {
    return WIDE ? (int64_t)(((uint64_t)hi[h] << 32) | lo[h]) : (int64_t)lo[h];
  }
};

// slot bytes of a table in the gain type GT (int64: one-word sums)
template <class GT>
constexpr bool wide_sums = sizeof(GT) > 8;
// a staged entry weight: below m, so one word with one-word sums
template <class GT>
using StageW = std::conditional_t<wide_sums<GT>, int64_t, uint32_t>;
template <class GT>
constexpr int tab_slot = wide_sums<GT> ? 12 : 8;

// A node's row offsets and lengths, label and strengths, loaded one node
// ahead of its sweep so that these dependent loads overlap the previous
// node's work.
struct NodeMeta {
  int32_t v, a, lo, li;
  int64_t oo, oi, ko, ki;
};

template <class WT>
__device__ inline NodeMeta node_meta(const SweepArgs<WT>& A, int32_t v) {
  NodeMeta m;
  m.v = v;
  m.lo = A.out.len[v];
  m.oo = A.out.off[v];
  m.li = A.directed ? A.in.len[v] : 0;
  m.oi = A.directed ? A.in.off[v] : 0;
  m.a = A.lab[v];
  m.ko = A.kout[v];
  m.ki = A.kin[v];
  return m;
}

// Adds a node's entries (its out-row, then its in-row) to its table; weights
// towards its own community (MODE 0; most entries, once communities have
// formed) are summed in a register instead, as they would all meet in one
// slot.
template <class WT, int MODE, bool WIDE, bool DIR>
__device__ inline void accumulate(const SweepArgs<WT>& A, const NodeMeta& m, const Tab<WIDE>& T, uint32_t mask,
                                  int tid, int nthreads, std::conditional_t<WIDE, int64_t, uint32_t>& own) {
  // ACC entries per thread per step: their loads and label gathers are all in
  // flight before the first insert
  constexpr int ACC = 4;
  const int32_t l = DIR ? m.lo + m.li : m.lo;
  for (int32_t k0 = tid; k0 < l; k0 += ACC * nthreads) {
    int32_t u[ACC];
    std::conditional_t<WIDE, int64_t, uint32_t> w[ACC];
#pragma unroll
    for (int j = 0; j < ACC; ++j) {
      const int32_t k = k0 + j * nthreads;
      const int64_t at = (!DIR || k < m.lo ? m.oo : m.oi - m.lo) + k;
      u[j] = k < l ? A.out.col[at] : -1;
      w[j] = k < l ? A.out.w[at] : 0;
    }
    int32_t key[ACC];
#pragma unroll
    for (int j = 0; j < ACC; ++j) {
      key[j] = -1;
      if (u[j] >= 0 && u[j] != m.v && (MODE == 0 || A.lab[u[j]] == m.a)) key[j] = MODE == 0 ? A.lab[u[j]] : A.par[u[j]];
    }
#pragma unroll
    for (int j = 0; j < ACC; ++j) {
      if (MODE == 0 && key[j] == m.a) own += w[j];
      else if (key[j] >= 0) T.add(mask, key[j], w[j]);
    }
  }
}

// Exact gain of v into key (see Eq. 2 with a' = a \ {v}).
template <int MODE>
__device__ inline i128 gain_of(int32_t key, int64_t acc, int64_t wa, int32_t a, int64_t ko, int64_t ki,
                               const int64_t* Tout, const int64_t* Tin, int64_t m, int64_t gn, int64_t gd,
                               int64_t mult) {
  if (MODE == 0) {
    const i128 dw = (i128)mult * (acc - wa);
    const i128 dd = (i128)ko * (Tin[key] - Tin[a] + ki) + (i128)ki * (Tout[key] - Tout[a] + ko);
    return (i128)gd * m * dw - (i128)gn * dd;
  } else {
    const i128 dw = (i128)mult * acc;
    const i128 dd = (i128)ko * Tin[key] + (i128)ki * Tout[key];
    return (i128)gd * m * dw - (i128)gn * dd;
  }
}

// Algorithmic bytes of a sweep (the minimum a sweep must move): per adjacency
// entry the neighbour id, its weight and its label (refinement: also its
// parent); per swept node its offsets, lengths, label and strengths; per
// evaluated (node, target) pair the target's totals.
template <class WT, int MODE>
__device__ inline int64_t sweep_bytes(bool directed, int64_t entries, int64_t nodes, int64_t pairs) {
  const int64_t per_entry = 4 + sizeof(WT) + 4 + (MODE == 1 ? 4 : 0);
  const int64_t per_node = (8 + 4) * (directed ? 2 : 1) + 4 + 16 + 4;
  const int64_t per_pair = directed ? 16 : 8;
  return per_entry * entries + per_node * nodes + per_pair * pairs;
}

// The argmax (gain desc, target asc) in the gain's integer type GT: int64 when
// the host has checked that no gain or intermediate product of this sweep can
// reach 2^62 (sweep_gain_fits_i64), else int128.  Both give the same exact
// gains, so the choice never changes a result.
template <class GT>
struct BestG {
  GT g;
  int32_t c;
  int32_t have;
};

template <class GT>
__device__ inline bool better(const BestG<GT>& a, const BestG<GT>& b) {
  if (!a.have) return false;
  if (!b.have) return true;
  if (a.g != b.g) return a.g > b.g;
  return a.c < b.c;
}

__device__ inline int64_t shfl_down_g(int64_t v, int d, int w) { return __shfl_down_sync(0xffffffffu, v, d, w); }
__device__ inline i128 shfl_down_g(i128 v, int d, int w) { return shfl_down_i128_w(v, d, w); }
__device__ inline int64_t shfl_g(int64_t v, int src, int w) { return __shfl_sync(0xffffffffu, v, src, w); }
__device__ inline i128 shfl_g(i128 v, int src, int w) { return shfl_i128_w(v, src, w); }

// Argmax over each segment of G lanes (every lane takes part; the result
// lands in every lane of the segment).  G = 32: the whole warp.
template <class GT, int G>
__device__ inline BestG<GT> seg_best(BestG<GT> x) {
  for (int d = G / 2; d > 0; d >>= 1) {
    BestG<GT> o;
    o.g = shfl_down_g(x.g, d, G);
    o.c = __shfl_down_sync(0xffffffffu, x.c, d, G);
    o.have = __shfl_down_sync(0xffffffffu, x.have, d, G);
    if (better(o, x)) x = o;
  }
  x.g = shfl_g(x.g, 0, G);
  x.c = __shfl_sync(0xffffffffu, x.c, 0, G);
  x.have = __shfl_sync(0xffffffffu, x.have, 0, G);
  return x;
}

// Evaluates a node's table (H slots, a multiple of 4; thread `start` of
// `step`): the exact gain (gain_of, with what does not depend on the target
// collected in g0) into every target but `self`, the best kept in b.  Most
// slots are empty, so the keys are read four at a time; the occupied ones are
// emptied on the way, which leaves a clean table for the next node.  The terms
// may wrap in GT where the gain itself fits, hence the unsigned arithmetic.
template <int MODE, class GT, class CT>
__device__ inline void eval_slots(const Tab<wide_sums<GT>>& T, uint32_t H, uint32_t start, uint32_t step, int32_t self,
                                  int32_t a, int64_t wa, int64_t ko, int64_t ki, int directed, const int64_t* Tout,
                                  const int64_t* Tin, int64_t m, int64_t gn, int64_t gd, int64_t mult, BestG<GT>& b,
                                  CT& pairs) {
  using UT = std::conditional_t<(sizeof(GT) > 8), unsigned __int128, uint64_t>;
  const UT cw = (UT)(gd * mult) * (UT)m, co = (UT)gn * (UT)ko, ci = (UT)gn * (UT)ki;
  UT g0 = 0;
  if (MODE == 0) g0 = co * (UT)(GT)(Tin[a] - ki) + ci * (UT)(GT)(Tout[a] - ko) - cw * (UT)wa;
  for (uint32_t k0 = 4 * start; k0 < H; k0 += 4 * step) {
    const int4 kk = *(const int4*)(T.K + k0);
    const int32_t key[4] = {kk.x, kk.y, kk.z, kk.w};
    if ((key[0] & key[1] & key[2] & key[3]) == -1) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (key[j] < 0 || (MODE == 1 && key[j] == self)) continue;
      ++pairs;
      const UT ti = (UT)Tin[key[j]];
      const UT dd = directed ? co * ti + ci * (UT)Tout[key[j]] : (co + ci) * ti;
      const GT g = (GT)(g0 + cw * (UT)T.sum(k0 + j) - dd);
      if (g > 0) {
        BestG<GT> c{g, key[j], 1};
        if (better(c, b)) b = c;
      }
    }
    T.clear4(k0);
  }
}

template <class WT>
__device__ inline void emit_cand(const SweepArgs<WT>& A, int32_t v, int32_t src, const Best& b) {
  const int32_t p = atomicAdd(A.ncand, 1);
  A.cv[p] = v;
  A.csrc[p] = src;
  A.cdst[p] = b.c;
  A.cghi[p] = (int64_t)(b.g >> 64);
  A.cglo[p] = (uint64_t)b.g;
}

template <class WT, class GT>
__device__ inline void emit_cand(const SweepArgs<WT>& A, int32_t v, int32_t src, const BestG<GT>& b) {
  const int32_t p = atomicAdd(A.ncand, 1);
  A.cv[p] = v;
  A.csrc[p] = src;
  A.cdst[p] = b.c;
  A.cghi[p] = (int64_t)((i128)b.g >> 64);
  A.cglo[p] = (uint64_t)b.g;
}

// One group of G lanes per node with a group-private shared hash of
// HG8 slots (G = 8, the lowest degrees) or HG32 slots (G = 32, a warp per
// node).  All groups
// of a warp advance together, so the warp-wide shuffles of the argmax see
// every lane; a group without a node in an iteration only takes part in them.
// Bound by instructions and by the latency of the dependent loads (row
// bounds, entries, labels, totals).  Occupancy hides the latter best: staging
// the next node as the block kernel does (64 registers, 4 blocks a SM) took
// 681 us where this form took 456.  Fewer instructions then brought warps to
// 206 us and groups to 176 (2M-vertex power-law graph, batch of 10^5): one
// multiply to hash, the target-independent terms of the gain collected, keys
// read four at a time, no separate clearing, no argmax without a candidate.
// Sweeps list[0..nl) as block blk of gridDim.x blocks of TPB threads.  A warp's
// tables take the same GROUP_SMEM / (TPB / 32) bytes of smem for both G.
template <class GT>
constexpr int GROUP_SMEM = TPB / 32 * HG32 * tab_slot<GT>;
static_assert(HG32 == 4 * HG8 && TPB / 32 * HG32 <= HB);

template <class WT, int MODE, int G, class GT>
__device__ inline void sweep_groups(const SweepArgs<WT>& A, const int32_t* list, uint32_t nl, unsigned char* smem,
                                    uint32_t blk) {
  constexpr int HG = G == 8 ? HG8 : HG32;
  constexpr int GPW = 32 / G;  // groups per warp
  constexpr bool WIDE = wide_sums<GT>;
  const int lane = threadIdx.x & 31, gl = threadIdx.x & (G - 1);
  int32_t* const hk = (int32_t*)(smem + (size_t)(threadIdx.x / G) * HG * tab_slot<GT>);
  const Tab<WIDE> T{hk, (uint32_t*)hk + HG, WIDE ? (uint32_t*)hk + 2 * HG : nullptr};
  const uint32_t warp = blk * (TPB / 32) + threadIdx.x / 32;
  const uint32_t ngroups = gridDim.x * (TPB / G);
  const int64_t mult = A.directed ? 1 : 2;
  uint32_t entries = 0, pairs = 0, nodes = 0;
  // the list is read one node ahead, off the chain of dependent loads
  uint32_t t = warp * GPW + lane / G;
  int32_t v_next = t < nl ? list[t] : 0;
  for (uint32_t k = 4 * gl; k < HG; k += 4 * G) T.clear4(k);
  __syncwarp();
  for (uint32_t base = warp * GPW; base < nl; base += ngroups, t += ngroups) {
    const bool act = t < nl;
    const int32_t v = v_next;
    v_next = t + ngroups < nl ? list[t + ngroups] : 0;
    NodeMeta cur{};
    if (act) cur = node_meta(A, v);
    const int32_t deg = cur.lo + cur.li, a = cur.a;
    int H = G;
    while (H < 2 * deg && H < HG) H <<= 1;
    BestG<GT> b{0, 0, 0};
    StageW<GT> wa = 0;
    if (A.directed) accumulate<WT, MODE, WIDE, true>(A, cur, T, H - 1, gl, G, wa);
    else accumulate<WT, MODE, WIDE, false>(A, cur, T, H - 1, gl, G, wa);
    if (act && gl == 0) {
      entries += deg;
      ++nodes;
    }
    __syncwarp();
    if (MODE == 0) {
#pragma unroll
      for (int d = G / 2; d > 0; d >>= 1) wa += __shfl_xor_sync(0xffffffffu, wa, d, G);
    }
    if (act)
      eval_slots<MODE, GT>(T, (uint32_t)H, (uint32_t)gl, (uint32_t)G, MODE == 0 ? a : v, a, (int64_t)wa, cur.ko,
                           cur.ki, A.directed, A.Tout, A.Tin, A.m, A.gn, A.gd, mult, b, pairs);
    // most nodes stay where they are: no argmax without a positive gain
    if (__any_sync(0xffffffffu, b.have)) {
      b = seg_best<GT, G>(b);
      if (act && gl == 0 && b.have) emit_cand(A, v, MODE == 0 ? a : v, b);
    }
    __syncwarp();
  }
  const int64_t bytes = warp_sum_i64(sweep_bytes<WT, MODE>(A.directed, entries, nodes, pairs));
  const int64_t scanned = warp_sum_i64(entries);
  if (lane == 0 && (scanned | bytes)) {
    atomic_add_i64(A.scanned, scanned);
    atomic_add_i64(&A.stats->sw_entries[G == 32 ? 1 : 0], scanned);
    atomic_add_i64(&A.stats->sw_bytes[G == 32 ? 1 : 0], bytes);
  }
}

template <class WT, int MODE, int G, class GT>
__global__ void __launch_bounds__(TPB, wide_sums<GT> ? 4 : 6) k_sweep_group(SweepArgs<WT> A, const int32_t* list,
                                                                             const int32_t* nlist) {
  pdl_enter();
  __shared__ __align__(16) unsigned char smem[GROUP_SMEM<GT>];
  sweep_groups<WT, MODE, G, GT>(A, list, *nlist, smem, blockIdx.x);
}

// Barrier of a block of NT threads, or of half `bar` of a block of 2 * NT.
template <int NT>
__device__ inline void sub_sync(int bar) {
  if (NT == TPB) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(bar + 1), "r"(NT) : "memory");
}

// Entries of a node's rows staged in registers: entry k of the node is its
// out-row entry k (k < lo) or its in-row entry k - lo; thread tid holds the
// entries tid + j * NT.  First the neighbour ids and weights ...
// Steps in which a warp has no entry are skipped by the whole warp: most rows
// of a bin are far shorter than its longest.
template <class WT, int NT, bool DIR, int ACC, class SW>
__device__ inline void stage_rows(const SweepArgs<WT>& A, const NodeMeta& m, int tid, int32_t (&u)[ACC], SW (&w)[ACC]) {
  const int32_t l = DIR ? m.lo + m.li : m.lo, w0 = tid & ~31;
#pragma unroll
  for (int j = 0; j < ACC; ++j) {
    u[j] = -1;
    if (w0 + j * NT < l) {
      const int32_t k = tid + j * NT;
      const int64_t at = (!DIR || k < m.lo ? m.oo : m.oi - m.lo) + k;
      if (k < l) {
        u[j] = A.out.col[at];
        w[j] = (SW)A.out.w[at];
      }
    }
  }
}

template <class WT, int NT, int ACC, class SW>
__device__ inline void stage_rows(const SweepArgs<WT>& A, const NodeMeta& m, int tid, int32_t (&u)[ACC], SW (&w)[ACC]) {
  if (A.directed) stage_rows<WT, NT, true>(A, m, tid, u, w);
  else stage_rows<WT, NT, false>(A, m, tid, u, w);
}

// ... then each id becomes its hash key (neighbour label, or for BestRef the
// neighbour's refined community when it shares v's label; -1: skipped).
template <class WT, int MODE, int NT, int ACC>
__device__ inline void stage_keys(const SweepArgs<WT>& A, int32_t v, int32_t a, int32_t l, int tid, int32_t (&u)[ACC]) {
  const int32_t w0 = tid & ~31;
#pragma unroll
  for (int j = 0; j < ACC; ++j) {
    if (w0 + j * NT >= l) continue;  // the whole warp
    const int32_t x = u[j];
    int32_t key = -1;
    if (x >= 0 && x != v) {
      const int32_t lx = A.lab[x];
      if (MODE == 0) key = lx;
      else if (lx == a) key = A.par[x];
    }
    u[j] = key;
  }
}

// One block of NT threads per node (a row of up to HMAX/2 entries, hash table
// of up to HMAX slots in shared memory).  Software-pipelined over the block's
// nodes: the row entries and labels of the next node are loaded into
// registers while the current node's table is evaluated, and the node after
// that has its offsets, lengths and strengths loaded one node further ahead,
// so a node's fill only inserts into shared memory.  The bins' bounds keep every
// row within the HMAX / 2 staged entries.
// With the evaluation emptying the table, two barriers a node instead of
// four: 263 -> 215 us for the rows of 97..1024 entries of a 10^5 batch on the
// 2M-vertex power-law graph, 249 -> 214 us for 10^4 on the R-MAT of 2^20.
// The caller may reuse smem right away: nothing reads it after the last barrier.
template <class WT, int MODE, int NT, int HMAX, class GT>
__device__ inline void sweep_blocks(const SweepArgs<WT>& A, const int32_t* list, uint32_t nl, unsigned char* smem,
                                    int tid, int bar, uint32_t blk, uint32_t nblk) {
  constexpr bool WIDE = wide_sums<GT>;
  __shared__ BestG<GT> wb_[2][NT / 32];
  __shared__ int64_t wown_[2][NT / 32];
  BestG<GT>* const wb = wb_[bar];
  int64_t* const wown = wown_[bar];
  constexpr int ACC = HMAX / (2 * NT);
  const int lane = tid & 31, wid = tid >> 5;
  const Tab<WIDE> T{(int32_t*)smem, (uint32_t*)smem + HMAX, WIDE ? (uint32_t*)smem + 2 * HMAX : nullptr};
  const int64_t mult = A.directed ? 1 : 2;
  int64_t ent_all = 0, nodes = 0, pairs_all = 0;
  NodeMeta cur{}, nxt{};
  int32_t ek[ACC];
  StageW<GT> ew[ACC];
  if (blk < nl) {
    cur = node_meta(A, list[blk]);
    stage_rows<WT, NT>(A, cur, tid, ek, ew);
    stage_keys<WT, MODE, NT>(A, cur.v, cur.a, cur.lo + cur.li, tid, ek);
  }
  if (blk + nblk < nl) nxt = node_meta(A, list[blk + nblk]);
  if (blk < nl)
    for (uint32_t k = 4 * tid; k < HMAX; k += 4 * NT) T.clear4(k);
  sub_sync<NT>(bar);
  for (uint32_t t = blk; t < nl; t += nblk) {
    const int32_t v = cur.v;
    const int64_t d = (int64_t)cur.lo + cur.li;
    uint32_t H = 256;
    while (H < 2 * d && H < HMAX) H <<= 1;
    const int32_t a = cur.a;
    StageW<GT> own = 0;
#pragma unroll
    for (int j = 0; j < ACC; ++j) {
      if ((tid & ~31) + j * NT >= d) continue;  // the whole warp
      if (MODE == 0 && ek[j] == a) own += ew[j];
      else if (ek[j] >= 0) T.add(H - 1, ek[j], ew[j]);
    }
    if (MODE == 0) {
      if constexpr (WIDE) own = warp_sum_i64(own);
      else own = __reduce_add_sync(0xffffffffu, own);
      if (lane == 0) wown[wid] = own;
    }
    sub_sync<NT>(bar);
    const bool has_next = t + nblk < nl;
    if (has_next) stage_rows<WT, NT>(A, nxt, tid, ek, ew);  // in flight during the evaluation
    int64_t wa = 0;
    if (MODE == 0) {
#pragma unroll
      for (int w = 0; w < NT / 32; ++w) wa += wown[w];
    }
    const int64_t ko = cur.ko, ki = cur.ki;
    BestG<GT> b{0, 0, 0};
    int64_t pairs = 0;
    eval_slots<MODE, GT>(T, H, (uint32_t)tid, (uint32_t)NT, MODE == 0 ? a : v, a, wa, ko, ki, A.directed,
                         A.Tout, A.Tin, A.m, A.gn, A.gd, mult, b, pairs);
    if (has_next) stage_keys<WT, MODE, NT>(A, nxt.v, nxt.a, nxt.lo + nxt.li, tid, ek);  // label gathers overlap the argmax
    if (__any_sync(0xffffffffu, b.have)) b = seg_best<GT, 32>(b);
    if (lane == 0) wb[wid] = b;
    pairs_all += pairs;
    // two barriers a node: this one also separates the evaluation (which
    // empties the table) from the next node's inserts, and the next node's
    // barrier separates thread 0's reads of wb from their next writes
    sub_sync<NT>(bar);
    if (tid == 0) {
      BestG<GT> r = wb[0];
      for (int w = 1; w < NT / 32; ++w)
        if (better(wb[w], r)) r = wb[w];
      if (r.have) emit_cand(A, v, MODE == 0 ? a : v, r);
      ent_all += d;
      ++nodes;
    }
    cur = nxt;
    if (t + 2 * nblk < nl) nxt = node_meta(A, list[t + 2 * nblk]);
  }
  // statistics once per block
  const int64_t bytes = warp_sum_i64(sweep_bytes<WT, MODE>(A.directed, ent_all, nodes, pairs_all));
  if (lane == 0 && bytes) atomic_add_i64(&A.stats->sw_bytes[NT == 128 ? 2 : 3], bytes);
  if (tid == 0 && ent_all) {
    atomic_add_i64(A.scanned, ent_all);
    atomic_add_i64(&A.stats->sw_entries[NT == 128 ? 2 : 3], ent_all);
  }
}

template <class WT, int MODE, int NT, int HMAX, class GT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_sweep_block(SweepArgs<WT> A, const int32_t* list,
                                                               const int32_t* nlist) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem[];
  sweep_blocks<WT, MODE, NT, HMAX, GT>(A, list, *nlist, smem, threadIdx.x, 0, blockIdx.x, gridDim.x);
}

// The four bins in one launch (see SWEEP_FUSE), each going on at the block
// where the one before it ended, the longest nodes first; the two halves of a
// block sweep the nodes of the lower mid bin on their own (as nodes of whole
// blocks they cost the 2M-vertex power-law graph 10%).  Bound by the longest
// chain of dependent loads of any block.
template <class WT, int MODE, class GT>
__global__ void __launch_bounds__(TPB, 4) k_sweep_bins(SweepArgs<WT> A, const int32_t* bt, const int32_t* nt,
                                                       const int32_t* bs, const int32_t* ns, const int32_t* bm,
                                                       const int32_t* nm, const int32_t* bm2, const int32_t* nm2) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int HALF = TPB / 2;
  const int half = threadIdx.x / HALF;
  uint32_t blk = blockIdx.x;
  int32_t n = *nm2;
  sweep_blocks<WT, MODE, TPB, HB, GT>(A, bm2, n, smem, threadIdx.x, 0, blk, gridDim.x);
  // the next bin starts at the block after this one's last node
  const auto turn = [&](uint32_t used) { blk = (blk + gridDim.x - used % gridDim.x) % gridDim.x; };
  turn(n);
  n = *nm;
  sweep_blocks<WT, MODE, HALF, HB / 2, GT>(A, bm, n, smem + (size_t)half * (HB / 2) * tab_slot<GT>,
                                           threadIdx.x % HALF, half, 2 * blk + half, 2 * gridDim.x);
  // a warp's tables lie in its half's part of smem, which the other half may still be using
  unsigned char* const sw = smem + (size_t)half * (HB / 2 * tab_slot<GT> - GROUP_SMEM<GT> / 2);
  turn((uint32_t)(n + 1) / 2);
  n = *ns;
  sweep_groups<WT, MODE, 32, GT>(A, bs, n, sw, blk);
  turn((uint32_t)(n + TPB / 32 - 1) / (TPB / 32));
  __syncwarp();
  sweep_groups<WT, MODE, 8, GT>(A, bt, *nt, sw, blk);
}

template <class WT>
__global__ void k_bin(Adj<WT> out, Adj<WT> in, int directed, const int32_t* list, const int32_t* nlist,
                      int32_t* bt, int32_t* nt, int32_t* bs, int32_t* ns, int32_t* bm, int32_t* nm, int32_t* bm2,
                      int32_t* nm2, int32_t* bc, int32_t* nc, int32_t* bl, int32_t* nlarge, int64_t* lsz,
                      int64_t* tabtop, int32_t t0_, int32_t t1, int32_t t2, int32_t t3,
                      int32_t cluster_max, Tail tail) {
  pdl_enter();
  // BI nodes per thread and step; the block counts its bins in shared memory
  // and takes its places with one global atomic per bin and step.  (With one
  // per warp, bin and 32 nodes the counters bound it: 28 us for the level-0
  // candidates of a 10^5 batch on the 2M-vertex power-law graph, now 10.)
  constexpr int BI = 4;
  __shared__ int32_t cnt[5], base[5];
  int32_t* const lists[5] = {bt, bs, bm, bm2, bc};
  const int32_t nl = *nlist;
  const int64_t span = (int64_t)blockDim.x * BI;
  const int lane = threadIdx.x & 31;
  for (int64_t t0 = blockIdx.x * span; t0 < nl; t0 += gridDim.x * span) {
    if (threadIdx.x < 5) cnt[threadIdx.x] = 0;
    int32_t v[BI], at[BI];
    int bin[BI];
    int64_t d[BI];
#pragma unroll
    for (int j = 0; j < BI; ++j) {
      const int64_t t = t0 + j * blockDim.x + threadIdx.x;
      v[j] = t < nl ? list[t] : -1;
    }
#pragma unroll
    for (int j = 0; j < BI; ++j) {
      d[j] = v[j] >= 0 ? (int64_t)out.len[v[j]] + (directed ? in.len[v[j]] : 0) : 0;
      bin[j] = v[j] < 0 ? -1 : d[j] <= t0_ ? 0 : d[j] <= t1 ? 1 : d[j] <= t2 ? 2 : d[j] <= t3 ? 3
               : d[j] <= cluster_max ? 4 : 5;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < BI; ++j) {
      const unsigned peers = __match_any_sync(0xffffffffu, bin[j]);
      int32_t first = 0;
      if (bin[j] >= 0 && bin[j] < 5 && lane == __ffs(peers) - 1) first = atomicAdd(&cnt[bin[j]], __popc(peers));
      at[j] = __shfl_sync(0xffffffffu, first, __ffs(peers) - 1) + __popc(peers & ((1u << lane) - 1u));
    }
    __syncthreads();
    if (threadIdx.x < 5) {
      int32_t* const n5[5] = {nt, ns, nm, nm2, nc};
      if (cnt[threadIdx.x]) base[threadIdx.x] = atomicAdd(n5[threadIdx.x], cnt[threadIdx.x]);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < BI; ++j) {
      if (bin[j] < 0) continue;
      if (bin[j] < 5) {
        lists[bin[j]][base[bin[j]] + at[j]] = v[j];
        continue;
      }
      int64_t sz = 1;
      while (sz < 2 * d[j]) sz <<= 1;
      const int32_t p = atomicAdd(nlarge, 1);
      bl[p] = v[j];
      lsz[p] = sz;
      atomicAdd((unsigned long long*)tabtop, (unsigned long long)sz);
    }
    __syncthreads();  // cnt and base are reused by the next step
  }
  pub_tail(tail);
}

// ---------------------------------------------------------------- cluster bin
// One thread-block cluster of CL blocks per node of MID_DEG < degree <=
// CLUSTER_DEG.  The node's hash table of H slots (a power of two >= 2 *
// degree) is spread over the blocks' shared memories: slot h lives in block
// h / (H / CL) at h % (H / CL), and every thread of the cluster inserts into
// it with distributed-shared-memory atomics.  Each block then evaluates its
// own slots, and the blocks' bests meet in block 0.  Every thread of the
// cluster runs every iteration, so the cluster barriers always complete.
template <class WT, int MODE>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(TPB)
    k_sweep_cluster(SweepArgs<WT> A, const int32_t* list, const int32_t* nlist) {
  pdl_enter();
  extern __shared__ unsigned char smem[];
  int64_t* V = (int64_t*)smem;
  int32_t* K = (int32_t*)(smem + sizeof(int64_t) * CL_SLOTS);
  __shared__ Best wb[TPB / 32];
  __shared__ Best cbest[CL];
  __shared__ int64_t s_wa;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t cid = blockIdx.x / CL, ncl = gridDim.x / CL;
  const int32_t nl = *nlist;
  const int64_t mult = A.directed ? 1 : 2;
  int64_t ent_all = 0, nodes = 0, pairs_all = 0;
  for (int64_t t = cid; t < nl; t += ncl) {
    const int32_t v = list[t];
    const int64_t d = (int64_t)A.out.len[v] + (A.directed ? A.in.len[v] : 0);
    uint32_t H = CL * 64;
    while (H < 2 * d && H < (uint32_t)(CL * CL_SLOTS)) H <<= 1;
    const uint32_t HL = H / CL;
    for (uint32_t k = threadIdx.x; k < HL; k += TPB) {
      K[k] = -1;
      V[k] = 0;
    }
    cl.sync();
    const int32_t a = A.lab[v];
    for (int side = 0; side < (A.directed ? 2 : 1); ++side) {
      const Adj<WT>& adj = side ? A.in : A.out;
      const int64_t o = adj.off[v];
      const int32_t l = adj.len[v];
      // warp-uniform trip count: lanes with equal keys find their slot once
      // (one remote compare-and-swap probe by the lowest such lane), then
      // every lane adds its weight with a remote reduction
      for (int32_t base = rank * TPB + wid * 32; base < l; base += CL * TPB) {
        const int32_t k = base + lane;
        int32_t key = -1;
        int64_t w = 0;
        if (k < l) {
          const int32_t u = adj.col[o + k];
          if (u != v && (MODE == 0 || A.lab[u] == a)) {
            key = MODE == 0 ? A.lab[u] : A.par[u];
            w = (int64_t)adj.w[o + k];
          }
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        const int leader = __ffs(peers) - 1;
        uint32_t h = 0;
        if (key >= 0 && lane == leader) {
          h = hash32((uint32_t)key) & (H - 1);
          while (true) {
            const int32_t prev = atomicCAS(&cl.map_shared_rank(K, (int)(h / HL))[h % HL], -1, key);
            if (prev == -1 || prev == key) break;
            h = (h + 1) & (H - 1);
          }
        }
        h = __shfl_sync(0xffffffffu, h, leader);
        if (key >= 0)
          atomicAdd((unsigned long long*)&cl.map_shared_rank(V, (int)(h / HL))[h % HL], (unsigned long long)w);
      }
    }
    cl.sync();
    if (threadIdx.x == 0) {
      int64_t wa = 0;
      if (MODE == 0) {
        uint32_t h = hash32((uint32_t)a) & (H - 1);
        while (true) {
          const int32_t k = cl.map_shared_rank(K, (int)(h / HL))[h % HL];
          if (k == a) {
            wa = cl.map_shared_rank(V, (int)(h / HL))[h % HL];
            break;
          }
          if (k == -1) break;
          h = (h + 1) & (H - 1);
        }
      }
      s_wa = wa;
    }
    __syncthreads();
    const int64_t wa = s_wa;
    const int64_t ko = A.kout[v], ki = A.kin[v];
    Best b{0, 0, 0};
    for (uint32_t k = threadIdx.x; k < HL; k += TPB) {
      const int32_t key = K[k];
      if (key < 0) continue;
      if (MODE == 0 ? key == a : key == v) continue;
      ++pairs_all;
      const i128 g = gain_of<MODE>(key, V[k], wa, a, ko, ki, A.Tout, A.Tin, A.m, A.gn, A.gd, mult);
      if (g > 0) {
        Best c{g, key, 1};
        if (best_better(c, b)) b = c;
      }
    }
    b = warp_best(b);
    if (lane == 0) wb[wid] = b;
    __syncthreads();
    if (threadIdx.x == 0) {
      Best r = wb[0];
      for (int w = 1; w < TPB / 32; ++w)
        if (best_better(wb[w], r)) r = wb[w];
      cl.map_shared_rank(cbest, 0)[rank] = r;
    }
    cl.sync();
    if (rank == 0 && threadIdx.x == 0) {
      Best r = cbest[0];
      for (int q = 1; q < CL; ++q)
        if (best_better(cbest[q], r)) r = cbest[q];
      if (r.have) emit_cand(A, v, MODE == 0 ? a : v, r);
      ent_all += d;
      ++nodes;
    }
  }
  cl.sync();  // no block leaves while another may still touch its shared memory
  const int64_t bytes = warp_sum_i64(sweep_bytes<WT, MODE>(A.directed, ent_all, nodes, pairs_all));
  if (lane == 0 && bytes) atomic_add_i64(&A.stats->sw_bytes[4], bytes);
  if (threadIdx.x == 0 && ent_all) {
    atomic_add_i64(A.scanned, ent_all);
    atomic_add_i64(&A.stats->sw_entries[4], ent_all);
  }
}

// ---------------------------------------------------------------- hubs
// Hub rows are spread over the whole GPU: one global hash table per hub
// (a power of two >= 2 * degree), filled by chunks of its rows.  A probe that
// claims an empty slot appends it to the hub's slot list (at most degree
// entries, so hub i's list fits at loff[i] / 2), and only the listed slots are
// evaluated, in chunks whose partial bests are reduced per hub, and then
// cleared, so the tables stay clean between sweeps without a full re-fill.
__global__ void k_hub_init(int32_t* K, int64_t* V, int64_t total) {
  pdl_enter();
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    K[t] = -1;
    V[t] = 0;
  }
}

// Exclusive scan over nh hubs by one block: their table offsets (from the
// table sizes, clearing slot counts and own weights), or their evaluation chunks (from
// the slot counts, with the total behind the last).
__global__ void __launch_bounds__(1024) k_hub_scan(int32_t nh, const int64_t* lsz, int32_t* hcnt, int64_t* hown,
                                                   int64_t* out) {
  pdl_enter();
  int64_t o = 0;
  for (int32_t i0 = 0; i0 < nh; i0 += 1024) {
    const int32_t i = i0 + threadIdx.x;
    const int64_t x = i >= nh ? 0 : lsz ? lsz[i] : (hcnt[i] + EVAL_CH - 1) / EVAL_CH;
    u64 tot;
    const u64 ex = block_scan<1024>((u64)x, &tot);
    if (i < nh) {
      out[i] = o + (int64_t)ex;
      if (lsz) {
        hcnt[i] = 0;
        hown[i] = 0;
      }
    }
    o += (int64_t)tot;
  }
  if (threadIdx.x == 0 && !lsz) out[nh] = o;
}

// The hub of evaluation chunk e.
__device__ inline int64_t hub_of(const int64_t* epre, int32_t nh, int64_t e) {
  int64_t lo = 0, hi = nh;
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (epre[mid] <= e) lo = mid; else hi = mid;
  }
  return lo;
}

template <class WT, int MODE>
__global__ void k_hub_acc(SweepArgs<WT> A, ChunkMap m, const int64_t* loff, const int64_t* lsz, int32_t* gK,
                          int64_t* gV, int32_t* glist, int32_t* hcnt, int64_t* hown) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  int64_t scanned = 0;
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const int32_t v = ch.v;
    const int32_t cv_ = A.lab[v];
    int32_t* K = gK + loff[ch.idx];
    int64_t* V = gV + loff[ch.idx];
    const uint32_t mask = (uint32_t)lsz[ch.idx] - 1;
    const Adj<WT>& adj = ch.row ? A.in : A.out;
    const int64_t o = adj.off[v];
    // HL entries per lane with their labels in flight together (2 and 4 measure
    // alike: the table atomics set the pace); weight towards the hub's own
    // community (MODE 0) is summed in a register and added once a chunk, as all
    // of it would meet in one slot (level 0 of a 10^4 batch on the R-MAT of
    // 2^20: 149 -> 127 us)
    constexpr int HL = 2;
    int64_t own = 0;
    for (int32_t base = ch.k0; base < ch.k1; base += 32 * HL) {  // warp-uniform
      int32_t u[HL];
      WT wt[HL];
#pragma unroll
      for (int j = 0; j < HL; ++j) {
        const int32_t k = base + j * 32 + lane;
        u[j] = k < ch.k1 ? adj.col[o + k] : -1;
        wt[j] = k < ch.k1 ? adj.w[o + k] : 0;
      }
#pragma unroll
      for (int j = 0; j < HL; ++j) {
        int32_t key = -1;
        if (u[j] >= 0 && u[j] != v) {
          const int32_t l = A.lab[u[j]];
          if (MODE == 0) key = l;
          else if (l == cv_) key = A.par[u[j]];
        }
        u[j] = key;
      }
#pragma unroll
      for (int j = 0; j < HL; ++j) {
        if (base + j * 32 >= ch.k1) break;  // warp-uniform
        int32_t key = u[j];
        if (MODE == 0 && key == cv_) {
          own += wt[j];
          key = -1;
        }
        // lanes with equal keys: one probe by the lowest, then one reduction each
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        const int leader = __ffs(peers) - 1;
        uint32_t h = 0;
        bool fresh = false;
        if (key >= 0 && lane == leader) {
          h = hash32((uint32_t)key) & mask;
          while (true) {
            const int32_t prev = atomicCAS(&K[h], -1, key);
            if (prev == -1 || prev == key) {
              fresh = prev == -1;
              break;
            }
            h = (h + 1) & mask;
          }
        }
        // new keys of the warp (all of one hub) are listed with one counter atomic
        const unsigned fm = __ballot_sync(0xffffffffu, fresh);
        if (fm) {
          int32_t at = 0;
          if (lane == __ffs(fm) - 1) at = atomicAdd(&hcnt[ch.idx], __popc(fm));
          at = __shfl_sync(0xffffffffu, at, __ffs(fm) - 1);
          if (fresh) glist[loff[ch.idx] / 2 + at + __popc(fm & ((1u << lane) - 1u))] = (int32_t)h;
        }
        h = __shfl_sync(0xffffffffu, h, leader);
        if (key >= 0) atomicAdd((unsigned long long*)&V[h], (unsigned long long)(int64_t)wt[j]);
      }
    }
    if (MODE == 0) {
      own = warp_sum_i64(own);
      if (lane == 0 && own) atomic_add_i64(&hown[ch.idx], own);
    }
    if (lane == 0) scanned += ch.k1 - ch.k0;
  }
  if (lane == 0 && scanned) {
    atomic_add_i64(A.scanned, scanned);
    atomic_add_i64(&A.stats->sw_entries[5], scanned);
    atomic_add_i64(&A.stats->sw_bytes[5], sweep_bytes<WT, MODE>(A.directed, scanned, 0, 0));
  }
}

template <class WT, int MODE>
__global__ void __launch_bounds__(TPB) k_hub_eval(SweepArgs<WT> A, const int32_t* hubs, int32_t nh,
                                                  const int64_t* loff, const int64_t* epre,
                                                  const int32_t* gK, const int64_t* gV, const int32_t* glist,
                                                  const int32_t* hcnt, const int64_t* hown, int64_t* pb_hi, uint64_t* pb_lo,
                                                  int32_t* pb_c) {
  pdl_enter();
  __shared__ Best wb[TPB / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t mult = A.directed ? 1 : 2;
  const int64_t total = epre[nh];
  for (int64_t e = blockIdx.x; e < total; e += gridDim.x) {
    const int64_t i = hub_of(epre, nh, e);
    const int32_t v = hubs[i];
    const int32_t* K = gK + loff[i];
    const int64_t* V = gV + loff[i];
    const int64_t s0 = (e - epre[i]) * EVAL_CH;
    const int64_t s1 = min((int64_t)hcnt[i], s0 + EVAL_CH);
    const int32_t* Lst = glist + loff[i] / 2;
    const int32_t a = A.lab[v];
    const int64_t wa = MODE == 0 ? hown[i] : 0;
    const int64_t ko = A.kout[v], ki = A.kin[v];
    Best b{0, 0, 0};
    int64_t pairs = 0;
    for (int64_t j = s0 + threadIdx.x; j < s1; j += TPB) {
      const int32_t slot = Lst[j];
      const int32_t key = K[slot];
      if (MODE == 1 && key == v) continue;
      ++pairs;
      const i128 g = gain_of<MODE>(key, V[slot], wa, a, ko, ki, A.Tout, A.Tin, A.m, A.gn, A.gd, mult);
      if (g > 0) {
        Best c{g, key, 1};
        if (best_better(c, b)) b = c;
      }
    }
    b = warp_best(b);
    pairs = warp_sum_i64(pairs);
    if (lane == 0) {
      wb[wid] = b;
      if (pairs) atomic_add_i64(&A.stats->sw_bytes[6], sweep_bytes<WT, MODE>(A.directed, 0, 0, pairs));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      Best r = wb[0];
      for (int w = 1; w < TPB / 32; ++w)
        if (best_better(wb[w], r)) r = wb[w];
      pb_hi[e] = r.have ? (int64_t)(r.g >> 64) : 0;
      pb_lo[e] = r.have ? (uint64_t)r.g : 0;
      pb_c[e] = r.have ? r.c : -1;
    }
    __syncthreads();
  }
}

// The best of each hub's chunks, and the listed slots back to empty.
template <class WT, int MODE>
__global__ void k_hub_final(SweepArgs<WT> A, const int32_t* hubs, int32_t nh, const int64_t* loff,
                            const int64_t* epre, const int64_t* pb_hi, const uint64_t* pb_lo, const int32_t* pb_c,
                            const int32_t* hcnt, const int32_t* glist, int32_t* gK, int64_t* gV) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < nh; i += nw) {
    Best b{0, 0, 0};
    for (int64_t e = epre[i] + lane; e < epre[i + 1]; e += 32) {
      if (pb_c[e] < 0) continue;
      Best c{i128_of(pb_hi[e], pb_lo[e]), pb_c[e], 1};
      if (best_better(c, b)) b = c;
    }
    b = warp_best(b);
    if (lane == 0) {
      const int32_t v = hubs[i];
      atomic_add_i64(&A.stats->sw_bytes[6], sweep_bytes<WT, MODE>(A.directed, 0, 1, 0));
      if (b.have) emit_cand(A, v, MODE == 0 ? A.lab[v] : v, b);
    }
  }
  const int64_t total = epre[nh];
  for (int64_t e = blockIdx.x; e < total; e += gridDim.x) {
    const int64_t i = hub_of(epre, nh, e);
    const int64_t s0 = (e - epre[i]) * EVAL_CH, s1 = min((int64_t)hcnt[i], s0 + EVAL_CH);
    const int32_t* L = glist + loff[i] / 2;
    for (int64_t j = s0 + threadIdx.x; j < s1; j += blockDim.x) {
      const int64_t slot = loff[i] + L[j];
      gK[slot] = -1;
      gV[slot] = 0;
    }
  }
}

// ---------------------------------------------------------------- decouple
// Candidate i precedes j when its gain is larger, or equal with a smaller node.
__device__ inline bool precedes(const int64_t* ghi, const uint64_t* glo, const int32_t* cv, int32_t i, int32_t j) {
  const i128 gi = i128_of(ghi[i], glo[i]), gj = i128_of(ghi[j], glo[j]);
  if (gi != gj) return gi > gj;
  return cv[i] < cv[j];
}

__device__ inline void claim(int32_t* best, int32_t c, int32_t i, const int64_t* ghi, const uint64_t* glo,
                             const int32_t* cv) {
  int32_t cur = best[c];
  while (cur == -1 || precedes(ghi, glo, cv, i, cur)) {
    const int32_t old = atomicCAS(&best[c], cur, i);
    if (old == cur) return;
    cur = old;
  }
}

// A candidate is decided once every earlier candidate touching its source and
// its target is decided: either the community already has a role (set by its
// first accepted candidate, which precedes every undecided one) or this
// candidate is the earliest undecided one touching it.  A round: every
// undecided candidate claims its still role-free communities (CAS keeping the
// earliest), then the decidable ones are decided, then accepted candidates
// give their communities roles (emitter / acceptor) and the claims are reset.

// Whole decoupling filter in one cooperative launch when the candidates are
// many: the three phases of a round, one grid barrier after each, and the
// round counters alternate between two slots (the
// next round's slot is cleared while the current one is still being read).
// Every block reads the same count after the barrier, so all leave together;
// at most nc + 1 rounds (each decides the earliest undecided candidate).
constexpr int DG_TPB = 1024;
__global__ void __launch_bounds__(DG_TPB) k_dec_grid(int32_t nc, int32_t* cst, const int32_t* cv, const int32_t* src,
                                                  const int32_t* dst, const int64_t* ghi, const uint64_t* glo,
                                                  int32_t* role, int32_t* best, int32_t* bv, int32_t* bsrc,
                                                  int32_t* bdst, int32_t* nb, int32_t* undecided, int32_t* stat) {
  pdl_enter();
  cg::grid_group grid = cg::this_grid();
  const int32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  for (int32_t i = tid; i < nc; i += nth) cst[i] = 0;
  if (tid == 0) undecided[0] = undecided[1] = 0;
  grid.sync();
  int32_t rounds = 0;
  bool ok = true;
  for (;;) {
    const int par = rounds & 1;
    for (int32_t i = tid; i < nc; i += nth) {
      if (cst[i] != 0) continue;
      if (role[src[i]] == 0) claim(best, src[i], i, ghi, glo, cv);
      if (role[dst[i]] == 0) claim(best, dst[i], i, ghi, glo, cv);
    }
    grid.sync();
    int32_t left = 0;
    for (int32_t i = tid; i < nc; i += nth) {
      if (cst[i] != 0) continue;
      const int32_t ra = role[src[i]], rb = role[dst[i]];
      const bool da = ra != 0 || best[src[i]] == i;
      const bool db = rb != 0 || best[dst[i]] == i;
      if (da && db) cst[i] = (ra != 2 && rb != 1) ? 3 : 2;
      else ++left;
    }
    left = warp_sum_i32(left);
    if ((threadIdx.x & 31) == 0 && left) atomicAdd(&undecided[par], left);
    grid.sync();
    for (int32_t i = tid; i < nc; i += nth) {
      best[src[i]] = -1;
      best[dst[i]] = -1;
      if (cst[i] == 3) {
        role[src[i]] = 1;
        role[dst[i]] = 2;
        cst[i] = 1;
      }
    }
    if (tid == 0) undecided[par ^ 1] = 0;
    grid.sync();
    const int32_t l = *(volatile int32_t*)&undecided[par];
    ++rounds;
    if (l == 0) break;
    if (rounds > nc + 1) {
      ok = false;
      break;
    }
  }
  for (int32_t i = tid; i < nc; i += nth) {
    role[src[i]] = 0;
    role[dst[i]] = 0;
    if (cst[i] == 1) {
      const int32_t p = atomicAdd(nb, 1);
      bv[p] = cv[i];
      bsrc[p] = src[i];
      bdst[p] = dst[i];
    }
  }
  if (tid == 0) *stat = ok ? rounds : -1;
}

// Whole decoupling filter in one block when the candidates are few: the
// claim / decide / role phases of every round are separated by block
// barriers, and the loop ends when no candidate is undecided (at most one
// round per candidate, since every round decides the earliest undecided
// one).  *stat receives the number of rounds, or -1 if that bound was hit.
constexpr int DEC_SMALL = 8192;
constexpr int DEC_THREADS = 1024;

constexpr int DEC_PER = DEC_SMALL / DEC_THREADS;  // candidates per thread
static_assert(DEC_PER * DEC_THREADS == DEC_SMALL, "whole candidates per thread");
// the candidates' gains and nodes, staged in shared memory for the claims
constexpr size_t DEC_SMEM = (size_t)DEC_SMALL * (sizeof(int64_t) + sizeof(uint64_t) + sizeof(int32_t));

// The same rounds in one block for up to DEC_SMALL candidates: thread tid
// owns candidates tid + j * DEC_THREADS, whose communities and state stay in
// registers; the gains and nodes that claims compare sit in shared memory.
__global__ void __launch_bounds__(DEC_THREADS) k_dec_block(const int32_t* ncp, const int32_t* cv, const int32_t* src,
                                                           const int32_t* dst, const int64_t* ghi,
                                                           const uint64_t* glo, int32_t* role, int32_t* best,
                                                           int32_t* bv, int32_t* bsrc, int32_t* bdst, int32_t* nb,
                                                           int32_t* stat, Tail tail) {
  pdl_enter();
  extern __shared__ unsigned char dsm[];
  int64_t* sghi = (int64_t*)dsm;
  uint64_t* sglo = (uint64_t*)(dsm + sizeof(int64_t) * DEC_SMALL);
  int32_t* scv = (int32_t*)(dsm + (sizeof(int64_t) + sizeof(uint64_t)) * DEC_SMALL);
  __shared__ int32_t left;
  const int tid = threadIdx.x;
  const int32_t nc = *ncp;
  if (nc > DEC_SMALL || nc <= 0) {  // left to the multi-block rounds, or nothing to filter
    if (tid == 0) *stat = nc > 0 ? -2 : 0;
    pub_tail(tail);
    return;
  }
  // state per owned candidate: 0 undecided, 1 accepted, 2 rejected, 3 accepted
  // this round (roles pending), 4 no candidate
  int32_t sa[DEC_PER], sb[DEC_PER], st[DEC_PER];
#pragma unroll
  for (int j = 0; j < DEC_PER; ++j) {
    const int32_t i = tid + j * DEC_THREADS;
    const bool have = i < nc;
    st[j] = have ? 0 : 4;
    sa[j] = have ? src[i] : 0;
    sb[j] = have ? dst[i] : 0;
    if (have) {
      sghi[i] = ghi[i];
      sglo[i] = glo[i];
      scv[i] = cv[i];
    }
  }
  __syncthreads();
  int32_t rounds = 0;
  bool ok = true;
  for (;;) {
#pragma unroll
    for (int j = 0; j < DEC_PER; ++j) {
      if (st[j] != 0) continue;
      const int32_t i = tid + j * DEC_THREADS;
      if (role[sa[j]] == 0) claim(best, sa[j], i, sghi, sglo, scv);
      if (role[sb[j]] == 0) claim(best, sb[j], i, sghi, sglo, scv);
    }
    if (tid == 0) left = 0;
    __syncthreads();
    int32_t mine = 0;
#pragma unroll
    for (int j = 0; j < DEC_PER; ++j) {
      if (st[j] != 0) continue;
      const int32_t i = tid + j * DEC_THREADS;
      const int32_t ra = role[sa[j]], rb = role[sb[j]];
      const bool da = ra != 0 || best[sa[j]] == i;
      const bool db = rb != 0 || best[sb[j]] == i;
      if (da && db) st[j] = (ra != 2 && rb != 1) ? 3 : 2;
      else ++mine;
    }
    if (mine) atomicAdd(&left, mine);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < DEC_PER; ++j) {
      if (st[j] == 4) continue;
      best[sa[j]] = -1;
      best[sb[j]] = -1;
      if (st[j] == 3) {
        role[sa[j]] = 1;
        role[sb[j]] = 2;
        st[j] = 1;
      }
    }
    ++rounds;
    __syncthreads();
    const int32_t l = left;
    __syncthreads();  // every thread has read `left` before it is reset
    if (l == 0) break;
    if (rounds > nc + 1) {
      ok = false;
      break;
    }
  }
#pragma unroll
  for (int j = 0; j < DEC_PER; ++j) {
    if (st[j] == 4) continue;
    role[sa[j]] = 0;
    role[sb[j]] = 0;
    if (st[j] == 1) {
      const int32_t p = atomicAdd(nb, 1);
      bv[p] = scv[tid + j * DEC_THREADS];
      bsrc[p] = sa[j];
      bdst[p] = sb[j];
    }
  }
  if (tid == 0) *stat = ok ? rounds : -1;
  pub_tail(tail);
}

// ---------------------------------------------------------------- commit (move)
// Labels and marks of the accepted moves; a touched community is listed with
// its totals as they are (they change in k_commit_e).
__device__ inline void touch(int32_t c, int32_t* stT, int32_t epT, int32_t* lT, int32_t* nT, const int64_t* Kout,
                             const int64_t* Kin, const int64_t* e, int64_t* sko, int64_t* ski, int64_t* se) {
  if (!stamp_claim(stT, epT, c)) return;
  const int32_t k = atomicAdd(nT, 1);
  lT[k] = c;
  sko[k] = Kout[c];
  ski[k] = Kin[c];
  se[k] = e[c];
}

__global__ void k_commit_mark(int32_t nb, const int32_t* bv, const int32_t* bsrc, const int32_t* bdst,
                              int32_t* lab, int32_t* oldlab, int32_t* stB, int32_t epB, int32_t* stT, int32_t epT,
                              int32_t* lT, int32_t* nT, int32_t* stCh, int32_t epCh, int32_t* lCh, int32_t* nCh,
                              int32_t* lab_before, int level0, const int64_t* Kout, const int64_t* Kin,
                              const int64_t* e, int64_t* sko, int64_t* ski, int64_t* se) {
  pdl_enter();
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    const int32_t v = bv[i];
    oldlab[v] = bsrc[i];
    stB[v] = epB;
    if (level0 && stamp_add(stCh, epCh, v, lCh, nCh)) lab_before[v] = bsrc[i];
    lab[v] = bdst[i];
    touch(bsrc[i], stT, epT, lT, nT, Kout, Kin, e, sko, ski, se);
    touch(bdst[i], stT, epT, lT, nT, Kout, Kin, e, sko, ski, se);
  }
}

// Internal-weight repair: every arc with a moved endpoint is counted once
// (from the moved tail's out-row, or from the moved head's in-row when the
// tail did not move).  The same launch moves the nodes' strengths between the
// community totals.
template <class WT>
__global__ void k_commit_e(Adj<WT> out, Adj<WT> in, ChunkMap m, const int32_t* bsrc, const int32_t* bdst,
                           const int32_t* lab, const int32_t* oldlab, const int32_t* stB, int32_t epB, int64_t* e,
                           int32_t nb, const int32_t* bv, const int64_t* kout, const int64_t* kin, int64_t* Kout,
                           int64_t* Kin, int directed) {
  pdl_enter();
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    const int32_t v = bv[i];
    atomic_add_i64(&Kout[bsrc[i]], -kout[v]);
    atomic_add_i64(&Kout[bdst[i]], kout[v]);
    if (directed) {
      atomic_add_i64(&Kin[bsrc[i]], -kin[v]);
      atomic_add_i64(&Kin[bdst[i]], kin[v]);
    }
  }
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const int32_t a = bsrc[ch.idx], b = bdst[ch.idx];
    int64_t da = 0, db = 0;
    if (ch.row == 0) {
      const int64_t o = out.off[ch.v];
      for (int32_t k = ch.k0 + lane; k < ch.k1; k += 32) {
        const int32_t u = out.col[o + k];
        const int64_t w = (int64_t)out.w[o + k];
        const bool mu = stB[u] == epB;
        const int32_t cold = mu ? oldlab[u] : lab[u];
        const int32_t cnew = lab[u];
        if (cold == a) da -= w;
        if (cnew == b) db += w;
      }
    } else {
      const int64_t o = in.off[ch.v];
      for (int32_t k = ch.k0 + lane; k < ch.k1; k += 32) {
        const int32_t u = in.col[o + k];
        if (stB[u] == epB) continue;
        const int64_t w = (int64_t)in.w[o + k];
        const int32_t cu = lab[u];
        if (cu == a) da -= w;
        if (cu == b) db += w;
      }
    }
    da = warp_sum_i64(da);
    db = warp_sum_i64(db);
    if (lane == 0) {
      if (da) atomic_add_i64(&e[a], da);
      if (db) atomic_add_i64(&e[b], db);
    }
  }
}

// dQ(B) = sum over touched communities of gd*m*de_C - gn*d(K_out K_in).
__global__ void k_commit_dq(const int32_t* lT, const int32_t* nT, const int64_t* Kout, const int64_t* Kin,
                            const int64_t* e, const int64_t* sko, const int64_t* ski, const int64_t* se, int64_t m,
                            int64_t gn, int64_t gd, CommitAcc* sc) {
  pdl_enter();
  const int32_t n = *nT;
  i128 dq = 0, dp = 0;
  int64_t de = 0;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t c = lT[k];
    const int64_t dec = e[c] - se[k];
    const i128 dpc = (i128)Kout[c] * Kin[c] - (i128)sko[k] * ski[k];
    de += dec;
    dp += dpc;
    dq += (i128)gd * m * dec - (i128)gn * dpc;
  }
  dq = warp_sum_i128(dq);
  dp = warp_sum_i128(dp);
  de = warp_sum_i64(de);
  if ((threadIdx.x & 31) == 0) {
    atomic_add_i128(&sc->dq, dq);
    atomic_add_i128(&sc->dp, dp);
    if (de) atomic_add_i64(&sc->de, de);
  }
}

__global__ void k_rollback(int32_t nb, const int32_t* bv, const int32_t* bsrc, int32_t* lab, const int32_t* lT,
                           const int32_t* nT, int64_t* Kout, int64_t* Kin, int64_t* e, const int64_t* sko,
                           const int64_t* ski, const int64_t* se, int directed) {
  pdl_enter();
  const int32_t n = *nT;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) lab[bv[i]] = bsrc[i];
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t c = lT[k];
    Kout[c] = sko[k];
    if (directed) Kin[c] = ski[k];
    e[c] = se[k];
  }
}

// After a mini-batch that stays: its nodes are moved nodes of the level (and
// of the pass, on level 0), and the next U joins U*.
__global__ void k_mark_moved(int32_t nb, const int32_t* bv, int32_t* stMv, int32_t epMv, int32_t* lMv, int32_t* nMv,
                             int32_t* stM0, int32_t epM0, int32_t* lM0, int32_t* nM0, int32_t nU, const int32_t* lU,
                             int32_t* stU, int32_t epU, int32_t* lUs, int32_t* nUs) {
  pdl_enter();
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    stamp_add(stMv, epMv, bv[i], lMv, nMv);
    if (stM0) stamp_add(stM0, epM0, bv[i], lM0, nM0);
  }
  const int32_t stride = gridDim.x * blockDim.x;
  for (int32_t base = blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < nU; base += stride) {
    const int32_t t = base + (threadIdx.x & 31);
    const int32_t v = t < nU ? lU[t] : 0;
    warp_append(t < nU && stamp_claim(stU, epU, v), v, lUs, nUs);
  }
}

// ---------------------------------------------------------------- refine commit
__global__ void k_commit_ref(int32_t nb, const int32_t* bv, const int32_t* bdst, int32_t* par, const int64_t* kout,
                             const int64_t* kin, int64_t* kout1, int64_t* kin1, int32_t* cnt1, int directed) {
  pdl_enter();
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    const int32_t v = bv[i], X = bdst[i];
    par[v] = X;
    atomic_add_i64(&kout1[X], kout[v]);
    atomic_add_i64(&kout1[v], -kout[v]);
    if (directed) {
      atomic_add_i64(&kin1[X], kin[v]);
      atomic_add_i64(&kin1[v], -kin[v]);
    }
    atomicAdd(&cnt1[X], 1);
    atomicAdd(&cnt1[v], -1);
  }
}

// SPExpand: dissolved, still-singleton neighbours of moved nodes inside the
// moved node's community.
template <class WT>
__global__ void k_spexpand(Adj<WT> out, Adj<WT> in, ChunkMap m, const int32_t* lab, const int32_t* par,
                           const int32_t* cnt1, const int32_t* stD, int32_t epD, int32_t* stR, int32_t epR,
                           int32_t* lR, int32_t* nR) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const Adj<WT>& A = ch.row ? in : out;
    const int64_t o = A.off[ch.v];
    const int32_t cv_ = lab[ch.v];
    for (int32_t base = ch.k0; base < ch.k1; base += 32) {
      const int32_t k = base + lane;
      bool want = false;
      int32_t u = 0;
      if (k < ch.k1) {
        u = A.col[o + k];
        want = stD[u] == epD && lab[u] == cv_ && par[u] == u && cnt1[u] == 1 && stamp_claim(stR, epR, u);
      }
      warp_append(want, u, lR, nR);
    }
  }
}

}  // namespace

// ================================================================== host side

static void expand_tail(ldl_ctx& c, int r, const int32_t* list, int idx_n, int32_t* stamp, int32_t ep, int32_t* olist,
                        int idx_out, int64_t n_hint, const Tail& tail) {
  const int g = chunk_grid(n_hint);
  if (r == 0) {
    Adj<int32_t> o = adj_out0(c), i = adj_in0(c);
    ChunkMap m = chunk_map(c, list, c.cp[idx_n], n_hint, o.len, c.directed ? i.len : nullptr);
    launch(k_expand<int32_t>, g, TPB, 0, c.s, o, i, m, stamp, ep, olist, c.cp[idx_out], tail);
  } else {
    Adj<int64_t> o = adj_out(c, r), i = adj_in(c, r);
    ChunkMap m = chunk_map(c, list, c.cp[idx_n], n_hint, o.len, c.directed ? i.len : nullptr);
    launch(k_expand<int64_t>, g, TPB, 0, c.s, o, i, m, stamp, ep, olist, c.cp[idx_out], tail);
  }
  CKL("k_expand");
}

void expand_set(ldl_ctx& c, int r, const int32_t* list, int idx_n, int32_t* stamp, int32_t ep, int32_t* olist,
                int idx_out, int64_t n_hint) {
  if (n_hint <= 0) return;
  expand_tail(c, r, list, idx_n, stamp, ep, olist, idx_out, n_hint, Tail{});
}

void frontier(ldl_ctx& c, int r, int32_t epU, const Tail& tail) {
  LevelState& L = c.lv[r];
  const int32_t* lo = r == 0 ? adj_out0(c).len : adj_out(c, r).len;
  const int32_t* li = !c.directed ? nullptr : r == 0 ? adj_in0(c).len : adj_in(c, r).len;
  launch(k_frontier, grid_for(L.ubA, TPB, 2), TPB, 0, c.s, L.lA.p, c.cp[K_A0 + r], r ? L.alive.p : nullptr, c.lU.p,
                                                       c.cp[K_U], c.stU.p, epU, c.lUstar.p, c.cp[K_USTAR], lo, li,
                                                       c.sums, tail);
  CKL("k_frontier");
}

void union_into(ldl_ctx& c, const int32_t* list, int idx_n, int32_t* stamp, int32_t ep, int32_t* olist, int idx_out,
                int64_t n_hint) {
  launch(k_union, grid_for(n_hint, TPB), TPB, 0, c.s, list, c.cp[idx_n], stamp, ep, olist, c.cp[idx_out]);
  CKL("k_union");
}

// No exact gain of a sweep, nor any intermediate product of it, reaches 2^62
// when (2 gamma_den + 4 gamma_num) m^2 < 2^62: |w(v,.)| <= m, strengths and
// totals are at most m, so gd*m*|dw| <= 2 gd m^2 and gn*|dd| <= 4 gn m^2.
static bool sweep_gain_fits_i64(const ldl_ctx& c) {
  const i128 m = (i128)c.m;
  const i128 bound = (i128)(2 * (int64_t)c.prm.gamma_den + 4 * (int64_t)c.prm.gamma_num) * m * m;
  return bound < ((i128)1 << 62);
}

// The bins of nodes with at most 2048 entries, in the gain type GT.
template <class WT, int MODE, class GT>
static void sweep_bins(ldl_ctx& c, const SweepArgs<WT>& A, int64_t n_hint, bool few, bool fused, cudaEvent_t* kev) {
  if (fused) {
    const size_t sm = (size_t)tab_slot<GT> * HB;
    CK(cudaFuncSetAttribute(k_sweep_bins<WT, MODE, GT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    launch(k_sweep_bins<WT, MODE, GT>, grid_for(n_hint, 1, 4), TPB, sm, c.s, A, c.binT.p, c.cp[K_TINY], c.binS.p,
           c.cp[K_SMALL], c.binM.p, c.cp[K_MID], c.binM2.p, c.cp[K_MID2]);
    CKL("k_sweep_bins");
    return;
  }
  if (!few) {
    launch(k_sweep_group<WT, MODE, 8, GT>, grid_for(n_hint * 8, TPB, 6), TPB, 0, c.s, A, c.binT.p, c.cp[K_TINY]);
    CKL("k_sweep_group<8>");
    if (kev) CK(cudaEventRecord(kev[1], c.s));
    launch(k_sweep_group<WT, MODE, 32, GT>, grid_for(n_hint * 32, TPB, 6), TPB, 0, c.s, A, c.binS.p, c.cp[K_SMALL]);
    CKL("k_sweep_group<32>");
    if (kev) CK(cudaEventRecord(kev[2], c.s));
    const size_t sm = (size_t)tab_slot<GT> * (HB / 2);
    launch(k_sweep_block<WT, MODE, TPB / 2, HB / 2, GT>, grid_for(n_hint, 1, 16), TPB / 2, sm, c.s, A, c.binM.p,
           c.cp[K_MID]);
    CKL("k_sweep_block(mid1)");
    if (kev) CK(cudaEventRecord(kev[3], c.s));
  }
  {
    const size_t sm = (size_t)tab_slot<GT> * HB;
    CK(cudaFuncSetAttribute(k_sweep_block<WT, MODE, 256, HB, GT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            (int)sm));
    launch(k_sweep_block<WT, MODE, 256, HB, GT>, grid_for(n_hint, 1, 4), 256, sm, c.s, A, c.binM2.p, c.cp[K_MID2]);
    CKL("k_sweep_block(mid2)");
  }
}

// the next KS_EVENTS statistics events of the context, created on first use
static cudaEvent_t* kstats_events(ldl_ctx& c) {
  while (c.kev.size() < c.kev_used + KS_EVENTS) {
    cudaEvent_t e;
    CK(cudaEventCreate(&e));
    c.kev.push_back(e);
  }
  cudaEvent_t* e = c.kev.data() + c.kev_used;
  c.kev_used += KS_EVENTS;
  return e;
}

template <class WT, int MODE>
static SweepOut sweep_t(ldl_ctx& c, int r, Adj<WT> out, Adj<WT> in, const int32_t* list, int idx_n,
                        int64_t n_hint, SplitRun* spec) {
  if (MODE == 0) stage_begin(c);  // refinement is timed as a whole
  zero_cnt(c, K_CAND);
  zero_cnts(c, K_LARGE, N_BINS);
  c.sums = (int64_t*)fresh(c, 2, c.d_sc->sums);
  LevelState& L = c.lv[r];
  SweepArgs<WT> A;
  A.out = out;
  A.in = in;
  A.directed = c.directed;
  A.lab = L.lab.p;
  A.par = L.par.p;
  A.kout = L.kout.p;
  A.kin = kin_of(c, r);
  if (MODE == 0) {
    A.Tout = c.Kout.p;
    A.Tin = Kin_of(c);
  } else {
    A.Tout = c.lv[r + 1].kout.p;
    A.Tin = kin_of(c, r + 1);
  }
  A.m = c.m;
  A.gn = c.prm.gamma_num;
  A.gd = c.prm.gamma_den;
  A.cv = c.cv.p;
  A.csrc = c.csrc.p;
  A.cdst = c.cdst.p;
  A.cghi = c.cghi.p;
  A.cglo = c.cglo.p;
  A.ncand = c.cp[K_CAND];
  A.scanned = &c.d_sc->scanned;
  A.stats = c.d_sc;
  // the bins' sizes, the hub tables' size and the list's length in one read
  int32_t bins[N_BINS] = {0}, nlist = 0;
  const int32_t& ch = bins[0];
  int64_t tab = 0;
  const HostRead rb[3] = {{c.cp[K_LARGE], bins, sizeof(bins)},
                          {c.cp[idx_n], &nlist, sizeof(int32_t)},
                          {c.sums, &tab, sizeof(int64_t)}};
  // Hub rows need their tables' size on the host before they are swept.  Where
  // the last sweep of this level and mode had none, the filter is launched
  // straight behind the sweeps and one read returns its outcome and the hub
  // count; should there be hubs after all, they are swept and the filter,
  // which leaves its scratch as it found it, runs again on all candidates.
  uint8_t& expect = c.hubs_seen[r][MODE];
  // Few nodes are swept by one block each, up to the last bin bound: a launch
  // per degree bin costs more than it saves (see SWEEP_FEW).  Statistics are
  // kept per bin, so they take a launch per bin, but no other order of waits.
  const bool is_short = n_hint <= SWEEP_FEW;
  const bool few = is_short && !c.kstats;
  const bool fused = !is_short && n_hint <= SWEEP_FUSE && !c.kstats;
  // The split is only launched ahead behind such short sweeps: they mostly end
  // the level's moves, and where moves are accepted its two launches are lost
  // (one edge on 10k vertices 508 -> 486 us a batch; with it behind every sweep,
  // batches of 10^3 and more on the R-MAT graphs lost up to 1%).
  // While stages are timed, filter and split wait for the stage that is theirs.
  if (spec) spec->done = false;
  if (!is_short || c.timing) spec = nullptr;
  const bool early = expect || c.timing;
  launch(k_bin<WT>, grid_for(n_hint, TPB), TPB, 0, c.s, out, in, c.directed, list, c.cp[idx_n], c.binT.p, c.cp[K_TINY],
                                                     c.binS.p, c.cp[K_SMALL], c.binM.p, c.cp[K_MID], c.binM2.p,
                                                     c.cp[K_MID2], c.binC.p, c.cp[K_CLU], c.binL.p, c.cp[K_LARGE],
                                                     c.binLsz.p, c.sums, few ? -1 : c.bin_deg[0],
                                                     few ? -1 : c.bin_deg[1], few ? -1 : c.bin_deg[2],
                                                     c.bin_deg[3],
                                                     std::min(c.prm.cluster_max_deg, CLUSTER_DEG),
                                                     early ? tail_begin(c, rb, 3) : Tail{});
  CKL("k_bin");
  // Every bin but the hubs is swept by a grid-stride kernel that reads its
  // bin's count on the device, so these launch before the counts come back
  // and the host's wait below overlaps them.  n_hint bounds every bin.
  cudaEvent_t* kev = c.kstats ? kstats_events(c) : nullptr;
  if (kev) CK(cudaEventRecord(kev[0], c.s));
  if (sweep_gain_fits_i64(c)) sweep_bins<WT, MODE, int64_t>(c, A, n_hint, few, fused, kev);
  else sweep_bins<WT, MODE, i128>(c, A, n_hint, few, fused, kev);
  if (kev) CK(cudaEventRecord(kev[4], c.s));
  if (c.prm.cluster_max_deg > c.bin_deg[3]) {
    const size_t sm = (sizeof(int64_t) + sizeof(int32_t)) * CL_SLOTS;
    CK(cudaFuncSetAttribute(k_sweep_cluster<WT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    const int ncl = (int)std::min<int64_t>(n_hint, std::max(1, device_sms() * 2 / CL));
    launch(k_sweep_cluster<WT, MODE>, ncl * CL, TPB, sm, c.s, A, c.binC.p, c.cp[K_CLU]);
    CKL("k_sweep_cluster");
  }
  if (kev) CK(cudaEventRecord(kev[5], c.s));
  DecoupleOut dd{};
  if (early) tail_wait(c, rb, 3);
  else dd = decouple(c, rb, 3, spec, r, true);
  if (kev) CK(cudaEventRecord(kev[6], c.s));  // the wait above (and the filter) is charged to no kernel
  if (ch > 0) {
    // Hub tables hold 2..4 slots per entry.  When all hubs' tables together
    // exceed the slot budget (static builds of the largest graphs), the hubs
    // are swept in consecutive groups whose tables fit, reusing the space.
    std::vector<int32_t> gb{0, ch};
    int64_t tab_use = tab;
    const int64_t budget = g_hub_table_slots.load();
    if (tab > budget) {
      std::vector<int64_t> sz((size_t)ch);
      CK(cudaMemcpyAsync(sz.data(), c.binLsz.p, sizeof(int64_t) * (size_t)ch, cudaMemcpyDeviceToHost, c.s));
      CK(cudaStreamSynchronize(c.s));
      ++c.syncs;
      gb.assign(1, 0);
      int64_t acc = 0;
      tab_use = 0;
      for (int32_t h = 0; h < ch; ++h) {
        if (acc + sz[(size_t)h] > budget && h > gb.back()) {
          gb.push_back(h);
          tab_use = std::max(tab_use, acc);
          acc = 0;
        }
        acc += sz[(size_t)h];
      }
      gb.push_back(ch);
      tab_use = std::max(tab_use, acc);
    }
    c.gkeys.reserve(tab_use, c.s);
    c.gvals.reserve(tab_use, c.s);
    if (c.gtab_clean != c.gkeys.cap || c.gvals.cap != c.gkeys.cap) {  // fresh tables: fill once
      launch(k_hub_init, grid_for(c.gkeys.cap, TPB), TPB, 0, c.s, c.gkeys.p, c.gvals.p, c.gkeys.cap);
      CKL("k_hub_init");
      c.gtab_clean = c.gkeys.cap;
    }
    c.glist.reserve(tab_use / 2 + 1, c.s);
    c.hcnt.reserve(ch + 1, c.s);
    c.hown.reserve(ch + 1, c.s);
    c.hub_epre.reserve(ch + 2, c.s);
    const int64_t ech = tab_use / 2 / EVAL_CH + ch + 1;  // bounds the evaluation chunks of any group
    c.pb_hi.reserve(ech, c.s);
    c.pb_lo.reserve(ech, c.s);
    c.pb_c.reserve(ech, c.s);
    if (kev) CK(cudaEventRecord(kev[7], c.s));
    for (size_t gi = 0; gi + 1 < gb.size(); ++gi) {
      const int32_t g0 = gb[gi], nh = gb[gi + 1] - g0;
      const int32_t* L = c.binL.p + g0;
      int64_t* Lsz = c.binLsz.p + g0;
      int64_t* Loff = c.binLoff.p + g0;
      const int32_t* cntp = c.cp[K_LARGE];
      if (gb.size() > 2) {
        set_cnt(c, K_HUBG, nh);
        cntp = c.cp[K_HUBG];
      }
      launch(k_hub_scan, 1, 1024, 0, c.s, nh, Lsz, c.hcnt.p, c.hown.p, Loff);
      CKL("k_hub_scan");
      ChunkMap m = chunk_map(c, L, cntp, nh, out.len, c.directed ? in.len : nullptr);
      launch(k_hub_acc<WT, MODE>, grid_for(tab_use / 4, HUB_ACC, 16), TPB, 0, c.s,
          A, m, Loff, Lsz, c.gkeys.p, c.gvals.p, c.glist.p, c.hcnt.p, c.hown.p);
      CKL("k_hub_acc");
      if (kev && gi + 2 == gb.size()) CK(cudaEventRecord(kev[8], c.s));
      launch(k_hub_scan, 1, 1024, 0, c.s, nh, nullptr, c.hcnt.p, nullptr, c.hub_epre.p);
      CKL("k_hub_scan");
      const int ge = grid_for(ech, 1, 8);
      launch(k_hub_eval<WT, MODE>, ge, TPB, 0, c.s, A, L, nh, Loff, c.hub_epre.p, c.gkeys.p, c.gvals.p, c.glist.p, c.hcnt.p,
                                                c.hown.p, c.pb_hi.p, c.pb_lo.p, c.pb_c.p);
      CKL("k_hub_eval");
      launch(k_hub_final<WT, MODE>, std::max(ge, grid_for((int64_t)nh * 32, TPB)), TPB, 0, c.s,
          A, L, nh, Loff, c.hub_epre.p, c.pb_hi.p, c.pb_lo.p, c.pb_c.p, c.hcnt.p, c.glist.p, c.gkeys.p, c.gvals.p);
      CKL("k_hub_final");
    }
  } else if (kev) {
    CK(cudaEventRecord(kev[7], c.s));
    CK(cudaEventRecord(kev[8], c.s));
  }
  if (kev) {
    // times and bytes are resolved when the statistics are read, so that
    // collecting them adds no host synchronisation to the sweep
    CK(cudaEventRecord(kev[9], c.s));
    for (int k = 0; k < 5; ++k) c.ks_launch[k] += bins[1 + k] > 0;
    c.ks_launch[5] += ch > 0;
    c.ks_launch[6] += ch > 0 ? 2 : 0;  // evaluation, final reduction with the clearing
  }
  if (MODE == 0) stage_end(c, ST_BEST);
  expect = ch > 0;
  if (early || ch > 0) {
    if (MODE == 0) stage_begin(c);
    dd = decouple(c, nullptr, 0, spec, r, false);
    if (MODE == 0) stage_end(c, ST_DECOUPLE);
  }
  c.res.decouple_rounds += dd.rounds;
  return {nlist, dd.nc, dd.nb};
}

extern "C" void ldl_debug_hub_table_slots(int64_t slots) {
  g_hub_table_slots.store(slots > 0 ? slots : HUB_TABLE_SLOTS);
}

SweepOut sweep(ldl_ctx& c, int r, int mode, const int32_t* list, int idx_n, int64_t n_hint, SplitRun* spec) {
  if (r == 0) {
    if (mode == 0) return sweep_t<int32_t, 0>(c, r, adj_out0(c), adj_in0(c), list, idx_n, n_hint, spec);
    return sweep_t<int32_t, 1>(c, r, adj_out0(c), adj_in0(c), list, idx_n, n_hint, spec);
  }
  if (mode == 0) return sweep_t<int64_t, 0>(c, r, adj_out(c, r), adj_in(c, r), list, idx_n, n_hint, spec);
  return sweep_t<int64_t, 1>(c, r, adj_out(c, r), adj_in(c, r), list, idx_n, n_hint, spec);
}

DecoupleOut decouple(ldl_ctx& c, const HostRead* extra, int n_extra, SplitRun* spec, int r, bool hubs) {
  // The single-block filter runs first and reads the candidate count on the
  // device; one read then returns the count, the accepted number and the
  // filter's status (-2: too many candidates for one block).
  zero_cnt(c, K_B);
  int32_t nc = 0, nb = 0, stat = 0;
  HostRead rr[TAIL_MAX] = {{c.cp[K_CAND], &nc, sizeof(int32_t)}, {c.cp[K_B], &nb, sizeof(int32_t)},
                           {c.cp[K_UNDEC], &stat, sizeof(int32_t)}};
  for (int i = 0; i < n_extra; ++i) rr[3 + i] = extra[i];
  CK(cudaFuncSetAttribute(k_dec_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DEC_SMEM));
  launch(k_dec_block, 1, DEC_THREADS, DEC_SMEM, c.s, c.cp[K_CAND], c.cv.p, c.csrc.p, c.cdst.p, c.cghi.p, c.cglo.p,
                                                 c.role.p, c.best.p, c.bv.p, c.bsrc.p, c.bdst.p, c.cp[K_B],
                                                 c.cp[K_UNDEC], spec ? Tail{} : tail_begin(c, rr, 3 + n_extra));
  CKL("k_dec_block");
  if (spec) split_launch(c, r, *spec, true, hubs, rr, 3 + n_extra);
  tail_wait(c, rr, 3 + n_extra + (spec ? 2 : 0));
  // the gate's own test (the first extra value is the hub count)
  if (spec) spec->done = nb == 0 && stat != -2 && !(hubs && *(const int32_t*)extra[0].dst != 0);
  if (nc <= 0) return {0, 0, 0};
  if (stat != -2) {
    if (stat < 0) ldl_throw(LDL_E_INVALID, "internal: decoupling did not converge");
    return {nc, nb, stat};
  }
  // many candidates: one cooperative launch of co-resident blocks runs all rounds
  // (at most one large block per SM: the grid barriers, three a round, take
  // longer with more blocks)
  const int g = std::min(div_up(nc, DG_TPB), device_sms());
  zero_cnt(c, K_B);
  int32_t ncv = nc;
  int32_t* cst = c.cst.p;
  const int32_t *cvp = c.cv.p, *srcp = c.csrc.p, *dstp = c.cdst.p;
  const int64_t* ghi = c.cghi.p;
  const uint64_t* glo = c.cglo.p;
  int32_t *role = c.role.p, *best = c.best.p, *bv = c.bv.p, *bsrc = c.bsrc.p, *bdst = c.bdst.p;
  int32_t* nbp = c.cp[K_B];
  int32_t* undec = (int32_t*)fresh(c, 2, c.d_sc->home);  // the two round counters
  int32_t* statp = c.cp[K_UNDEC];
  void* args[] = {&ncv, &cst, &cvp, &srcp, &dstp, &ghi, &glo, &role, &best, &bv, &bsrc, &bdst, &nbp, &undec, &statp};
  CK(cudaLaunchCooperativeKernel((const void*)k_dec_grid, dim3(g), dim3(DG_TPB), args, 0, c.s));
  CKL("k_dec_grid");
  const HostRead rf[2] = {{c.cp[K_B], &nb, sizeof(int32_t)}, {c.cp[K_UNDEC], &stat, sizeof(int32_t)}};
  host_read(c, rf, 2);
  if (stat < 0) ldl_throw(LDL_E_INVALID, "internal: decoupling did not converge");
  return {nc, nb, stat};
}

void commit_move(ldl_ctx& c, int r, int32_t nb, int32_t epB, int32_t epT, int32_t epCh) {
  LevelState& L = c.lv[r];
  const int g = grid_for(nb, TPB);
  zero_cnt(c, K_T);
  c.acc = (CommitAcc*)fresh(c, sizeof(CommitAcc) / 4, c.d_sc->home);
  launch(k_commit_mark, g, TPB, 0, c.s, nb, c.bv.p, c.bsrc.p, c.bdst.p, L.lab.p, c.oldlab.p, c.stB.p, epB, c.stT.p, epT,
                                    c.lT.p, c.cp[K_T], c.stCh.p, epCh, c.lCh.p, c.cp[K_CH], c.lab_before.p, r == 0,
                                    c.Kout.p, Kin_of(c), c.e.p, c.snapKo.p, c.snapKi.p, c.snapE.p);
  CKL("k_commit_mark");
  const int gw = chunk_grid(nb);
  if (r == 0) {
    Adj<int32_t> o = adj_out0(c), i = adj_in0(c);
    ChunkMap m = chunk_map(c, c.bv.p, c.cp[K_B], nb, o.len, i.len);
    launch(k_commit_e<int32_t>, gw, TPB, 0, c.s, o, i, m, c.bsrc.p, c.bdst.p, L.lab.p, c.oldlab.p, c.stB.p, epB, c.e.p, nb,
                                          c.bv.p, L.kout.p, kin_of(c, r), c.Kout.p, Kin_of(c), c.directed);
  } else {
    Adj<int64_t> o = adj_out(c, r), i = adj_in(c, r);
    ChunkMap m = chunk_map(c, c.bv.p, c.cp[K_B], nb, o.len, i.len);
    launch(k_commit_e<int64_t>, gw, TPB, 0, c.s, o, i, m, c.bsrc.p, c.bdst.p, L.lab.p, c.oldlab.p, c.stB.p, epB, c.e.p, nb,
                                          c.bv.p, L.kout.p, kin_of(c, r), c.Kout.p, Kin_of(c), c.directed);
  }
  CKL("k_commit_e");
  launch(k_commit_dq, grid_for(2 * (int64_t)nb, TPB), TPB, 0, c.s, c.lT.p, c.cp[K_T], c.Kout.p, Kin_of(c), c.e.p,
                                                               c.snapKo.p, c.snapKi.p, c.snapE.p, c.m,
                                                               c.prm.gamma_num, c.prm.gamma_den, c.acc);
  CKL("k_commit_dq");
}

CommitOut commit_expand(ldl_ctx& c, int r, int32_t nb, int32_t ep, int32_t* nU) {
  CommitOut o;
  CommitAcc a{};
  const HostRead rr[3] = {{c.acc, &a, sizeof(a)}, {c.cp[K_T], &o.ntc, sizeof(int32_t)}, {c.cp[K_U], nU, sizeof(int32_t)}};
  expand_tail(c, r, c.bv.p, K_B, c.stS.p, ep, c.lU.p, K_U, nb, tail_begin(c, rr, 3));
  tail_wait(c, rr, 3);
  o.dq = i128_of(a.dq.hi, a.dq.lo);
  o.dp = i128_of(a.dp.hi, a.dp.lo);
  o.de = a.de;
  return o;
}

void rollback_move(ldl_ctx& c, int r, int32_t nb, int32_t ntc) {
  LevelState& L = c.lv[r];
  const int64_t m = nb > ntc ? nb : ntc;
  launch(k_rollback, grid_for(m, TPB), TPB, 0, c.s, nb, c.bv.p, c.bsrc.p, L.lab.p, c.lT.p, c.cp[K_T], c.Kout.p,
                                                Kin_of(c), c.e.p, c.snapKo.p, c.snapKi.p, c.snapE.p, c.directed);
  CKL("k_rollback");
}

void mark_moved(ldl_ctx& c, int r, int32_t nb, int32_t epMv, int32_t epM0, int32_t epU, int32_t nU) {
  c.ubU = std::min<int64_t>(c.n, c.ubU + nU);
  launch(k_mark_moved, grid_for(std::max(nb, nU), TPB), TPB, 0, c.s,
      nb, c.bv.p, c.stMv.p, epMv, c.lMv.p, c.cp[K_MV], r == 0 ? c.stM0.p : nullptr, epM0, c.lM0.p, c.cp[K_M0], nU,
      c.lU.p, c.stU.p, epU, c.lUstar.p, c.cp[K_USTAR]);
  CKL("k_mark_moved");
}

void commit_ref(ldl_ctx& c, int r, int32_t nb) {
  LevelState& L = c.lv[r];
  LevelState& N = c.lv[r + 1];
  launch(k_commit_ref, grid_for(nb, TPB), TPB, 0, c.s, nb, c.bv.p, c.bdst.p, L.par.p, L.kout.p, kin_of(c, r), N.kout.p,
                                                   kin_of(c, r + 1), N.cnt.p, c.directed);
  CKL("k_commit_ref");
}

void spexpand(ldl_ctx& c, int r, int32_t nb, int32_t epD, int32_t epR, int32_t* lR, int idx_R) {
  LevelState& L = c.lv[r];
  const int g = chunk_grid(nb);
  if (r == 0) {
    Adj<int32_t> o = adj_out0(c), i = adj_in0(c);
    ChunkMap m = chunk_map(c, c.bv.p, c.cp[K_B], nb, o.len, c.directed ? i.len : nullptr);
    launch(k_spexpand<int32_t>, g, TPB, 0, c.s, o, i, m, L.lab.p, L.par.p, c.lv[r + 1].cnt.p, c.stD.p, epD, c.stR.p,
                                            epR, lR, c.cp[idx_R]);
  } else {
    Adj<int64_t> o = adj_out(c, r), i = adj_in(c, r);
    ChunkMap m = chunk_map(c, c.bv.p, c.cp[K_B], nb, o.len, c.directed ? i.len : nullptr);
    launch(k_spexpand<int64_t>, g, TPB, 0, c.s, o, i, m, L.lab.p, L.par.p, c.lv[r + 1].cnt.p, c.stD.p, epD, c.stR.p,
                                            epR, lR, c.cp[idx_R]);
  }
  CKL("k_spexpand");
}
