// Hierarchy maintenance of Algorithm 1: batch ingest and validation (the
// batch's application to level 0), statistic repair along the parent chain
// and InitFrontier, label push-down after supernode moves, the refined-community
// split of TouchedRefined, and the Eq. 3 subtract-add aggregate repair with
// NextFrontier.
#include "chunks.cuh"
#include "kern.cuh"

namespace {

constexpr int TPB = 256;

#define GRID_STRIDE(i, n) \
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

// ---------------------------------------------------------------- ingest
__device__ inline void set_err(unsigned long long* err, int64_t idx, int code) {
  atomicMin(err, ((unsigned long long)idx << 8) | (unsigned long long)code);
}

// Start of a batch: every counter, and the scalars that ingest adds to.
__global__ void k_batch_begin(int32_t* dcnt, int32_t* arena, DevScalars* sc) {
  pdl_enter();
  const int t = threadIdx.x;
  if (t < K_COUNT) dcnt[t] = 0;
  for (int i = t; i < ARENA_WORDS / 4; i += blockDim.x) ((int4*)arena)[i] = make_int4(0, 0, 0, 0);
  if (t == 0) {
    sc->scanned = 0;
    sc->dm = 0;
    sc->agg_recs = 0;
    sc->err_key = -1;
    sc->err_seq = -1;
  }
}

// Checks each update by itself and makes its edge key (an update that fails
// gets key 0: the batch is rejected before anything uses it).
__global__ void k_upd_keys(const ldl_update* u, int64_t cnt, int64_t n, int bits, int directed, u64* keys, u64* vals,
                           unsigned long long* err) {
  pdl_enter();
  GRID_STRIDE(i, cnt) {
    const ldl_update x = u[i];
    int code = 0;
    if (x.src < 0 || x.src >= n || x.dst < 0 || x.dst >= n) code = LDL_E_RANGE;
    else if (x.op != LDL_INSERT && x.op != LDL_DELETE && x.op != LDL_REWEIGHT) code = LDL_E_INVALID;
    else if (x.op == LDL_INSERT && x.w < 1) code = LDL_E_INVALID;
    else if (x.op == LDL_REWEIGHT && x.w < 0) code = LDL_E_NEG_WEIGHT;
    int64_t a = x.src, b = x.dst;
    if (code) {
      set_err(err, i, code);
      a = b = 0;
    }
    if (!directed && a > b) {
      int64_t t = a; a = b; b = t;
    }
    keys[i] = ((u64)a << bits) | (u64)b;
    vals[i] = (u64)i;
  }
}

// The distinct keys of a sorted list and where each starts, in one pass with
// look-back (their number in *nu).
constexpr int UQ_TPB = 512;
__global__ void __launch_bounds__(UQ_TPB) k_unique(const u64* keys, int64_t n, u64* ukeys, int64_t* ustart,
                                                   int32_t* nu, LookBack q) {
  pdl_enter();
  __shared__ int64_t s_tile, s_pre;
  if (threadIdx.x == 0) s_tile = atomicAdd(q.ctr, 1);
  __syncthreads();
  const int64_t tile = s_tile, i = tile * UQ_TPB + threadIdx.x;
  const u64 k = i < n ? keys[i] : 0;
  const bool head = i < n && (i == 0 || keys[i - 1] != k);
  u64 tot;
  const u64 ex = block_scan<UQ_TPB>(head ? 1 : 0, &tot);
  if (threadIdx.x < 32) {
    const int64_t agg[1] = {(int64_t)tot};
    int64_t pre[1];
    look_back<1>(q.st, tile, agg, pre, q.ep, q.err);
    if (threadIdx.x == 0) {
      s_pre = pre[0];
      if ((tile + 1) * UQ_TPB >= n) *nu = (int32_t)(pre[0] + agg[0]);
    }
  }
  __syncthreads();
  if (head) {
    ukeys[s_pre + (int64_t)ex] = k;
    ustart[s_pre + (int64_t)ex] = i;
  }
}

// Per distinct edge: its current weight, its updates in array order on top,
// and the arcs whose weight changes (an undirected edge's mirror too).
__global__ void k_seq(const ldl_update* u, int64_t cnt, const u64* vals, const int64_t* ustart, const int32_t* nup,
                      const u64* ukeys, const int64_t* off, const int32_t* len, const int32_t* col, const int32_t* wt,
                      int bits, int directed, unsigned long long* err, int64_t* dm, u64* ok, u64* ov, int32_t* na) {
  pdl_enter();
  const int64_t nu = *nup, stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  int64_t total = 0;
  // warp-uniform trip counts: one counter atomic per warp and step (one per
  // edge took 108 us for 10^5 updates, this 11)
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; base < nu; base += stride) {
    const int64_t k = base + lane;
    int64_t d = 0;
    u64 key = 0, a = 0, b = 0;
    if (k < nu) {
      const int64_t s = ustart[k], e = (k + 1 < nu) ? ustart[k + 1] : cnt;
      key = ukeys[k];
      a = key >> bits;
      b = key & ((((u64)1) << bits) - 1);
      const int64_t o = off[a];
      const int32_t l = len[a];
      const int32_t at = row_lower_bound(col, o, l, (int32_t)b);
      const int64_t w0 = at < l && col[o + at] == (int32_t)b ? wt[o + at] : 0;
      int64_t cur = w0;
      for (int64_t t = s; t < e; ++t) {
        const int64_t idx = (int64_t)vals[t];
        const ldl_update x = u[idx];
        int bad = 0;
        if (x.op == LDL_INSERT) {
          cur += x.w;
          if (cur > INT32_MAX) bad = LDL_E_OVERFLOW;
        } else if (x.op == LDL_DELETE) {
          if (cur == 0) bad = LDL_E_NO_EDGE;
          cur = 0;
        } else {
          if (cur == 0) bad = LDL_E_NO_EDGE;
          cur = x.w;
        }
        if (bad) {
          set_err(err, idx, bad);
          cur = w0;
          break;
        }
      }
      d = cur - w0;
    }
    const bool two = d && !directed && a != b;
    total += two ? 2 * d : d;
    const unsigned m1 = __ballot_sync(0xffffffffu, d != 0), m2 = __ballot_sync(0xffffffffu, two);
    int32_t p = 0;
    if (lane == 0 && m1) p = atomicAdd(na, __popc(m1) + __popc(m2));
    p = __shfl_sync(0xffffffffu, p, 0);
    if (d) {
      const unsigned lt = (1u << lane) - 1u;
      p += __popc(m1 & lt) + __popc(m2 & lt);
      ok[p] = key;
      ov[p] = (u64)d;
      if (two) {
        ok[p + 1] = (b << bits) | a;
        ov[p + 1] = (u64)d;
      }
    }
  }
  total = warp_sum_i64(total);
  if (lane == 0 && total) atomic_add_i64(dm, total);
}

// (row, col) -> (col + row_off, row): the in-direction records of a level
// whose in-rows live at row_off (directed graphs keep both in one CSR).
__global__ void k_transpose(const u64* k, const u64* v, int64_t n, int bits, u64* ok, u64* ov, int64_t row_off) {
  pdl_enter();
  const u64 mask = (((u64)1) << bits) - 1;
  GRID_STRIDE(i, n) {
    ok[i] = (((k[i] & mask) + (u64)row_off) << bits) | (k[i] >> bits);
    ov[i] = v[i];
  }
}

// ---------------------------------------------------------------- repair
// The communities that the changed arcs touch, and the sum of their K_out *
// K_in as it is (the totals change in k_stat_arcs).
__global__ void k_dirty(const u64* keys, int64_t na, int bits, const int32_t* lab, int32_t* stT, int32_t epT,
                        int32_t* lT, int32_t* nT, const int64_t* Kout, const int64_t* Kin, I128* acc) {
  pdl_enter();
  const u64 mask = (((u64)1) << bits) - 1;
  i128 s = 0;
  GRID_STRIDE(i, na) {
    const int32_t a = lab[keys[i] >> bits], b = lab[keys[i] & mask];
    if (stamp_add(stT, epT, a, lT, nT)) s += (i128)Kout[a] * Kin[a];
    if (stamp_add(stT, epT, b, lT, nT)) s += (i128)Kout[b] * Kin[b];
  }
  s = warp_sum_i128(s);
  if ((threadIdx.x & 31) == 0) atomic_add_i128(acc, s);
}

// sum over listed communities of K_out * K_in into an int128 accumulator
__global__ void k_psum(const int32_t* list, const int32_t* nlist, const int64_t* Kout, const int64_t* Kin,
                       I128* acc) {
  pdl_enter();
  const int32_t n = *nlist;
  i128 s = 0;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t c = list[k];
    s += (i128)Kout[c] * Kin[c];
  }
  s = warp_sum_i128(s);
  if ((threadIdx.x & 31) == 0) atomic_add_i128(acc, s);
}

__global__ void k_stat_arcs(const u64* keys, const int64_t* delta, int64_t na, int bits, int directed,
                            const int32_t* lab, int64_t* kout, int64_t* kin, int64_t* Kout, int64_t* Kin, int64_t* e,
                            int64_t* de, int32_t* stA, int32_t epA, int32_t* lA, int32_t* nA) {
  pdl_enter();
  const u64 mask = (((u64)1) << bits) - 1;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t sde = 0;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; base < na; base += stride) {
    const int64_t t = base + lane;
    int32_t i = 0, j = 0;
    bool wi = false, wj = false;
    if (t < na) {
      i = (int32_t)(keys[t] >> bits);
      j = (int32_t)(keys[t] & mask);
      const int64_t d = delta[t];
      atomic_add_i64(&kout[i], d);
      if (directed) atomic_add_i64(&kin[j], d);
      const int32_t ci = lab[i], cj = lab[j];
      atomic_add_i64(&Kout[ci], d);
      if (directed) atomic_add_i64(&Kin[cj], d);
      if (ci == cj) {
        atomic_add_i64(&e[ci], d);
        sde += d;
      }
      wi = stamp_claim(stA, epA, i);
      wj = stamp_claim(stA, epA, j);
    }
    warp_append(wi, i, lA, nA);
    warp_append(wj, j, lA, nA);
  }
  sde = warp_sum_i64(sde);
  if (lane == 0 && sde) atomic_add_i64(de, sde);
}

// Per-level pointers for walks up the parent chain (levels 0..7).
struct Chain {
  const int32_t* par[8];  // pi_q
  int64_t* kout[8];
  int64_t* kin[8];
  u64* pk[8];             // pending weight records of level q
  u64* pv[8];
  int32_t* stA[8];        // frontier A^q: stamp, epoch, list
  int32_t epA[8];
  int32_t* lA[8];
  int32_t* nA[8];         // its length
  int32_t* np[8];         // pending records of level q
};

// Warp-aggregated append of one record per lane that wants one (every lane
// of the warp calls it together): one atomic per warp.
__device__ inline void warp_append_rec(bool want, u64 key, int64_t v, u64* pk, u64* pv, int32_t* count) {
  const unsigned m = __ballot_sync(0xffffffffu, want);
  if (!m) return;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  int32_t base = 0;
  if (lane == leader) base = atomicAdd(count, __popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (want) {
    const int32_t p = base + __popc(m & ((1u << lane) - 1u));
    pk[p] = key;
    pv[p] = (u64)v;
  }
}

// Weight records (keys, vals) of level q0 carried up the hierarchy: with
// `self` a record joins level q0's pending list; mapped through pi_q0,
// pi_q0+1, ... it joins the pending list of every level above up to `top`,
// until an endpoint has no parent (W_{q+1}(pi(i), pi(j)) takes the weight of
// every level-q arc (i, j)).  With `add_k` the strengths of those levels take
// the weight as well.  Records are not reduced here: the pending list of a
// level is sorted, summed and applied when the level is next read.
__global__ void k_chain_records(const u64* keys, const int64_t* vals, int64_t n, const int32_t* n_dev, int bits, int q0, int top, int self,
                                int add_k, int directed, Chain ch) {
  pdl_enter();
  if (n_dev) n = min(n, (int64_t)*n_dev);
  const u64 mask = (((u64)1) << bits) - 1;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // warp-uniform trip counts, so that appends aggregate over the warp
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; base < n; base += stride) {
    const int64_t t = base + lane;
    bool on = t < n;
    u64 key = 0;
    int64_t d = 0;
    if (on) {
      key = keys[t];
      d = vals[t];
    }
    int32_t x = (int32_t)(key >> bits), y = (int32_t)(key & mask);
    if (self) warp_append_rec(on, key, d, ch.pk[q0], ch.pv[q0], ch.np[q0]);
    for (int q = q0; q < top; ++q) {
      if (on) {
        x = ch.par[q][x];
        y = ch.par[q][y];
        on = x >= 0 && y >= 0;
      }
      if (!__any_sync(0xffffffffu, on)) break;
      if (on && add_k) {
        atomic_add_i64(&ch.kout[q + 1][x], d);
        if (directed) atomic_add_i64(&ch.kin[q + 1][y], d);
      }
      warp_append_rec(on, ((u64)x << bits) | (u64)(uint32_t)y, d, ch.pk[q + 1], ch.pv[q + 1], ch.np[q + 1]);
    }
  }
}

// InitFrontier above level 0: A^{q+1} = pi_q(A^q) for every q < top, by
// walking each node of A^0 up its parent chain.  A walk stops at a node that
// is already marked: the walk that marked it goes on above it.
__global__ void k_chain_frontier(const int32_t* l0, const int32_t* n0, int top, Chain ch) {
  pdl_enter();
  const int32_t m = *n0, stride = gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (int32_t base = blockIdx.x * blockDim.x + threadIdx.x - lane; base < m; base += stride) {
    int32_t x = base + lane < m ? l0[base + lane] : -1;
    for (int q = 0; q < top; ++q) {
      if (x >= 0) x = ch.par[q][x];
      const bool on = x >= 0 && stamp_claim(ch.stA[q + 1], ch.epA[q + 1], x);
      warp_append(on, x, ch.lA[q + 1], ch.nA[q + 1]);
      if (!on) x = -1;
      if (!__any_sync(0xffffffffu, on)) break;
    }
  }
}

// ---------------------------------------------------------------- push-down
// Children of each listed level-(q+1) node take its label at level q.
__global__ void k_push(ChunkMap m, const int32_t* lab_up, Adj<int32_t> ch_adj, const int32_t* par, int32_t* lab,
                       int32_t* olist, int32_t* nout, int32_t* stCh, int32_t epCh, int32_t* lCh, int32_t* nCh,
                       int32_t* lab_before, Tail tail) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const int32_t L = lab_up[ch.v];
    const int64_t o = ch_adj.off[ch.v];
    for (int32_t base = ch.k0; base < ch.k1; base += 32) {
      const int32_t k = base + lane;
      int32_t u = k < ch.k1 ? ch_adj.col[o + k] : 0;
      const bool valid = k < ch.k1 && par[u] == ch.v;  // a listed node that left (emptied) is skipped
      bool first = false;
      if (valid) {
        if (stCh) {
          first = stamp_claim(stCh, epCh, u);
          if (first) lab_before[u] = lab[u];
        }
        lab[u] = L;
      }
      if (stCh) warp_append(first, u, lCh, nCh);
      if (olist) warp_append(valid, u, olist, nout);
    }
  }
  pub_tail(tail);
}

// ---------------------------------------------------------------- dissolve
__global__ void k_stamp_list(const int32_t* l, const int32_t* n, int32_t* st, int32_t ep) {
  pdl_enter();
  const int32_t m = *n;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < m; k += gridDim.x * blockDim.x) st[l[k]] = ep;
}

__global__ void k_dissolve(const int32_t* lD, const int32_t* nD, int32_t* par, int32_t* par_old,
                           const int64_t* kout, const int64_t* kin, int64_t* kout1, int64_t* kin1, int32_t* cnt1,
                           int directed) {
  pdl_enter();
  const int32_t n = *nD;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t u = lD[k];
    const int32_t p = par[u];
    par_old[u] = p;
    if (p >= 0) {
      atomic_add_i64(&kout1[p], -kout[u]);
      if (directed) atomic_add_i64(&kin1[p], -kin[u]);
      atomicAdd(&cnt1[p], -1);
    }
    par[u] = u;
    atomic_add_i64(&kout1[u], kout[u]);
    if (directed) atomic_add_i64(&kin1[u], kin[u]);
    atomicAdd(&cnt1[u], 1);
  }
}

__global__ void k_reset_par(const int32_t* lD, int32_t nD, int32_t* par, int64_t* kout1, int64_t* kin1,
                            int32_t* cnt1, int directed) {
  pdl_enter();
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < nD; k += gridDim.x * blockDim.x) {
    const int32_t u = lD[k];
    par[u] = -1;
    kout1[u] = 0;
    if (directed) kin1[u] = 0;
    cnt1[u] = 0;
  }
}

// ---------------------------------------------------------------- split
// The split may be launched behind a sweep before the host knows whether the
// sweep ends the level's moves.  It runs only if it does: no move was accepted,
// no hub row is still to be swept and the filter finished.
struct SplitGate {
  const int32_t *nb, *hubs, *stat;  // null: open
  __device__ bool open() const { return !nb || (*nb == 0 && (!hubs || *hubs == 0) && *stat != -2); }
};

// TouchedRefined of a batch update (see split()).  The refined communities
// holding an endpoint of a deleted level-r arc are re-checked (before any
// node leaves, so with their current parents).
__global__ void k_brk_check(const int32_t* lK, const int32_t* nK, const uint8_t* alive, const int32_t* par,
                            int32_t* stX, int32_t epX, int32_t* lX, int32_t* nX, int32_t* ckf, int32_t epF,
                            SplitGate gate) {
  pdl_enter();
  const int32_t n = gate.open() ? *nK : 0;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t z = lK[k];
    if (alive[z] && par[z] >= 0) {
      stamp_add(stX, epX, par[z], lX, nX);
      ckf[par[z]] = epF;  // an arc inside it may be gone: its components are computed
    }
  }
}

// A node of U* whose label differs from its refined community's label (or
// that has no refined community) leaves it as a singleton named by its own
// id; its old refined community is re-checked.
__global__ void k_leave(const int32_t* lU, const int32_t* nU, const uint8_t* alive, const int32_t* lab,
                        const int32_t* labN, int32_t* par, int32_t* par_old, const int64_t* kout, const int64_t* kin,
                        int64_t* kout1, int64_t* kin1, int32_t* cnt1, int directed, int32_t* stL, int32_t epL,
                        int32_t* stD, int32_t epD, int32_t* lD, int32_t* nD, int32_t* stX, int32_t epX, int32_t* lX,
                        int32_t* nX, int32_t* nbr, SplitGate gate, Tail tail) {
  pdl_enter();
  const int32_t n = gate.open() ? *nU : 0;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t u = lU[k];
    if (!alive[u]) continue;
    const int32_t X = par[u];
    if (X >= 0 && labN[X] == lab[u]) continue;
    stL[u] = epL;
    par_old[u] = X;
    nbr[u] = 0;
    if (X >= 0) {
      stamp_add(stX, epX, X, lX, nX);
      atomic_add_i64(&kout1[X], -kout[u]);
      if (directed) atomic_add_i64(&kin1[X], -kin[u]);
      atomicAdd(&cnt1[X], -1);
    }
    par[u] = u;
    atomic_add_i64(&kout1[u], kout[u]);
    if (directed) atomic_add_i64(&kin1[u], kin[u]);
    atomicAdd(&cnt1[u], 1);
    stamp_add(stD, epD, u, lD, nD);
  }
  pub_tail(tail);
}

// A refined community that lost nodes stays connected when every node that
// left had at most one neighbour in it and no arc inside it was deleted
// (removing leaves keeps a connected graph connected).  Counts each leaving
// node's neighbours in its old refined community (an arc seen from both
// rows of a directed pair counts twice: the test only errs towards a check)
// and flags the community for a connectivity check at the second one.
template <class WT>
__global__ void k_leave_degree(Adj<WT> out, Adj<WT> in, ChunkMap m, const int32_t* par, const int32_t* par_old,
                               const int32_t* stL, int32_t epL, int32_t* nbr, int32_t* ckf, int32_t epF) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const int32_t v = ch.v;
    const int32_t X = par_old[v];
    if (X < 0 || stL[v] != epL) continue;
    const Adj<WT>& A = ch.row ? in : out;
    const int64_t o = A.off[v];
    for (int32_t k = ch.k0 + lane; k < ch.k1; k += 32) {
      const int32_t y = A.col[o + k];
      if (y == v) continue;
      const bool inX = stL[y] == epL ? par_old[y] == X : par[y] == X;
      if (inX && atomicAdd(&nbr[v], 1) == 1) ckf[X] = epF;
    }
  }
}

// Remaining members of the re-checked refined communities whose connectivity
// is in doubt (flagged, or their seed node left); each starts as its own
// component.
__global__ void k_members(Adj<int32_t> ch_adj, ChunkMap m, const int32_t* par, const int32_t* stL, int32_t epL,
                          const int32_t* ckf, int32_t epF, int32_t* comp, int32_t* lG, int32_t* nG, Tail tail) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const int32_t X = ch.v;
    if (ckf[X] != epF && stL[X] != epL) continue;
    const int64_t o = ch_adj.off[X];
    for (int32_t base = ch.k0; base < ch.k1; base += 32) {
      const int32_t k = base + lane;
      bool want = false;
      int32_t u = 0;
      if (k < ch.k1) {
        u = ch_adj.col[o + k];
        want = stL[u] != epL && par[u] == X;  // listed nodes that emptied or left are skipped
        if (want) comp[u] = u;
      }
      warp_append(want, u, lG, nG);
    }
  }
  pub_tail(tail);
}

// Root of x's tree.  Parent links only point to smaller ids of the same
// component and a root never becomes a root again, so reads that lag behind
// other threads still lead to a node of x's component; they bypass L1 so that
// a thread sees links other SMs made.  With `halve`, x's link is shortened to
// its grandparent on the way (only a non-root's link is ever written, and
// compare-and-swap hooks only roots, so the two never collide).
__device__ inline int32_t uf_find(int32_t* comp, int32_t x, bool halve) {
  int32_t p = __ldcg(&comp[x]);
  while (p != x) {
    const int32_t q = __ldcg(&comp[p]);
    if (halve && q != p) comp[x] = q;
    x = p;
    p = q;
  }
  return x;
}

// Joins the trees of u and y: always hooks the larger root under the smaller
// one (a compare-and-swap that fails because another thread hooked first is
// retried), so every component ends rooted at its lowest member.
__device__ inline void uf_union(int32_t* comp, int32_t u, int32_t y) {
  for (;;) {
    const int32_t a = uf_find(comp, u, true), b = uf_find(comp, y, true);
    if (a == b) return;
    const int32_t hi = a > b ? a : b, lo = a > b ? b : a;
    if (atomicCAS(&comp[hi], hi, lo) == hi) return;
  }
}

// Connected components of the collected members over the arcs between two
// remaining members of the same refined community, by a lock-free union-find
// with neighbour sampling (the Afforest scheme of Sutton, Ben-Nun and Barak,
// IPDPS 2018).  First every member is joined along at most UF_SAMPLE of the
// qualifying arcs among the first 32 entries of its rows (k_uf_sample); in a
// community that is still connected this already puts most members into the
// seed node's tree.  Then k_uf walks all arcs of the members that are not (yet)
// in their community seed's tree.  The components are exact: every arc with an
// endpoint outside the seed's tree is joined from that endpoint's side (both
// rows of a member are walked, so the arc is seen from either end), and an arc
// whose two endpoints were both in the seed's tree when they were checked
// joins nothing new, because trees only ever merge.
constexpr int UF_SAMPLE = 2;

template <class WT>
__global__ void k_uf_sample(Adj<WT> out, Adj<WT> in, int directed, const int32_t* lG, const int32_t* nG,
                            const int32_t* par, const int32_t* stL, int32_t epL, int32_t* comp) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int32_t n = *nG;
  for (int64_t t = warp; t < n; t += nw) {
    const int32_t u = lG[t];
    const int32_t X = par[u];
    int taken = 0;  // warp-uniform
    for (int side = 0; side < (directed ? 2 : 1) && taken < UF_SAMPLE; ++side) {
      const Adj<WT>& A = side ? in : out;
      const int32_t l = A.len[u];
      bool q = false;
      int32_t y = 0;
      if (lane < l) {
        y = A.col[A.off[u] + lane];
        q = y != u && par[y] == X && stL[y] != epL;
      }
      const unsigned mask = __ballot_sync(0xffffffffu, q);
      const int before = __popc(mask & ((1u << lane) - 1u));
      if (q && before < UF_SAMPLE - taken) uf_union(comp, u, y);
      taken += min(__popc(mask), UF_SAMPLE - taken);
    }
  }
}

template <class WT>
__global__ void k_uf(Adj<WT> out, Adj<WT> in, ChunkMap m, const int32_t* par, const uint8_t* alive,
                     const int32_t* stL, int32_t epL, int32_t* comp) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const int32_t u = ch.v;
    const int32_t X = par[u];
    // the community's seed node X is a member when it is alive, stays and is
    // its own parent (then the members gathering set its tree)
    const bool seed = alive[X] && stL[X] != epL && par[X] == X;
    if (seed && uf_find(comp, u, true) == uf_find(comp, X, true)) continue;
    const Adj<WT>& A = ch.row ? in : out;
    const int64_t o = A.off[u];
    for (int32_t k = ch.k0 + lane; k < ch.k1; k += 32) {
      const int32_t y = A.col[o + k];
      if (y == u || par[y] != X || stL[y] == epL) continue;
      uf_union(comp, u, y);
    }
  }
}

// Every member's label becomes its component's root (its lowest member).
// The find here writes nothing but the member's own label: a shortening
// write could otherwise replace another member's final root by an ancestor
// read before that root was written.  Every own write is a node of the same
// component (the root, or before it an ancestor), so other threads' finds
// still end at the root.
__global__ void k_uf_final(const int32_t* lG, const int32_t* nG, int32_t* comp) {
  pdl_enter();
  const int32_t n = *nG;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t u = lG[k];
    comp[u] = uf_find(comp, u, false);
  }
}

// A component keeps its refined community's id when it holds the community's
// seed node (the node with that id, still a member); any other component is
// renamed after its lowest member.
__global__ void k_rename(const int32_t* lG, const int32_t* nG, const int32_t* comp, const uint8_t* alive,
                         const int32_t* stL, int32_t epL, int32_t* par, int32_t* par_old, const int64_t* kout,
                         const int64_t* kin, int64_t* kout1, int64_t* kin1, int32_t* cnt1, int directed,
                         int32_t* stD, int32_t epD, int32_t* lD, int32_t* nD, Tail tail) {
  pdl_enter();
  const int32_t n = *nG;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t u = lG[k];
    const int32_t X = par[u];
    const int32_t root = comp[u];
    const bool keep = alive[X] && stL[X] != epL && par[X] == X && comp[X] == root;
    if (keep) continue;
    par_old[u] = X;
    par[u] = root;
    atomic_add_i64(&kout1[X], -kout[u]);
    if (directed) atomic_add_i64(&kin1[X], -kin[u]);
    atomicAdd(&cnt1[X], -1);
    atomic_add_i64(&kout1[root], kout[u]);
    if (directed) atomic_add_i64(&kin1[root], kin[u]);
    atomicAdd(&cnt1[root], 1);
    stamp_add(stD, epD, u, lD, nD);
  }
  pub_tail(tail);
}

// the listed nodes that are singleton refined communities
__global__ void k_singletons(const int32_t* l, const int32_t* n, const int32_t* par, const int32_t* cnt1, int32_t* out,
                             int32_t* nout) {
  pdl_enter();
  const int32_t m = *n;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < m; base += stride) {
    const int64_t k = base + (threadIdx.x & 31);
    int32_t u = 0;
    bool want = false;
    if (k < m) {
      u = l[k];
      want = par[u] == u && cnt1[u] == 1;
    }
    warp_append(want, u, out, nout);
  }
}

// ---------------------------------------------------------------- aggregate
// The nodes of D whose parent changed, and the entries of their rows.
__global__ void k_changed(const int32_t* lD, const int32_t* nD, const int32_t* par, const int32_t* par_old,
                          int32_t* stC, int32_t epC, int32_t* lC, int32_t* nC, const int32_t* len_out,
                          const int32_t* len_in, int64_t* acc_out, int64_t* acc_in, Tail tail) {
  pdl_enter();
  const int32_t n = *nD;
  int64_t so = 0, si = 0;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t u = lD[k];
    if (par[u] != par_old[u] && stamp_add(stC, epC, u, lC, nC)) {
      so += len_out[u];
      si += len_in[u];
    }
  }
  so = warp_sum_i64(so);
  si = warp_sum_i64(si);
  if ((threadIdx.x & 31) == 0 && so) atomic_add_i64(acc_out, so);
  if ((threadIdx.x & 31) == 0 && si) atomic_add_i64(acc_in, si);
  pub_tail(tail);
}

// Subtract-add records of Eq. 3 for every arc incident to a changed node,
// each arc counted once (from its changed tail's out-row, or from its changed
// head's in-row when the tail is unchanged).
template <class WT>
__global__ void k_emit(Adj<WT> out, Adj<WT> in, ChunkMap m, const int32_t* par, const int32_t* par_old,
                       const int32_t* stC, int32_t epC, int bits, u64* rk, u64* rv, int32_t* cnt, int64_t cap,
                       int32_t* err) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ ChunkPre sh;
  const int64_t total = chunk_begin(m, sh);
  for (int64_t c = warp; c < total; c += nw) {
    const Chunk ch = chunk_of(m, sh, c);
    if (ch.row < 0) continue;
    const int32_t u = ch.v;
    const int32_t po = par_old[u], pn = par[u];
    const Adj<WT>& A = ch.row ? in : out;
    const int64_t o = A.off[u];
    // 64 entries per step, up to four records per lane, one counter atomic
    // per warp and step
    for (int32_t base = ch.k0; base < ch.k1; base += 64) {
      u64 rkey[4] = {0, 0, 0, 0}, rval[4] = {0, 0, 0, 0};
      bool ok[4] = {false, false, false, false};  // fixed slots: (first entry -, +), (second entry -, +)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int32_t k = base + h * 32 + lane;
        if (k >= ch.k1) continue;
        const int32_t v = A.col[o + k];
        const int64_t w = (int64_t)A.w[o + k];
        const bool vc = stC[v] == epC;
        if (ch.row == 0) {  // arc (u, v) from u's out-row
          const int32_t pvo = vc ? par_old[v] : par[v];
          const int32_t pvn = par[v];
          ok[2 * h] = po >= 0 && pvo >= 0;
          rkey[2 * h] = ((u64)po << bits) | (u64)pvo;
          rval[2 * h] = (u64)(-w);
          ok[2 * h + 1] = true;
          rkey[2 * h + 1] = ((u64)pn << bits) | (u64)pvn;
          rval[2 * h + 1] = (u64)w;
        } else if (!vc) {  // arc (v, u) from u's in-row, v unchanged
          const int32_t pv = par[v];
          ok[2 * h] = po >= 0;
          rkey[2 * h] = ((u64)pv << bits) | (u64)po;
          rval[2 * h] = (u64)(-w);
          ok[2 * h + 1] = true;
          rkey[2 * h + 1] = ((u64)pv << bits) | (u64)pn;
          rval[2 * h + 1] = (u64)w;
        }
      }
      const int nrec = (int)ok[0] + (int)ok[1] + (int)ok[2] + (int)ok[3];
      int incl = nrec;  // warp inclusive scan of the per-lane counts
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
      }
      const int wtot = __shfl_sync(0xffffffffu, incl, 31);
      int32_t wbase = 0;
      if (lane == 31 && wtot) wbase = atomicAdd(cnt, wtot);
      wbase = __shfl_sync(0xffffffffu, wbase, 31);
      int64_t p = (int64_t)wbase + incl - nrec;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (ok[j]) {
          if (p < cap) {
            rk[p] = rkey[j];
            rv[p] = rval[j];
          } else {
            atomicExch(err, 3);  // the record bound was wrong: reported, nothing written past it
          }
          ++p;
        }
    }
  }
}

// Children-list records of the changed nodes; their strengths move from the
// old parent's ancestors to the new one's, up to level `top` (the parents'
// own strengths moved with the members; a supernode's are its members' sums).
__global__ void k_emit_nodes(const int32_t* lC, const int32_t* nC, const int32_t* par, const int32_t* par_old,
                             const int64_t* kout, const int64_t* kin, int bits, int q0, int top, int directed,
                             Chain ch, u64* ck, u64* cv, int32_t* ncr) {
  pdl_enter();
  const int32_t n = *nC;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t u = lC[k];
    const int32_t po = par_old[u], pn = par[u];
    const int32_t p = atomicAdd(ncr, po >= 0 ? 2 : 1);
    ck[p] = ((u64)pn << bits) | (u64)u;
    cv[p] = (u64)(int64_t)1;
    if (po >= 0) {
      ck[p + 1] = ((u64)po << bits) | (u64)u;
      cv[p + 1] = (u64)(int64_t)-1;
    }
    const int64_t ko = kout[u], ki = kin[u];
    for (int side = 0; side < 2; ++side) {
      int32_t x = side ? pn : po;
      for (int q = q0; q < top && x >= 0; ++q) {
        x = ch.par[q][x];
        if (x < 0) break;
        atomic_add_i64(&ch.kout[q + 1][x], side ? ko : -ko);
        if (directed) atomic_add_i64(&ch.kin[q + 1][x], side ? ki : -ki);
      }
    }
  }
}

// Existence after a level-q0 aggregate step, for the candidate level-q0 nodes
// (old and new parents of the changed nodes, each handled by the thread that
// claims it): a node with members appears (it has no parent yet); a node left
// without members dies and leaves its parent, and a parent that thereby loses
// its last member dies in turn, up the chain to level top.  The walk that
// takes a parent's member count to zero carries on with that parent, so each
// death is handled once, and the counts above q0 only fall meanwhile.  (An
// emptied node stays listed among its parent's children; readers of the
// lists check the parent.)
struct ExistChain {
  int32_t* cnt[8];
  uint8_t* alive[8];
  int32_t* par[8];
};

__global__ void k_exist_chain(const int32_t* lC, const int32_t* nC, const int32_t* par, const int32_t* par_old,
                              int32_t* stE, int32_t epE, int q0, int top, ExistChain ch, int32_t* err) {
  pdl_enter();
  const int32_t n = *nC;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < 2 * n; k += gridDim.x * blockDim.x) {
    const int32_t u = lC[k >> 1];
    int32_t x = (k & 1) ? par_old[u] : par[u];
    if (x < 0 || !stamp_claim(stE, epE, x)) continue;
    int q = q0;
    const int32_t c = ch.cnt[q][x];
    if (!ch.alive[q][x]) {
      if (c > 0) {
        ch.alive[q][x] = 1;
        if (q < top && ch.par[q][x] >= 0) atomicExch(err, 2);
      }
      continue;
    }
    if (c != 0) continue;
    for (;;) {  // x at level q has no members left
      ch.alive[q][x] = 0;
      if (q >= top) break;
      const int32_t p = ch.par[q][x];
      if (p < 0) break;
      ch.par[q][x] = -1;
      if (atomicAdd(&ch.cnt[q + 1][p], -1) != 1) break;
      x = p;
      ++q;
    }
  }
}

// Level r + 1 after level r's aggregate step: the images of the frontier and
// dissolved nodes take their labels, and NextFrontier is marked: the images of
// U* and D (D's old parents too) and the endpoints of the level's nr weight
// records, as far as they exist.  (Stamps make the three lists one set, so one
// launch goes through them all; without stA only the labels are written.)
__global__ void k_next_level(const int32_t* lU, const int32_t* nU, const int32_t* lD, const int32_t* nD,
                             const int32_t* par, const int32_t* par_old, const int32_t* lab, int32_t* lab_up,
                             const u64* keys, const int32_t* nr, int64_t nr_max, int bits, const uint8_t* alive,
                             int32_t* stA, int32_t epA, int32_t* lA, int32_t* nA, int64_t* agg_recs) {
  pdl_enter();
  const int64_t mu = *nU, md = *nD;
  const int64_t mr = keys ? min((int64_t)*nr, nr_max) : 0;
  const u64 mask = (((u64)1) << bits) - 1;
  if (blockIdx.x == 0 && threadIdx.x == 0 && mr) atomic_add_i64(agg_recs, mr);
  GRID_STRIDE(t, mu + md + mr) {
    if (t < mu + md) {
      const int32_t u = t < mu ? lU[t] : lD[t - mu];
      const int32_t p = par[u];
      lab_up[p] = lab[u];
      if (!stA) continue;
      if (p >= 0 && alive[p]) stamp_add(stA, epA, p, lA, nA);
      if (t >= mu) {
        const int32_t q = par_old[u];
        if (q >= 0 && alive[q]) stamp_add(stA, epA, q, lA, nA);
      }
    } else if (stA) {
      const u64 key = keys[t - mu - md];
      const int32_t x = (int32_t)(key >> bits), y = (int32_t)(key & mask);
      if (alive[x]) stamp_add(stA, epA, x, lA, nA);
      if (alive[y]) stamp_add(stA, epA, y, lA, nA);
    }
  }
}

// ---------------------------------------------------------------- static set-up
// Records of a CSR snapshot (nnz entries, rp[0] = 0, rp[n] = nnz), entry by
// entry so that a hub row spreads over the GPU (a warp per row took 2.1 ms on
// the R-MAT of 2^20, all of it the longest row).  *unsorted is set where a
// row's columns are not strictly increasing.
__global__ void k_csr_records(const int64_t* rp, const int32_t* col, const int32_t* w, int64_t n, int64_t nnz, int bits,
                              u64* rk, u64* rv, unsigned long long* err, int32_t* unsorted) {
  pdl_enter();
  GRID_STRIDE(v, n) {
    if (rp[v + 1] < rp[v]) set_err(err, 0, LDL_E_INVALID);
  }
  bool bad = false;
  for_seg_runs(rp, n, nnz, [&](int64_t t0, int cnt, int64_t slo, int64_t shi) {
    for (int64_t t = t0 + (threadIdx.x & 31); t < t0 + cnt; t += 32) {
      const int64_t v = seg_of(rp, slo, shi, t);
      const int32_t c = col[t], x = w[t];
      if (c < 0 || c >= n) set_err(err, 0, LDL_E_RANGE);
      if (x < 1) set_err(err, 0, LDL_E_INVALID);
      bad |= t > 0 && t > rp[v] && col[t - 1] >= c;
      rk[t] = ((u64)v << bits) | (u64)(uint32_t)c;
      rv[t] = (u64)(int64_t)x;
    }
  });
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicExch(unsorted, 1);
}

__global__ void k_check_max(const int64_t* s, int64_t n, unsigned long long* err) {
  pdl_enter();
  GRID_STRIDE(i, n) {
    if (s[i] > INT32_MAX) set_err(err, 0, LDL_E_OVERFLOW);
  }
}

__global__ void k_compare(const u64* a, const int64_t* av, const u64* b, const u64* bv, int64_t n,
                          unsigned long long* err) {
  pdl_enter();
  GRID_STRIDE(i, n) {
    if (a[i] != b[i] || (u64)av[i] != bv[i]) set_err(err, 0, LDL_E_INVALID);
  }
}

// Row sums (cleared before) of sorted records, rows counted from row0, the
// weight on the diagonal and the sum of all.  A thread sums RS_RUN consecutive
// records and adds once per row it meets, so a hub row is no longer than others
// (a warp per row took 337 us on the R-MAT of 2^20).
constexpr int RS_RUN = 8;
__global__ void k_row_sums(const u64* keys, const int64_t* w, int64_t nrec, int bits, int64_t row0, int64_t* out,
                           int64_t* self, int64_t* total) {
  pdl_enter();
  const u64 mask = (((u64)1) << bits) - 1;
  int64_t tot = 0;
  GRID_STRIDE(r, (nrec + RS_RUN - 1) / RS_RUN) {
    int64_t row = -1, s = 0;
    for (int64_t i = r * RS_RUN; i < min(nrec, (r + 1) * RS_RUN); ++i) {
      const int64_t v = (int64_t)(keys[i] >> bits) - row0;
      if (v != row && row >= 0) {
        atomic_add_i64(&out[row], s);
        tot += s;
        s = 0;
      }
      row = v;
      s += w[i];
      if (self && (int64_t)(keys[i] & mask) == v) atomic_add_i64(&self[v], w[i]);
    }
    if (row >= 0) atomic_add_i64(&out[row], s);
    tot += s;
  }
  tot = warp_sum_i64(tot);
  if ((threadIdx.x & 31) == 0 && total && tot) atomic_add_i64(total, tot);
}

__global__ void k_iota(int32_t* a, int64_t n) {
  pdl_enter();
  GRID_STRIDE(i, n) a[i] = (int32_t)i;
}

__global__ void k_fill_i32(int32_t* a, int64_t n, int32_t v) {
  pdl_enter();
  GRID_STRIDE(i, n) a[i] = v;
}

__global__ void k_alive_list(const uint8_t* alive, int64_t n, int32_t* l, int32_t* cnt) {
  pdl_enter();
  GRID_STRIDE(i, n) {
    if (!alive || alive[i]) l[atomicAdd(cnt, 1)] = (int32_t)i;
  }
}

__global__ void k_esum(const int64_t* e, const int64_t* Kout, const int64_t* Kin, int64_t n, int64_t* E, I128* P) {
  pdl_enter();
  int64_t se = 0;
  i128 sp = 0;
  GRID_STRIDE(i, n) {
    se += e[i];
    sp += (i128)Kout[i] * Kin[i];
  }
  se = warp_sum_i64(se);
  sp = warp_sum_i128(sp);
  if ((threadIdx.x & 31) == 0) {
    if (se) atomic_add_i64(E, se);
    atomic_add_i128(P, sp);
  }
}

__global__ void k_changed_final(const int32_t* lCh, const int32_t* nCh, const int32_t* lab,
                                const int32_t* lab_before, int32_t* out, int32_t* nout, Tail tail) {
  pdl_enter();
  const int32_t n = *nCh;
  for (int32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int32_t u = lCh[k];
    if (lab[u] != lab_before[u]) out[atomicAdd(nout, 1)] = u;
  }
  pub_tail(tail);
}

__global__ void k_gather(const int32_t* ids, int32_t k, const int32_t* lab, int32_t* out) {
  pdl_enter();
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) out[i] = lab[ids[i]];
}

}  // namespace

// ================================================================== host side
void gather_labels(ldl_ctx& c, const int32_t* ids, int32_t k, int32_t* out) {
  if (k <= 0) return;
  launch(k_gather, grid_for(k, TPB), TPB, 0, c.s, ids, k, c.lv[0].lab.p, out);
  CKL("k_gather");
}
static void throw_err(ldl_ctx& c, unsigned long long* d_err, const char* what) {
  unsigned long long e = 0;
  const HostRead r{d_err, &e, sizeof(e)};
  host_read(c, &r, 1);
  if (e != ~0ull) {
    const int code = (int)(e & 255);
    const long long idx = (long long)(e >> 8);
    char buf[160];
    snprintf(buf, sizeof buf, "%s: status %d at update %lld", what, code, idx);
    ldl_throw((ldl_status)code, buf);
  }
}

static void reset_err(ldl_ctx& c) {
  CK(cudaMemsetAsync(&c.d_sc->err_key, 0xff, sizeof(int64_t), c.s));
}

static unsigned long long* err_ptr(ldl_ctx& c) { return (unsigned long long*)&c.d_sc->err_key; }

static void throw_at(int64_t key, const char* what) {
  char buf[160];
  snprintf(buf, sizeof buf, "%s: status %d at update %lld", what, (int)(key & 255), (long long)(key >> 8));
  ldl_throw((ldl_status)(key & 255), buf);
}

int64_t ingest(ldl_ctx& c, const ldl_update* upd, int64_t count, int on_device, int64_t* dm) {
  *dm = 0;
  c.arena_top = 0;
  for (int k = 0; k < K_COUNT; ++k) c.cp[k] = c.dcnt + k;
  launch(k_batch_begin, 1, 1024, 0, c.s, c.dcnt, c.arena, c.d_sc);
  CKL("k_batch_begin");
  if (count <= 0) return 0;
  const ldl_update* du = upd;
  if (!on_device) {
    c.upd.reserve(count, c.s);
    CK(cudaMemcpyAsync(c.upd.p, upd, sizeof(ldl_update) * (size_t)count, cudaMemcpyHostToDevice, c.s));
    du = c.upd.p;
  }
  // (rk, rv) may change places with (tk, tv) in the sort, and takes the arcs
  // of both directions at the end
  const int64_t arcs = c.directed ? count : 2 * count;
  for (DBuf<u64>* b : {&c.rk, &c.rv, &c.tk, &c.tv, &c.trk, &c.trv}) b->reserve(2 * count + 2, c.s);
  c.rk2.reserve(count + 1, c.s);
  c.rsum.reserve(count + 1, c.s);
  unsigned long long* err = (unsigned long long*)&c.d_sc->err_key;
  unsigned long long* err_seq = (unsigned long long*)&c.d_sc->err_seq;
  const int g = grid_for(count, TPB);
  launch(k_upd_keys, g, TPB, 0, c.s, du, count, c.n, c.bits, c.directed, c.rk.p, c.rv.p, err);
  CKL("k_upd_keys");
  sort_pairs(c.rk, c.rv, c.tk, c.tv, count, 2 * c.bits, c.P, c.s);
  const int tiles = div_up(count, UQ_TPB);
  const LookBack q = look_back_begin(c.P, tiles, c.s);
  launch(k_unique, tiles, UQ_TPB, 0, c.s, c.rk.p, count, c.rk2.p, c.rsum.p, c.cp[K_NU], q);
  CKL("k_unique");
  const auto& g0 = c.lv[0].out0;
  launch(k_seq, g, TPB, 0, c.s, du, count, c.rv.p, c.rsum.p, c.cp[K_NU], c.rk2.p, g0.off.p, g0.len.p, g0.col.p, g0.w.p,
                            c.bits, c.directed, err_seq, &c.d_sc->dm, c.trk.p, c.trv.p, c.cp[K_REC]);
  CKL("k_seq");
  // the changed arcs in order (each once, no change zero), on directed graphs
  // followed by their in-direction records
  sort_reduce(c.trk, c.trv, c.tk, c.tv, arcs, c.cp[K_REC], c.bits, c.directed, c.n, c.rk.p, (int64_t*)c.rv.p,
              c.cp[K_NR], c.P, c.s);
  int64_t e1 = -1, e2 = -1;
  int32_t na = 0;
  const HostRead rr[4] = {{err, &e1, sizeof(int64_t)}, {err_seq, &e2, sizeof(int64_t)},
                          {&c.d_sc->dm, dm, sizeof(int64_t)}, {c.cp[K_NR], &na, sizeof(int32_t)}};
  host_read(c, rr, 4);
  if (e1 != -1) throw_at(e1, "invalid update");
  if (e2 != -1) throw_at(e2, "invalid update sequence");
  if (c.m + *dm >= ((int64_t)1 << 50) || c.m + *dm < 0) ldl_throw(LDL_E_OVERFLOW, "total weight m would reach 2^50");
  return na;
}

// Sorted unique out-records of a directed level -> the same records followed
// by their in-direction copies (rows n..2n-1), still sorted: (rk2, rv2), 2*nr.
static void combine_in_out(ldl_ctx& c, const u64* keys, const u64* vals, int64_t nr) {
  c.rk2.reserve(2 * nr + 1, c.s);
  c.rv2.reserve(2 * nr + 1, c.s);
  c.trk.reserve(nr + 1, c.s);
  c.trv.reserve(nr + 1, c.s);
  launch(k_transpose, grid_for(nr, TPB), TPB, 0, c.s, keys, vals, nr, c.bits, c.trk.p, c.trv.p, c.n);
  CKL("k_transpose");
  // the out-records are ordered by row, so a stable sort on the new row alone
  // gives (in-row, col) order
  sort_pairs(c.trk, c.trv, c.tk, c.tv, nr, 2 * c.bits + 1, c.P, c.s, c.bits);
  CK(cudaMemcpyAsync(c.rk2.p, keys, sizeof(u64) * (size_t)nr, cudaMemcpyDeviceToDevice, c.s));
  CK(cudaMemcpyAsync(c.rv2.p, vals, sizeof(u64) * (size_t)nr, cudaMemcpyDeviceToDevice, c.s));
  CK(cudaMemcpyAsync(c.rk2.p + nr, c.trk.p, sizeof(u64) * (size_t)nr, cudaMemcpyDeviceToDevice, c.s));
  CK(cudaMemcpyAsync(c.rv2.p + nr, c.trv.p, sizeof(u64) * (size_t)nr, cudaMemcpyDeviceToDevice, c.s));
}

// Where level r's update records the endpoints of arcs that disappear.  A
// deleted arc can only disconnect the refined community holding both of its
// endpoints (refined communities are connected); until the level's next split
// its parents change only where a node empties and leaves its parent.
static DelTrack del_track(ldl_ctx& c, int r) {
  LevelState& L = c.lv[r];
  return DelTrack{L.stK.p, L.brk_ep, L.lK.p, c.cp[K_BRK0 + r], c.n, r < c.T ? L.par.p : nullptr};
}

// m records (both directions of a directed level) were applied: arcs
static int64_t applied(ldl_ctx& c, int r, int64_t m) {
  if (c.directed) m /= 2;
  c.lv[r].ubK = std::min<int64_t>(c.n, c.lv[r].ubK + 2 * m);
  return m;
}

// Applies sorted unique records (directed: followed by their in-direction
// copies) to a level's adjacency; the endpoints of arcs that disappear are
// recorded for the level's next refinement.  nr records, or *n_dev of them
// with nr an upper bound; returns their number.
static int64_t apply_records(ldl_ctx& c, int r, const u64* keys, const int64_t* vals, int64_t nr,
                             const int32_t* n_dev) {
  const CsrRecords rec{keys, vals, (c.directed ? 2 : 1) * nr, n_dev, c.directed ? 2 : 1, c.bits};
  const DelTrack trk = del_track(c, r);
  const int64_t m = r == 0 ? csr_apply<int32_t>(c.lv[0].out0, rec, c.CS, c.P, c.s, c.d_sc, &trk)
                           : csr_apply<int64_t>(c.lv[r].out, rec, c.CS, c.P, c.s, c.d_sc, &trk);
  return applied(c, r, m);
}

static Chain chain_of(ldl_ctx& c, const int32_t* epA) {
  Chain ch{};
  for (int q = 0; q <= c.T && q < 8; ++q) {
    LevelState& L = c.lv[q];
    ch.par[q] = L.par.p;
    ch.kout[q] = L.kout.p;
    ch.kin[q] = kin_of(c, q);
    ch.pk[q] = L.pk.p;
    ch.pv[q] = L.pv.p;
    ch.stA[q] = L.stA.p;
    ch.lA[q] = L.lA.p;
    ch.epA[q] = epA ? epA[q] : 0;
    ch.nA[q] = c.cp[K_A0 + q];
    ch.np[q] = c.cp[K_PEND0 + q];
  }
  return ch;
}

// Records of level q0 onto the pending lists of level q0 (with `self`) and
// of every level above: each list is grown (keeping its contents) to hold n
// more (n_dev: their device count, n bounds it).
static void chain_records(ldl_ctx& c, const u64* keys, const int64_t* vals, int64_t n, const int32_t* n_dev, int q0,
                          bool self, bool add_k) {
  if (n <= 0 || (!self && q0 >= c.T)) return;
  if (n > INT32_MAX / 2) ldl_throw(LDL_E_OVERFLOW, "too many weight records in one step for the 32-bit counters");
  for (int q = self ? q0 : q0 + 1; q <= c.T; ++q) {
    LevelState& L = c.lv[q];
    // the device counters are 32-bit: a list that would pass them is applied first
    if (L.pend_ub + n > INT32_MAX - 1) flush_level(c, q);
    L.pk.reserve(L.pend_ub + n + 1, c.s, true);
    L.pv.reserve(L.pend_ub + n + 1, c.s, true);
    L.pend_ub += n;
  }
  launch(k_chain_records, grid_for(n, TPB), TPB, 0, c.s, keys, vals, n, n_dev, c.bits, q0, c.T, self ? 1 : 0, add_k ? 1 : 0,
                                                     c.directed, chain_of(c, nullptr));
  CKL("k_chain_records");
}

void pending_reset(ldl_ctx& c) {  // the device counters are cleared by ingest
  for (auto& L : c.lv) L.pend_ub = 0;
}

// Level q's pending records, sorted by (row, col) and summed per arc (zero
// sums dropped), applied to its adjacency: the level's weights become
// current before anything reads them.
void flush_level(ldl_ctx& c, int q, int64_t known) {
  LevelState& L = c.lv[q];
  if (L.pend_ub == 0) return;
  const int64_t n = known >= 0 ? known : rd_cnt(c, K_PEND0 + q);
  L.pend_ub = 0;
  zero_cnt(c, K_PEND0 + q);
  if (n <= 0) return;
  // own output buffers: a flush may run while the caller's records sit in rk / rv
  c.flk.reserve((c.directed ? 2 : 1) * n + 1, c.s);
  c.flv.reserve((c.directed ? 2 : 1) * n + 1, c.s);
  int32_t* nr = c.cp[K_FL];
  sort_reduce(L.pk, L.pv, c.tk, c.tv, n, nullptr, c.bits, c.directed, c.n, c.flk.p, c.flv.p, nr, c.P, c.s);
  c.res.pending_records += n;
  c.res.pending_applied += apply_records(c, q, c.flk.p, c.flv.p, n, nr);
}

static CsrRecords flush_records(ldl_ctx& c, int64_t n, const int32_t* gate) {
  const int mul = c.directed ? 2 : 1;
  return CsrRecords{c.flk.p, c.flv.p, mul * n, c.cp[K_FL], mul, c.bits, gate};
}

void flush_plan(ldl_ctx& c, int q, const int32_t* gate, HostRead* rr, int n, int64_t (&tot)[6]) {
  LevelState& L = c.lv[q];
  const int64_t ub = L.pend_ub;
  c.flk.reserve((c.directed ? 2 : 1) * ub + 1, c.s);
  c.flv.reserve((c.directed ? 2 : 1) * ub + 1, c.s);
  zero_cnt(c, K_FL);
  // sorting the list changes its order only: it stays valid if the gate is shut
  sort_reduce(L.pk, L.pv, c.tk, c.tv, ub, c.cp[K_PEND0 + q], c.bits, c.directed, c.n, c.flk.p, c.flv.p, c.cp[K_FL], c.P,
              c.s);
  rr[n] = {c.d_sc->plan, tot, sizeof(tot)};
  const DelTrack trk = del_track(c, q);
  csr_plan<int64_t>(c.lv[q].out, flush_records(c, ub, gate), c.CS, c.P, c.s, c.d_sc, &trk, tail_begin(c, rr, n + 1));
  tail_wait(c, rr, n + 1);
}

void flush_finish(ldl_ctx& c, int q, int64_t n, const int64_t (&tot)[6]) {
  LevelState& L = c.lv[q];
  const int64_t ub = L.pend_ub;
  L.pend_ub = 0;
  zero_cnt(c, K_PEND0 + q);
  c.res.pending_records += n;
  c.res.pending_applied +=
      applied(c, q, csr_finish<int64_t>(c.lv[q].out, flush_records(c, ub, nullptr), tot, c.CS, c.P, c.s, c.d_sc));
}

void repair_done(ldl_ctx& c, const RepairAcc& a, int64_t dm) {
  c.m += dm;
  c.E += a.de;
  c.Psum += i128_of(a.p_new.hi, a.p_new.lo) - i128_of(a.p_old.hi, a.p_old.lo);
}

void repair_batch(ldl_ctx& c, int64_t na, const int32_t* epA, int32_t epT) {
  if (na <= 0) return;
  // Algorithm 1, applying the batch: it changes level 0
  apply_records(c, 0, c.rk.p, (const int64_t*)c.rv.p, na, nullptr);
  // statistic repair: degrees, community totals (exactly, with sum_C K_out K_in)
  LevelState& L0 = c.lv[0];
  zero_cnt(c, K_T);
  c.racc = (RepairAcc*)fresh(c, sizeof(RepairAcc) / 4, c.d_sc->home2);
  launch(k_dirty, grid_for(na, TPB), TPB, 0, c.s, c.rk.p, na, c.bits, L0.lab.p, c.stT.p, epT, c.lT.p, c.cp[K_T], c.Kout.p,
                                              Kin_of(c), &c.racc->p_old);
  CKL("k_dirty");
  launch(k_stat_arcs, grid_for(na, TPB), TPB, 0, c.s, c.rk.p, (const int64_t*)c.rv.p, na, c.bits, c.directed, L0.lab.p,
                                                  L0.kout.p, kin_of(c, 0), c.Kout.p, Kin_of(c), c.e.p, &c.racc->de,
                                                  L0.stA.p, epA[0], L0.lA.p, c.cp[K_A0]);
  CKL("k_stat_arcs");
  launch(k_psum, grid_for(2 * na, TPB), TPB, 0, c.s, c.lT.p, c.cp[K_T], c.Kout.p, Kin_of(c), &c.racc->p_new);
  CKL("k_psum");
  if (c.T == 0) return;
  // InitFrontier: A^{q+1} = pi_q(A^q) along the chain
  launch(k_chain_frontier, grid_for(2 * na, TPB), TPB, 0, c.s, L0.lA.p, c.cp[K_A0], c.T, chain_of(c, epA));
  CKL("k_chain_frontier");
  // the aggregate chain: W_q(anc(i), anc(j)) += delta and the strengths of
  // every level above 0; the weights are applied when each level is next read
  chain_records(c, c.rk.p, (const int64_t*)c.rv.p, na, nullptr, 0, false, true);
}

void pushdown(ldl_ctx& c, int r, int32_t epCh, int64_t moved_ub) {
  // lMv holds the level-r nodes moved in this level's move loop; its count
  // stays on the device and moved_ub bounds it (0 exactly when it is empty)
  int32_t* src = c.lMv.p;
  int idx = K_MV;
  int64_t n = std::min<int64_t>(moved_ub, c.n);
  int32_t* bufs[2] = {c.lTmp.p, c.lE2.p};
  int idxs[2] = {K_TMP, K_TMP2};
  int flip = 0;
  for (int q = r - 1; q >= 0 && n > 0; --q) {
    LevelState& L = c.lv[q];
    Adj<int32_t> ch{L.children.off.p, L.children.len.p, L.children.col.p, L.children.w.p};
    int32_t* dst = q > 0 ? bufs[flip] : nullptr;
    zero_cnt(c, idxs[flip]);
    ChunkMap m = chunk_map(c, src, c.cp[idx], n, L.children.len.p, nullptr);
    int32_t nn = 0;
    const HostRead rr{c.cp[idxs[flip]], &nn, sizeof(int32_t)};
    launch(k_push, chunk_grid(n), TPB, 0, c.s,
        m, c.lv[q + 1].lab.p, ch, L.par.p, L.lab.p, dst, c.cp[idxs[flip]], q == 0 ? c.stCh.p : nullptr, epCh,
        c.lCh.p, c.cp[K_CH], c.lab_before.p, q > 0 ? tail_begin(c, &rr, 1) : Tail{});
    CKL("k_push");
    if (q > 0) {
      tail_wait(c, &rr, 1);
      src = bufs[flip];
      idx = idxs[flip];
      n = nn;
      flip ^= 1;
    }
  }
}

// Static build: every alive level-r node becomes a singleton refined
// community (refinement starts from singletons).  Returns |D| (list lD).
int32_t dissolve_all(ldl_ctx& c, int r, int32_t epD) {
  LevelState& L = c.lv[r];
  LevelState& N = c.lv[r + 1];
  zero_cnt(c, K_D);
  launch(k_alive_list, grid_for(c.n, TPB), TPB, 0, c.s, r ? L.alive.p : nullptr, c.n, c.lD.p, c.cp[K_D]);
  CKL("k_alive_list");
  launch(k_stamp_list, grid_for(c.n, TPB), TPB, 0, c.s, c.lD.p, c.cp[K_D], c.stD.p, epD);
  CKL("k_stamp_list");
  const int32_t nd = rd_cnt(c, K_D);
  if (nd > 0) {
    launch(k_dissolve, grid_for(nd, TPB), TPB, 0, c.s, c.lD.p, c.cp[K_D], L.par.p, c.par_old.p, L.kout.p,
                                                   kin_of(c, r), N.kout.p, kin_of(c, r + 1), N.cnt.p, c.directed);
    CKL("k_dissolve");
  }
  return nd;
}

void singletons_of(ldl_ctx& c, int r, const int32_t* list, int idx_n, int64_t n_hint, int32_t* out, int idx_out) {
  zero_cnt(c, idx_out);
  if (n_hint > 0) {
    launch(k_singletons, grid_for(n_hint, TPB), TPB, 0, c.s, list, c.cp[idx_n], c.lv[r].par.p, c.lv[r + 1].cnt.p, out,
                                                         c.cp[idx_out]);
    CKL("k_singletons");
  }
}

void reset_par(ldl_ctx& c, int r, int32_t nD) {
  if (nD <= 0) return;
  launch(k_reset_par, grid_for(nD, TPB), TPB, 0, c.s, c.lD.p, nD, c.lv[r].par.p, c.lv[r + 1].kout.p,
                                                  kin_of(c, r + 1), c.lv[r + 1].cnt.p, c.directed);
  CKL("k_reset_par");
}

template <class WT>
static void leave_degree(ldl_ctx& c, int r, Adj<WT> out, Adj<WT> in, int32_t nD, int32_t epL, int32_t epF) {
  ChunkMap m = chunk_map(c, c.lD.p, c.cp[K_D], nD, out.len, c.directed ? in.len : nullptr);
  launch(k_leave_degree<WT>, chunk_grid(nD), TPB, 0, c.s, out, in, m, c.lv[r].par.p, c.par_old.p,
                                                                           c.stL.p, epL, c.nbr.p, c.ckf.p, epF);
  CKL("k_leave_degree");
}

template <class WT>
static void union_find(ldl_ctx& c, int r, Adj<WT> out, Adj<WT> in, int32_t nG, int32_t epL) {
  LevelState& L = c.lv[r];
  launch(k_uf_sample<WT>, grid_for((int64_t)nG * 32, TPB, 16), TPB, 0, c.s, out, in, c.directed, c.lG.p, c.cp[K_G],
                                                                       L.par.p, c.stL.p, epL, c.comp.p);
  CKL("k_uf_sample");
  ChunkMap m = chunk_map(c, c.lG.p, c.cp[K_G], nG, out.len, c.directed ? in.len : nullptr);
  launch(k_uf<WT>, chunk_grid(nG), TPB, 0, c.s, out, in, m, L.par.p, L.alive.p, c.stL.p, epL,
                                                                  c.comp.p);
  CKL("k_uf");
}

// TouchedRefined of a batch update at level r < T (Sec. III-C: refinement
// revisits the communities touched by accepted moves).  A refined community
// lies inside one community, so every node of U* whose label differs from its
// refined community's label (moved at level r, or relabelled from its members'
// moves at level r-1), and every parentless new node, leaves it as a
// singleton named by its own id.  The refined communities that lost a node or
// hold an endpoint of a level-r arc deleted since the level was last refined
// are re-checked for connectivity over the arcs among their remaining members
// (connected components by hooking and pointer jumping): the component with
// the community's seed node keeps the id, any other is renamed after its
// lowest member.  Returns |D|, the nodes whose refined community changed
// (list lD, stamp epD, old parents in par_old); the level's deletion list is
// consumed.
void split_launch(ldl_ctx& c, int r, SplitRun& sr, bool gated, bool hubs, HostRead* rr, int n) {
  LevelState& L = c.lv[r];
  LevelState& N = c.lv[r + 1];
  zero_cnt(c, K_D);
  zero_cnt(c, K_X);
  sr.epD = c.next_epoch();
  sr.epF = c.next_epoch();  // communities whose connectivity is in doubt
  sr.epL = c.next_epoch();
  const int32_t epX = c.next_epoch();
  const SplitGate gate{gated ? c.cp[K_B] : nullptr, hubs ? c.cp[K_LARGE] : nullptr, c.cp[K_UNDEC]};
  // The level's deleted-arc endpoints and U* stay on the device: both kernels
  // stride over their lists' counts with grids sized by the host's bounds.
  launch(k_brk_check, grid_for(L.ubK, TPB, 4), TPB, 0, c.s, L.lK.p, c.cp[K_BRK0 + r], L.alive.p, L.par.p, c.stX.p, epX,
                                                        c.lX.p, c.cp[K_X], c.ckf.p, sr.epF, gate);
  CKL("k_brk_check");
  rr[n] = {c.cp[K_D], &sr.nleft, sizeof(int32_t)};
  rr[n + 1] = {c.cp[K_X], &sr.nx, sizeof(int32_t)};
  launch(k_leave, grid_for(c.ubU, TPB, 4), TPB, 0, c.s, c.lUstar.p, c.cp[K_USTAR], L.alive.p, L.lab.p, N.lab.p, L.par.p,
                                                    c.par_old.p, L.kout.p, kin_of(c, r), N.kout.p, kin_of(c, r + 1),
                                                    N.cnt.p, c.directed, c.stL.p, sr.epL, c.stD.p, sr.epD, c.lD.p,
                                                    c.cp[K_D], c.stX.p, epX, c.lX.p, c.cp[K_X], c.nbr.p, gate,
                                                    tail_begin(c, rr, n + 2));
  CKL("k_leave");
}

int32_t split(ldl_ctx& c, int r, SplitRun& sr) {
  LevelState& L = c.lv[r];
  LevelState& N = c.lv[r + 1];
  if (!sr.done) {
    HostRead rr[2];
    split_launch(c, r, sr, false, false, rr, 0);
    tail_wait(c, rr, 2);
  }
  const int32_t nleft = sr.nleft, nx = sr.nx, epL = sr.epL, epF = sr.epF, epD = sr.epD;
  int32_t nD = nleft;  // k_rename appends to lD
  if (nx > 0) {
    if (nleft > 0) {
      if (r == 0) leave_degree<int32_t>(c, r, adj_out0(c), adj_in0(c), nleft, epL, epF);
      else leave_degree<int64_t>(c, r, adj_out(c, r), adj_in(c, r), nleft, epL, epF);
    }
    zero_cnt(c, K_G);
    int32_t nG = 0;
    const HostRead rg{c.cp[K_G], &nG, sizeof(int32_t)};
    Adj<int32_t> ch{L.children.off.p, L.children.len.p, L.children.col.p, L.children.w.p};
    ChunkMap m = chunk_map(c, c.lX.p, c.cp[K_X], nx, L.children.len.p, nullptr);
    launch(k_members, chunk_grid(nx), TPB, 0, c.s, ch, m, L.par.p, c.stL.p, epL, c.ckf.p, epF,
                                                                   c.comp.p, c.lG.p, c.cp[K_G], tail_begin(c, &rg, 1));
    CKL("k_members");
    tail_wait(c, &rg, 1);
    c.res.split_members += nG;
    if (nG > 0) {
      if (r == 0) union_find<int32_t>(c, r, adj_out0(c), adj_in0(c), nG, epL);
      else union_find<int64_t>(c, r, adj_out(c, r), adj_in(c, r), nG, epL);
      launch(k_uf_final, grid_for(nG, TPB), TPB, 0, c.s, c.lG.p, c.cp[K_G], c.comp.p);
      CKL("k_uf_final");
      const HostRead rn{c.cp[K_D], &nD, sizeof(int32_t)};
      launch(k_rename, grid_for(nG, TPB), TPB, 0, c.s, c.lG.p, c.cp[K_G], c.comp.p, L.alive.p, c.stL.p, epL, L.par.p,
                                                   c.par_old.p, L.kout.p, kin_of(c, r), N.kout.p, kin_of(c, r + 1),
                                                   N.cnt.p, c.directed, c.stD.p, epD, c.lD.p, c.cp[K_D], tail_begin(c, &rn, 1));
      CKL("k_rename");
      tail_wait(c, &rn, 1);
    }
  }
  // the deletions of this level are consumed
  L.brk_ep = c.next_epoch();
  L.ubK = 0;
  zero_cnt(c, K_BRK0 + r);
  return nD;
}

// deg: out-row and in-row entries of the changed nodes (k_changed); returns
// the bound on the records (their count is at cp[K_REC])
template <class WT>
static int64_t emit_records(ldl_ctx& c, int r, Adj<WT> out, Adj<WT> in, int32_t nC, int32_t epC, bool build,
                            const int64_t (&deg)[2]) {
  // at most a subtract and an add record per visited entry; in the static
  // build no node had a parent (no subtract records) and every node is
  // changed (no in-row records), so one record per out-row entry
  const int64_t cap = (build ? deg[0] : 2 * (deg[0] + deg[1])) + 16;
  if (cap > INT32_MAX) ldl_throw(LDL_E_OVERFLOW, "aggregate records beyond the 32-bit record counter");
  c.rk2.reserve(cap, c.s);
  c.rv2.reserve(cap, c.s);
  // (in the static build the in-rows would be walked for nothing)
  ChunkMap m = chunk_map(c, c.lC.p, c.cp[K_C], nC, out.len, build ? nullptr : in.len);
  launch(k_emit<WT>, chunk_grid(nC), TPB, 0, c.s, out, in, m, c.lv[r].par.p, c.par_old.p,
                                                                          c.stC.p, epC, c.bits, c.rk2.p, c.rv2.p,
                                                                          c.cp[K_REC], cap, c.cp[K_ERR]);
  CKL("k_emit");
  return cap;
}

// Above this many records a step reads their exact number before it sorts them
// and queues them on the levels above: up to four times as many are reserved
// as come, which costs memory where the buffers are large and nothing but the
// read (about 8 us) to avoid.
// (Device memory that 14 batches add to a new context, against exact counts in
// separate buffers: 926 MB for 1040 with 10^3 on the R-MAT of 131k, 8022 for
// 9074 with 10^4 on the R-MAT of 2^20, 942 for 920 with 10^5 on the 2M-vertex
// power-law graph.)
constexpr int64_t AGG_EXACT = 1 << 20;

void aggregate(ldl_ctx& c, int r, int32_t epD, int32_t epC, int32_t epA_next, bool build, int32_t nD) {
  (void)epD;
  LevelState& L = c.lv[r];
  LevelState& N = c.lv[r + 1];
  // changed nodes
  sub_begin(c);
  for (int k : {K_C, K_REC, K_CREC}) zero_cnt(c, k);
  c.sums = (int64_t*)fresh(c, 4, c.d_sc->sums);
  int32_t nC = 0;
  int64_t deg[2] = {0, 0};
  if (nD > 0) {
    const int32_t* lo = r == 0 ? adj_out0(c).len : adj_out(c, r).len;
    const int32_t* li = r == 0 ? adj_in0(c).len : adj_in(c, r).len;
    const HostRead rr[2] = {{c.cp[K_C], &nC, sizeof(int32_t)}, {c.sums, deg, 2 * sizeof(int64_t)}};
    launch(k_changed, grid_for(nD, TPB), TPB, 0, c.s, c.lD.p, c.cp[K_D], L.par.p, c.par_old.p, c.stC.p, epC, c.lC.p,
                                                  c.cp[K_C], lo, li, c.sums, c.sums + 1, tail_begin(c, rr, 2));
    CKL("k_changed");
    tail_wait(c, rr, 2);
  }
  int64_t nr = 0;  // bound on the level r+1 records (their number is at cp[K_NR])
  if (nC > 0) {
    int64_t nrec = r == 0 ? emit_records<int32_t>(c, r, adj_out0(c), adj_in0(c), nC, epC, build, deg)
                          : emit_records<int64_t>(c, r, adj_out(c, r), adj_in(c, r), nC, epC, build, deg);
    c.crk.reserve(2 * (int64_t)nC + 2, c.s);
    c.crv.reserve(2 * (int64_t)nC + 2, c.s);
    launch(k_emit_nodes, grid_for(nC, TPB), TPB, 0, c.s, c.lC.p, c.cp[K_C], L.par.p, c.par_old.p, L.kout.p,
                                                     kin_of(c, r), c.bits, r + 1, build ? r + 1 : c.T, c.directed,
                                                     chain_of(c, nullptr), c.crk.p, c.crv.p, c.cp[K_CREC]);
    CKL("k_emit_nodes");
    sub_end(c, SU_AGG_EMIT);
    sub_begin(c);
    if (build) {
      // level r+1 starts empty: build its adjacency and the children lists
      int32_t nrec32 = 0, ncr32 = 0;
      {
        const HostRead rr[2] = {{c.cp[K_REC], &nrec32, sizeof(int32_t)},
                                {c.cp[K_CREC], &ncr32, sizeof(int32_t)}};
        host_read(c, rr, 2);
      }
      const int64_t cnt = nrec32, ncr = ncr32;
      if (cnt > nrec) ldl_throw(LDL_E_INVALID, "internal: aggregate records exceed their bound");
      sort_pairs(c.rk2, c.rv2, c.tk, c.tv, cnt, 2 * c.bits, c.P, c.s);
      c.rk.reserve(cnt + 1, c.s);
      c.rsum.reserve(cnt + 1, c.s);
      nr = reduce_by_key(c.rk2.p, c.rv2.p, cnt, c.rk.p, c.rsum.p, c.P, c.s);
      c.res.agg_records += nr;
      sub_end(c, SU_AGG_SORT);
      sub_begin(c);
      sort_pairs(c.crk, c.crv, c.tk, c.tv, ncr, 2 * c.bits, c.P, c.s);
      if (c.directed) {
        combine_in_out(c, c.rk.p, (const u64*)c.rsum.p, nr);
        csr_build<int64_t>(N.out, 2 * c.n, c.rk2.p, (const int64_t*)c.rv2.p, 2 * nr, c.bits, 25, c.CS, c.P, c.s);
      } else {
        csr_build<int64_t>(N.out, c.n, c.rk.p, c.rsum.p, nr, c.bits, 25, c.CS, c.P, c.s);
      }
      csr_build<int32_t>(L.children, c.n, c.crk.p, (const int64_t*)c.crv.p, ncr, c.bits, 25, c.CS, c.P, c.s);
    } else {
      const int32_t* cnt_dev = c.cp[K_REC];
      if (nrec > AGG_EXACT) {
        const int64_t cnt = rd_cnt(c, K_REC);
        if (cnt > nrec) ldl_throw(LDL_E_INVALID, "internal: aggregate records exceed their bound");
        nrec = cnt;
        cnt_dev = nullptr;
      }
      c.rk.reserve(nrec + 1, c.s);
      c.rsum.reserve(nrec + 1, c.s);
      if (nrec > 0)
        sort_reduce(c.rk2, c.rv2, c.tk, c.tv, nrec, cnt_dev, c.bits, false, 0, c.rk.p, c.rsum.p, c.cp[K_NR], c.P,
                    c.s);
      nr = nrec;
      if (nrec > AGG_EXACT) nr = rd_cnt(c, K_NR);
      sub_end(c, SU_AGG_SORT);
      sub_begin(c);
      // the level r+1 records join its pending list and, mapped through the
      // current parents, the lists of the levels above
      chain_records(c, c.rk.p, c.rsum.p, nr, c.cp[K_NR], r + 1, true, false);
      sort_pairs(c.crk, c.crv, c.tk, c.tv, 2 * (int64_t)nC, 2 * c.bits, c.P, c.s, 0, c.cp[K_CREC]);
      csr_apply<int32_t>(L.children,
                         CsrRecords{c.crk.p, (const int64_t*)c.crv.p, 2 * (int64_t)nC, c.cp[K_CREC], 1, c.bits}, c.CS,
                         c.P, c.s, c.d_sc);
    }
    sub_end(c, SU_AGG_APPLY);
    sub_begin(c);
    // existence: appear at r+1, emptied nodes cascade upwards
    ExistChain ech{};
    for (int q = 0; q <= c.T && q < 8; ++q) {
      ech.cnt[q] = c.lv[q].cnt.p;
      ech.alive[q] = c.lv[q].alive.p;
      ech.par[q] = c.lv[q].par.p;
    }
    launch(k_exist_chain, grid_for(2 * (int64_t)nC, TPB), TPB, 0, c.s, c.lC.p, c.cp[K_C], L.par.p, c.par_old.p,
                                                                    c.stE.p, c.next_epoch(), r + 1, c.T, ech,
                                                                    c.cp[K_ERR]);
    CKL("k_exist_chain");
    // the error flag K_ERR is read once at the end of the batch (or of the static build)
  } else {
    sub_end(c, SU_AGG_EMIT);
    sub_begin(c);
  }
  if (!build) N.ubA = std::min<int64_t>(c.n, N.ubA + c.ubU + 2 * (int64_t)nD + 2 * nr);
  // |U*| stays on the device
  const bool recs = nC > 0 && epA_next;
  launch(k_next_level, grid_for(build ? c.n : c.ubU + nD + nr, TPB, 2), TPB, 0, c.s, c.lUstar.p, c.cp[K_USTAR], c.lD.p, c.cp[K_D], L.par.p,
                                                  c.par_old.p, L.lab.p, N.lab.p, recs ? c.rk.p : nullptr,
                                                  c.cp[K_NR], nr, c.bits, N.alive.p, epA_next ? N.stA.p : nullptr,
                                                  epA_next, N.lA.p, c.cp[K_A0 + r + 1], &c.d_sc->agg_recs);
  CKL("k_next_level");
  sub_end(c, SU_AGG_EXIST);
}

void level_alloc(ldl_ctx& c, int r) {
  LevelState& L = c.lv[r];
  if (L.allocated) return;
  const int64_t n = c.n;
  // (the cleared arrays first: one clear)
  Slab& S = L.nodes;
  S.add(L.stK, n);
  S.add(L.lab, n);
  S.add(L.cnt, n);
  S.add(L.kout, n);
  if (c.directed) S.add(L.kin, n);
  S.add(L.alive, n);
  S.add(L.stA, n);
  const size_t cleared = S.parts.size();
  S.add(L.par, n);
  S.add(L.lA, n);
  S.add(L.lK, n);
  S.alloc();
  CK(cudaMemsetAsync(S.base, 0, S.span(0, cleared), c.s));
  CK(cudaMemsetAsync(L.par.p, 0xff, sizeof(int32_t) * (size_t)n, c.s));
  L.allocated = true;
}

void level_free(ldl_ctx& c, int r) { c.lv[r].release(); }

int32_t alive_list(ldl_ctx& c, int r, int32_t* list, int idx) {
  zero_cnt(c, idx);
  launch(k_alive_list, grid_for(c.n, TPB), TPB, 0, c.s, r ? c.lv[r].alive.p : nullptr, c.n, list, c.cp[idx]);
  CKL("k_alive_list");
  return rd_cnt(c, idx);
}

void changed_labels(ldl_ctx& c, const HostRead* rr, int n) {
  // strides over the candidates' device count with a grid bounded by the node count
  launch(k_changed_final, grid_for(c.n, TPB, 2), TPB, 0, c.s, c.lCh.p, c.cp[K_CH], c.lv[0].lab.p, c.lab_before.p, c.lChg.p,
                                                          c.cp[K_CHG], tail_begin(c, rr, n));
  CKL("k_changed_final");
  tail_wait(c, rr, n);
}

void upload_graph(ldl_ctx& c, int64_t nnz, const int64_t* row_ptr, const int32_t* col, const int32_t* w) {
  const int64_t n = c.n;
  DBuf<int64_t> drp;
  DBuf<int32_t> dcol, dw;
  drp.exact(n + 1);
  dcol.exact(nnz + 1);
  dw.exact(nnz + 1);
  CK(cudaMemcpyAsync(drp.p, row_ptr, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyHostToDevice, c.s));
  if (nnz) {
    CK(cudaMemcpyAsync(dcol.p, col, sizeof(int32_t) * (size_t)nnz, cudaMemcpyHostToDevice, c.s));
    CK(cudaMemcpyAsync(dw.p, w, sizeof(int32_t) * (size_t)nnz, cudaMemcpyHostToDevice, c.s));
  }
  c.rk.reserve(nnz + 1, c.s);
  c.rv.reserve(nnz + 1, c.s);
  reset_err(c);
  zero_cnt(c, K_TMP);
  launch(k_csr_records, grid_for(std::max(n, nnz / 8), TPB), TPB, 0, c.s, drp.p, dcol.p, dw.p, n, nnz, c.bits, c.rk.p,
                                                                      c.rv.p, err_ptr(c), c.cp[K_TMP]);
  CKL("k_csr_records");
  CK(cudaStreamSynchronize(c.s));
  drp.release();
  dcol.release();
  dw.release();
  throw_err(c, err_ptr(c), "invalid CSR");
  int64_t na = nnz;
  // rows in strictly increasing column order are unique sorted arcs already
  if (rd_cnt(c, K_TMP)) {
    sort_pairs(c.rk, c.rv, c.tk, c.tv, nnz, 2 * c.bits, c.P, c.s);
    c.rk2.reserve(nnz + 1, c.s);
    c.rsum.reserve(nnz + 1, c.s);
    na = reduce_by_key(c.rk.p, c.rv.p, nnz, c.rk2.p, c.rsum.p, c.P, c.s);
    reset_err(c);
    launch(k_check_max, grid_for(na, TPB), TPB, 0, c.s, c.rsum.p, na, err_ptr(c));
    CKL("k_check_max");
    throw_err(c, err_ptr(c), "summed weight above INT32_MAX");
    // (rk2, rsum) = unique arcs
    CK(cudaMemcpyAsync(c.rk.p, c.rk2.p, sizeof(u64) * (size_t)na, cudaMemcpyDeviceToDevice, c.s));
    CK(cudaMemcpyAsync(c.rv.p, c.rsum.p, sizeof(int64_t) * (size_t)na, cudaMemcpyDeviceToDevice, c.s));
  }
  if (na) {
    c.rk2.reserve(na + 1, c.s);
    c.rv2.reserve(na + 1, c.s);
    if (!c.directed) {
      launch(k_transpose, grid_for(na, TPB), TPB, 0, c.s, c.rk.p, c.rv.p, na, c.bits, c.rk2.p, c.rv2.p, 0);
      CKL("k_transpose");
      sort_pairs(c.rk2, c.rv2, c.tk, c.tv, na, 2 * c.bits, c.P, c.s, c.bits);  // rows already ordered
      reset_err(c);
      launch(k_compare, grid_for(na, TPB), TPB, 0, c.s, c.rk.p, (const int64_t*)c.rv.p, c.rk2.p, c.rv2.p, na,
                                                    err_ptr(c));
      CKL("k_compare");
      throw_err(c, err_ptr(c), "undirected CSR is not symmetric");
    }
  }
  LevelState& L0 = c.lv[0];
  if (c.directed) {
    combine_in_out(c, c.rk.p, c.rv.p, na);
    csr_build<int32_t>(L0.out0, 2 * n, c.rk2.p, (const int64_t*)c.rv2.p, 2 * na, c.bits, 25, c.CS, c.P, c.s);
  } else {
    csr_build<int32_t>(L0.out0, n, c.rk.p, (const int64_t*)c.rv.p, na, c.bits, 25, c.CS, c.P, c.s);
  }
  // strengths, m, labels, community totals
  CK(cudaMemsetAsync(&c.d_sc->dm, 0, sizeof(int64_t), c.s));
  CK(cudaMemsetAsync(L0.kout.p, 0, sizeof(int64_t) * (size_t)n, c.s));
  CK(cudaMemsetAsync(c.e.p, 0, sizeof(int64_t) * (size_t)n, c.s));
  const int gr = grid_for((na + RS_RUN - 1) / RS_RUN, TPB);
  launch(k_row_sums, gr, TPB, 0, c.s, c.rk.p, (const int64_t*)c.rv.p, na, c.bits, 0, L0.kout.p, c.e.p, &c.d_sc->dm);
  CKL("k_row_sums");
  if (c.directed) {
    CK(cudaMemsetAsync(L0.kin.p, 0, sizeof(int64_t) * (size_t)n, c.s));
    launch(k_row_sums, gr, TPB, 0, c.s, c.rk2.p + na, (const int64_t*)c.rv2.p + na, na, c.bits, n, L0.kin.p, nullptr,
                                    nullptr);
    CKL("k_row_sums(in)");
  }
  launch(k_iota, grid_for(n, TPB), TPB, 0, c.s, L0.lab.p, n);
  CKL("k_iota");
  launch(k_fill_i32, grid_for(n, TPB), TPB, 0, c.s, L0.cnt.p, n, 1);
  CKL("k_fill_i32");
  CK(cudaMemsetAsync(L0.alive.p, 1, (size_t)n, c.s));
  CK(cudaMemcpyAsync(c.Kout.p, L0.kout.p, sizeof(int64_t) * (size_t)n, cudaMemcpyDeviceToDevice, c.s));
  if (c.directed) CK(cudaMemcpyAsync(c.Kin.p, L0.kin.p, sizeof(int64_t) * (size_t)n, cudaMemcpyDeviceToDevice, c.s));
  c.racc = (RepairAcc*)c.d_sc->home2;
  CK(cudaMemsetAsync(c.racc, 0, sizeof(RepairAcc), c.s));
  launch(k_esum, grid_for(n, TPB), TPB, 0, c.s, c.e.p, c.Kout.p, Kin_of(c), n, &c.racc->de, &c.racc->p_new);
  CKL("k_esum");
  DevScalars h;
  CK(cudaMemcpyAsync(&h, c.d_sc, sizeof(DevScalars), cudaMemcpyDeviceToHost, c.s));
  CK(cudaStreamSynchronize(c.s));
  c.m = h.dm;
  if (c.m >= ((int64_t)1 << 50)) ldl_throw(LDL_E_OVERFLOW, "total weight m reaches 2^50");
  RepairAcc ra;
  memcpy(&ra, h.home2, sizeof(ra));
  c.E = ra.de;
  c.Psum = i128_of(ra.p_new.hi, ra.p_new.lo);
}
