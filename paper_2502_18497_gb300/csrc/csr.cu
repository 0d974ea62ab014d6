// Device-resident CSR with per-row slack (Sec. III-A keeps adjacency at
// every level; inserts go into the row's slack, deletes shrink the row, a row
// out of slack moves to the end of the pool).
//
// Every row is kept sorted by neighbour id.  Records are (key, delta) pairs
// with key = row << bshift | col, sorted by key and unique.  Matching a record
// is a binary search in its row (one thread per record); a row that gains or
// loses entries is rebuilt by a flattened scatter in which every kept entry
// and every inserted entry computes its own destination, so hub rows spread
// over the whole GPU instead of one warp.
#include <algorithm>

#include "csr.cuh"
#include "prims.cuh"

namespace {

#define GRID_STRIDE(i, n) \
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

constexpr int TPB = 256;

// ---- planning an update: records -> rows (segments) -> what each row needs
// A record list: n records, or mul * *n_dev of them with n an upper bound; none
// where the gate is given and zero.
struct RecN {
  int64_t n;
  const int32_t* n_dev;
  int mul;
  const int32_t* gate;
  __device__ int64_t count() const {
    if (gate && *gate == 0) return 0;
    return n_dev ? min(n, (int64_t)mul * *n_dev) : n;
  }
};

// Per-record and per-segment arrays of an update (see CsrScratch).
struct PlanOut {
  int32_t *pos, *lb, *segid, *pins, *pdel;
  int64_t* oldw;
  int64_t *seg, *segrow;
  int32_t* newcap;
  int64_t *soff, *woff, *noff;
  int64_t* nseg;  // device: number of segments
  u64* bad;       // device: the last plan number that met an impossible record
  u64 plan;       // this plan's number
  const void* totals;  // DevScalars::plan: names the totals in a tail
};

struct Rec {
  int32_t ins, del, head;
};

// Matches record i in its (sorted) row and says what it does to it; the
// endpoints of an entry it removes go to *t (rows below t.rows).
template <class WT>
__device__ inline Rec match_record(const int64_t* off, const int32_t* len, const int32_t* col, const WT* w,
                                   const u64* keys, const int64_t* delta, int64_t i, int bshift, const PlanOut& o,
                                   const DelTrack& t) {
  const u64 cmask = (((u64)1) << bshift) - 1;
  const u64 key = keys[i];
  const int64_t row = (int64_t)(key >> bshift);
  const int32_t c = (int32_t)(key & cmask);
  const int64_t at = off[row];
  const int32_t l = len[row];
  const int64_t d = delta[i];
  Rec r;
  r.head = i == 0 || (int64_t)(keys[i - 1] >> bshift) != row;
  const int32_t p = row_lower_bound(col, at, l, c);
  const bool found = p < l && col[at + p] == c;
  const int64_t ow = found ? (int64_t)w[at + p] : 0;
  const int64_t nv = ow + d;
  o.pos[i] = found ? p : -1;
  o.lb[i] = p;
  o.oldw[i] = ow;
  if (nv < 0 || (!found && nv == 0)) atomicMax((unsigned long long*)o.bad, (unsigned long long)o.plan);
  r.ins = !found && nv > 0;
  r.del = found && nv == 0;
  if (r.del && t.stamp && row < t.rows) {
    // an arc between two different refined communities cannot disconnect
    // either; a parentless endpoint may have just left its community (an
    // emptied node), so such arcs are kept
    if (!(t.par && (row == c || (t.par[row] >= 0 && t.par[c] >= 0 && t.par[row] != t.par[c])))) {
      stamp_add(t.stamp, t.ep, (int32_t)row, t.list, t.cnt);
      stamp_add(t.stamp, t.ep, c, t.list, t.cnt);
    }
  }
  return r;
}

struct SegNeed {
  int64_t scratch, work, pool;  // old entries to copy, items of the rebuild, pool slots of a relocation
};

// Segment s (records [a, b)): its new capacity when the row no longer fits,
// and what its rebuild needs.
__device__ inline SegNeed plan_segment(const PlanOut& o, int64_t s, int64_t a, int64_t b, const int32_t* len,
                                       const int32_t* cap) {
  const int64_t row = o.segrow[s];
  const int64_t ins = o.pins[b] - o.pins[a], del = o.pdel[b] - o.pdel[a];
  const int64_t l = len[row];
  const int64_t nl = l - del + ins;
  SegNeed q{0, 0, 0};
  if (nl > cap[row]) {
    q.pool = nl + (nl >> 1) + 4;
    q.pool = (q.pool + 3) & ~(int64_t)3;
  }
  o.newcap[s] = (int32_t)q.pool;
  if (ins > 0 || del > 0) {
    q.scratch = l;
    q.work = l + ins;
  }
  return q;
}

// The plan's totals straight into the tail's entry for them (its other values
// are of earlier kernels).
__device__ inline void put_totals(const Tail& t, const PlanOut& o, int64_t need, int64_t nseg, int64_t stot,
                                  int64_t wtot, int64_t nrec) {
  const int64_t v[6] = {need, nseg, stot, wtot, nrec, (int64_t)(*(volatile u64*)o.bad == o.plan)};
  put_values(t, o.totals, v);
}

constexpr int PL_TPB = 512;  // records (segments) per tile: one each per thread, as a match is a chain of loads

// Records: one pass over tiles of PL_TPB, with a look-back for the running
// counts of inserts, deletes and segments.
template <class WT>
__global__ void __launch_bounds__(PL_TPB) k_plan_records(const int64_t* off, const int32_t* len, const int32_t* col,
                                                         const WT* w, const u64* keys, const int64_t* delta, RecN rn,
                                                         int bshift, PlanOut o, DelTrack t, LookBack q) {
  pdl_enter();
  __shared__ int64_t s_tile, s_pre[3];
  if (threadIdx.x == 0) s_tile = atomicAdd(q.ctr, 1);
  __syncthreads();
  const int64_t n = rn.count(), tile = s_tile, i = tile * PL_TPB + threadIdx.x;
  if (tile * PL_TPB >= n && tile > 0) return;
  Rec r{0, 0, 0};
  if (i < n) r = match_record<WT>(off, len, col, w, keys, delta, i, bshift, o, t);
  u64 tot;
  const u64 ex = block_scan<PL_TPB>((u64)r.ins | ((u64)r.del << 20) | ((u64)r.head << 40), &tot);
  if (threadIdx.x < 32) {
    const int64_t agg[3] = {(int64_t)(tot & 0xfffff), (int64_t)((tot >> 20) & 0xfffff), (int64_t)(tot >> 40)};
    int64_t pre[3];
    look_back<3>(q.st, tile, agg, pre, q.ep, q.err);
    if (threadIdx.x == 0) {
      for (int k = 0; k < 3; ++k) s_pre[k] = pre[k];
      if ((tile + 1) * PL_TPB >= n) {
        o.pins[n] = (int32_t)(pre[0] + agg[0]);
        o.pdel[n] = (int32_t)(pre[1] + agg[1]);
        *o.nseg = pre[2] + agg[2];
      }
    }
  }
  __syncthreads();
  if (i < n) {
    o.pins[i] = (int32_t)(s_pre[0] + (int64_t)(ex & 0xfffff));
    o.pdel[i] = (int32_t)(s_pre[1] + (int64_t)((ex >> 20) & 0xfffff));
    const int64_t seg = s_pre[2] + (int64_t)(ex >> 40);  // heads before i
    o.segid[i] = (int32_t)(seg + r.head - 1);
    if (r.head) {
      o.seg[seg] = i;
      o.segrow[seg] = (int64_t)(keys[i] >> bshift);
    }
  }
}

// Segments: scratch, rebuild and pool offsets by one pass; the last tile hands
// the totals to the host.
__global__ void __launch_bounds__(PL_TPB) k_plan_segments(const int32_t* len, const int32_t* cap, RecN rn, PlanOut o,
                                                          LookBack q, Tail tail) {
  pdl_enter();
  __shared__ int64_t s_tile, s_pre[3];
  __shared__ int64_t s_sum[3];
  if (threadIdx.x == 0) s_tile = atomicAdd(q.ctr, 1);
  __syncthreads();
  const int64_t n = rn.count(), nseg = *o.nseg, tile = s_tile, s = tile * PL_TPB + threadIdx.x;
  if (tile * PL_TPB >= nseg && tile > 0) return;
  SegNeed d{0, 0, 0};
  if (s < nseg) d = plan_segment(o, s, o.seg[s], s + 1 < nseg ? o.seg[s + 1] : n, len, cap);
  u64 ex[3];
  u64 tot[3];
  ex[0] = block_scan<PL_TPB>((u64)d.scratch, &tot[0]);
  ex[1] = block_scan<PL_TPB>((u64)d.work, &tot[1]);
  ex[2] = block_scan<PL_TPB>((u64)d.pool, &tot[2]);
  if (threadIdx.x < 32) {
    const int64_t agg[3] = {(int64_t)tot[0], (int64_t)tot[1], (int64_t)tot[2]};
    int64_t pre[3];
    look_back<3>(q.st, tile, agg, pre, q.ep, q.err);
    if (threadIdx.x == 0)
      for (int k = 0; k < 3; ++k) {
        s_pre[k] = pre[k];
        s_sum[k] = pre[k] + agg[k];
      }
  }
  __syncthreads();
  if (s < nseg) {
    o.soff[s] = s_pre[0] + (int64_t)ex[0];
    o.woff[s] = s_pre[1] + (int64_t)ex[1];
    o.noff[s] = s_pre[2] + (int64_t)ex[2];
  }
  if ((tile + 1) * PL_TPB >= nseg) {
    if (threadIdx.x == 0) {
      o.soff[nseg] = s_sum[0];
      o.woff[nseg] = s_sum[1];
      put_totals(tail, o, s_sum[2], nseg, s_sum[0], s_sum[1], n);
    }
    put_tail(tail, o.totals);
  }
}

// Both steps in one block for up to PS_TPB records (one launch).
constexpr int PS_TPB = 1024;
template <class WT>
__global__ void __launch_bounds__(PS_TPB) k_plan_small(const int64_t* off, const int32_t* len, const int32_t* cap,
                                                       const int32_t* col, const WT* w, const u64* keys,
                                                       const int64_t* delta, RecN rn, int bshift, PlanOut o,
                                                       DelTrack t, Tail tail) {
  pdl_enter();
  const int64_t n = rn.count(), i = threadIdx.x;
  Rec r{0, 0, 0};
  if (i < n) r = match_record<WT>(off, len, col, w, keys, delta, i, bshift, o, t);
  u64 tot;
  const u64 ex = block_scan<PS_TPB>((u64)r.ins | ((u64)r.del << 20) | ((u64)r.head << 40), &tot);
  const int64_t nseg = (int64_t)(tot >> 40);
  if (i < n) {
    const int64_t seg = (int64_t)(ex >> 40);
    o.pins[i] = (int32_t)(ex & 0xfffff);
    o.pdel[i] = (int32_t)((ex >> 20) & 0xfffff);
    o.segid[i] = (int32_t)(seg + r.head - 1);
    if (r.head) {
      o.seg[seg] = i;
      o.segrow[seg] = (int64_t)(keys[i] >> bshift);
    }
  }
  if (i == 0) {
    o.pins[n] = (int32_t)(tot & 0xfffff);
    o.pdel[n] = (int32_t)((tot >> 20) & 0xfffff);
    *o.nseg = nseg;
  }
  __syncthreads();
  SegNeed d{0, 0, 0};
  if (i < nseg) d = plan_segment(o, i, o.seg[i], i + 1 < nseg ? o.seg[i + 1] : n, len, cap);
  u64 ts, tw, tp;
  const u64 es = block_scan<PS_TPB>((u64)d.scratch, &ts);
  const u64 ew = block_scan<PS_TPB>((u64)d.work, &tw);
  const u64 en = block_scan<PS_TPB>((u64)d.pool, &tp);
  if (i < nseg) {
    o.soff[i] = (int64_t)es;
    o.woff[i] = (int64_t)ew;
    o.noff[i] = (int64_t)en;
  }
  if (i == 0) {
    o.soff[nseg] = (int64_t)ts;
    o.woff[nseg] = (int64_t)tw;
    put_totals(tail, o, (int64_t)tp, nseg, (int64_t)ts, (int64_t)tw, n);
  }
  put_tail(tail, o.totals);
}

// ---- undo log (batches that may be rolled back)
// Rollback of one row chunk: offsets, lengths and capacities come back; a
// rewritten row's old contents go back where they were when they lie in the
// batch's first pool below its first free slot (anything else was written
// into space that held no data of the state being restored).
template <class WT>
__global__ void k_undo_rows(int64_t nr, const int64_t* lrow, const int64_t* loff, const int32_t* llen,
                            const int32_t* lcap, const int64_t* lsrc, const int32_t* lcol, const WT* lw,
                            int64_t* off, int32_t* len, int32_t* cap, int32_t* col, WT* w, int restore_content,
                            int64_t top0) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < nr; i += nw) {
    const int64_t row = lrow[i], o = loff[i], src = lsrc[i];
    const int32_t l = llen[i];
    if (lane == 0) {
      off[row] = o;
      len[row] = l;
      cap[row] = lcap[i];
    }
    if (restore_content && src >= 0 && o + l <= top0)
      for (int32_t k = lane; k < l; k += 32) {
        col[o + k] = lcol[src + k];
        w[o + k] = lw[src + k];
      }
  }
}

template <class WT>
__global__ void k_undo_weights(int64_t nw, const int64_t* lpos, const WT* lold, WT* w, int64_t top0) {
  pdl_enter();
  GRID_STRIDE(i, nw) {
    const int64_t p = lpos[i];
    if (p >= 0 && p < top0) w[p] = lold[i];
  }
}

// First half of an update: the weights of rows that keep their entries change
// in place, and the rows to rebuild are copied out as they are (into the undo
// log while a batch is logged).  With a log also: per row its old offset,
// length and capacity and where its contents went (-1: not rewritten), per
// record the pool position of its entry (-1: absent) and its old weight.  The
// three parts touch different entries, so one launch does them all.
template <class WT>
struct UndoOut {  // null pointers without a log
  int64_t *lrow, *loff, *lsrc, *lpos;
  int32_t *llen, *lcap;
  WT* lold;
  int64_t c0;  // first free slot of the content log
};

template <class WT>
__global__ void k_apply(int64_t nrec, int64_t nseg, int64_t stotal, const u64* keys, const int64_t* delta, int bshift,
                        PlanOut o, const int64_t* off, const int32_t* len, const int32_t* cap, const int32_t* col,
                        WT* w, int32_t* scol, WT* sw, UndoOut<WT> u) {
  pdl_enter();
  GRID_STRIDE(i, nrec) {
    const int32_t p = o.pos[i];
    const int64_t at = p >= 0 ? off[(int64_t)(keys[i] >> bshift)] + p : -1;
    const int64_t ow = o.oldw[i];
    if (u.lpos) {
      u.lpos[i] = at;
      u.lold[i] = (WT)ow;
    }
    const int32_t s = o.segid[i];
    if (p >= 0 && o.woff[s + 1] == o.woff[s]) w[at] = (WT)(ow + delta[i]);
  }
  if (u.lrow) {
    GRID_STRIDE(s, nseg) {
      const int64_t row = o.segrow[s];
      u.lrow[s] = row;
      u.loff[s] = off[row];
      u.llen[s] = len[row];
      u.lcap[s] = cap[row];
      u.lsrc[s] = o.soff[s + 1] > o.soff[s] ? u.c0 + o.soff[s] : -1;
    }
  }
  // a lane's entries of a run are in flight together (one after the other, with
  // two 17-step searches per run, took 49 us a level on the R-MAT of 2^20
  // where this takes 25)
  for_seg_runs(o.soff, nseg, stotal, [&](int64_t t0, int n, int64_t slo, int64_t shi) {
    const int lane = threadIdx.x & 31;
    int32_t c[SEG_PL];
    WT x[SEG_PL];
#pragma unroll
    for (int j = 0; j < SEG_PL; ++j) {
      const int64_t t = t0 + j * 32 + lane;
      c[j] = 0;
      x[j] = 0;
      if (j * 32 + lane < n) {
        const int64_t s = seg_of(o.soff, slo, shi, t);
        const int64_t at = off[o.segrow[s]] + (t - o.soff[s]);
        c[j] = col[at];
        x[j] = w[at];
      }
    }
#pragma unroll
    for (int j = 0; j < SEG_PL; ++j)
      if (j * 32 + lane < n) {
        scol[t0 + j * 32 + lane] = c[j];
        sw[t0 + j * 32 + lane] = x[j];
      }
  });
}

// Second half, for rows with inserts or deletes.  Item t is either a kept old
// entry (from the copy; its record, if it has one, changes its weight, and a
// weight of zero drops it) or an inserted record; each computes its sorted
// position.  A row that outgrew its capacity moves to base + noff.  The row
// table is written by the same launch: only relocated rows change their
// offset, and nobody reads that.
template <class WT>
__global__ void k_rebuild(int64_t nrec, int64_t nseg, int64_t total, int64_t base, PlanOut o, const int32_t* scol,
                          const WT* sw, const u64* keys, const int64_t* delta, int bshift, int64_t* off, int32_t* len,
                          int32_t* cap, int32_t* col, WT* w) {
  pdl_enter();
  const u64 cmask = (((u64)1) << bshift) - 1;
  GRID_STRIDE(s, nseg) {
    if (o.woff[s + 1] == o.woff[s]) continue;
    const int64_t a = o.seg[s], b = s + 1 < nseg ? o.seg[s + 1] : nrec;
    const int64_t row = o.segrow[s];
    len[row] += (o.pins[b] - o.pins[a]) - (o.pdel[b] - o.pdel[a]);
    if (o.newcap[s]) {
      off[row] = base + o.noff[s];
      cap[row] = o.newcap[s];
    }
  }
  for_seg_runs(o.woff, nseg, total, [&](int64_t t0, int n, int64_t slo, int64_t shi) {
    const int lane = threadIdx.x & 31;
    if (slo == shi && t0 + n <= o.woff[slo + 1] - (o.pins[slo + 1 < nseg ? o.seg[slo + 1] : nrec] - o.pins[o.seg[slo]])) {
      // kept entries of one row: the records between its first and its last
      // column are few, so one search per run leaves each entry next to none
      // (57 -> 45 us a level on the R-MAT of 2^20)
      const int64_t s = slo, a = o.seg[s], b = s + 1 < nseg ? o.seg[s + 1] : nrec;
      const int64_t to = o.newcap[s] ? base + o.noff[s] : off[o.segrow[s]];
      const int64_t from = o.soff[s], k0 = t0 - o.woff[s];
      const int32_t ia = o.pins[a], da = o.pdel[a];
      int32_t c[SEG_PL];
      WT x[SEG_PL];
#pragma unroll
      for (int j = 0; j < SEG_PL; ++j) {
        const int64_t i = from + k0 + j * 32 + lane;
        c[j] = j * 32 + lane < n ? scol[i] : 0;
        x[j] = j * 32 + lane < n ? sw[i] : 0;
      }
      // lane 0: records before the run's first column; the others: up to its last
      int64_t lo = a, hi = b;
      const int32_t cs = lane == 0 ? scol[from + k0] : scol[from + k0 + n - 1];
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int32_t)(keys[mid] & cmask) < cs) lo = mid + 1; else hi = mid;
      }
      const int64_t l0 = __shfl_sync(0xffffffffu, lo, 0), l1 = __shfl_sync(0xffffffffu, lo, 31);
#pragma unroll
      for (int j = 0; j < SEG_PL; ++j) {
        if (j * 32 + lane >= n) continue;
        int64_t q = l0, h = l1;  // records with a smaller column
        while (q < h) {
          const int64_t mid = (q + h) >> 1;
          if ((int32_t)(keys[mid] & cmask) < c[j]) q = mid + 1; else h = mid;
        }
        if (q < b && (int32_t)(keys[q] & cmask) == c[j]) {
          x[j] = (WT)((int64_t)x[j] + delta[q]);
          if (x[j] == 0) continue;  // deleted
        }
        const int64_t dst = to + k0 + j * 32 + lane - (o.pdel[q] - da) + (o.pins[q] - ia);
        col[dst] = c[j];
        w[dst] = x[j];
      }
      return;
    }
    for (int j = lane; j < n; j += 32) {
      const int64_t t = t0 + j, s = seg_of(o.woff, slo, shi, t);
      const int64_t a = o.seg[s];
      const int64_t b = s + 1 < nseg ? o.seg[s + 1] : nrec;
      const int64_t to = o.newcap[s] ? base + o.noff[s] : off[o.segrow[s]];
      const int32_t ia = o.pins[a], da = o.pdel[a];
      const int64_t lold = (o.woff[s + 1] - o.woff[s]) - (o.pins[b] - ia);
      const int64_t k = t - o.woff[s];
      if (k < lold) {
        const int32_t c = scol[o.soff[s] + k];
        WT x = sw[o.soff[s] + k];
        // records of this segment with a smaller column
        int64_t lo = a, hi = b;
        while (lo < hi) {
          const int64_t mid = (lo + hi) >> 1;
          if ((int32_t)(keys[mid] & cmask) < c) lo = mid + 1; else hi = mid;
        }
        if (lo < b && (int32_t)(keys[lo] & cmask) == c) {
          x = (WT)((int64_t)x + delta[lo]);
          if (x == 0) continue;  // deleted
        }
        const int64_t dst = to + k - (o.pdel[lo] - da) + (o.pins[lo] - ia);
        col[dst] = c;
        w[dst] = x;
      } else {
        const int64_t q = k - lold;  // q-th insert of the segment
        int64_t lo = a, hi = b - 1;
        while (lo < hi) {  // the record J with q inserts before it that is one itself
          const int64_t mid = (lo + hi) >> 1;
          if (o.pins[mid + 1] - ia <= q) lo = mid + 1; else hi = mid;
        }
        const int64_t dst = to + (int64_t)o.lb[lo] - (o.pdel[lo] - da) + q;
        col[dst] = (int32_t)(keys[lo] & cmask);
        w[dst] = (WT)delta[lo];
      }
    }
  });
}

// compaction: every live entry is one item (rows located through the scan of
// the row lengths), copied to its row's new offset (the scan of the caps)
template <class WT>
__global__ void k_compact_rows(int64_t n, const int64_t* off, const int64_t* lpre, int64_t total,
                               const int64_t* noff, const int32_t* col, const WT* w, int32_t* ncol, WT* nw) {
  pdl_enter();
  for_seg_runs(lpre, n, total, [&](int64_t t0, int cnt, int64_t slo, int64_t shi) {
    for (int64_t t = t0 + (threadIdx.x & 31); t < t0 + cnt; t += 32) {
      const int64_t v = seg_of(lpre, slo, shi, t), k = t - lpre[v];
      ncol[noff[v] + k] = col[off[v] + k];
      nw[noff[v] + k] = w[off[v] + k];
    }
  });
}

// ---------------------------------------------------------------- build
// Row lengths (cleared before) and first records of sorted records: a row's
// first and last record each add their share, where an atomic per record took
// 220 us for 16M records (neighbouring threads meet in one counter).
__global__ void k_row_bounds(const u64* keys, int64_t nrec, int bshift, int32_t* len, int64_t* start) {
  pdl_enter();
  GRID_STRIDE(i, nrec) {
    const int64_t row = (int64_t)(keys[i] >> bshift);
    if (i == 0 || (int64_t)(keys[i - 1] >> bshift) != row) {
      start[row] = i;
      atomicAdd((unsigned*)&len[row], 0u - (unsigned)i);  // modulo 2^32, as the length fits
    }
    if (i + 1 == nrec || (int64_t)(keys[i + 1] >> bshift) != row) atomicAdd((unsigned*)&len[row], (unsigned)(i + 1));
  }
}

__global__ void k_caps(const int32_t* cnt, int64_t n, int32_t* cap, int slack_pct) {
  pdl_enter();
  GRID_STRIDE(v, n) {
    const int64_t d = cnt[v];
    int64_t c = d + (d * slack_pct) / 100 + (d ? 2 : 0);
    c = (c + 1) & ~(int64_t)1;
    cap[v] = (int32_t)c;
  }
}

template <class WT>
__global__ void k_scatter_build(const u64* keys, const int64_t* vals, int64_t nrec, int bshift, const int64_t* rs,
                                const int64_t* off, int32_t* col, WT* w) {
  pdl_enter();
  const u64 cmask = (((u64)1) << bshift) - 1;
  GRID_STRIDE(i, nrec) {
    const int64_t row = (int64_t)(keys[i] >> bshift);
    const int64_t p = off[row] + (i - rs[row]);
    col[p] = (int32_t)(keys[i] & cmask);
    w[p] = (WT)vals[i];
  }
}

__global__ void k_i32_to_i64(const int32_t* a, int64_t* b, int64_t n) {
  pdl_enter();
  GRID_STRIDE(i, n) b[i] = a[i];
}

}  // namespace

// ---------------------------------------------------------------- host side
template <class WT>
void csr_build(SlackCSR<WT>& g, int64_t n, const u64* keys, const int64_t* vals, int64_t nrec, int bshift,
               int slack_pct, CsrScratch& S, Prims& P, cudaStream_t s) {
  g.n = n;
  if (g.off.cap < n + 1) {
    g.off.release(); g.len.release(); g.cap.release(); g.tables.release();
    g.tables.add(g.off, n + 1);
    g.tables.add(g.len, n + 1);
    g.tables.add(g.cap, n + 1);
    g.tables.alloc();
  }
  CK(cudaMemsetAsync(g.len.p, 0, sizeof(int32_t) * (size_t)(n + 1), s));
  S.rs.reserve(n + 1, s);
  if (nrec > 0) {
    launch(k_row_bounds, grid_for(nrec, TPB), TPB, 0, s, keys, nrec, bshift, g.len.p, S.rs.p);
    CKL("k_row_bounds");
  }
  launch(k_caps, grid_for(n, TPB), TPB, 0, s, g.len.p, n, g.cap.p, slack_pct);
  CKL("k_caps");
  const int64_t total = scan_exclusive_i32(g.cap.p, g.off.p, n, P, s, true);
  const int64_t pool = total + total / 8 + 1024;
  g.col.release();
  g.w.release();
  g.col.exact(pool);
  g.w.exact(pool);
  g.pool_top = total;
  if (nrec > 0) {
    launch(k_scatter_build<WT>, grid_for(nrec, TPB), TPB, 0, s, keys, vals, nrec, bshift, S.rs.p, g.off.p, g.col.p, g.w.p);
    CKL("k_scatter_build");
  }
}

// Copy every row into a fresh pool of `cap_total + extra` slots.
template <class WT>
static void compact_pool(SlackCSR<WT>& g, int64_t extra, CsrScratch& S, Prims& P, cudaStream_t s) {
  const int64_t n = g.n;
  S.tmp64.reserve(n + 1, s);
  S.rs.reserve(n + 1, s);
  launch(k_i32_to_i64, grid_for(n, TPB), TPB, 0, s, g.cap.p, S.tmp64.p, n);
  CKL("k_i32_to_i64");
  const int64_t total = scan_exclusive(S.tmp64.p, S.rs.p, n, P, s, true);  // new offsets
  // the same headroom again: rows that outgrow their slack move to the pool's
  // end, so a level whose rows churn refills it quickly
  const int64_t pool = 2 * (total + extra) + 4096;
  int32_t* c2 = (int32_t*)dalloc(sizeof(int32_t) * (size_t)pool);
  WT* w2 = (WT*)dalloc(sizeof(WT) * (size_t)pool);
  const int64_t live = scan_exclusive_i32(g.len.p, S.tmp64.p, n, P, s, true);
  if (live > 0) {
    launch(k_compact_rows<WT>, grid_for((live + 7) / 8, TPB), TPB, 0, s, n, g.off.p, S.tmp64.p, live, S.rs.p, g.col.p,
                                                                     g.w.p, c2, w2);
    CKL("k_compact_rows");
  }
  if (g.logging) {  // the offset table as it was, for a rollback
    g.lofs.reserve(g.otop + n, s, true);
    CK(cudaMemcpyAsync(g.lofs.p + g.otop, g.off.p, sizeof(int64_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
    g.events.push_back({true, 0, 0, 0, 0, g.otop, g.col.p});
    g.otop += n;
  }
  CK(cudaMemcpyAsync(g.off.p, S.rs.p, sizeof(int64_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
  CK(cudaStreamSynchronize(s));
  if (g.logging) {
    g.retired.emplace_back(g.col.p, g.w.p);  // freed when the batch commits
  } else {
    dfree(g.col.p);
    dfree(g.w.p);
  }
  g.col.p = c2;
  g.col.cap = pool;
  g.w.p = w2;
  g.w.cap = pool;
  g.pool_top = total;
}

static PlanOut plan_out(CsrScratch& S, DevScalars* d_sc) {
  return PlanOut{S.pos.p,    S.lb.p,     S.segid.p, S.pins.p, S.pdel.p, S.oldw.p,     S.seg.p,
                 S.segrow.p, S.newcap.p, S.soff.p,  S.woff.p, S.noff.p, &d_sc->seg_n, (u64*)&d_sc->plan_bad,
                 S.plans,    d_sc->plan};
}

template <class WT>
void csr_plan(const SlackCSR<WT>& g, const CsrRecords& r, CsrScratch& S, Prims& P, cudaStream_t s, DevScalars* d_sc,
              const DelTrack* trk, const Tail& tail) {
  const int64_t n_max = r.n_max;
  S.reserve_recs(n_max, s);  // the segment count stays on the device: one segment per record bounds it
  const RecN rn{n_max, r.n_dev, r.mul, r.gate};
  ++S.plans;
  const PlanOut o = plan_out(S, d_sc);
  const DelTrack t = trk ? *trk : DelTrack{};
  // Up to one record per thread of a block, one launch plans the update: 6.2 us
  // for a few records and 7.5 for some hundred, where the two tiled launches
  // take 8.9 and 9.9 and the gap between them.  Beyond, one block would match
  // several records per thread one after the other.
  if (n_max <= PS_TPB) {
    launch(k_plan_small<WT>, 1, PS_TPB, 0, s, g.off.p, g.len.p, g.cap.p, g.col.p, g.w.p, r.keys, r.delta, rn, r.bshift, o,
                                          t, tail);
    CKL("k_plan_small");
  } else {
    const int tiles = div_up(n_max, PL_TPB);
    const LookBack q1 = look_back_begin(P, 3 * (int64_t)tiles, s);
    launch(k_plan_records<WT>, tiles, PL_TPB, 0, s, g.off.p, g.len.p, g.col.p, g.w.p, r.keys, r.delta, rn, r.bshift, o, t,
                                                q1);
    CKL("k_plan_records");
    const LookBack q2 = look_back_begin(P, 3 * (int64_t)tiles, s);
    launch(k_plan_segments, tiles, PL_TPB, 0, s, g.len.p, g.cap.p, rn, o, q2, tail);
    CKL("k_plan_segments");
  }
}

template <class WT>
int64_t csr_apply(SlackCSR<WT>& g, const CsrRecords& r, CsrScratch& S, Prims& P, cudaStream_t s, DevScalars* d_sc,
                  const DelTrack* trk) {
  if (r.n_max <= 0) return 0;
  int64_t tot[6];
  const HostRead rr{d_sc->plan, tot, sizeof(tot)};
  csr_plan<WT>(g, r, S, P, s, d_sc, trk, P.tail_begin(P.rd_owner, &rr, 1));
  P.tail_wait(P.rd_owner, &rr, 1);
  return csr_finish<WT>(g, r, tot, S, P, s, d_sc);
}

template <class WT>
int64_t csr_finish(SlackCSR<WT>& g, const CsrRecords& r, const int64_t (&tot)[6], CsrScratch& S, Prims& P,
                   cudaStream_t s, DevScalars* d_sc) {
  const u64* keys = r.keys;
  const int64_t* delta = r.delta;
  const int bshift = r.bshift;
  const PlanOut o = plan_out(S, d_sc);
  const int64_t need = tot[0], nseg = tot[1], stotal = tot[2], wtotal = tot[3], nrec = tot[4];
  if (tot[5]) ldl_throw(LDL_E_INVALID, "internal: adjacency update would make a weight negative");
  if (nrec <= 0) return 0;
  if (g.pool_top + need > g.col.cap) compact_pool<WT>(g, need, S, P, s);
  DBuf<WT>& sw = S.template sw_of<WT>();
  UndoOut<WT> u{};
  int32_t* scol = nullptr;
  WT* swp = nullptr;
  if (g.logging) {
    // everything a rollback needs, reserved before any change
    g.reserve_log(g.rtop + nseg + 1, g.wtop + nrec + 1, g.ctop + stotal + 1, s);
    u = {g.lrow.p + g.rtop, g.loff.p + g.rtop, g.lsrc.p + g.rtop, g.lpos.p + g.wtop,
         g.llen.p + g.rtop, g.lcap.p + g.rtop, g.lold.p + g.wtop, g.ctop};
    scol = g.lcol.p + g.ctop;
    swp = g.lw.p + g.ctop;
  } else {
    S.scol.reserve(stotal + 1, s);
    sw.reserve(stotal + 1, s);
    scol = S.scol.p;
    swp = sw.p;
  }
  launch(k_apply<WT>, grid_for(std::max(nrec, (stotal + 7) / 8), TPB), TPB, 0, s,
      nrec, nseg, stotal, keys, delta, bshift, o, g.off.p, g.len.p, g.cap.p, g.col.p, g.w.p, scol, swp, u);
  CKL("k_apply");
  if (g.logging) {
    g.events.push_back({false, g.rtop, nseg, g.wtop, nrec, 0, g.col.p});
    g.rtop += nseg;
    g.wtop += nrec;
    g.ctop += stotal;
  }
  if (wtotal > 0) {
    launch(k_rebuild<WT>, grid_for(std::max(nseg, (wtotal + 7) / 8), TPB), TPB, 0, s,
        nrec, nseg, wtotal, g.pool_top, o, scol, swp, keys, delta, bshift, g.off.p, g.len.p, g.cap.p, g.col.p, g.w.p);
    CKL("k_rebuild");
    g.pool_top += need;
  }
  return nrec;
}

template <class WT>
void csr_txn_begin(SlackCSR<WT>& g) {
  g.logging = true;
  g.col0 = g.col.p;
  g.w0 = g.w.p;
  g.cap0 = g.col.cap;
  g.top0 = g.pool_top;
  g.retired.clear();
  g.events.clear();
  g.rtop = g.wtop = g.ctop = g.otop = 0;
}

template <class WT>
void csr_txn_commit(SlackCSR<WT>& g, cudaStream_t s) {
  if (!g.retired.empty()) {
    CK(cudaStreamSynchronize(s));
    for (auto& x : g.retired) {
      dfree(x.first);
      dfree(x.second);
    }
  }
  g.retired.clear();
  g.events.clear();
  g.logging = false;
}

template <class WT>
cudaError_t csr_txn_rollback(SlackCSR<WT>& g, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  // undo in reverse order; contents go back only into the batch's first pool
  for (size_t k = g.events.size(); k-- > 0 && e == cudaSuccess;) {
    const auto& ev = g.events[k];
    if (ev.offsets) {
      e = cudaMemcpyAsync(g.off.p, g.lofs.p + ev.o0, sizeof(int64_t) * (size_t)g.n, cudaMemcpyDeviceToDevice, s);
      continue;
    }
    const int restore = ev.col == g.col0 ? 1 : 0;
    if (ev.nr > 0) {
      const int grid = (int)std::min<int64_t>((ev.nr + 7) / 8, 4096);
      launch(k_undo_rows<WT>, grid, TPB, 0, s, ev.nr, g.lrow.p + ev.r0, g.loff.p + ev.r0, g.llen.p + ev.r0,
                                           g.lcap.p + ev.r0, g.lsrc.p + ev.r0, g.lcol.p, g.lw.p, g.off.p, g.len.p,
                                           g.cap.p, g.col0, g.w0, restore, g.top0);
      g_launches.fetch_add(1, std::memory_order_relaxed);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess && restore && ev.nw > 0) {
      const int grid = (int)std::min<int64_t>((ev.nw + TPB - 1) / TPB, 4096);
      launch(k_undo_weights<WT>, grid, TPB, 0, s, ev.nw, g.lpos.p + ev.w0, g.lold.p + ev.w0, g.w0, g.top0);
      g_launches.fetch_add(1, std::memory_order_relaxed);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  // back to the first pool; pools made during the batch go
  auto drop = [&](int32_t* cp, WT* wp) {
    if (cp != g.col0) dfree(cp);
    if (wp != g.w0) dfree(wp);
  };
  drop(g.col.p, g.w.p);
  for (auto& x : g.retired) drop(x.first, x.second);
  g.retired.clear();
  g.col.p = g.col0;
  g.w.p = g.w0;
  g.col.cap = g.w.cap = g.cap0;
  g.pool_top = g.top0;
  g.events.clear();
  g.logging = false;
  return e;
}

template void csr_txn_begin<int32_t>(SlackCSR<int32_t>&);
template void csr_txn_begin<int64_t>(SlackCSR<int64_t>&);
template void csr_txn_commit<int32_t>(SlackCSR<int32_t>&, cudaStream_t);
template void csr_txn_commit<int64_t>(SlackCSR<int64_t>&, cudaStream_t);
template cudaError_t csr_txn_rollback<int32_t>(SlackCSR<int32_t>&, cudaStream_t);
template cudaError_t csr_txn_rollback<int64_t>(SlackCSR<int64_t>&, cudaStream_t);

template void csr_build<int32_t>(SlackCSR<int32_t>&, int64_t, const u64*, const int64_t*, int64_t, int, int,
                                 CsrScratch&, Prims&, cudaStream_t);
template void csr_build<int64_t>(SlackCSR<int64_t>&, int64_t, const u64*, const int64_t*, int64_t, int, int,
                                 CsrScratch&, Prims&, cudaStream_t);
template void csr_plan<int32_t>(const SlackCSR<int32_t>&, const CsrRecords&, CsrScratch&, Prims&, cudaStream_t, DevScalars*,
                                const DelTrack*, const Tail&);
template int64_t csr_finish<int32_t>(SlackCSR<int32_t>&, const CsrRecords&, const int64_t (&)[6], CsrScratch&, Prims&,
                                     cudaStream_t, DevScalars*);
template int64_t csr_apply<int32_t>(SlackCSR<int32_t>&, const CsrRecords&, CsrScratch&, Prims&, cudaStream_t, DevScalars*,
                                    const DelTrack*);
template void csr_plan<int64_t>(const SlackCSR<int64_t>&, const CsrRecords&, CsrScratch&, Prims&, cudaStream_t, DevScalars*,
                                const DelTrack*, const Tail&);
template int64_t csr_finish<int64_t>(SlackCSR<int64_t>&, const CsrRecords&, const int64_t (&)[6], CsrScratch&, Prims&,
                                     cudaStream_t, DevScalars*);
template int64_t csr_apply<int64_t>(SlackCSR<int64_t>&, const CsrRecords&, CsrScratch&, Prims&, cudaStream_t, DevScalars*,
                                    const DelTrack*);
