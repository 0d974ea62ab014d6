// Declarations of the slack-CSR operations (csr.cu).
#pragma once
#include "common.cuh"
#include "prims.cuh"

// last s in [lo, hi] with pre[s] <= t
__device__ inline int64_t seg_in(const int64_t* pre, int64_t lo, int64_t hi, int64_t t) {
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Items [0, total) split into segments by the exclusive scan pre.  Each warp
// takes runs of SEG_RUN consecutive items: two warp-wide searches bound the
// run's segments.  f(t0, n, slo, shi) is called by the whole warp for the n
// items from t0 on, whose segments are slo .. shi; lane l's items are t0 + l,
// t0 + l + 32, ...
constexpr int SEG_RUN = 256;
constexpr int SEG_PL = SEG_RUN / 32;  // items per lane
template <class F>
__device__ inline void for_seg_runs(const int64_t* pre, int64_t nseg, int64_t total, F f) {
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t0 = warp * SEG_RUN; t0 < total; t0 += nwarps * SEG_RUN) {
    const int n = (int)min((int64_t)SEG_RUN, total - t0);
    const int64_t slo = warp_find(pre, nseg, t0);
    const int64_t shi =
        slo + 1 >= nseg || pre[slo + 1] > t0 + n - 1 ? slo : warp_find(pre, nseg, t0 + n - 1, slo + 1);
    f(t0, n, slo, shi);
  }
}

// The segment of item t of such a run.
__device__ inline int64_t seg_of(const int64_t* pre, int64_t slo, int64_t shi, int64_t t) {
  return slo == shi ? slo : seg_in(pre, slo, shi, t);
}

struct CsrScratch {
  // per record and per segment of an update (for max_rec of them, in one slab)
  DBuf<int64_t> seg, segrow, oldw, soff, woff, noff;
  DBuf<int32_t> pos, lb, newcap, pins, pdel, segid;
  Slab recs;
  int64_t max_rec = 0;
  DBuf<int64_t> rs, tmp64, sw64;
  DBuf<int32_t> scol, sw32;
  u64 plans = 0;  // updates planned so far
  template <class WT>
  DBuf<WT>& sw_of();
  void drop_recs() {
    for (auto* b : {&seg, &segrow, &oldw, &soff, &woff, &noff}) b->release();
    for (auto* b : {&pos, &lb, &newcap, &pins, &pdel, &segid}) b->release();
    recs.release();
    max_rec = 0;
  }
  void reserve_recs(int64_t n, cudaStream_t s) {
    if (n <= max_rec) return;
    int64_t nc = max_rec ? max_rec : 1024;
    while (nc < n) nc = nc * 3 / 2 + 1024;
    CK(cudaStreamSynchronize(s));
    drop_recs();
    for (auto* b : {&seg, &segrow, &oldw, &soff, &woff, &noff}) recs.add(*b, nc + 2);
    for (auto* b : {&pos, &lb, &newcap, &pins, &pdel, &segid}) recs.add(*b, nc + 2);
    recs.alloc();
    max_rec = nc;
  }
  void release() {
    drop_recs();
    for (auto* b : {&rs, &tmp64, &sw64}) b->release();
    for (auto* b : {&scol, &sw32}) b->release();
  }
};
template <>
inline DBuf<int32_t>& CsrScratch::sw_of<int32_t>() { return sw32; }
template <>
inline DBuf<int64_t>& CsrScratch::sw_of<int64_t>() { return sw64; }

// Build g over rows [0,n) from sorted unique records (key = row<<bshift|col,
// vals = weights), with slack_pct percent spare capacity per row.
template <class WT>
void csr_build(SlackCSR<WT>& g, int64_t n, const u64* keys, const int64_t* vals, int64_t nrec, int bshift,
               int slack_pct, CsrScratch& S, Prims& P, cudaStream_t s);

// Binary search of col in a sorted row: the lower bound index.
__device__ inline int32_t row_lower_bound(const int32_t* col, int64_t off, int32_t len, int32_t c) {
  int32_t lo = 0, hi = len;
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if (col[off + mid] < c) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Where csr_apply records the endpoints (row and column) of the entries it
// removes, for records whose row is below `rows`: a dedup stamp with its
// epoch, a list and its device counter.
struct DelTrack {
  int32_t* stamp;
  int32_t ep;
  int32_t* list;
  int32_t* cnt;
  int64_t rows;
  const int32_t* par;  // with it, arcs between two different parents are not recorded
};

// Batch transactions on a CSR (see SlackCSR's undo log): begin logging,
// commit (free pools replaced during the batch), or roll back to the state
// at begin.  Rollback only copies (no allocation) and synchronises s.
template <class WT>
void csr_txn_begin(SlackCSR<WT>& g);
template <class WT>
void csr_txn_commit(SlackCSR<WT>& g, cudaStream_t s);
template <class WT>
cudaError_t csr_txn_rollback(SlackCSR<WT>& g, cudaStream_t s);

// Records of an update, key (row << bshift | col) and delta, sorted by key and
// unique: n_max of them, or mul * *n_dev (device count, n_max an upper bound);
// none where the gate is given and *gate is zero when the update is planned.
struct CsrRecords {
  const u64* keys;
  const int64_t* delta;
  int64_t n_max;
  const int32_t* n_dev;
  int mul;
  int bshift;
  const int32_t* gate = nullptr;
};

// Add delta to each record's entry: absent entries are inserted, entries that
// reach zero are removed (their endpoints go to *trk when given).  In two
// halves: csr_plan launches the planning, whose last kernel hands over `tail`
// (the caller reads d_sc->plan with it and waits), and csr_finish, given those
// totals, applies the update and returns the number of records.  No other
// update is planned in between.
template <class WT>
void csr_plan(const SlackCSR<WT>& g, const CsrRecords& r, CsrScratch& S, Prims& P, cudaStream_t s, DevScalars* d_sc,
              const DelTrack* trk, const Tail& tail);
template <class WT>
int64_t csr_finish(SlackCSR<WT>& g, const CsrRecords& r, const int64_t (&tot)[6], CsrScratch& S, Prims& P,
                   cudaStream_t s, DevScalars* d_sc);
// both, with the wait between them
template <class WT>
int64_t csr_apply(SlackCSR<WT>& g, const CsrRecords& r, CsrScratch& S, Prims& P, cudaStream_t s, DevScalars* d_sc,
                  const DelTrack* trk = nullptr);
