// Host-side launchers of the algorithm kernels (sweep.cu, hier.cu).
#pragma once
#include "ctx.cuh"

struct CommitOut {
  i128 dq;     // exact change of the Eq. 1 numerator
  i128 dp;     // change of sum_C K_out K_in
  int64_t de;  // change of sum_C e_C
  int32_t ntc; // touched communities
};

// Degree bins of the sweeps: a node with d adjacency entries goes to the
// first bin whose bound is >= d (8-lane groups, warps, 128-thread blocks,
// 256-thread blocks; beyond: clusters / hub path).  Default bounds, and the
// largest bound each bin's hash table allows while staying at most half full.
constexpr int32_t BIN_DEFAULT[4] = {24, 96, 1024, 2048};
constexpr int32_t BIN_MAX[4] = {32, 128, 1024, 2048};

// The state of a level's split (TouchedRefined): `done` when its first kernels
// have run behind the sweep that ended the level's moves.
struct SplitRun {
  bool done = false;
  int32_t epD = 0, epL = 0, epF = 0;
  int32_t nleft = 0, nx = 0;  // nodes that left, refined communities to check
};

// ---- sweep.cu
void expand_set(ldl_ctx& c, int r, const int32_t* list, int idx_n, int32_t* stamp, int32_t ep, int32_t* olist,
                int idx_out, int64_t n_hint);
// U = U* = the existing nodes of A^r (lists lU and lUstar, stamp stU with
// epU) and the entries of their rows (c.sums).
void frontier(ldl_ctx& c, int r, int32_t epU, const Tail& tail);
void union_into(ldl_ctx& c, const int32_t* list, int idx_n, int32_t* stamp, int32_t ep, int32_t* olist, int idx_out,
                int64_t n_hint);
// BestMove (mode 0) / BestRef (mode 1) over the listed nodes, then the
// decoupling filter over the candidates: the list's length, the number of
// candidates and the number accepted (in bv / bsrc / bdst).
struct SweepOut {
  int32_t nlist, nc, nb;
};
// With `spec` the level's split starts in the same launch sequence if no move
// is accepted.
SweepOut sweep(ldl_ctx& c, int r, int mode, const int32_t* list, int idx_n, int64_t n_hint, SplitRun* spec = nullptr);
// Decoupling filter over the last sweep's candidates; the values of `extra`
// arrive in the same host wait.
struct DecoupleOut {
  int32_t nc, nb, rounds;
};
// (With spec: see sweep; `hubs`: the candidates may lack those of hub rows.)
DecoupleOut decouple(ldl_ctx& c, const HostRead* extra = nullptr, int n_extra = 0, SplitRun* spec = nullptr, int r = 0,
                     bool hubs = false);
// Launches the commit of a mini-batch; commit_expand then expands the next
// frontier U = V + N(V) and reads the outcome and |U|.
void commit_move(ldl_ctx& c, int r, int32_t nb, int32_t epB, int32_t epT, int32_t epCh);
CommitOut commit_expand(ldl_ctx& c, int r, int32_t nb, int32_t ep, int32_t* nU);
void rollback_move(ldl_ctx& c, int r, int32_t nb, int32_t ntc);
// moved nodes into lMv (level 0: lM0 too), and the next U (nU nodes) into U*
void mark_moved(ldl_ctx& c, int r, int32_t nb, int32_t epMv, int32_t epM0, int32_t epU, int32_t nU);
void commit_ref(ldl_ctx& c, int r, int32_t nb);
void spexpand(ldl_ctx& c, int r, int32_t nb, int32_t epD, int32_t epR, int32_t* lR, int idx_R);

// ---- hier.cu
// Batch validation and net deltas; leaves the sorted arcs in (c.rk, c.rv)
// and returns their count.  Throws (state untouched) on a bad batch.
int64_t ingest(ldl_ctx& c, const ldl_update* upd, int64_t count, int on_device, int64_t* dm);
// Apply the level-0 arcs to the adjacency and repair every statistic along
// the parent chain; marks InitFrontier in the A lists (epA per level).
// The sums that change m, E and P stay on the device (c.racc) until repair_done.
void repair_batch(ldl_ctx& c, int64_t na, const int32_t* epA, int32_t epT);
void repair_done(ldl_ctx& c, const RepairAcc& a, int64_t dm);
void pending_reset(ldl_ctx& c);
// known: the level's pending record count when the caller has read it, else -1
void flush_level(ldl_ctx& c, int q, int64_t known = -1);
// The same in two halves for a list that has records: flush_plan sorts it and
// plans the update, unless *gate is zero by then, and waits for the read rr (n
// values, room for one more) with the plan's totals; flush_finish applies it
// (n: the list's length).  Without the second half the list stays as it was.
void flush_plan(ldl_ctx& c, int q, const int32_t* gate, HostRead* rr, int n, int64_t (&tot)[6]);
void flush_finish(ldl_ctx& c, int q, int64_t n, const int64_t (&tot)[6]);
// moved_ub: an upper bound of the level's moved nodes (0 when none moved)
void pushdown(ldl_ctx& c, int r, int32_t epCh, int64_t moved_ub);
int32_t dissolve_all(ldl_ctx& c, int r, int32_t epD);
// TouchedRefined's first kernels, with the values rr[0..n) and the two of the
// split (room for them) handed over by the last; `gated`: only if no move was
// accepted (and, with `hubs`, no hub row is left).
void split_launch(ldl_ctx& c, int r, SplitRun& sr, bool gated, bool hubs, HostRead* rr, int n);
int32_t split(ldl_ctx& c, int r, SplitRun& sr);
// the listed level-r nodes that are singleton refined communities -> out
// (their count stays on the device, at cp[idx_out])
void singletons_of(ldl_ctx& c, int r, const int32_t* list, int idx_n, int64_t n_hint, int32_t* out, int idx_out);
// nD = |D| (list lD), the nodes whose refined community changed.
void aggregate(ldl_ctx& c, int r, int32_t epD, int32_t epC, int32_t epA_next, bool build, int32_t nD);
// context set-up and tear-down (ldl.cu)
void alloc_globals(ldl_ctx& c);
void free_all(ldl_ctx& c);
ldl_status ctx_new(const ldl_params& p, int64_t n, ldl_ctx** out);
void set_create_error(const std::string& msg);
// static set-up of level 0 from a host CSR
void upload_graph(ldl_ctx& c, int64_t nnz, const int64_t* row_ptr, const int32_t* col, const int32_t* w);
void level_alloc(ldl_ctx& c, int r);
void level_free(ldl_ctx& c, int r);
int32_t alive_list(ldl_ctx& c, int r, int32_t* list, int idx);
void reset_par(ldl_ctx& c, int r, int32_t nD);
// the level-0 nodes whose label differs from the batch's start -> lChg
// (count at cp[K_CHG], which the caller clears); the read rr ends it
void changed_labels(ldl_ctx& c, const HostRead* rr, int n);
void gather_labels(ldl_ctx& c, const int32_t* ids, int32_t k, int32_t* out);
