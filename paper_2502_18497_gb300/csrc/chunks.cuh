// Load-balanced iteration over the rows of a node list.
//
// Every listed node is split into chunks of CH adjacency entries (out-row
// chunks first, then in-row chunks); a node with empty rows still gets one
// chunk so that per-node work has a place to run.  An exclusive scan of the
// chunk counts maps a global chunk id back to (node, row, range) by binary
// search, so a hub row is spread over many warps instead of one.
#pragma once
#include "ctx.cuh"

constexpr int CH = 256;

struct ChunkMap {
  const int32_t* list;   // nodes
  const int64_t* pre;    // exclusive scan of chunk counts, length n_hint + 1 (null: see chunk_begin)
  int64_t n_hint;        // list capacity used for the scan
  const int32_t* len_a;  // first row lengths (out)
  const int32_t* len_b;  // second row lengths (in) or nullptr
  const int32_t* nlist;  // device count of the list
};

// Lists of up to CH_SMALL nodes are scanned by every block of the kernel that
// walks them, into shared memory.  As a launch of its own the one-block scan
// of so short a list took 3.8 us and the gap in front of it 2.9, 36 times a
// batch of 10^4 on the R-MAT of 2^20, and the searches went to L2.  Longer
// lists keep the separate scan (10 us at some 10^4 nodes): every block would
// read all of their lengths.
constexpr int CH_SMALL = 1024;
struct ChunkPre {
  int32_t pre[CH_SMALL + 1];
  int32_t wsum[32];
};

struct Chunk {
  int64_t idx;    // position in the list
  int32_t v;      // node
  int32_t first;  // 1 for the node's first chunk
  int32_t row;    // 0: first row, 1: second row, -1: none
  int32_t k0, k1; // entry range in that row
};

// Called by every thread of the block (a multiple of 32, at most 1024) before
// chunk_of; returns the number of chunks.
__device__ inline int64_t chunk_begin(const ChunkMap& m, ChunkPre& sh) {
  if (m.pre) return m.pre[m.n_hint];
  const int n = min((int)m.n_hint, *m.nlist), nt = blockDim.x, tid = threadIdx.x;
  const int lane = tid & 31, wid = tid >> 5;
  int base = 0;
  for (int i0 = 0; i0 < n; i0 += nt) {
    const int i = i0 + tid;
    int c = 0;
    if (i < n) {
      const int32_t v = m.list[i];
      c = (m.len_a[v] + CH - 1) / CH + (m.len_b ? (m.len_b[v] + CH - 1) / CH : 0);
      if (c == 0) c = 1;
    }
    int x = c;
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) sh.wsum[wid] = x;
    __syncthreads();
    int before = base, all = base;
    for (int w = 0; w < nt / 32; ++w) {
      if (w < wid) before += sh.wsum[w];
      all += sh.wsum[w];
    }
    if (i < n) sh.pre[i] = before + x - c;
    base = all;
    __syncthreads();
  }
  if (tid == 0) sh.pre[n] = base;
  __syncthreads();
  return base;
}

// Chunk c, the same in every lane of a warp that calls it together.
__device__ inline Chunk chunk_of(const ChunkMap& m, const ChunkPre& sh, int64_t c) {
  const int64_t lo = m.pre ? warp_find(m.pre, m.n_hint, c) : warp_find(sh.pre, min(m.n_hint, (int64_t)*m.nlist), c);
  const int64_t start = m.pre ? m.pre[lo] : sh.pre[lo];
  Chunk r;
  r.idx = lo;
  r.v = m.list[lo];
  const int64_t j = c - start;
  r.first = j == 0;
  const int32_t la = m.len_a[r.v];
  const int32_t lb = m.len_b ? m.len_b[r.v] : 0;
  const int64_t ca = (la + CH - 1) / CH;
  if (j < ca) {
    r.row = 0;
    r.k0 = (int32_t)(j * CH);
    r.k1 = min(la, r.k0 + CH);
  } else if (lb > 0) {
    r.row = 1;
    r.k0 = (int32_t)((j - ca) * CH);
    r.k1 = min(lb, r.k0 + CH);
  } else {
    r.row = -1;
    r.k0 = r.k1 = 0;
  }
  return r;
}

// The map of `list` (device count *nlist <= n_hint); lists above CH_SMALL are
// scanned here, the total chunk count at pre[n_hint] on the device (no sync).
ChunkMap chunk_map(ldl_ctx& c, const int32_t* list, const int32_t* nlist, int64_t n_hint, const int32_t* len_a,
                   const int32_t* len_b);
// Blocks of 256 threads for a kernel that walks the chunks of n_hint nodes: a
// warp per four nodes, and two blocks per SM where that is more, as a short
// list may hold hubs.
int chunk_grid(int64_t n_hint);
