// Pieces shared by the tensor-core attention kernels: bounded mbarrier waits, the row-block
// decomposition of the chunked mask (Section 3.2, Attn-Fill 1/2), TMA descriptor creation.
#pragma once

#include "lrsa_internal.h"
#include "sm100_ptx.h"

namespace lrsa {

constexpr int kTile = 128;                 // rows of a query tile, keys of a key tile
constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz: no wait in a correct run gets close

// Waits for the phase with the given parity; gives up (returns false, raises *abort) when another
// thread of the CTA has given up or after kWaitCycles.  For a branch of one thread: every lane reads the clock and *abort
// by itself, so the lanes of a warp may give up apart from one another.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  if (ptx::mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t it = 0;; ++it) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 63u) {
      if (*abort) return false;
      if (clock64() - t0 > kWaitCycles) { *abort = 1; return false; }
    }
  }
}

// The same wait executed by all 32 lanes of a converged warp, with one verdict for the warp: what follows is
// warp-wide (tensor-memory accesses, __syncwarp) and must be reached by all lanes or by none.  The
// warps that issue tcgen05.mma run in warp-uniform control flow with descriptors computed once
// outside the loops (building a descriptor per instruction in a single-lane branch costs ~100
// cycles per MMA, more than the MMA itself) and issue through one lane, by predicate.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort) {
  const bool ok = mbar_wait(bar, parity, abort);
  return __all_sync(0xffffffffu, ok);
}

// The same wait executed by all 32 lanes, with a verdict for each: the caller must not branch on them before it has voted
// (__all_sync), so that the lanes stay together.
__device__ __forceinline__ bool mbar_wait_lanes(uint32_t bar, uint32_t parity, volatile int* abort) {
  return mbar_wait(bar, parity, abort);
}

// A block of query rows that share one key list: rows [q0, q_end) (at most `rows_per_block`), all in
// one query chunk (or the sink region).  Their keys are the first n_front rows of the compact
// (sinks + kept) buffer followed by original positions [dense_start, own position].
struct RowBlock {
  int q0, q_end;      // query rows of this block
  int n_front;        // compact rows visible: S + n_c*K (0 for sink queries)
  int dense_start;    // first position of the contiguous key range
};

struct BlockPlan {
  int S, L, K, N, W, T, Wsel, ndp;
  int rows;           // rows per block (128 or 256)
  int per_chunk;      // blocks per full chunk
  int per_tail;       // blocks of the tail chunk
  int per_sink;       // blocks of the sink region
  int total;          // per (batch, head)
};

inline BlockPlan make_plan(const Geom& g, int rows) {
  BlockPlan p;
  p.S = g.S; p.L = g.L; p.K = g.K; p.N = g.N; p.W = g.W; p.T = g.T; p.Wsel = g.Wsel; p.ndp = g.ndp;
  p.rows = rows;
  p.per_chunk = (g.L + rows - 1) / rows;
  p.per_tail = (g.T + rows - 1) / rows;
  p.per_sink = (g.S + rows - 1) / rows;
  p.total = g.W * p.per_chunk + p.per_tail + p.per_sink;
  return p;
}

// Blocks are numbered from the end of the sequence: tail chunk, then full chunks from the last to the first (inside a chunk
// from the last rows to the first), then the sink region.  That is roughly heaviest first: the list grows from chunk to chunk, but with
// L > K the first rows of a chunk have fewer keys than the last rows of the chunk in front of it.
__device__ __forceinline__ RowBlock decode_block(const BlockPlan& p, int blk) {
  RowBlock r;
  int c, i;
  if (blk < p.per_tail) {
    c = p.W; i = p.per_tail - 1 - blk;
  } else if (blk < p.per_tail + p.W * p.per_chunk) {
    blk -= p.per_tail;
    c = p.W - 1 - blk / p.per_chunk;
    i = p.per_chunk - 1 - blk % p.per_chunk;
  } else {
    i = blk - p.per_tail - p.W * p.per_chunk;
    r.q0 = i * p.rows;
    r.q_end = min(p.S, r.q0 + p.rows);
    r.n_front = 0;
    r.dense_start = 0;
    return r;
  }
  const int c0 = p.S + c * p.L;
  const int c1 = min(p.N, c0 + p.L);
  r.q0 = c0 + i * p.rows;
  r.q_end = min(c1, r.q0 + p.rows);
  const int nh = n_hist_windows(c, p.ndp, p.Wsel);
  r.n_front = p.S + nh * p.K;
  r.dense_start = p.S + nh * p.L;
  return r;
}

// 3-D bf16 tensor map over [outer][rows][d] with a (64 x box_rows x 1) box and 128-byte swizzle.
// `row_stride`: rows between consecutive `outer` slices in memory (0: rows); larger when the map covers
// one sequence of a packed row.
int make_tmap_bf16(CUtensorMap* map, const void* base, int d, long long rows, long long outer, int box_rows,
                   long long row_stride = 0);

// The sequences of a packed batch are taken up to kMaxSeqs at a time by one launch of each kernel (their tensor maps travel
// as kernel parameters), longest first.  An unpacked batch is one sequence.  row0: first row of the sequence's part of the
// compact buffers.
constexpr int kMaxSeqs = 16;
struct SeqBatch {
  int n;
  Geom g[kMaxSeqs];
  long long row0[kMaxSeqs];
};
struct SeqBatches {
  const Geom& whole;
  int s = 0, woff = 0;
  explicit SeqBatches(const Geom& w) : whole(w) {}
  bool next(SeqBatch* b);   // false: none left
};

// Rows of the compact buffers per KV head: what the largest batch of a call takes, and what a batch takes at most in any
// packing of rows of this shape (k sequences have k - 1 times the sinks more than the row unpacked, and never more kept rows).
inline long long compact_rows_used(const Geom& g) {
  if (g.n_seqs == 0) return g.Rc > 0 ? g.Rc : 1;
  long long most = 1, sum = 0;
  for (int s = 0; s < g.n_seqs; ++s) {
    if (s % kMaxSeqs == 0) sum = 0;
    const int n = g.cu[s + 1] - g.cu[s], S = g.S < n ? g.S : n, w = (n - S) / g.L;
    sum += S + (long long)(w > 1 ? w - 1 : 0) * g.K;
    if (sum > most) most = sum;
  }
  return most;
}
inline long long compact_rows_bound(const Geom& g) {
  const long long rows = g.Rc + (kMaxSeqs - 1LL) * g.S;
  return rows < 1 ? 1 : rows < g.N ? rows : g.N;
}

// Gather of the sink rows and the kept rows of K and V into the compact buffers: per sequence Kc, Vc [B*Hkv][Rc][d] (the
// condensed KV cache of Section 3.2) for the query-outer kernels, which stream the list once per query tile (a TMA row
// gather in their main loops was measured at about 6 bytes per clock and SM, a fifth of what they consume).  256 threads
// a block, 16 bytes of K and of V each.
struct CompactArgs {
  const __nv_bfloat16 *K, *V;
  const int32_t* idx;
  __nv_bfloat16 *Kc, *Vc;
  int* status;                 // cleared when not null
  int Nrow, cpr, kept_stride, n;   // cpr: 16-byte chunks per row
  int item0[kMaxSeqs + 1];     // rows before the sequence's, over all (batch, KV head) pairs
  int Rc[kMaxSeqs], S[kMaxSeqs], tok0[kMaxSeqs], kept_off[kMaxSeqs];
  long long row0[kMaxSeqs];
  int blocks() const { return (int)(((long long)item0[n] * cpr + 255) / 256); }
};
inline CompactArgs compact_args(const Geom& whole, const SeqBatch& b, const __nv_bfloat16* K, const __nv_bfloat16* V,
                                const int32_t* idx, __nv_bfloat16* Kc, __nv_bfloat16* Vc, int* status) {
  CompactArgs c;
  c.K = K; c.V = V; c.idx = idx; c.Kc = Kc; c.Vc = Vc; c.status = status;
  c.Nrow = whole.Nrow; c.cpr = whole.d / 8; c.kept_stride = whole.Wtot * whole.K; c.n = b.n;
  c.item0[0] = 0;
  for (int s = 0; s < b.n; ++s) {
    const Geom& g = b.g[s];
    c.item0[s + 1] = c.item0[s] + g.B * g.Hkv * g.Rc;
    c.Rc[s] = g.Rc; c.S[s] = g.S; c.tok0[s] = g.tok0; c.kept_off[s] = g.woff * g.K; c.row0[s] = b.row0[s];
  }
  return c;
}
__device__ __forceinline__ void compact_rows(const CompactArgs& c, int block) {
  const int item = block * (256 / c.cpr) + (int)threadIdx.x / c.cpr, ch = threadIdx.x % c.cpr;
  if (item >= c.item0[c.n]) return;
  int s = 0;
  while (item >= c.item0[s + 1]) ++s;
  const int i = item - c.item0[s], bh = i / c.Rc[s], r = i - bh * c.Rc[s];
  const int pos = r < c.S[s] ? r + c.tok0[s] : c.idx[(size_t)bh * c.kept_stride + c.kept_off[s] + (r - c.S[s])];
  const size_t src = ((size_t)bh * c.Nrow + pos) * c.cpr + ch, dst = (size_t)(c.row0[s] + i) * c.cpr + ch;
  const uint4 k = reinterpret_cast<const uint4*>(c.K)[src], v = reinterpret_cast<const uint4*>(c.V)[src];
  reinterpret_cast<uint4*>(c.Kc)[dst] = k;
  reinterpret_cast<uint4*>(c.Vc)[dst] = v;
}

// Writes `BYTES` bytes (whole 16-byte chunks) of each of a warp's 32 rows from shared memory, `stride` bytes apart, to rows
// `row_bytes` apart in global memory: neighbouring lanes take neighbouring chunks of a row.  Rows at or beyond n_rows are skipped.
template <int BYTES>
__device__ __forceinline__ void store_rows(const unsigned char* src, int stride, unsigned char* dst, int row_bytes, int n_rows, int lane) {
  constexpr int kLanes = BYTES / 16, kRows = 32 / kLanes;   // lanes per row, rows per instruction
  const int chunk = lane % kLanes * 16;
#pragma unroll
  for (int r = lane / kLanes; r < 32; r += kRows)
    if (r < n_rows)
      *reinterpret_cast<uint4*>(dst + (size_t)r * row_bytes + chunk) = *reinterpret_cast<const uint4*>(src + r * stride + chunk);
}

// 2-D bf16 tensor map over [rows][d] with a (64 x 1) box and 128-byte swizzle, for row gathers
// (tile::gather4).  The key-outer dK/dV kernel loads its one list tile per CTA this way, four rows per
// copy, straight from K and V into the swizzled operand tile.
int make_tmap_bf16_rows(CUtensorMap* map, const void* base, int d, long long rows);

// Original position of row r of the compact (sinks + kept) key list of one (batch, KV head); `kept`
// points at that head's idx entries.  Rows at or beyond n_rows are never used by a product (their scores
// are masked); they map to position 0 so that the row fetched for them is valid, finite data.
// Positions are local to the sequence (kept entries are positions in the whole row, tok0 + local).
__device__ __forceinline__ int compact_row_pos(const int32_t* kept, int S, int n_rows, int r, int tok0) {
  if (r >= n_rows) return 0;
  return r < S ? r : kept[r - S] - tok0;
}

}  // namespace lrsa
