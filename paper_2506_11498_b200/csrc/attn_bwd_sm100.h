// What the kernels of the backward share: the tiles and launch order of the dK/dV kernel, the pointers of a call.
#pragma once

#include "attn_common_sm100.h"

namespace lrsa {

constexpr int kQRows = 128;   // query rows per inner tile
// Inner iterations per CTA of the dK/dV kernel, from their number in the whole call: at most 128 (a CTA's start and its
// additions to the accumulators are then lost in the rest), fewer in small problems, so that the longest list does not
// outlast an even share (iterations / 148) by much, and never below 16.  Whole backward, us, at 8 | 16 | 32 | 64 | 128 iterations a CTA (the
// rule's), windows of 512 and a quarter kept where nothing else stands:
// 8/8 heads, d = 64: 2K tokens 42 | 52 | 52 | 52 | 52 (16), 4K 83 | 81 | 90 | 90 | 90 (16), 8K 192 | 181 | 175 | 174 | 173 (16), windows of 1024
// 240 | 216 | 212 | 212 | 212 (16), 16K 555 | 509 | 496 | 488 | 484 (37: 489), of 1024 649 | 579 | 570 | 563 | 562 (45: 560);
// 16/2, d = 64: 4K 138 | 132 | 126 | 157 | 240 (16), 8K 334 | 310 | 297 | 297 | 314 (23: 307);
// 28/4, d = 128: 1777 105 | 98 | 99 | 139 | 213 (16), 4K 298 | 278 | 276 | 268 | 306 (16), 8K 819 | 750 | 734 | 739 | 715 (41: 725), windows of
// 1024 995 | 922 | 892 | 886 | 915 (53: 878), 16K 2910 | 2628 | 2508 | 2414 | 2420 (128), 32K 9197 | 8269 | 7771 | 7555 | 7480 (128);
// 32/8: 2K 141 | 129 | 133 | 180 | 179 (16), 4K 348 | 326 | 321 | 312 | 362 (16), 20K of 256 3785 | 3416 | 3264 | 3113 | 3093 (128).
// At d = 64 the rule is 4 % off around 8K tokens and a fifth at 2K, where 8 would fill the SMs better.
constexpr int kSegMax = 128;
inline int dkv_segment(long long iters) {
  const long long s = iters / (kSms * 4);
  return s < 16 ? 16 : s > kSegMax ? kSegMax : (int)s;
}

// Launch order of the dK/dV kernel: by length (see dkv_setup), with segments of a tile made about equally long?  Up to four CTAs per SM what
// the last ones leave idle is what counts, beyond that the query tiles that neighbours share in L2.  Whole backward, us, by length
// up to 0 | 4 | 6 | 8 CTAs per SM (windows of 512, a quarter kept): 1777 tokens (28/4 heads, d = 128) 107 | 99 | 99 | 99, 5K (16/2, d = 64)
// 155 | 153 | 153 | 153; 4K (28/4) 278 | 279 | 285 | 285, 8K (8/8, d = 64) 181 | 181 | 187 | 187; windows of 1024 (28/4): 8K 875 | 874 | 904 | 914,
// 16K 2430 | 2440 | 2446 | 2509.
inline bool order_by_length(long long ctas) {
  return ctas <= 4 * kSms;
}

struct DkvPlan {
  int S, L, K, N, W, T, C, Wsel, ndp, Rc, G;
  int n_cmp;       // compact tiles
  int n_sink;      // dense tiles of the sink region
  int per_win;     // dense tiles per full window
  int per_tail;    // dense tiles of the tail
  int n_tiles;
  int seg;         // inner iterations per CTA at most
  int by_length;   // launch order
};

struct KvTile {
  int kind;      // 0 compact, 1 dense
  int row0;      // first compact row / first key position
  int key_end;   // rows at or beyond this are not part of the tile
  int qb, qend;  // query positions [qb, qend) see (part of) the tile
  int nq;        // query tiles (kQRows rows) per head
};

inline DkvPlan make_dkv_plan(const Geom& g, int seg) {
  DkvPlan p;
  p.S = g.S; p.L = g.L; p.K = g.K; p.N = g.N; p.W = g.W; p.T = g.T; p.C = g.C; p.Wsel = g.Wsel;
  p.ndp = g.ndp; p.Rc = g.Rc; p.G = g.G;
  p.n_cmp = (g.Rc + kTile - 1) / kTile;
  p.n_sink = (g.S + kTile - 1) / kTile;
  p.per_win = (g.L + kTile - 1) / kTile;
  p.per_tail = (g.T + kTile - 1) / kTile;
  p.n_tiles = p.n_cmp + p.n_sink + g.W * p.per_win + p.per_tail;
  p.seg = seg;
  p.by_length = 0;
  return p;
}

__host__ __device__ inline KvTile describe_tile(const DkvPlan& p, int tile) {
  KvTile t;
  if (tile < p.n_cmp) {
    t.kind = 0;
    t.row0 = tile * kTile;
    t.key_end = p.Rc;
    int cmin = 0;
    if (t.row0 >= p.S) cmin = first_compressed_chunk((t.row0 - p.S) / p.K, p.ndp, p.Wsel, p.C);
    t.qb = p.S + cmin * p.L;
    t.qend = cmin >= p.C ? t.qb : p.N;
  } else {
    t.kind = 1;
    int d = tile - p.n_cmp;
    if (d < p.n_sink) {
      t.row0 = d * kTile; t.key_end = p.S; t.qend = p.S;
    } else {
      d -= p.n_sink;
      int w;
      if (d < p.W * p.per_win) {
        w = d / p.per_win;
        t.row0 = p.S + w * p.L + (d % p.per_win) * kTile;
        t.key_end = p.S + (w + 1) * p.L;
      } else {
        w = p.W;
        t.row0 = p.S + p.W * p.L + (d - p.W * p.per_win) * kTile;
        t.key_end = p.N;
      }
      const int cc = first_compressed_chunk(w, p.ndp, p.Wsel, p.C);
      t.qend = cc >= p.C ? p.N : (p.S + cc * p.L < p.N ? p.S + cc * p.L : p.N);
    }
    t.qb = t.row0;
  }
  t.nq = t.qend > t.qb ? (t.qend - t.qb + kQRows - 1) / kQRows : 0;
  return t;
}

__host__ __device__ inline int tile_segments(const DkvPlan& p, const KvTile& t) {
  return (p.G * t.nq + p.seg - 1) / p.seg;
}

// Iterations per segment of a tile with `iters` of them (the last segment may have fewer).
__host__ __device__ inline int segment_length(const DkvPlan& p, int iters) {
  if (!p.by_length) return p.seg;
  const int k = (iters + p.seg - 1) / p.seg;   // as many segments, of about the same length
  return (iters + k - 1) / k;
}

// Exclusive prefix sums over a block of 256 threads; *total: the sum.  Ends with a barrier.
__device__ inline int block_prefix(int v, int* total) {
  __shared__ int warp_sum[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  int before = incl - v, sum = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    if (w < warp) before += warp_sum[w];
    sum += warp_sum[w];
  }
  *total = sum;
  __syncthreads();
  return before;
}

// Launch order of the (tile, segment) pairs (one block of 256 threads).  Iteration i of a tile is query tile
// nq-1 - i/G (counted from the last query) of head i%G, so segment s of every compact tile covers the
// same queries of the same heads.
//   by length  (small grids): the longest segments of the sequence first, so that its last ones to start are short (the sequences of
//              a packed row come one after another).
//   otherwise  compact tiles are issued segment-major: the CTAs that run at the same time then stream the same Q_i / dO_i
//              tiles and share them through L2 instead of fetching them from DRAM once per key tile.  Dense tiles (short
//              lists, neighbours already overlap) follow in position order.
// seg_cnt: scratch of n_tiles + 1 ints; seg_map[x] = (tile, segment of the tile).
constexpr int kMaxSegsPerTile = 2048;
__device__ inline void dkv_setup(const DkvPlan& p, int* seg_cnt, int2* seg_map) {
  __shared__ int off[kMaxSegsPerTile];   // off[s] = pairs of compact tiles with a segment index below s; by length: see below
  const int tid = threadIdx.x, nt = blockDim.x;   // 256
  int total;
  if (p.by_length) {
    // off[k]: where the next segment of p.seg - k iterations goes
    for (int k = tid; k < p.seg; k += nt) off[k] = 0;
    __syncthreads();
    for (int i = tid; i < p.n_tiles; i += nt) {
      const int iters = p.G * describe_tile(p, i).nq;
      if (iters == 0) continue;
      const int len = segment_length(p, iters), full = (iters - 1) / len;
      if (full) atomicAdd(&off[p.seg - len], full);
      atomicAdd(&off[p.seg - (iters - full * len)], 1);
    }
    __syncthreads();
    const int at = block_prefix(tid < p.seg ? off[tid] : 0, &total);   // p.seg <= kSegMax < 256
    if (tid < p.seg) off[tid] = at;
    __syncthreads();
    for (int i = tid; i < p.n_tiles; i += nt) {
      const int iters = p.G * describe_tile(p, i).nq;
      if (iters == 0) continue;
      const int len = segment_length(p, iters), full = (iters - 1) / len;
      const int pos = full ? atomicAdd(&off[p.seg - len], full) : 0;
      for (int k = 0; k < full; ++k) seg_map[pos + k] = make_int2(i, k);
      seg_map[atomicAdd(&off[p.seg - (iters - full * len)], 1)] = make_int2(i, full);
    }
    return;
  }
  for (int i = tid; i < p.n_tiles; i += nt) seg_cnt[i] = tile_segments(p, describe_tile(p, i));
  __syncthreads();
  // segment-major order needs the compact tiles' segment counts to be non-increasing (later rows are
  // seen by later chunks only) and few enough for the table; otherwise every tile is taken in position order
  bool mono = p.n_cmp > 0 && seg_cnt[0] <= kMaxSegsPerTile;
  for (int c = 1 + tid; c < p.n_cmp; c += nt) mono = mono && seg_cnt[c] <= seg_cnt[c - 1];
  mono = __syncthreads_and(mono);
  int base = 0;
  if (mono) {
    const int maxs = seg_cnt[0], per = (maxs + nt - 1) / nt;
    const int lo = min(maxs, tid * per), hi = min(maxs, lo + per);
    int c = p.n_cmp, mine = 0;   // tiles [0, c) have more than s segments
    auto more_than = [&](int sgm, int c1) {
      int a = 0, b = c1;
      while (a < b) { const int m = (a + b) >> 1; if (seg_cnt[m] > sgm) a = m + 1; else b = m; }
      return a;
    };
    for (int sgm = lo; sgm < hi; ++sgm) { c = more_than(sgm, c); off[sgm] = mine; mine += c; }
    const int at = block_prefix(mine, &base);
    for (int sgm = lo; sgm < hi; ++sgm) off[sgm] += at;
    __syncthreads();
    for (int t = tid; t < p.n_cmp; t += nt)
      for (int sgm = 0; sgm < seg_cnt[t]; ++sgm) seg_map[off[sgm] + t] = make_int2(t, sgm);
  }
  // position order: every thread takes a run of consecutive tiles
  const int first = mono ? p.n_cmp : 0, nd = p.n_tiles - first, per = (nd + nt - 1) / nt;
  const int d_lo = min(p.n_tiles, first + tid * per), d_hi = min(p.n_tiles, d_lo + per);
  int mine = 0;
  for (int t = d_lo; t < d_hi; ++t) mine += seg_cnt[t];
  int pos = base + block_prefix(mine, &total);
  for (int t = d_lo; t < d_hi; ++t) {
    for (int sgm = 0; sgm < seg_cnt[t]; ++sgm) seg_map[pos + sgm] = make_int2(t, sgm);
    pos += seg_cnt[t];
  }
}

// Pointers of one backward call (whole rows; the workspace's parts among them).
struct BwdPtrs {
  const __nv_bfloat16 *Q, *K, *V, *O, *Olo, *dO;
  const float* LSE;
  const int32_t* idx;
  __nv_bfloat16 *dQ, *dK, *dV;
  __nv_bfloat16 *Kc, *Vc;   // compact buffers
  float2* stats;            // per query row: (-LSE * log2(e), D~ = rowsum(dO * O))
  float* Dacc;              // per query row: sum_j P dP, the accurate D (zeroed, then filled by the dK/dV kernel)
  float *kbar, *kpart;      // mean key per (batch, KV head); its partial sums [kMeanSplits][B*Hkv][d]
  int* seg_cnt;             // dK/dV launch order: scratch, and (tile, segment) pairs
  int2* seg_map;
  float *dKf, *dVf;         // fp32 accumulators [B*Hkv][N][d], zeroed
  int* status;
};
// Parts of the sum for the mean key: at most kMeanSplits, of about 256 rows or more (a row of fewer is one part; the last may be shorter).
constexpr int kMeanSplits = 64;
inline int mean_splits(int rows) { return rows >= 256 * kMeanSplits ? kMeanSplits : rows > 256 ? rows / 256 : 1; }

// Per sequence of the batch: its plan, where its parts of seg_cnt and seg_map start, its number of (tile, segment) pairs.
struct DkvBatch {
  DkvPlan plan[kMaxSeqs];
  int cnt0[kMaxSeqs], map0[kMaxSeqs], segs[kMaxSeqs];
};

int launch_bwd_dq_sm100(const Geom& whole, const SeqBatch& b, const BwdPtrs& p, cudaStream_t st);
// `mean`: also finish the mean key from its partial sums (once per call).
int launch_bwd_dkv_sm100(const Geom& whole, const SeqBatch& b, const DkvBatch& db, const BwdPtrs& p, bool mean, cudaStream_t st);

}  // namespace lrsa
