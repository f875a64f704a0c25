// LRSA attention backward: workspace layout, the kernels in front of and behind the tensor-core kernels, the sequence of
// launches: prep (statistics, zeroed accumulators, compact K/V, launch order, partial mean key), dK/dV (also the accurate
// D of every query row and the mean key), dQ, conversion of dK, dV to bf16.
#include <algorithm>

#include "attn_bwd_sm100.h"

namespace lrsa {
namespace {

using namespace ptx;

constexpr int kPrepUnroll = 4;
constexpr int kZeroPerThread = 16;   // float4 per thread of a zeroing block
constexpr int kMeanPrefetch = 256;   // rows of K that a block of the mean key brings into L2 ahead

struct PrepArgs {
  const __nv_bfloat16 *O, *Olo, *dO, *K;
  const float* LSE;
  float2* stats;
  float* Dacc;
  float* kpart;
  float4* zero;          // the fp32 accumulators
  long long zero_n, rows;
  int N, d, BHkv, splits;
  int* status;           // cleared when not null
  int* seg_cnt;
  int2* seg_map;
  DkvBatch db;
  int b_setup, b_mean, b_compact, b_stats;   // last block + 1 of each part; the rest zeroes
  CompactArgs c;
};

// Per query row: D~_t = sum_c dO[t,c] * O[t,c] and -LSE_t * log2(e); the row's accurate D starts at zero.  d/8 lanes share
// a row (16 bytes each) and a warp takes kPrepUnroll groups of 256/d rows with all loads issued before the arithmetic:
// this part only streams O and dO once.  With the rounding remainder of O (Olo, optional) the sum runs over O + Olo,
// which is O to fp32 accuracy.
__device__ __forceinline__ void prep_stats(const PrepArgs& a, long long block) {
  const int lane = threadIdx.x & 31, d = a.d;
  const int lpr = d >> 3, rpw = 32 / lpr;   // lanes per row, rows per warp-wide load (d = 64: 8, 4; d = 128: 16, 2)
  const long long warp_id = block * 8 + (threadIdx.x >> 5);
  const long long row0 = warp_id * (kPrepUnroll * rpw) + lane / lpr;
  const int c = (lane % lpr) * 8;
  uint4 o[kPrepUnroll], l[kPrepUnroll], g[kPrepUnroll];
#pragma unroll
  for (int u = 0; u < kPrepUnroll; ++u) {
    const long long row = row0 + u * rpw;
    o[u] = l[u] = g[u] = make_uint4(0, 0, 0, 0);
    if (row < a.rows) {
      o[u] = *reinterpret_cast<const uint4*>(a.O + row * d + c);
      g[u] = *reinterpret_cast<const uint4*>(a.dO + row * d + c);
      if (a.Olo) l[u] = *reinterpret_cast<const uint4*>(a.Olo + row * d + c);
    }
  }
#pragma unroll
  for (int u = 0; u < kPrepUnroll; ++u) {
    const uint32_t ow[4] = {o[u].x, o[u].y, o[u].z, o[u].w}, gw[4] = {g[u].x, g[u].y, g[u].z, g[u].w};
    const uint32_t lw[4] = {l[u].x, l[u].y, l[u].z, l[u].w};
    float acc = 0.f, acc_lo = 0.f;   // the remainder's products are 2^-9 of the others: summed apart, added last
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc = fmaf(__uint_as_float(ow[j] << 16), __uint_as_float(gw[j] << 16), acc);
      acc = fmaf(__uint_as_float(ow[j] & 0xffff0000u), __uint_as_float(gw[j] & 0xffff0000u), acc);
      acc_lo = fmaf(__uint_as_float(lw[j] << 16), __uint_as_float(gw[j] << 16), acc_lo);
      acc_lo = fmaf(__uint_as_float(lw[j] & 0xffff0000u), __uint_as_float(gw[j] & 0xffff0000u), acc_lo);
    }
    acc += acc_lo;
    for (int off = lpr >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    const long long row = row0 + u * rpw;
    if ((lane % lpr) == 0 && row < a.rows) {
      a.stats[row] = make_float2(-a.LSE[row] * 1.4426950408889634f, acc);
      a.Dacc[row] = 0.f;
    }
  }
}

// kpart[split][bh][c] = (1/N) * sum of K[bh][t][c] over the split's rows (a.splits of them).
__device__ __forceinline__ void prep_mean(const PrepArgs& a, int block) {
  __shared__ float red[256 * 8];
  const int bh = block / a.splits, split = block % a.splits, tid = threadIdx.x, d = a.d;
  const int lpr = d / 8, rps = 256 / lpr;          // lanes per row (16 bytes each), rows per step
  const int chunk = tid % lpr, r_in = tid / lpr, per = (a.N + a.splits - 1) / a.splits;
  const int r0 = split * per, r1 = min(a.N, r0 + per);
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll 4
  for (int r = r0 + r_in; r < r1; r += rps) {
    const uint4 q = *reinterpret_cast<const uint4*>(a.K + ((size_t)bh * a.N + r) * d + chunk * 8);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      acc[2 * e] += __uint_as_float(w[e] << 16);
      acc[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) red[tid * 8 + e] = acc[e];
  __syncthreads();
  if (tid < d) {
    const int ch = tid / 8, e = tid % 8;
    float sum = 0.f;
    for (int r = 0; r < rps; ++r) sum += red[(r * lpr + ch) * 8 + e];
    a.kpart[((size_t)split * a.BHkv + bh) * d + tid] = sum / (float)a.N;
  }
}

// Everything that has to be in place before the dK/dV kernel, in one launch: its parts are bound by memory (O, dO and K
// read once, the accumulators written) or by one block's serial work (launch order) and overlap.  As four kernels and two
// memsets they took 206 us of a 32K step (28/4 heads, d = 128) and 33 us with the gaps of a 4K one (8 heads, d = 64).  In
// small problems the block of the launch order and the number of blocks bound it: with one thread adding up the order's table and 64 parts
// of the mean key per head whatever its length 7.8 us at 4K (8 heads, d = 64), now 5.7.
__global__ void __launch_bounds__(256) bwd_prep_kernel(const __grid_constant__ PrepArgs a) {
  const int b = blockIdx.x;
  // While the kernel in front ends: the rows of dO or the first rows of K that the block reads, into L2 (a hint).  Whole backward with
  // neither | dO | both, us: 1000 tokens (28/4 heads, d = 128) 62.3 | 62.0 | 61.5, 1777 102.0 | 101.2 | 101.0, 4K (8/8, d = 64) 83.6 | 83.1 | 82.7; with
  // a kernel in front that writes dO and lets nothing start early 67.5 | 67.5 | 65.9, 110.6 | 110.6 | 110.3, 87.4 | 87.5 | 86.3 (1777 tokens of 8/8
  // 55.4 | 55.5 | 56.0).  Bounded, because at 128K tokens the parts of K are together several times as large as L2.
  if (threadIdx.x == 0) {
    if (b >= a.b_compact && b < a.b_stats) {
      const long long per = 8LL * kPrepUnroll * (32 / (a.d >> 3)), row = (b - a.b_compact) * per;
      prefetch_l2(a.dO + row * a.d, (uint32_t)(min(per, a.rows - row) * a.d * 2));
    } else if (b >= a.b_setup && b < a.b_mean) {
      const int bh = (b - a.b_setup) / a.splits, split = (b - a.b_setup) % a.splits, per = (a.N + a.splits - 1) / a.splits;
      const int r0 = split * per, r1 = min(a.N, r0 + per);
      if (r1 > r0) prefetch_l2(a.K + ((size_t)bh * a.N + r0) * a.d, (uint32_t)(min(r1 - r0, kMeanPrefetch) * a.d * 2));
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (b == 0 && threadIdx.x == 0 && a.status) *a.status = 0;
  if (b < a.b_setup) {
    dkv_setup(a.db.plan[b], a.seg_cnt + a.db.cnt0[b], a.seg_map + a.db.map0[b]);
  } else if (b < a.b_mean) {
    prep_mean(a, b - a.b_setup);
  } else if (b < a.b_compact) {
    compact_rows(a.c, b - a.b_mean);
  } else if (b < a.b_stats) {
    prep_stats(a, b - a.b_compact);
  } else {
    const long long i0 = (long long)(b - a.b_stats) * (256 * kZeroPerThread) + threadIdx.x;
#pragma unroll
    for (int k = 0; k < kZeroPerThread; ++k)
      if (i0 + k * 256 < a.zero_n) a.zero[i0 + k * 256] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// bf16 outputs from the fp32 accumulators [BHkv][N][d]; n4 = number of float4 groups
__global__ void __launch_bounds__(256) convert_dkv_kernel(const float* dKf, const float* dVf, __nv_bfloat16* dK,
                                                          __nv_bfloat16* dV, long long n4) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const long long e = i * 4;
  const float4 k = *reinterpret_cast<const float4*>(dKf + e);
  const float4 v = *reinterpret_cast<const float4*>(dVf + e);
  uint2 ko, vo;
  ko.x = pack_bf16(k.x, k.y); ko.y = pack_bf16(k.z, k.w);
  vo.x = pack_bf16(v.x, v.y); vo.y = pack_bf16(v.z, v.w);
  *reinterpret_cast<uint2*>(dK + e) = ko;
  *reinterpret_cast<uint2*>(dV + e) = vo;
}

// What a call needs per batch of sequences: inner iterations per CTA; compact rows, and entries of the launch order tables.
struct BwdSizes {
  int seg;
  long long rows, tiles, segs;
};
BwdSizes bwd_sizes(const Geom& g) {
  BwdSizes z = {kSegMax, compact_rows_used(g), 0, 0};
  SeqBatch b;
  long long iters = 0;
  for (SeqBatches it(g); it.next(&b);) {
    long long tiles = 0;
    for (int s = 0; s < b.n; ++s) {
      const DkvPlan p = make_dkv_plan(b.g[s], kSegMax);
      tiles += p.n_tiles;
      for (int i = 0; i < p.n_tiles; ++i) iters += (long long)p.G * describe_tile(p, i).nq;
    }
    z.tiles = std::max(z.tiles, tiles);
  }
  iters *= (long long)g.B * g.Hkv;
  z.seg = dkv_segment(iters);
  for (SeqBatches it(g); it.next(&b);) {
    long long segs = 0;
    for (int s = 0; s < b.n; ++s) {
      const DkvPlan p = make_dkv_plan(b.g[s], z.seg);
      for (int i = 0; i < p.n_tiles; ++i) segs += tile_segments(p, describe_tile(p, i));
    }
    z.segs = std::max(z.segs, segs);
  }
  return z;
}

// The same for any packing of rows of this shape, from above.  Tiles: every sequence rounds its list, its sinks and its last window
// up.  Query tiles of a tile: all of the row for a list tile; a window is seen whole for at most two windows' length (from its own tokens on), a
// sink by the sinks.  Segments: one more per tile than iterations / seg, and seg is 128 or keeps iterations / seg below 592 * 17 / 16.
BwdSizes bwd_sizes_bound(const Geom& g) {
  auto up = [](long long x, long long y) { return (x + y - 1) / y; };
  const long long seqs = std::min(kMaxSeqs, g.N), rows = compact_rows_bound(g);
  const long long list = rows / kTile + seqs, sinks = seqs * up(g.S, kTile), dense = (g.N / g.L + seqs) * up(g.L, kTile);
  const long long iters = list * up(g.N, kQRows) + sinks * up(g.S, kQRows) + dense * up(2LL * g.L, kQRows);
  BwdSizes z = {kSegMax, rows, list + sinks + dense, 0};
  z.segs = z.tiles + 630 + g.G * iters / kSegMax;
  return z;
}

struct BwdWs {
  size_t kbar, kpart, dacc, kc, vc, stats, cnt, map, dkf, acc, total;
};
BwdWs bwd_ws_layout(const Geom& g, const BwdSizes& z) {
  BwdWs w;
  const size_t BHkv = (size_t)g.B * g.Hkv;
  const size_t cbytes = align_up(BHkv * z.rows * g.d * sizeof(__nv_bfloat16), 1024);
  size_t off = 1024;
  w.kbar = off; off += align_up(BHkv * g.d * sizeof(float), 1024);
  w.kpart = off; off += align_up(kMeanSplits * BHkv * g.d * sizeof(float), 1024);
  w.dacc = off; off += align_up((size_t)g.B * g.Hq * g.N * sizeof(float), 1024);
  w.kc = off; off += cbytes;   // compact K/V for the query-outer dQ kernel
  w.vc = off; off += cbytes;
  w.stats = off; off += align_up((size_t)g.B * g.Hq * g.N * sizeof(float2), 1024);
  w.cnt = off; off += align_up((size_t)(z.tiles + 1) * sizeof(int), 1024);
  w.map = off; off += align_up((size_t)(z.segs + 1) * sizeof(int2), 1024);
  w.acc = align_up(BHkv * g.Nrow * g.d * sizeof(float), 1024);
  w.dkf = off; off += 2 * w.acc;   // dK, then dV
  w.total = off;
  return w;
}

}  // namespace

size_t attn_bwd_ws_bytes(const Geom& g) { return bwd_ws_layout(g, bwd_sizes(g)).total; }
size_t attn_bwd_ws_bound(const Geom& g) { return bwd_ws_layout(g, bwd_sizes_bound(g)).total; }

int launch_attn_bwd_sm100(const lrsa_params_t* params, const Geom& g, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                          const __nv_bfloat16* V, const __nv_bfloat16* O, const __nv_bfloat16* dO,
                          const float* LSE, const int32_t* idx, __nv_bfloat16* dQ, __nv_bfloat16* dK,
                          __nv_bfloat16* dV, void* ws, cudaStream_t st) {
  const BwdSizes z = bwd_sizes(g);
  const BwdWs lay = bwd_ws_layout(g, z);
  unsigned char* base = static_cast<unsigned char*>(ws);
  auto at = [&](size_t off) { return base + off; };
  BwdPtrs p;
  p.Q = Q; p.K = K; p.V = V; p.O = O; p.dO = dO; p.LSE = LSE; p.idx = idx; p.dQ = dQ; p.dK = dK; p.dV = dV;
  p.Olo = static_cast<const __nv_bfloat16*>(params->o_residual);
  p.Kc = reinterpret_cast<__nv_bfloat16*>(at(lay.kc));
  p.Vc = reinterpret_cast<__nv_bfloat16*>(at(lay.vc));
  p.stats = reinterpret_cast<float2*>(at(lay.stats));
  p.Dacc = reinterpret_cast<float*>(at(lay.dacc));
  p.kbar = reinterpret_cast<float*>(at(lay.kbar));
  p.kpart = reinterpret_cast<float*>(at(lay.kpart));
  p.seg_cnt = reinterpret_cast<int*>(at(lay.cnt));
  p.seg_map = reinterpret_cast<int2*>(at(lay.map));
  p.dKf = reinterpret_cast<float*>(at(lay.dkf));
  p.dVf = reinterpret_cast<float*>(at(lay.dkf + lay.acc));
  p.status = &reinterpret_cast<WsHeader*>(base)->status;

  const int BHkv = g.B * g.Hkv;
  SeqBatches batches(g);
  SeqBatch b;
  for (bool first = true; batches.next(&b); first = false) {
    PrepArgs a;
    int cnt = 0, map = 0;
    for (int s = 0; s < b.n; ++s) {
      const DkvPlan dp = make_dkv_plan(b.g[s], z.seg);
      a.db.plan[s] = dp;
      a.db.cnt0[s] = cnt;
      a.db.map0[s] = map;
      a.db.segs[s] = 0;
      for (int i = 0; i < dp.n_tiles; ++i) a.db.segs[s] += tile_segments(dp, describe_tile(dp, i));
      cnt += dp.n_tiles;
      map += a.db.segs[s];
    }
    const bool by_length = order_by_length((long long)map * BHkv);
    for (int s = 0; s < b.n; ++s) a.db.plan[s].by_length = by_length;
    a.O = O; a.Olo = p.Olo; a.dO = dO; a.K = K; a.LSE = LSE; a.stats = p.stats; a.Dacc = p.Dacc; a.kpart = p.kpart;
    a.seg_cnt = p.seg_cnt; a.seg_map = p.seg_map;
    a.N = g.Nrow; a.d = g.d; a.BHkv = BHkv; a.splits = mean_splits(g.Nrow);
    a.c = compact_args(g, b, K, V, idx, p.Kc, p.Vc, nullptr);
    a.status = first ? p.status : nullptr;
    a.zero = reinterpret_cast<float4*>(p.dKf);
    // what belongs to whole rows comes with the first batch of sequences
    a.zero_n = first ? (long long)(2 * lay.acc / sizeof(float4)) : 0;
    a.rows = first ? (long long)g.B * g.Hq * g.Nrow : 0;
    const long long rows_per_block = 8LL * kPrepUnroll * (32 / (g.d >> 3));
    long long nb = b.n;
    a.b_setup = (int)nb; nb += first ? a.splits * BHkv : 0;
    a.b_mean = (int)nb; nb += a.c.blocks();
    a.b_compact = (int)nb; nb += (a.rows + rows_per_block - 1) / rows_per_block;
    a.b_stats = (int)nb; nb += (a.zero_n + 256 * kZeroPerThread - 1) / (256 * kZeroPerThread);
    if (nb > 0x7fffffffLL) return LRSA_ERR_UNSUPPORTED;
    LRSA_CUDA_CHECK(launch_dependent(bwd_prep_kernel, dim3((unsigned)nb), dim3(256), 0, st, 1, a));
    launch_counter().n++;
    int rc = launch_bwd_dkv_sm100(g, b, a.db, p, first, st);
    if (rc == LRSA_OK) rc = launch_bwd_dq_sm100(g, b, p, st);
    if (rc != LRSA_OK) return rc;
  }
  const long long n4 = (long long)BHkv * g.Nrow * g.d / 4;
  LRSA_CUDA_CHECK(launch_dependent(convert_dkv_kernel, dim3((unsigned)((n4 + 255) / 256)), dim3(256), 0, st, 1,
                                   (const float*)p.dKf, (const float*)p.dVf, dK, dV, n4));
  launch_counter().n++;
  return LRSA_OK;
}

}  // namespace lrsa
