// Inference side of LRSA (Section 3.2: the KV-cache update of Attn-Fill 1 / Attn-Fill 2 and the condensed
// cache of its last paragraph): a physically condensed KV cache that grows token by token, and decode
// attention over it.
//
// Cache of one (batch, KV head), all bf16:
//   list  [S + Wcap*K][d]  the sinks, then K kept rows of every compressed window, in window order
//   ring  [2L][d]          the uncompressed recent tokens: position p >= S sits at row (p - S) mod 2L
// for K and for V, plus idx [Wcap][K] (the kept positions, for inspection and parity).  A query of chunk
// c sees the sinks, windows 0..c-2 through their kept rows, window c-1 and its own chunk causally, so the
// ring only ever needs the last full window and the chunk being filled.  Window c-2 is scored (Eq. 4-8,
// with window c-1 as its reference) and its kept rows are appended to the list when the first token of
// chunk c arrives: not earlier, because the queries of chunk c-1 still see it whole.
//
// Decode attention reads the list prefix and the ring once per KV head for (up to 16) query heads of the group
// (HBM-bound: 4*d bytes per key, a few FMAs per byte).  Two kernels: in decode_kernel the keys are split over CTAs and
// warps, every warp keeps an online softmax of its keys, and the CTAs of a head form a cluster that merges the partial
// results; decode_split_kernel (groups of more than eight heads, use_split_kernel) takes 128 keys a CTA and a merge kernel.
#include "lrsa_internal.h"
#include "sm100_ptx.h"

namespace lrsa {
namespace {

struct CacheLayout {
  int rows_list;   // S + Wcap*K
  int Wcap;        // windows that can ever be compressed with seq_len tokens of capacity
  size_t k_list, v_list, k_ring, v_ring, idx, total;
};

CacheLayout cache_layout(const Geom& g) {
  CacheLayout c;
  // the last token of the capacity sits in chunk (N-1-S)/L; windows up to that chunk minus two get compressed
  const int c_last = g.N > g.S ? (g.N - 1 - g.S) / g.L : 0;
  c.Wcap = c_last >= 2 ? c_last - 1 : 0;
  c.rows_list = g.S + c.Wcap * g.K;
  const size_t BH = (size_t)g.B * g.Hkv;
  const size_t list = align_up(BH * (c.rows_list > 0 ? c.rows_list : 1) * g.d * sizeof(__nv_bfloat16), 256);
  const size_t ring = align_up(BH * 2 * g.L * g.d * sizeof(__nv_bfloat16), 256);
  size_t off = 256;
  c.k_list = off; off += list;
  c.v_list = off; off += list;
  c.k_ring = off; off += ring;
  c.v_ring = off; off += ring;
  c.idx = off; off += align_up(BH * (c.Wcap > 0 ? c.Wcap : 1) * g.K * sizeof(int32_t), 256);
  c.total = off;
  return c;
}

// ---- growing the cache ----
struct CacheRows {
  const __nv_bfloat16 *k_new, *v_new;               // [BH][n_new][d], token p at row p - p_first
  __nv_bfloat16 *k_list, *v_list, *k_ring, *v_ring;
  const int32_t* idx;                                // [BH][Wcap][K]
  int* status;                                       // cleared when not null
  int n_new, p_first, S, L, K, Wcap, rows_list, cpr; // cpr: 16-byte chunks per row (d / 8)
  int n_sink;           // the new tokens of the call up to the last sink, when p0 lies beyond them
  int p0, n_ins;        // tokens [p0, p0 + n_ins) go to the sink rows of the list or to the ring
  int w0, n_keep;       // kept rows: n_keep = windows * K rows of windows w0 ...
  int blocks;           // thread blocks per (batch, KV head)
  int wait_first;       // see below
  int keep_from_ring;   // their source: the ring (a window that had entered the cache before) or the new tokens
};

__device__ __forceinline__ void wait_for_front() {
  asm volatile("griddepcontrol.wait;" ::: "memory");   // may be launched before the kernel in front of it has ended
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// New tokens into the sink rows of the list or into the ring, and the kept rows of newly compressed windows into
// the list (items: tokens first, then kept rows; a thread moves 16 bytes of K and of V).  Bound by the rows it moves
// (one read and one write each); one launch for a whole prompt, whose tokens go to the ring only if they stay there.
// A 32K prompt (windows of 1024 tokens, 4 KV heads, d = 128): window after window, three launches each, 1.25 ms;
// scoring all windows in one launch and this kernel behind it 34 us.
__global__ void __launch_bounds__(256) cache_rows_kernel(const CacheRows a) {
  if (a.wait_first) wait_for_front();
  const int rpb = 256 / a.cpr;   // rows per block
  const int bh = blockIdx.x / a.blocks, item = (blockIdx.x % a.blocks) * rpb + threadIdx.x / a.cpr, ch = threadIdx.x % a.cpr;
  const int n_tok = a.n_sink + a.n_ins;
  const size_t list0 = (size_t)bh * a.rows_list, ring0 = (size_t)bh * 2 * a.L;
  size_t src = 0, dst = 0;
  bool from_ring = false, to_list = true;
  if (item < n_tok) {
    const int p = item < a.n_sink ? a.p_first + item : a.p0 + (item - a.n_sink);
    src = (size_t)bh * a.n_new + (p - a.p_first);
    to_list = p < a.S;
    dst = to_list ? list0 + p : ring0 + (p - a.S) % (2 * a.L);
  }
  if (!a.wait_first) wait_for_front();
  if (a.status && blockIdx.x == 0 && threadIdx.x == 0) *a.status = 0;
  if (item >= n_tok + a.n_keep) return;
  if (item >= n_tok) {
    const int r = item - n_tok;
    const int pos = a.idx[((size_t)bh * a.Wcap + a.w0) * a.K + r];
    from_ring = a.keep_from_ring != 0;
    src = from_ring ? ring0 + (pos - a.S) % (2 * a.L) : (size_t)bh * a.n_new + (pos - a.p_first);
    dst = list0 + a.S + (size_t)a.w0 * a.K + r;
  }
  const uint4 k = reinterpret_cast<const uint4*>(from_ring ? a.k_ring : a.k_new)[src * a.cpr + ch];
  const uint4 v = reinterpret_cast<const uint4*>(from_ring ? a.v_ring : a.v_new)[src * a.cpr + ch];
  reinterpret_cast<uint4*>(to_list ? a.k_list : a.k_ring)[dst * a.cpr + ch] = k;
  reinterpret_cast<uint4*>(to_list ? a.v_list : a.v_ring)[dst * a.cpr + ch] = v;
}

// Does the wait for the kernel in front come ahead of the index work?  With the index work first most tokens take 0.1 to 0.4 us less.  But the
// decode kernel that follows starts when every block here has passed the wait, and its clusters, whose CTAs take an SM each, go where there is room
// then: where they about fill the GPU, shorter blocks here leave some of them a round late.  us a token, wait first | index work first, 16 to 32
// (batch, KV head) pairs: 8/8 heads, d = 64, four sequences at 33K 18.8 | 21.9, at 16K 14.6 | 16.5; 16/2, sixteen at 33K 22.6 | 24.4; 32/8, d = 128,
// two at 120K 47.2 | 49.7, four at 66K 52.2 | 55.1; 28/4, eight at 33K 37.3 | 38.3 (at 16K 28.6 | 25.6).  Others: 28/4, one at 33K 14.7 | 14.4, two at
// 120K 30.1 | 32.0 (in a CUDA graph 29.3 | 29.8); 8/8, d = 64, one at 33K 12.3 | 11.9, eight at 16K 19.1 | 18.8; 16/2, four at 16K 11.1 | 10.7,
// thirty-two 16.3 | 15.9.  What finds room differs between GPUs: a second one gave 18.9 | 19.0 for four of 8/8,
// 22.7 | 21.2 for sixteen of 16/2 and 47.6 | 50.1 for two of 32/8.  (Only for a token: behind the rows of a prompt comes its next piece, or nothing.)
inline int wait_first(int n_new, int BH) { return n_new == 1 && BH >= 16 && BH <= 32; }

int launch_cache_rows(CacheRows a, int BH, cudaStream_t st) {
  const int rows = a.n_sink + a.n_ins + a.n_keep, rpb = 256 / a.cpr;
  a.blocks = (rows + rpb - 1) / rpb;
  a.wait_first = wait_first(a.n_new, BH);
  LRSA_CUDA_CHECK(launch_dependent(cache_rows_kernel, dim3((unsigned)a.blocks * BH), dim3(256), 0, st, 1, a));
  launch_counter().n++;
  return LRSA_OK;
}

// ---- decode attention ----
constexpr int kDecMaxWarps = 16;
constexpr int kDecThreads = 128;  // of the split kernel
constexpr int kDecHeads = 16;     // its query heads of a group per pass over the keys (the M of the tensor-core product)
constexpr int kDecKeys = 128;     // its keys per CTA (32 per warp), staged in shared memory
// Warps of the largest CTA: 128 registers hold the operands of one group of 8 heads; two groups take more.
__host__ __device__ constexpr int dec_max_warps(int nh) { return nh == 1 ? kDecMaxWarps : kDecMaxWarps / 2; }

// Blocks of keys that a warp brings into L2 while the kernel in front ends, where every warp has at least kDecPrefetchMin to do: the
// transfers then start about 2 us earlier.  us a token, without | with 2 blocks: 16 sequences of 28/4 heads at 33K (16 blocks a warp) 53.1 |
// 52.4, four of 32/8 34.3 | 33.7, eight of 8/8, d = 64, 30.1 | 28.3, one of 28/4 at 120K 22.0 | 21.5.  More is slower (16 sequences of 28/4 with 2 | 4 | 16
// blocks 53.9 | 54.6 | 72, four of 32/8 30.7 | 32.8 | 38), and so it is for warps of fewer blocks (eight sequences at 8K, 3 blocks, without | with 2
// 19.9 | 20.1, one at 32K, 2.3 blocks, in L2 already 12.9 | 13.7).
constexpr int kDecPrefetch = 2, kDecPrefetchMin = 4;

struct DecodeArgs {
  const __nv_bfloat16 *q, *k_list, *k_ring;
  long long v_of_list, v_of_ring;   // bytes from a K row to its V row
  float* part;          // [BHkv][n_group, or splits][G][D + 2]: unnormalised output, maximum (log2 domain), sum
  __nv_bfloat16* o;     // [B][Hq][D]
  float* lse;           // [B][Hq], optional
  int* status;          // workspace status word
  int Hq, Hkv, G, rows_list, ring_rows;
  int n_list, n_keys, ring0;   // keys: list rows [0, n_list), then ring rows from ring row ring0 on (wrapping)
  int n_split, n_group, blocks;   // key blocks per (batch, KV head), dealt out evenly to n_group clusters of n_split CTAs
                                  // (split kernel: n_split CTAs of kDecKeys keys)
  float scale_log2;
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// D (16x8, fp32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// transpose of an 8x8 matrix of 16-bit elements held two per lane
__device__ __forceinline__ uint32_t transpose_8x8(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
// this CTA's variable at `p` as CTA `rank` of the cluster has it
__device__ __forceinline__ float ld_cluster(const float* p, int rank) {
  float v;
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(ptx::smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint4 ld_stream(const void* p) {   // read once: no place in L1
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Grid (n_group * n_split, BHkv), clusters of n_split CTAs of 4 to 16 warps.  One query token per (batch, head) over a few hundred to a few thousand keys
// per KV head: the work is the transfer of K and V (two bytes per multiply-add of one head), so the kernel is built
// around the loads.  A warp takes blocks of 2048 / D keys; it loads the block's K and V rows straight into the
// registers in which the warp-level tensor-core products want them and has 8 KB in flight while the other warps of
// the SM compute; nothing is staged in shared memory (with one bulk copy per row into it, a barrier and ldmatrix the
// kernel took 90.6 us for 16 sequences of 9471 keys, 4 KV heads, d = 128; now 52.7 us = 5.9 TB/s, 90 % of a copy's rate;
// one such sequence, where latency counts: 7.3 -> 7.1 us).  The query heads of the KV group are the n of the products
// (8 at a time; a 128-row tcgen05 product would be nine tenths padding):
//   S^T = K Q^T    A = K  (m = keys, k = channels): lane (g, t) = (lane / 4, lane % 4) loads 16-byte chunks t, t+4, ...
//                  of rows g and g + 8; the order of the channels in the contraction is free, and Q is read alike
//   O^T = V^T P^T  A = V^T (m = channels, k = keys): chunk g (+8) of rows 2t, 2t+1, 2t+8, 2t+9; a byte permute pairs
//                  the keys.  P^T comes out of the first product with keys and heads the other way round: one
//                  movmatrix per eight keys turns it.
// The maximum is raised only when it grew by more than 2^8 (then O is rescaled); it is common to the warp, since the
// second product sums over the keys of all its lanes.  The warps are merged through shared memory, the CTAs through the
// shared memory of their cluster (a second kernel for that, partial results in global memory, took 4.4 us beside 7.1 us of
// this one for one sequence at 32K, and a launch on top: 26 us a token with it, 16 without).  Only where one cluster for
// each head would leave most of the GPU idle for long (decode_plan), a head gets several and decode_merge_kernel
// merges them.
template <int D, int NH>
__global__ void __launch_bounds__(dec_max_warps(NH) * 32, 1) decode_kernel(const DecodeArgs a) {
  constexpr int U = 128 / D;                // 16-key groups per block
  constexpr int KC = D / 32, VC = D / 64;   // 16-byte chunks per lane and row, of K and of V
  constexpr int MT = D / 16;                // channel tiles of the output
  constexpr int kSlots = dec_max_warps(NH) / 2;
  __shared__ __align__(16) float sm_o[kSlots][8][D + 4];   // padded: lanes of a store differ in the head
  __shared__ float sm_m[kSlots][8], sm_l[kSlots][8];
  __shared__ __align__(16) uint4 sm_q[NH][KC][32];
  __shared__ float fin_o[8][D], fin_m[8], fin_l[8];   // the CTA's result, read by the cluster
  const int bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nw = blockDim.x >> 5, g = lane >> 2, t = lane & 3;
  const int b = bh / a.Hkv, hkv = bh % a.Hkv;
  const unsigned char* kl = reinterpret_cast<const unsigned char*>(a.k_list) + (size_t)bh * a.rows_list * (D * 2);
  const unsigned char* kr = reinterpret_cast<const unsigned char*>(a.k_ring) + (size_t)bh * a.ring_rows * (D * 2);
  // K row of key `key`, and what leads from there to its V row
  auto row_of = [&](int key, long long& to_v) {
    key = min(key, a.n_keys - 1);       // beyond the end: any row that is there (its probability is zero)
    const bool in_list = key < a.n_list;
    int r = key - a.n_list + a.ring0;
    if (r >= a.ring_rows) r -= a.ring_rows;
    to_v = in_list ? a.v_of_list : a.v_of_ring;
    return in_list ? kl + (size_t)key * (D * 2) : kr + (size_t)r * (D * 2);
  };
  const int nx = a.n_split * a.n_group;
  const int blk0 = (int)((long long)a.blocks * blockIdx.x / nx), blk1 = (int)((long long)a.blocks * (blockIdx.x + 1) / nx);
  // While the kernel in front of this one ends, the warp's first blocks of the list are brought into L2 (a hint: what that kernel
  // writes is read from L2 all the same, after the wait).
  if (lane < 2 && blk1 - blk0 >= kDecPrefetchMin * nw) {
    for (int blk = blk0 + warp, i = 0; blk < blk1 && i < kDecPrefetch && (blk + 1) * 16 * U <= a.n_list; blk += nw, ++i)
      ptx::prefetch_l2(kl + (size_t)blk * (16 * U * D * 2) + (lane ? a.v_of_list : 0), 16 * U * D * 2);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the cache rows of the kernel in front of this one
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (blockIdx.x == 0 && bh == 0 && tid == 0) *a.status = 0;

  for (int g0 = 0; g0 < a.G; g0 += 8 * NH) {
    // Q of head g0 + 8h + g as the B operand: the chunks this lane also takes of every key row.  The same for every warp;
    // in shared memory, because the registers are full of K, V and O.
    for (int i = tid; i < NH * KC * 32; i += blockDim.x) {
      const int h = i / (KC * 32), j = i / 32 % KC, head = g0 + 8 * h + (i & 31) / 4;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (head < a.G)
        v = *reinterpret_cast<const uint4*>(a.q + ((size_t)(b * a.Hq + hkv * a.G + head)) * D + ((i & 3) + 4 * j) * 8);
      sm_q[h][j][i & 31] = v;
    }
    __syncthreads();
    float o[NH][MT][4];        // tile 4j + f: channels 8(g + 8j) + 2f, + 1 of heads 2t, 2t + 1
    float m[NH][2], l[NH][2];  // heads 2t, 2t + 1: maximum (the warp's), sum (this lane's keys)
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      m[h][0] = m[h][1] = -INFINITY;
      l[h][0] = l[h][1] = 0.f;
#pragma unroll
      for (int i = 0; i < MT; ++i) o[h][i][0] = o[h][i][1] = o[h][i][2] = o[h][i][3] = 0.f;
    }
    for (int blk = blk0 + warp; blk < blk1; blk += nw) {
      const int key0 = blk * (16 * U);
      uint4 kq[U][2][KC], vq[U][4][VC];
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          long long to_v;
          const unsigned char* r = row_of(key0 + 16 * u + g + 8 * i, to_v);
#pragma unroll
          for (int j = 0; j < KC; ++j) kq[u][i][j] = ld_stream(r + (t + 4 * j) * 16);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          long long to_v;
          const unsigned char* r = row_of(key0 + 16 * u + 2 * t + (i & 1) + 8 * (i >> 1), to_v);
#pragma unroll
          for (int j = 0; j < VC; ++j) vq[u][i][j] = ld_stream(r + to_v + (g + 8 * j) * 16);
        }
      }
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        float s[U][4];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          s[u][0] = s[u][1] = s[u][2] = s[u][3] = 0.f;
#pragma unroll
          for (int j = 0; j < KC; ++j) {
            uint4 q;
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                         : "r"(ptx::smem_u32(&sm_q[h][j][lane])));
            mma_16816(s[u], kq[u][0][j].x, kq[u][1][j].x, kq[u][0][j].y, kq[u][1][j].y, q.x, q.y);
            mma_16816(s[u], kq[u][0][j].z, kq[u][1][j].z, kq[u][0][j].w, kq[u][1][j].w, q.z, q.w);
          }
        }
        // elements: e = 0, 1: key g, heads 2t, 2t + 1; e = 2, 3: key g + 8
        float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            s[u][e] = key0 + 16 * u + g + 8 * (e >> 1) < a.n_keys ? s[u][e] * a.scale_log2 : -INFINITY;
            mx[e & 1] = fmaxf(mx[e & 1], s[u][e]);
          }
        if (__any_sync(0xffffffffu, mx[0] > m[h][0] + 8.f || mx[1] > m[h][1] + 8.f)) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
#pragma unroll
            for (int x = 4; x < 32; x <<= 1) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], x));
            const float mn = fmaxf(m[h][e], mx[e]);   // -inf while every score has been (f = 0 then)
            const float f = m[h][e] == -INFINITY ? 0.f : exp2f(m[h][e] - mn);
            m[h][e] = mn;
            l[h][e] *= f;
#pragma unroll
            for (int i = 0; i < MT; ++i) { o[h][i][e] *= f; o[h][i][e + 2] *= f; }
          }
        }
        const float ref[2] = {m[h][0] == -INFINITY ? 0.f : m[h][0], m[h][1] == -INFINITY ? 0.f : m[h][1]};
#pragma unroll
        for (int u = 0; u < U; ++u) {
          float p[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            p[e] = exp2f(s[u][e] - ref[e & 1]);
            l[h][e & 1] += p[e];
          }
          const uint32_t b0 = transpose_8x8(ptx::pack_bf16(p[0], p[1])), b1 = transpose_8x8(ptx::pack_bf16(p[2], p[3]));
#pragma unroll
          for (int j = 0; j < VC; ++j)
#pragma unroll
            for (int f = 0; f < 4; ++f) {
              auto w = [&](int i) { return f == 0 ? vq[u][i][j].x : f == 1 ? vq[u][i][j].y : f == 2 ? vq[u][i][j].z : vq[u][i][j].w; };
              mma_16816(o[h][4 * j + f], __byte_perm(w(0), w(1), 0x5410), __byte_perm(w(0), w(1), 0x7632),
                        __byte_perm(w(2), w(3), 0x5410), __byte_perm(w(2), w(3), 0x7632), b0, b1);
            }
        }
      }
    }
    // Merge the warps: the upper half hands its state to the lower half, then all threads add what is left.
    const int half = nw / 2;
    const bool upper = warp >= half;
    const int slot = upper ? warp - half : warp;   // nw is even and half <= kSlots
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      float lh[2], mh[2];
      auto put = [&]() {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float* dst = sm_o[slot][2 * t + e];
#pragma unroll
          for (int i = 0; i < MT; ++i)
            *reinterpret_cast<float2*>(dst + 8 * (g + 8 * (i >> 2)) + 2 * (i & 3)) = make_float2(o[h][i][e], o[h][i][e + 2]);
          if (g == 0) { sm_m[slot][2 * t + e] = mh[e]; sm_l[slot][2 * t + e] = lh[e]; }
        }
      };
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        mh[e] = m[h][e];
        lh[e] = l[h][e];
#pragma unroll
        for (int y = 4; y < 32; y <<= 1) lh[e] += __shfl_xor_sync(0xffffffffu, lh[e], y);
      }
      __syncthreads();   // the buffer is free
      if (upper) put();
      __syncthreads();
      if (!upper) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float mo = sm_m[slot][2 * t + e], mn = fmaxf(mh[e], mo);
          const float f0 = mh[e] == -INFINITY ? 0.f : exp2f(mh[e] - mn), f1 = mo == -INFINITY ? 0.f : exp2f(mo - mn);
          lh[e] = lh[e] * f0 + sm_l[slot][2 * t + e] * f1;
          mh[e] = mn;
          const float* srcp = sm_o[slot][2 * t + e];
#pragma unroll
          for (int i = 0; i < MT; ++i) {
            const float2 v = *reinterpret_cast<const float2*>(srcp + 8 * (g + 8 * (i >> 2)) + 2 * (i & 3));
            o[h][i][e] = o[h][i][e] * f0 + v.x * f1;
            o[h][i][e + 2] = o[h][i][e + 2] * f0 + v.y * f1;
          }
        }
        __syncwarp();   // every lane has read the slot before it is overwritten
        put();
      }
      __syncthreads();
      const int ng = min(8, a.G - g0 - 8 * h);
      for (int i = tid; i < ng * D; i += blockDim.x) {
        const int hd = i / D, c = i % D;
        float M = -INFINITY;
        for (int w = 0; w < half; ++w) M = fmaxf(M, sm_m[w][hd]);
        float ov = 0.f, ls = 0.f;
        for (int w = 0; w < half; ++w) {
          const float f = sm_m[w][hd] == -INFINITY ? 0.f : exp2f(sm_m[w][hd] - M);
          ov = fmaf(sm_o[w][hd][c], f, ov);
          ls = fmaf(sm_l[w][hd], f, ls);
        }
        fin_o[hd][c] = ov;
        if (c == 0) { fin_m[hd] = M; fin_l[hd] = ls; }
      }
      cluster_sync();
      // the CTAs of the cluster share the elements of the output
      const int group = blockIdx.x / a.n_split, rank = blockIdx.x - group * a.n_split;
      for (int i = rank * blockDim.x + tid; i < ng * D; i += a.n_split * blockDim.x) {
        const int hd = i / D, c = i % D;
        float M = -INFINITY;
#pragma unroll 4
        for (int r = 0; r < a.n_split; ++r) M = fmaxf(M, ld_cluster(&fin_m[hd], r));
        float ov = 0.f, ls = 0.f;
#pragma unroll 4
        for (int r = 0; r < a.n_split; ++r) {
          const float f = M == -INFINITY ? 0.f : exp2f(ld_cluster(&fin_m[hd], r) - M);   // -inf: no score of the head was finite
          ov = fmaf(ld_cluster(&fin_o[hd][c], r), f, ov);
          ls = fmaf(ld_cluster(&fin_l[hd], r), f, ls);
        }
        if (a.n_group > 1) {
          float* dst = a.part + (((size_t)bh * a.n_group + group) * a.G + g0 + 8 * h + hd) * (D + 2);
          dst[c] = ov;
          if (c == 0) { dst[D] = M; dst[D + 1] = ls; }
          continue;
        }
        const size_t head = (size_t)b * a.Hq + hkv * a.G + g0 + 8 * h + hd;
        a.o[head * D + c] = __float2bfloat16(ov / ls);
        if (c == 0 && a.lse) a.lse[head] = (M + log2f(ls)) * 0.6931471805599453f;
      }
      cluster_sync();   // the other CTAs have read this one's result: it may be overwritten, or the CTA may leave
    }
  }
}

// Decode of groups of more than eight query heads where the whole work is a wave or so of small CTAs (use_split_kernel).
// Grid (n_split, BHkv), one CTA of four warps per kDecKeys keys.  The query heads of the group are the rows of the products
// (16 a pass; the unused ones zero), so a 16-head group costs what one head does, where decode_kernel above repeats its products
// for every eight heads and, with the second group's operands, has half as many warps an SM.  Every key row of the CTA is
// fetched at once (a bulk copy each of K and of V per thread) into rows padded by 16 bytes, and everything after
// that is short: a warp takes 32 keys, Q, K and V fragments through ldmatrix, the softmax of its keys in registers, P as the A operand
// of the second product.  The four warps are merged through shared memory, the splits by decode_merge_kernel.
// A layer of a model (caches in turn, larger together than L2; CUDA graph), decode_kernel | this one, us: 20/1 heads, d = 64,
// 9471 keys 22.7 | 10.6; 24/2, d = 128 17.0 | 11.4; 40/2 24.7 | 14.1, 38 000 keys 39.0 | 42.5; 320/8 62.7 | 47.4.
template <int D>
__global__ void __launch_bounds__(kDecThreads) decode_split_kernel(const DecodeArgs a) {
  constexpr int CPR = D / 8;                 // 16-byte chunks per row
  constexpr int KS = D / 16;                 // k-steps of Q K^T
  constexpr int NT = D / 8;                  // 8-channel tiles of the output
  constexpr int kRowBytes = D * 2, kStride = kRowBytes + 16;
  extern __shared__ __align__(128) unsigned char dec_smem[];   // K rows [kDecKeys], V rows [kDecKeys], Q rows [16]
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_fail;
  const int bh = blockIdx.y, split = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_keys = a.n_keys;
  const int k_lo = split * kDecKeys, k_hi = min(n_keys, k_lo + kDecKeys), nk = k_hi - k_lo;
  const int b = bh / a.Hkv, hkv = bh % a.Hkv;
  const uint32_t sK = ptx::smem_u32(dec_smem), sV = sK + kDecKeys * kStride, sQ = sV + kDecKeys * kStride;
  unsigned char* gQ = dec_smem + 2 * kDecKeys * kStride;
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the cache rows of the kernel in front of this one
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) {
    s_fail = 0;
    ptx::mbar_init(ptx::smem_u32(&bar), 1);
    ptx::fence_barrier_init();
    ptx::mbar_expect_tx(ptx::smem_u32(&bar), (uint32_t)nk * kRowBytes * 2);   // every row copy below reports here
    // the only writer of the status word before a wait below can expire (seconds later)
    if (split == 0 && bh == 0) *a.status = 0;
  }
  __syncthreads();
  {
    // this thread's row of K and of V
    const int r = tid;
    if (r < nk) {
      const int k = k_lo + r;
      const bool in_list = k < a.n_list;
      const size_t row = in_list ? (size_t)bh * a.rows_list + k
                                 : (size_t)bh * a.ring_rows + (a.ring0 + (k - a.n_list)) % a.ring_rows;
      const unsigned char* ks = reinterpret_cast<const unsigned char*>(in_list ? a.k_list : a.k_ring) + row * kRowBytes;
      bulk_load(sK + r * kStride, ks, kRowBytes, ptx::smem_u32(&bar));
      bulk_load(sV + r * kStride, ks + (in_list ? a.v_of_list : a.v_of_ring), kRowBytes, ptx::smem_u32(&bar));
    } else {
      // rows beyond the split's keys: their probabilities are zero, their V must not be NaN
#pragma unroll
      for (int c = 0; c < CPR; ++c) {
        *reinterpret_cast<uint4*>(dec_smem + r * kStride + c * 16) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(dec_smem + (kDecKeys + r) * kStride + c * 16) = make_uint4(0, 0, 0, 0);
      }
    }
  }

  const int row = lane >> 2, cpair = (lane & 3) * 2;   // fragment coordinates of this lane
  for (int g0 = 0; g0 < a.G; g0 += kDecHeads) {
    const int ng = min(kDecHeads, a.G - g0);
    // Q of this pass: 16 rows (heads g0 ..., zero beyond the group) into shared memory, 16 bytes per thread and step
    for (int i = tid; i < kDecHeads * CPR; i += kDecThreads) {
      const int g = i / CPR, cch = i % CPR;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (g < ng) v = *reinterpret_cast<const uint4*>(a.q + ((size_t)(b * a.Hq + hkv * a.G + g0 + g)) * D + cch * 8);
      *reinterpret_cast<uint4*>(gQ + g * kStride + cch * 16) = v;
    }
    if (g0 == 0) {
      // bounded wait for the copies; a CTA that gives up records it, waits once more for its copies (they write
      // this CTA's shared memory) and leaves its partial result empty
      bool got = ptx::mbar_try_wait(ptx::smem_u32(&bar), 0);
      const long long t0 = clock64();
      while (!got) {
        got = ptx::mbar_try_wait(ptx::smem_u32(&bar), 0);
        if (!got && clock64() - t0 > 4000000000LL) { s_fail = 1; break; }
      }
    }
    __syncthreads();
    if (s_fail) {
      if (tid == 0) {
        atomicExch(a.status, (int)LRSA_ERR_TIMEOUT);
        const long long t0 = clock64();
        while (!ptx::mbar_try_wait(ptx::smem_u32(&bar), 0) && clock64() - t0 < 4000000000LL) {}
      }
      __syncthreads();
      // empty partial results: maximum -inf, the merge kernel skips them
      for (int i = tid; i < ng; i += kDecThreads) {
        float* dst = a.part + (((size_t)bh * a.n_split + split) * a.G + g0 + i) * (D + 2);
        dst[D] = -INFINITY; dst[D + 1] = 0.f;
      }
      continue;
    }
    // Q as A fragments: matrices (heads 0-7, channels k..k+7), (heads 8-15, same), then channels k+8..k+15
    uint32_t qa[KS][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
      ldmatrix_x4(sQ + ((lane & 7) + 8 * ((lane >> 3) & 1)) * kStride + (2 * ks + (lane >> 4)) * 16, qa[ks]);
    // S = Q K^T for this warp's 32 keys: four tiles of 8 keys
    float s[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
      const int key = warp * 32 + 8 * j + (lane & 7);
#pragma unroll
      for (int q4 = 0; q4 < CPR / 4; ++q4) {
        uint32_t kb[4];
        ldmatrix_x4(sK + key * kStride + (4 * q4 + (lane >> 3)) * 16, kb);
        const uint32_t (&q0)[4] = qa[2 * q4], (&q1)[4] = qa[2 * q4 + 1];
        mma_16816(s[j], q0[0], q0[1], q0[2], q0[3], kb[0], kb[1]);
        mma_16816(s[j], q1[0], q1[1], q1[2], q1[3], kb[2], kb[3]);
      }
    }
    // scale, mask the keys beyond the split, row maxima and sums (rows: head `row` -> index 0, `row + 8` -> 1)
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int key = warp * 32 + 8 * j + cpair + (e & 1);
        s[j][e] = key < nk ? s[j][e] * a.scale_log2 : -INFINITY;
        mx[e >> 1] = fmaxf(mx[e >> 1], s[j][e]);
      }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
      mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
    }
    float sum[2] = {0.f, 0.f};
    uint32_t pa[2][4];   // P as A fragments of the two 16-key steps
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float pr[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        pr[e] = mx[e >> 1] == -INFINITY ? 0.f : exp2f(s[j][e] - mx[e >> 1]);
        sum[e >> 1] += pr[e];
      }
      pa[j >> 1][(j & 1) * 2 + 0] = ptx::pack_bf16(pr[0], pr[1]);
      pa[j >> 1][(j & 1) * 2 + 1] = ptx::pack_bf16(pr[2], pr[3]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], 1);
      sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], 2);
    }
    // O = P V: V fragments transposed on the way out of shared memory (keys are the contraction index)
    float o[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
      uint32_t vb[4];
      ldmatrix_x4_trans(sV + (warp * 32 + lane) * kStride + nt * 16, vb);
      mma_16816(o[nt], pa[0][0], pa[0][1], pa[0][2], pa[0][3], vb[0], vb[1]);
      mma_16816(o[nt], pa[1][0], pa[1][1], pa[1][2], pa[1][3], vb[2], vb[3]);
    }
    // merge the four warps through shared memory (the K rows are no longer needed once every warp is here;
    // with more than one pass over the heads they are needed again, so the merge buffer then follows V)
    __syncthreads();
    float* mrg = reinterpret_cast<float*>(dec_smem + (a.G > kDecHeads ? (2 * kDecKeys + kDecHeads) * kStride : 0));
    float* mo = mrg;                                   // [4 warps][16 heads][D]
    float* mm_ = mrg + 4 * kDecHeads * D;              // [4][16] maxima
    float* ml = mm_ + 4 * kDecHeads;                   // [4][16] sums
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      *reinterpret_cast<float2*>(mo + ((warp * kDecHeads + row) * D + nt * 8 + cpair)) = make_float2(o[nt][0], o[nt][1]);
      *reinterpret_cast<float2*>(mo + ((warp * kDecHeads + row + 8) * D + nt * 8 + cpair)) = make_float2(o[nt][2], o[nt][3]);
    }
    if ((lane & 3) == 0) {
      mm_[warp * kDecHeads + row] = mx[0]; mm_[warp * kDecHeads + row + 8] = mx[1];
      ml[warp * kDecHeads + row] = sum[0]; ml[warp * kDecHeads + row + 8] = sum[1];
    }
    __syncthreads();
    for (int i = tid; i < ng * D; i += kDecThreads) {
      const int g = i / D, c = i % D;
      float M = -INFINITY;
#pragma unroll
      for (int w = 0; w < 4; ++w) M = fmaxf(M, mm_[w * kDecHeads + g]);
      float ov = 0.f, lsum = 0.f;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const float mw = mm_[w * kDecHeads + g];
        const float f = mw == -INFINITY ? 0.f : exp2f(mw - M);
        ov = fmaf(mo[(w * kDecHeads + g) * D + c], f, ov);
        lsum = fmaf(ml[w * kDecHeads + g], f, lsum);
      }
      float* dst = a.part + (((size_t)bh * a.n_split + split) * a.G + g0 + g) * (D + 2);
      dst[c] = ov;
      if (c == 0) { dst[D] = M; dst[D + 1] = lsum; }
    }
    __syncthreads();   // the merge buffer is reused by the next pass
  }
}

// One CTA per (batch, query head): merges the partial results of its splits, or of its clusters.  kRows thread rows (one
// for clusters, of which there are at most kDecMaxGroups) take alternate results, four at a time with all their loads issued before the
// arithmetic (the kernel is a chain of L2 round trips otherwise), then the rows are merged through shared memory.
constexpr int kMergeRows = 8;
template <int D, int kRows>
__global__ void __launch_bounds__(kRows * D) decode_merge_kernel(const float* part, __nv_bfloat16* o, float* lse, int Hq,
                                                                  int Hkv, int G, int n_split) {
  __shared__ float sm_m[kRows], sm_l[kRows], sm_o[kRows][D];
  const int bhq = blockIdx.x, b = bhq / Hq, hq = bhq % Hq, hkv = hq / G, g = hq % G;
  const int c = threadIdx.x % D, row = threadIdx.x / D;
  const float* base = part + (((size_t)(b * Hkv + hkv) * n_split) * G + g) * (D + 2);
  const size_t stride = (size_t)G * (D + 2);
  float M = -INFINITY, acc = 0.f, l = 0.f;
  constexpr int kBatch = 4;
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the partial results of the kernel in front of this one
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int s0 = row; s0 < n_split; s0 += kRows * kBatch) {
    float ms[kBatch], vs[kBatch], ls[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int s = s0 + u * kRows;
      const bool in = s < n_split;
      ms[u] = in ? __ldcg(base + s * stride + D) : -INFINITY;
      vs[u] = in ? __ldcg(base + s * stride + c) : 0.f;
      ls[u] = in ? __ldcg(base + s * stride + D + 1) : 0.f;
    }
    float mn = M;
#pragma unroll
    for (int u = 0; u < kBatch; ++u) mn = fmaxf(mn, ms[u]);
    if (mn == -INFINITY) continue;
    const float f0 = exp2f(M - mn);   // exp2f(-inf) = 0 while nothing has been merged
    acc *= f0; l *= f0;
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const float f = exp2f(ms[u] - mn);
      acc = fmaf(vs[u], f, acc);
      l = fmaf(ls[u], f, l);
    }
    M = mn;
  }
  sm_o[row][c] = acc;
  if (c == 0) { sm_m[row] = M; sm_l[row] = l; }
  __syncthreads();
  if (row == 0) {
    float Mt = -INFINITY;
    for (int r = 0; r < kRows; ++r) Mt = fmaxf(Mt, sm_m[r]);
    float at = 0.f, lt = 0.f;
    for (int r = 0; r < kRows; ++r) {
      const float f = sm_m[r] == -INFINITY ? 0.f : exp2f(sm_m[r] - Mt);
      at = fmaf(sm_o[r][c], f, at);
      lt = fmaf(sm_l[r], f, lt);
    }
    o[(size_t)bhq * D + c] = __float2bfloat16(at / lt);
    if (c == 0 && lse) lse[bhq] = (Mt + log2f(lt)) * 0.6931471805599453f;
  }
}

// Groups of more than eight query heads: the split kernel up to three of its CTAs an SM (what is resident), four when
// decode_kernel goes over the keys more than once (more than 16 heads); beyond, decode_kernel's transfers are the better ones.  Its merge
// has a CTA per query head: not for hundreds of them.  us, decode_kernel | split kernel (data as in that kernel's head):
// 18/2 heads, 148 CTAs 16.4 | 11.0, 600 23.6 | 28.1; 72/8, 112 CTAs 12.1 | 9.2, 592 24.1 | 23.8; batch 16 of 18/2, 448 16.5 | 21.5;
// 160/8, 592 CTAs 40.4 | 32.6; batch 16 of 40/2, 448 CTAs 29.3 | 33.9.
int decode_splits(int n_keys) { return n_keys > 0 ? (n_keys + kDecKeys - 1) / kDecKeys : 1; }
long long split_ctas_limit(const Geom& g) { return kSms * (g.G > kDecHeads ? 4LL : 3LL); }
bool use_split_kernel(const Geom& g, int n_keys) {
  return g.G > 8 && (long long)g.B * g.Hq <= 512 && (long long)g.B * g.Hkv * decode_splits(n_keys) <= split_ctas_limit(g);
}

// How the keys of the (batch, KV head) pairs are dealt out: to `groups` clusters of `splits` CTAs of `warps` warps each.
struct DecodePlan { int nh, warps, blocks, splits, groups; };
constexpr int kDecMaxSplits = 16, kDecMaxGroups = 16;
DecodePlan decode_plan(const Geom& g, int n_keys, int max_splits = kDecMaxSplits) {
  DecodePlan p;
  p.nh = g.G > 8 ? 2 : 1;
  const int per_block = 2048 / g.d;
  const long long BH = (long long)g.B * g.Hkv;
  p.blocks = n_keys > 0 ? (n_keys + per_block - 1) / per_block : 1;
  // 16 warps (8 with two groups of heads) are resident per SM, as one large CTA or several small ones.  Large ones
  // have fewer partial results to merge; small ones fill the SMs more evenly when every SM has several blocks per warp
  // to do.  A round of blocks takes about 1.3 us, a CTA's start and merge as long as two, the second kernel as three; a
  // cluster lies in one group of SMs (ClusterRoom).  (One sequence, 4 heads, d = 128: 9471 keys, one cluster for a
  // head 17.7 us a token with 8 CTAs, 15.8 with 16; 66 000 keys 107 us with one cluster of 16, 34.5 with two.)
  const int max_warps = dec_max_warps(p.nh);
  p.warps = BH * p.blocks > 2LL * kSms * max_warps ? 4 : max_warps;
  const int per_sm = max_warps / p.warps;
  const ClusterRoom& room = cluster_room();
  long long best = -1;
  for (int s = 1; s <= max_splits; s *= 2) {
    const long long at_once = room.at_once(per_sm, s);
    for (int grp = 1; grp <= kDecMaxGroups; grp *= 2) {
      const int n = s * grp;
      if (n > 1 && ((n - 1) * p.warps >= p.blocks || BH * n > (long long)kSms * per_sm * 4)) break;
      const long long waves = (BH * grp + at_once - 1) / at_once;
      const int per_cta = (p.blocks + n - 1) / n;
      const long long cost = waves * ((per_cta + p.warps - 1) / p.warps + 2) + (grp > 1 ? 3 : 0);
      if (best < 0 || cost < best) { best = cost; p.splits = s; p.groups = grp; }
    }
  }
  return p;
}

template <int D, int NH>
cudaError_t launch_decode_t(DecodeArgs& a, const DecodePlan& pl, int BHkv, cudaStream_t st) {
  a.n_split = pl.splits; a.n_group = pl.groups; a.blocks = pl.blocks;
  auto kern = decode_kernel<D, NH>;
  if (pl.splits > 8) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  return launch_dependent(kern, dim3(pl.splits * pl.groups, BHkv), dim3(pl.warps * 32), 0, st, pl.splits, a);
}

template <int D>
cudaError_t launch_split_t(const Geom& g, DecodeArgs& a, cudaStream_t st) {
  // K and V rows; the merge buffer (4 warps x 16 heads x (d + 2) floats) lies over them, or behind them when the
  // group has more than 16 query heads and the rows are read again
  const size_t rows_bytes = (size_t)(2 * kDecKeys + kDecHeads) * (D * sizeof(__nv_bfloat16) + 16);   // K, V and Q rows, padded
  const size_t merge_bytes = (size_t)4 * kDecHeads * (D + 2) * sizeof(float);
  const size_t smem = g.G > kDecHeads ? rows_bytes + merge_bytes : (rows_bytes > merge_bytes ? rows_bytes : merge_bytes);
  const cudaError_t e = cudaFuncSetAttribute(decode_split_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(decode_split_kernel<D>, dim3(a.n_split, g.B * g.Hkv), dim3(kDecThreads), smem, st, 1, a);
}

template <int kRows>
cudaError_t launch_merge(const Geom& g, const DecodeArgs& a, int n, cudaStream_t st) {
  return launch_dependent(g.d == 128 ? decode_merge_kernel<128, kRows> : decode_merge_kernel<64, kRows>, dim3(g.B * g.Hq),
                          dim3(kRows * g.d), 0, st, 1, (const float*)a.part, a.o, a.lse, g.Hq, g.Hkv, g.G, n);
}

cudaError_t launch_decode(const Geom& g, DecodeArgs& a, const DecodePlan& pl, cudaStream_t st) {
  const int BHkv = g.B * g.Hkv;
  if (g.d == 128) return pl.nh == 1 ? launch_decode_t<128, 1>(a, pl, BHkv, st) : launch_decode_t<128, 2>(a, pl, BHkv, st);
  return pl.nh == 1 ? launch_decode_t<64, 1>(a, pl, BHkv, st) : launch_decode_t<64, 2>(a, pl, BHkv, st);
}

}  // namespace
}  // namespace lrsa

using namespace lrsa;

extern "C" {

int lrsa_cache_bytes(const lrsa_params_t* params, size_t* cache_bytes, size_t* workspace_bytes) {
  Geom g;
  const int rc = make_geom(params, &g);
  if (rc != LRSA_OK) return rc;
  if (params->n_seqs > 0 || g.ndp != 1) return LRSA_ERR_UNSUPPORTED;
  if (cache_bytes) *cache_bytes = cache_layout(g).total;
  if (workspace_bytes) {
    // scoring scratch of the windows of a whole prompt
    Geom all = g;
    const int wcap = cache_layout(g).Wcap;
    all.W = wcap + 1 > 2 ? wcap + 1 : 2; all.Wsel = all.W - 1;
    const size_t a = score_select_ws_bytes(all);
    // or the partial results of decode (see decode_plan: several clusters for a head only below 592 CTAs of 16 warps)
    const long long BH = (long long)g.B * g.Hkv;
    size_t parts = BH <= 4 * 592 ? (size_t)BH * kDecMaxGroups : 0;
    // (or those of the split kernel; a query never sees more than S + Wcap*K + 2L keys)
    const size_t splits = (size_t)BH * decode_splits(cache_layout(g).rows_list + 2 * g.L);
    const size_t most = splits < (size_t)split_ctas_limit(g) ? splits : (size_t)split_ctas_limit(g);
    if (g.G > 8 && most > parts) parts = most;
    const size_t b = sizeof(WsHeader) + parts * g.G * (g.d + 2) * sizeof(float);
    *workspace_bytes = a > b ? a : b;
  }
  return LRSA_OK;
}

int lrsa_cache_append(const lrsa_params_t* params, void* cache, size_t cache_bytes, const void* k_new,
                      const void* v_new, int32_t n_prev, int32_t n_new, void* workspace, size_t workspace_bytes,
                      void* cuda_stream) {
  NvtxRange nvtx_range("lrsa_cache_append");
  launch_counter().n = 0;
  Geom g;
  int rc = make_geom(params, &g);
  if (rc != LRSA_OK) return rc;
  if (params->n_seqs > 0 || g.ndp != 1) return LRSA_ERR_UNSUPPORTED;
  if (!cache || !k_new || !v_new || !workspace || n_prev < 0 || n_new < 1 || (long long)n_prev + n_new > g.N)
    return LRSA_ERR_INVALID_ARG;
  auto mis = [](const void* p, size_t al) { return reinterpret_cast<uintptr_t>(p) % al != 0; };
  if (mis(cache, 256) || mis(workspace, 256) || mis(k_new, 16) || mis(v_new, 16)) return LRSA_ERR_INVALID_ARG;
  const CacheLayout lay = cache_layout(g);
  size_t need_ws = 0;
  lrsa_cache_bytes(params, nullptr, &need_ws);
  if (cache_bytes < lay.total || workspace_bytes < need_ws) return LRSA_ERR_WORKSPACE_TOO_SMALL;
  auto st = static_cast<cudaStream_t>(cuda_stream);
  unsigned char* cb = static_cast<unsigned char*>(cache);
  auto* k_list = reinterpret_cast<__nv_bfloat16*>(cb + lay.k_list);
  auto* v_list = reinterpret_cast<__nv_bfloat16*>(cb + lay.v_list);
  auto* k_ring = reinterpret_cast<__nv_bfloat16*>(cb + lay.k_ring);
  auto* v_ring = reinterpret_cast<__nv_bfloat16*>(cb + lay.v_ring);
  auto* idx = reinterpret_cast<int32_t*>(cb + lay.idx);
  const int BH = g.B * g.Hkv;
  CacheRows rows = {};
  rows.k_new = static_cast<const __nv_bfloat16*>(k_new); rows.v_new = static_cast<const __nv_bfloat16*>(v_new);
  rows.k_list = k_list; rows.v_list = v_list; rows.k_ring = k_ring; rows.v_ring = v_ring;
  rows.idx = idx; rows.n_new = n_new; rows.p_first = n_prev;
  rows.S = g.S; rows.L = g.L; rows.K = g.K; rows.Wcap = lay.Wcap; rows.rows_list = lay.rows_list; rows.cpr = g.d / 8;
  // The status word is cleared by the first kernel of the call: a scoring kernel that can, else a memset in front of
  // it, else the row copies.
  int* status = &reinterpret_cast<WsHeader*>(workspace)->status;
  bool cleared = false;
  auto score = [&](const Geom& w, const __nv_bfloat16* k, const __nv_bfloat16* v) -> int {
    const bool self = !cleared && score_select_clears_status(w);
    if (!cleared && !self) {
      LRSA_CUDA_CHECK(cudaMemsetAsync(workspace, 0, sizeof(WsHeader), st));
      launch_counter().n++;
    }
    cleared = true;
    return launch_score_select(&w, 1, k, v, idx, nullptr, workspace, st, self);
  };
  auto copy_rows = [&]() -> int {
    if (rows.n_sink + rows.n_ins + rows.n_keep == 0) return LRSA_OK;
    rows.status = cleared ? nullptr : status;
    cleared = true;
    return launch_cache_rows(rows, BH, st);
  };
  const int end = n_prev + n_new;
  int pos = n_prev;                                     // tokens before it are in the list or the ring
  int c = pos > g.S ? (pos - g.S + g.L - 1) / g.L : 0;  // next chunk whose first token has not arrived yet
  if (c < 2) c = 2;
  // Chunk start after chunk start while the window c-2 that leaves the ring holds tokens of earlier calls (at most
  // two): the tokens up to it enter the ring, the window is scored with window c-1 as its reference (the two halves
  // of the ring, in either order), and its kept rows join the list before its half is overwritten.
  for (; g.S + c * g.L < end && g.S + (c - 2) * g.L < n_prev; ++c) {
    const int w = c - 2;
    rows.p0 = pos; rows.n_ins = g.S + c * g.L - pos; rows.n_keep = 0;
    rc = copy_rows();
    if (rc != LRSA_OK) return rc;
    Geom two = g;
    two.N = 2 * g.L; two.Nrow = 2 * g.L; two.S = 0; two.W = 2; two.Wsel = 1; two.T = 0; two.C = 2;
    two.tok0 = (w % 2) * g.L;
    two.win_stride = (w % 2) ? -g.L : g.L;
    two.emit_off = g.S + w * g.L;
    two.Wtot = lay.Wcap; two.woff = w;
    rc = score(two, k_ring, v_ring);
    if (rc != LRSA_OK) return rc;
    rows.n_ins = 0; rows.w0 = w; rows.n_keep = g.K; rows.keep_from_ring = 1;
    rc = copy_rows();
    if (rc != LRSA_OK) return rc;
    pos = g.S + c * g.L;
  }
  rows.n_keep = 0;
  rows.p0 = pos; rows.n_ins = end - pos;
  if (g.S + c * g.L < end) {
    // Windows c-2 .. c_last-2 lie in the new tokens as a whole: one scoring launch for all of them, then one for their
    // kept rows, the sinks and the tokens that stay in the ring.
    const int w0 = c - 2, nw = (end - 1 - g.S) / g.L - c + 1;
    Geom many = g;
    many.N = n_new; many.Nrow = n_new; many.S = 0; many.W = nw + 1; many.Wsel = nw; many.T = 0; many.C = nw + 1;
    many.tok0 = g.S + w0 * g.L - n_prev;
    many.emit_off = g.S + w0 * g.L;
    many.Wtot = lay.Wcap; many.woff = w0;
    rc = score(many, rows.k_new, rows.v_new);
    if (rc != LRSA_OK) return rc;
    rows.n_sink = pos < g.S ? g.S - pos : 0;
    rows.p0 = end - 2 * g.L > pos ? end - 2 * g.L : pos;   // beyond the sinks: the call ends in chunk 2 or later
    rows.n_ins = end - rows.p0;
    rows.w0 = w0; rows.n_keep = nw * g.K; rows.keep_from_ring = 0;
  }
  return copy_rows();
}

int lrsa_cache_kept(const lrsa_params_t* params, const void* cache, const int32_t** idx, int32_t* w_cap) {
  Geom g;
  const int rc = make_geom(params, &g);
  if (rc != LRSA_OK) return rc;
  if (!cache || !idx) return LRSA_ERR_INVALID_ARG;
  const CacheLayout lay = cache_layout(g);
  *idx = reinterpret_cast<const int32_t*>(static_cast<const unsigned char*>(cache) + lay.idx);
  if (w_cap) *w_cap = lay.Wcap;
  return LRSA_OK;
}

int lrsa_attn_decode(const lrsa_params_t* params, const void* cache, size_t cache_bytes, const void* q,
                     int32_t n_tokens, void* o, float* lse, void* workspace, size_t workspace_bytes,
                     void* cuda_stream) {
  NvtxRange nvtx_range("lrsa_attn_decode");
  launch_counter().n = 0;
  Geom g;
  const int rc = make_geom(params, &g);
  if (rc != LRSA_OK) return rc;
  if (params->n_seqs > 0 || g.ndp != 1) return LRSA_ERR_UNSUPPORTED;
  if (!cache || !q || !o || !workspace || n_tokens < 1 || n_tokens > g.N) return LRSA_ERR_INVALID_ARG;
  auto mis = [](const void* p, size_t al) { return reinterpret_cast<uintptr_t>(p) % al != 0; };
  if (mis(cache, 256) || mis(workspace, 256) || mis(q, 16) || mis(o, 16) || mis(lse, 4)) return LRSA_ERR_INVALID_ARG;
  const CacheLayout lay = cache_layout(g);
  size_t need_ws = 0;
  lrsa_cache_bytes(params, nullptr, &need_ws);
  if (cache_bytes < lay.total || workspace_bytes < need_ws) return LRSA_ERR_WORKSPACE_TOO_SMALL;
  auto st = static_cast<cudaStream_t>(cuda_stream);
  const unsigned char* cb = static_cast<const unsigned char*>(cache);
  DecodeArgs a;
  a.q = static_cast<const __nv_bfloat16*>(q);
  a.k_list = reinterpret_cast<const __nv_bfloat16*>(cb + lay.k_list);
  a.k_ring = reinterpret_cast<const __nv_bfloat16*>(cb + lay.k_ring);
  a.v_of_list = (long long)(lay.v_list - lay.k_list);
  a.v_of_ring = (long long)(lay.v_ring - lay.k_ring);
  a.part = reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + sizeof(WsHeader));
  a.o = static_cast<__nv_bfloat16*>(o);
  a.lse = lse;
  a.Hq = g.Hq; a.Hkv = g.Hkv; a.G = g.G; a.rows_list = lay.rows_list > 0 ? lay.rows_list : 1;
  a.ring_rows = 2 * g.L;
  // the keys the query at position t = n_tokens - 1 sees (Attn-Fill 1/2): a sink query its causal prefix;
  // otherwise the sinks, the kept rows of windows 0..c-2, and positions [S + (c-1)L, t] from the ring
  const int t = n_tokens - 1;
  if (t < g.S) {
    a.n_list = t + 1; a.n_keys = t + 1; a.ring0 = 0;
  } else {
    const int c = (t - g.S) / g.L, nc = c >= 1 ? c - 1 : 0;
    a.n_list = g.S + nc * g.K;
    a.n_keys = a.n_list + t - (g.S + nc * g.L) + 1;
    a.ring0 = (nc * g.L) % (2 * g.L);
  }
  a.scale_log2 = g.scale * 1.4426950408889634f;
  a.status = &reinterpret_cast<WsHeader*>(workspace)->status;
  if (use_split_kernel(g, a.n_keys)) {
    a.n_split = decode_splits(a.n_keys);
    LRSA_CUDA_CHECK(g.d == 128 ? launch_split_t<128>(g, a, st) : launch_split_t<64>(g, a, st));
    LRSA_CUDA_CHECK(launch_merge<kMergeRows>(g, a, a.n_split, st));
    launch_counter().n += 2;
    return LRSA_OK;
  }
  DecodePlan pl = decode_plan(g, a.n_keys);
  cudaError_t e = launch_decode(g, a, pl, st);
  if (e != cudaSuccess && pl.splits > 8) {   // clusters of 16 are not portable: a part of a GPU may not have room for them
    (void)cudaGetLastError();
    pl = decode_plan(g, a.n_keys, 8);
    e = launch_decode(g, a, pl, st);
  }
  LRSA_CUDA_CHECK(e);
  launch_counter().n++;
  if (pl.groups > 1) {
    LRSA_CUDA_CHECK(launch_merge<1>(g, a, pl.groups, st));
    launch_counter().n++;
  }
  return LRSA_OK;
}

}  // extern "C"
