// LagKV scoring and top-K selection (Section 3.2, Eq. 4-8 and the selection rule after Eq. 8).
//
// Two kernels, chosen by the lag window size:
//   * score_select_cluster_kernel (lag windows of up to 4096 tokens: the hot path).  A cluster of CTAs owns a run of
//     consecutive scored windows of one (batch, KV head); statistics and spreads stay on the SMs.  Described in front
//     of the kernel below.
//   * score_select_kernel (longer windows).  The work unit is a slice of TOK tokens of one lag window; a
//     CTA takes one unit from a ticket counter in DESCENDING window order and keeps its slice of K and V
//     in registers for both phases:
//       phase 1  per-channel min/max of the slice (packed bf16x2 compares, exact), folded into the
//                window's statistics in global memory with order-preserving integer atomics, then
//                a release-increment of the window's `ready` counter            (Eq. 4, Eq. 5)
//       phase 2  wait (bounded) until the FOLLOWING window's statistics are complete, normalise
//                the slice held in registers (Eq. 6), per-token standard deviation over head_dim
//                (Eq. 7, inner part), written to a small fp32 scratch
//       select   the CTA that finishes a window last soft-maxes the window's K and V spreads
//                (Eq. 7), adds them (Eq. 8), radix-selects the top_k scores and emits the kept
//                positions in ascending order.
//     A unit of window w waits only on units of window w+1, all of which hold smaller tickets, were
//     therefore picked up by CTAs that already run, and publish before they wait on anything: the
//     wait always ends, whatever the number of resident CTAs.  It is bounded all the same.
// Both see one sequence: rows of N tokens per (batch, KV head), of which the sequence starts at token tok0
// (packed batches), windows win_stride tokens apart (negative for the two-window ring of the inference cache).
#include <stddef.h>

#include "lrsa_internal.h"
#include "sm100_ptx.h"

namespace lrsa {
namespace {

constexpr int kThreads = 256;
constexpr int kSteps = 4;  // 16-byte row chunks of K (and of V) each thread keeps in registers

struct ScoreArgs {
  const __nv_bfloat16* K;
  const __nv_bfloat16* V;
  int32_t* idx;
  float* score;   // optional
  WsHeader* hdr;
  int* ready;     // [BH, W]     slices of window w whose min/max are folded in
  int* done;      // [BH, Wsel]  slices of window w whose spreads are written
  uint32_t* mm;   // [BH, W, 2 (K,V), 2 (min,max), d] order-preserving keys, zero = identity
  float* spread;  // [BH, Wsel, 2 (K,V), L]
  int BH, N, L, Kk, S, W, Wsel, n_slices, ddof;   // N: tokens per (batch, head) row of K and V (the row stride)
  int tok0, Wtot, woff;   // the sequence starts at token tok0 of the rows; its windows are [woff, woff + Wsel) of the
                          // Wtot windows per head of idx and score
  int emit_off;           // added to S + w*L + i when a position is written to idx
  int win_stride;         // tokens from window w to window w+1 in memory (L; -L or L for a two-window ring buffer)
  int clear_status;       // the cluster kernel's first CTA clears the status word itself (saves a memset node)
  int unit_wait_limit;    // polls of the one-slice-per-CTA kernel's wait for the next window; negative: give up at once
};

// fp32 bits -> uint32 whose unsigned order is the float order (and back).
__device__ __forceinline__ uint32_t order_key(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_to_float(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k ^ 0x80000000u) : ~k);
}

__device__ __forceinline__ uint32_t bmin2(uint32_t a, uint32_t b) {
  __nv_bfloat162 r = __hmin2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
  return *reinterpret_cast<uint32_t*>(&r);
}
__device__ __forceinline__ uint32_t bmax2(uint32_t a, uint32_t b) {
  __nv_bfloat162 r = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
  return *reinterpret_cast<uint32_t*>(&r);
}
__device__ __forceinline__ float bf_lo(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf_hi(uint32_t p) { return __uint_as_float(p & 0xffff0000u); }

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Top-K of the window by the last CTA to finish it.  smem: sk[L], sv[L] floats, then scratch.
// Bytes of the selection scratch: sk[L], sv[L] (rounded up to 16 bytes), two histograms of 256 bins, 32 floats, 16 + 8 words.
// Rounded up to 16 bytes: the cluster kernel has two of them one behind the other.
__host__ __device__ inline size_t select_scratch_bytes(int L) {
  return (((size_t)2 * L * 4 + 15) & ~(size_t)15) + 2 * 256 * 4 + 32 * 4 + 16 * 4 + 8 * 4;
}

// Barrier of the 256 scoring threads (named barrier 1): the whole block in the one-unit-per-CTA kernel,
// or of the cluster kernel.
__device__ __forceinline__ void scoring_warps_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// `in_smem`: the spreads are already in sk / sv (the cluster kernel keeps them there) instead of in a.spread.
// `wi`: the window's place among all windows of idx and score; `pos0`: position of its first token; `gk`: its spreads in global
// memory otherwise.
__device__ void select_window(const ScoreArgs& a, int bh, int wi, int pos0, unsigned char* smem, bool in_smem,
                              const float* gk = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, L = a.L;
  float* sk = reinterpret_cast<float*>(smem);
  float* sv = sk + L;
  uint32_t* hist = reinterpret_cast<uint32_t*>(smem + (((size_t)2 * L * 4 + 15) & ~(size_t)15));   // two of 256 bins
  float* red = reinterpret_cast<float*>(hist + 512);            // [maxima of K, V][sums of K, V] of the eight warps
  uint32_t* kred = reinterpret_cast<uint32_t*>(red + 32);       // [least, largest key] of the eight warps
  int* wtot = reinterpret_cast<int*>(kred + 16);                // kept keys of the eight warps
  const float* gv = gk + L;
  hist[tid] = hist[256 + tid] = 0;

  // Eq. 7: softmax over the L tokens of the window, for K and for V
  float mk = -INFINITY, mv = -INFINITY;
  for (int i = tid; i < L; i += kThreads) {
    const float x = in_smem ? sk[i] : __ldcg(gk + i), y = in_smem ? sv[i] : __ldcg(gv + i);
    sk[i] = x; sv[i] = y;
    mk = fmaxf(mk, x); mv = fmaxf(mv, y);
  }
  mk = warp_max(mk); mv = warp_max(mv);
  if (lane == 0) { red[warp] = mk; red[8 + warp] = mv; }
  scoring_warps_sync();
  mk = red[0]; mv = red[8];
#pragma unroll
  for (int i = 1; i < 8; ++i) { mk = fmaxf(mk, red[i]); mv = fmaxf(mv, red[8 + i]); }
  float ek = 0.f, ev = 0.f;
  for (int i = tid; i < L; i += kThreads) {
    const float x = expf(sk[i] - mk), y = expf(sv[i] - mv);
    sk[i] = x; sv[i] = y;
    ek += x; ev += y;
  }
  ek = warp_sum(ek); ev = warp_sum(ev);
  if (lane == 0) { red[16 + warp] = ek; red[24 + warp] = ev; }
  scoring_warps_sync();
  ek = 0.f; ev = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) { ek += red[16 + i]; ev += red[24 + i]; }
  // Eq. 8
  float* gs = a.score ? a.score + (size_t)(bh * a.Wtot + wi) * L : nullptr;
  uint32_t kmin = 0xffffffffu, kmax = 0u;   // range of the keys (scores are positive: bit order = value order)
  for (int i = tid; i < L; i += kThreads) {
    const float s = sk[i] / ek + sv[i] / ev;
    sk[i] = s;
    if (gs) gs[i] = s;
    kmin = min(kmin, __float_as_uint(s));
    kmax = max(kmax, __float_as_uint(s));
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) { kred[warp] = kmin; kred[8 + warp] = kmax; }
  scoring_warps_sync();
#pragma unroll
  for (int i = 0; i < 8; ++i) { kmin = min(kmin, kred[i]); kmax = max(kmax, kred[8 + i]); }

  // radix select of the K-th largest score; scores are positive, so bit order = value order
  // The keys of a window share their leading bits (the scores of one window lie within a small factor of
  // each other): those bits are fixed at once, and the 8-bit passes start at the highest bit in which two
  // keys differ.  (A pass over shared bits would also send every key to one histogram bin: a thousand
  // serialised shared-memory atomics.)
  const uint32_t* key = reinterpret_cast<const uint32_t*>(sk);
  const uint32_t diff = kmin ^ kmax;
  const int top = diff ? 31 - __clz(diff) : -1;                  // highest differing bit, -1: all keys equal
  uint32_t mask = top >= 31 ? 0u : ~((2u << (top < 0 ? 0 : top)) - 1u);
  if (top < 0) mask = 0xffffffffu;
  uint32_t prefix = kmax & mask;
  int remaining = a.Kk;
  // One barrier per pass: every warp finds the bin of the K-th key itself, and the histograms take turns.  (With one warp
  // searching and four barriers a pass a call took 28.9 us instead of 27.4 at 32K tokens in windows of 1024.)
  int pass = 0;
  for (int shift = top < 0 ? -1 : max(top - 7, 0); shift >= 0; shift = shift == 0 ? -1 : max(shift - 8, 0), ++pass) {
    uint32_t* h = hist + (pass & 1) * 256;
    for (int i = tid; i < L; i += kThreads) {
      const uint32_t k = key[i];
      if ((k & mask) == prefix) atomicAdd(&h[(k >> shift) & 255u], 1u);
    }
    scoring_warps_sync();
    // lane l owns bins 255-8l ... 248-8l, highest first
    const uint4 hi = *reinterpret_cast<const uint4*>(h + 252 - 8 * lane), lo = *reinterpret_cast<const uint4*>(h + 248 - 8 * lane);
    const uint32_t c[8] = {hi.w, hi.z, hi.y, hi.x, lo.w, lo.z, lo.y, lo.x};
    uint32_t tot = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) tot += c[e];
    uint32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t n = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += n;
    }
    uint32_t above = incl - tot;   // elements in bins above this lane's
    const bool mine = above < (uint32_t)remaining && (uint32_t)remaining <= incl;
    uint32_t bin = 255 - 8 * lane, cnt = c[0];
    bool more = true;
#pragma unroll
    for (int e = 0; e < 7; ++e) {
      more = more && above + c[e] < (uint32_t)remaining;
      if (more) { above += c[e]; --bin; cnt = c[e + 1]; }
    }
    const int src = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
    bin = __shfl_sync(0xffffffffu, bin, src);
    cnt = __shfl_sync(0xffffffffu, cnt, src);              // keys in the chosen bin
    remaining -= (int)__shfl_sync(0xffffffffu, above, src);
    prefix |= bin << shift;
    mask |= 255u << shift;
    // Every key of the chosen bin is kept: the remaining bits need not be resolved.  (With 8-bit digits a
    // thousand keys are alone in their bin after two passes, so this ends the search at half its length.)
    // The threshold is then the bin's lowest possible key: keys above it are kept as "greater", keys equal to
    // it as "equal", of which `remaining` is at least as many as exist.
    if ((int)cnt == remaining) break;
    if (pass > 0) {   // a third pass needs the first histogram again (windows of keys that differ in their last bits only)
      hist[((pass + 1) & 1) * 256 + tid] = 0;
      scoring_warps_sync();
    }
  }
  const uint32_t kth = prefix;    // K-th largest key
  const int need_eq = remaining;  // how many keys equal to it are kept (lowest positions first)

  // emit kept positions in ascending order: every thread takes a run of consecutive tokens, one block
  // scan gives the number of kept tokens before the run
  int32_t* out = a.idx + (size_t)(bh * a.Wtot + wi) * a.Kk;
  const int per = (L + kThreads - 1) / kThreads;
  const int i_lo = min(L, tid * per), i_hi = min(L, i_lo + per);
  int packed = 0;   // tokens above the K-th score | tokens equal to it << 16
  for (int i = i_lo; i < i_hi; ++i) {
    const uint32_t k = key[i];
    packed += (k > kth ? 1 : 0) | (k == kth ? 1 << 16 : 0);
  }
  int incl = packed;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  if (lane == 31) wtot[warp] = incl;
  scoring_warps_sync();
  int excl = incl - packed;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j < warp) excl += wtot[j];
  int gt_before = excl & 0xffff, eq_before = excl >> 16;
  for (int i = i_lo; i < i_hi; ++i) {
    const uint32_t k = key[i];
    if (k > kth) {
      out[gt_before + min(eq_before, need_eq)] = pos0 + i;
      ++gt_before;
    } else if (k == kth) {
      if (eq_before < need_eq) out[gt_before + eq_before] = pos0 + i;
      ++eq_before;
    }
  }
  scoring_warps_sync();   // the scratch may be reused by the caller
}

template <int D>
__global__ void __launch_bounds__(kThreads) score_select_kernel(const ScoreArgs a) {
  constexpr int LPR = D / 8;              // lanes per token row, 16 bytes each
  constexpr int RPS = kThreads / LPR;     // rows per step
  constexpr int TOK = kSteps * RPS;       // tokens per unit
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_ticket, s_flag;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) { s_ticket = atomicAdd(&a.hdr->ticket, 1); s_flag = 0; }
  __syncthreads();
  const int per_w = a.BH * a.n_slices;
  const int w = a.W - 1 - s_ticket / per_w;   // descending windows
  const int r = s_ticket % per_w;
  const int bh = r / a.n_slices, slice = r % a.n_slices;
  const int chunk = tid % LPR, row = tid / LPR;

  // the slice of K and of V, held in registers for both phases
  uint4 kq[kSteps], vq[kSteps];
  bool valid[kSteps];
  const long long row0 = (long long)bh * a.N + a.tok0 + a.S + (long long)w * a.win_stride;
#pragma unroll
  for (int s = 0; s < kSteps; ++s) {
    const int i = slice * TOK + s * RPS + row;
    valid[s] = i < a.L;
    if (valid[s]) {
      const long long off = (row0 + i) * D + chunk * 8;
      kq[s] = __ldcs(reinterpret_cast<const uint4*>(a.K + off));
      vq[s] = __ldcs(reinterpret_cast<const uint4*>(a.V + off));
    } else {
      kq[s] = make_uint4(0, 0, 0, 0);
      vq[s] = make_uint4(0, 0, 0, 0);
    }
  }

  // ---- phase 1: Eq. 4, Eq. 5 (window 0 is never a reference) ----
  if (w >= 1) {
    const uint32_t PINF = 0x7F807F80u, NINF = 0xFF80FF80u;
    uint32_t st[2][2][4];  // [K,V][min,max][4 bf16 pairs]
#pragma unroll
    for (int j = 0; j < 4; ++j) { st[0][0][j] = st[1][0][j] = PINF; st[0][1][j] = st[1][1][j] = NINF; }
#pragma unroll
    for (int s = 0; s < kSteps; ++s) {
      if (!valid[s]) continue;
      const uint32_t kk[4] = {kq[s].x, kq[s].y, kq[s].z, kq[s].w};
      const uint32_t vv[4] = {vq[s].x, vq[s].y, vq[s].z, vq[s].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        st[0][0][j] = bmin2(st[0][0][j], kk[j]); st[0][1][j] = bmax2(st[0][1][j], kk[j]);
        st[1][0][j] = bmin2(st[1][0][j], vv[j]); st[1][1][j] = bmax2(st[1][1][j], vv[j]);
      }
    }
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1)
#pragma unroll
      for (int z = 0; z < 2; ++z)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          st[z][0][j] = bmin2(st[z][0][j], __shfl_xor_sync(0xffffffffu, st[z][0][j], o));
          st[z][1][j] = bmax2(st[z][1][j], __shfl_xor_sync(0xffffffffu, st[z][1][j], o));
        }
    // cross-warp: smem [warp][z*2+stat][D] bf16
    __nv_bfloat16* sm = reinterpret_cast<__nv_bfloat16*>(smem);
    if (lane < LPR) {
#pragma unroll
      for (int z = 0; z < 2; ++z)
#pragma unroll
        for (int m = 0; m < 2; ++m)
          *reinterpret_cast<uint4*>(sm + ((warp * 4 + z * 2 + m) * D + lane * 8)) =
              make_uint4(st[z][m][0], st[z][m][1], st[z][m][2], st[z][m][3]);
    }
    __syncthreads();
    uint32_t* mm = a.mm + (size_t)(bh * a.W + w) * 4 * D;
    for (int v = tid; v < 4 * D; v += kThreads) {
      const int zs = v / D, ch = v % D;
      const bool is_max = zs & 1;
      float acc = __bfloat162float(sm[zs * D + ch]);
#pragma unroll
      for (int ww = 1; ww < kThreads / 32; ++ww) {
        const float x = __bfloat162float(sm[(ww * 4 + zs) * D + ch]);
        acc = is_max ? fmaxf(acc, x) : fminf(acc, x);
      }
      const uint32_t k = order_key(acc);
      atomicMax(mm + v, is_max ? k : ~k);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicAdd(a.ready + bh * a.W + w, 1);
  }
  if (w >= a.Wsel) return;  // the last full window is a reference only

  // ---- phase 2: Eq. 6 and the per-token Std of Eq. 7 ----
  if (tid == 0) {
    const int* flag = a.ready + bh * a.W + w + 1;
    int it = 0;
    while (a.unit_wait_limit < 0 || ld_acquire(flag) < a.n_slices) {
      if (++it > a.unit_wait_limit) { s_flag = 1; atomicExch(&a.hdr->status, (int)LRSA_ERR_TIMEOUT); break; }
      __nanosleep(64);
    }
  }
  __syncthreads();
  if (s_flag) return;
  __threadfence();

  const uint32_t* mm = a.mm + (size_t)(bh * a.W + w + 1) * 4 * D;
  const float inv_dof = 1.0f / (float)(D - a.ddof);
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    // z' = x*sa + sb = zbar - 1/2; a channel with zero range has zbar = 0
    float sa[8], sb[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4 kmn = __ldcg(reinterpret_cast<const uint4*>(mm + (z * 2 + 0) * D + chunk * 8 + h * 4));
      const uint4 kmx = __ldcg(reinterpret_cast<const uint4*>(mm + (z * 2 + 1) * D + chunk * 8 + h * 4));
      const uint32_t a_mn[4] = {kmn.x, kmn.y, kmn.z, kmn.w}, a_mx[4] = {kmx.x, kmx.y, kmx.z, kmx.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float mn = key_to_float(~a_mn[j]), mx = key_to_float(a_mx[j]);
        const float range = mx - mn;
        const float inv = range > 0.f ? 1.0f / range : 0.f;
        sa[h * 4 + j] = inv;
        sb[h * 4 + j] = range > 0.f ? -(0.5f * (mn + mx)) * inv : -0.5f;
      }
    }
    float* out = a.spread + ((size_t)(bh * a.Wsel + w) * 2 + z) * a.L;
#pragma unroll
    for (int s = 0; s < kSteps; ++s) {
      const uint4 q = z == 0 ? kq[s] : vq[s];
      const uint32_t pk[4] = {q.x, q.y, q.z, q.w};
      float sum = 0.f, sq = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float z0 = fmaf(bf_lo(pk[j]), sa[2 * j], sb[2 * j]);
        const float z1 = fmaf(bf_hi(pk[j]), sa[2 * j + 1], sb[2 * j + 1]);
        sum += z0 + z1;
        sq = fmaf(z0, z0, sq);
        sq = fmaf(z1, z1, sq);
      }
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
      }
      if (chunk == 0 && valid[s]) {
        const float var = (sq - sum * sum * (1.0f / D)) * inv_dof;
        out[slice * TOK + s * RPS + row] = sqrtf(fmaxf(var, 0.f));
      }
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_flag = (atomicAdd(a.done + bh * a.Wsel + w, 1) == a.n_slices - 1) ? 2 : 0;
  __syncthreads();
  if (s_flag != 2) return;
  __threadfence();
  select_window(a, bh, a.woff + w, a.emit_off + a.S + w * a.L, smem, false, a.spread + (size_t)(bh * a.Wsel + w) * 2 * a.L);
}

// ---------------------------------------------------------------------------------------------
// Cluster kernel (lag windows up to kClusterMaxL tokens).
//
// A cluster of C CTAs owns a run of consecutive scored windows [w_a, w_b) of one (batch, KV head) and walks it
// downwards; every CTA takes 1/C of the tokens of each window.  It first reads its part of window w_b only for the
// channel minima and maxima (Eq. 4-5), which the CTAs exchange through shared memory; then for w = w_b-1 ... w_a its
// tokens are normalised with the statistics of window w+1 (Eq. 6), reduced to per-token spreads (Eq. 7) that go to the
// shared memory of the CTA that selects the window (the ranks take turns), and folded into the statistics of window w
// for the next step.  The selecting CTA soft-maxes, adds (Eq. 8) and selects while the others go on.
//
// K and V are loaded straight into registers (nothing is staged): four lanes share a token's row (16-byte chunks t,
// t + 4, ... of lane t), eight tokens a warp-wide load, T such groups in flight per warp; half of the warps take K, half
// V.  The channels' scale and offset come from shared memory, one 16-byte broadcast per channel pair for T tokens, and
// the sum over a token's channels ends with two shuffle levels.  A row per 16 lanes with scale and offset in registers,
// the layout of the kernel this one replaces, spent twice the instructions (12 per channel pair, 6 here) on exchanges, and
// one CTA per window left most of the GPU idle when there were few.  Calls back to back on one set of tensors, that kernel | this one, us:
// 4 KV heads, d = 128: 32K tokens in windows of 1024 32.8 | 22.5 (with inputs that change from call to call 35.9 | 25.5, 2.6 TB/s of
// algorithmic bytes; every window is read twice, the second time from L2), 64K of 2048 61.2 | 48.4, 32K of 256 41.0 | 26.7, 1777 tokens
// of 512 20.5 | 9.0; 8 KV heads, 128K of 4096 184 | 160.  What is left is a chain: two streams
// of at most 16 warps' loads an SM, the exchange, the selection (about 3 us).
constexpr int kClusterMaxL = 4096;
constexpr int kClusterMax = 8;

__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {   // p as CTA `rank` of the cluster has it
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(ptx::smem_u32(p)), "r"(rank));
  return addr;
}
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Where the sequences of a launch lie (up to kScoreSeqs of a packed row; the windows of all of them have the same length).
constexpr int kScoreSeqs = 16;
struct ScoreSeqs {
  int n;
  int item0[kScoreSeqs + 1];    // clusters of the sequences before
  int runs[kScoreSeqs], Wsel[kScoreSeqs], first[kScoreSeqs];   // runs per (batch, KV head); scored windows; token of window 0
  int woff[kScoreSeqs], emit0[kScoreSeqs];                     // first window in idx and score; position of window 0
};

template <int D, bool FOLD>
__global__ void __launch_bounds__(kThreads, 2)
score_select_cluster_kernel(const __grid_constant__ ScoreArgs a, const __grid_constant__ ScoreSeqs seqs, int run, int C) {
  constexpr int KC = D / 32;              // 16-byte chunks per lane and row
  constexpr int T = FOLD ? 2 : 4;         // groups of eight tokens in flight
  constexpr int kStatBytes = 4 * D * 2;   // [K, V][min, max][D] bf16
  extern __shared__ __align__(16) unsigned char smem[];
  // [2 (K,V)][KC][4 pairs][4 lanes] (sa, sa, sb, sb); two buffers of statistics; per-warp partial statistics; two
  // selection scratch areas (spreads sk[L], sv[L], histogram, ...)
  float4* sasb = reinterpret_cast<float4*>(smem);
  unsigned char* stat = smem + D * 16;
  __nv_bfloat16* part = reinterpret_cast<__nv_bfloat16*>(stat + 2 * kStatBytes);   // [8 warps][min, max][D]
  unsigned char* sel = stat + 2 * kStatBytes + 8 * 2 * D * 2;
  const size_t sel_bytes = select_scratch_bytes(a.L);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int z = warp & 1, wz = warp >> 1;                 // tensor of this warp (0: K, 1: V), its place among four
  const int rank = blockIdx.x % C;
  int item = blockIdx.x / C, sq = 0;
  while (sq + 1 < seqs.n && item >= seqs.item0[sq + 1]) ++sq;
  item -= seqs.item0[sq];
  const int bh = item / seqs.runs[sq], seg = item % seqs.runs[sq];
  const int w_a = seg * run, w_b = min(seqs.Wsel[sq], w_a + run);   // scored windows [w_a, w_b); reference w_b <= W-1
  const int per = (a.L + C - 1) / C;
  const int i0 = min(a.L, rank * per), i1 = min(a.L, i0 + per);   // this CTA's tokens of every window
  const __nv_bfloat16* base = (z == 0 ? a.K : a.V) + ((long long)bh * a.N + seqs.first[sq]) * D;
  const float inv_dof = 1.0f / (float)(D - a.ddof);

  const int first = i0 + wz * 8 * T;   // this warp's first token
  // While the kernel in front of this one ends: the warps' first two rounds of loads, into L2 (a hint: what that kernel writes is read from
  // L2 all the same, after the wait).  It pays behind a kernel that lets this one start early and has not just written K and V, such as this library's.
  // Behind one that has written them without | with two rounds, us, both kernels: 32K tokens (28/4 heads, d = 128, windows of 1024) 49.4 | 49.9,
  // of 256 53.6 | 54.8, 128K of 4096 184.4 | 183.5, 32K (8/8, d = 64) 51.1 | 50.2, of 256 62.9 | 61.1.  Calls back to back with inputs that change, us, without | with one | two | all rounds:
  // 32K tokens (4 heads, d = 128, windows of 1024) 27.0 | 26.3 | 25.5 | 25.9, as part of a prompt's append 34.0 | 33.0 | 33.2 | 33.4, of a 4K training
  // step 120.6 | 119.4 | 119.5 | 119.4; a call for which the GPU is waited 42.2 | 42.2 | 42.4 | 45.
  if (lane == 0 && wz == 0 && i1 > i0)
    ptx::prefetch_l2(base + ((long long)w_b * a.win_stride + i0) * D, min(i1 - i0, 2 * 32 * T) * D * 2);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (a.clear_status && blockIdx.x == 0 && tid == 0) a.hdr->status = 0;
  for (int w = w_b; w >= w_a; --w) {
    const int it = w_b - w, buf = it & 1;
    const bool scoring = it > 0, want_stats = w > w_a;
    const __nv_bfloat16* win = base + (long long)w * a.win_stride * D;
    const int sel_rank = it % C;
    uint32_t mn[KC][4], mx[KC][4];
#pragma unroll
    for (int j = 0; j < KC; ++j)
#pragma unroll
      for (int p = 0; p < 4; ++p) { mn[j][p] = 0x7F807F80u; mx[j][p] = 0xFF80FF80u; }
    for (int r0 = first; r0 < i1; r0 += 4 * 8 * T) {
      uint4 x[T][KC];
#pragma unroll
      for (int s = 0; s < T; ++s) {
        const int row = min(r0 + 8 * s + g, i1 - 1);    // beyond the part: its last token again (not written)
#pragma unroll
        for (int j = 0; j < KC; ++j)
          x[s][j] = *reinterpret_cast<const uint4*>(win + (long long)row * D + (t + 4 * j) * 8);
      }
      if (want_stats && (FOLD || !scoring)) {
#pragma unroll
        for (int s = 0; s < T; ++s)
#pragma unroll
          for (int j = 0; j < KC; ++j) {
            const uint32_t v[4] = {x[s][j].x, x[s][j].y, x[s][j].z, x[s][j].w};
#pragma unroll
            for (int p = 0; p < 4; ++p) { mn[j][p] = bmin2(mn[j][p], v[p]); mx[j][p] = bmax2(mx[j][p], v[p]); }
          }
      }
      if (scoring) {
        // Eq. 6 with the statistics of window w+1 (z' = x*sa + sb = zbar - 1/2), sums for the Std of Eq. 7
        // The sums are formed chunk by chunk (eight channels) and the chunks added in a tree over the distances 8, 4, 2, 1,
        // whatever the layout: a score that ties with the K-th one falls on the same side in every version of this kernel.
        float v[T][2], first2[T][2];
#pragma unroll
        for (int k = 0; k < KC; ++k) {
          const int j = KC == 4 ? (k & 1) * 2 + (k >> 1) : k;   // 0, 2, 1, 3
          uint64_t sum2[T], sq2[T];
#pragma unroll
          for (int s = 0; s < T; ++s) sum2[s] = sq2[s] = 0ull;   // (+0, +0)
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            const float4 f = sasb[((z * KC + j) * 4 + p) * 4 + t];
            const uint64_t sa = ptx::f2_pack(f.x, f.y), sb = ptx::f2_pack(f.z, f.w);
#pragma unroll
            for (int s = 0; s < T; ++s) {
              const uint32_t u = p == 0 ? x[s][j].x : p == 1 ? x[s][j].y : p == 2 ? x[s][j].z : x[s][j].w;
              const uint64_t z2 = ptx::f2_fma(ptx::f2_pack(bf_lo(u), bf_hi(u)), sa, sb);
              sum2[s] = ptx::f2_add(sum2[s], z2);
              sq2[s] = ptx::f2_fma(z2, z2, sq2[s]);
            }
          }
#pragma unroll
          for (int s = 0; s < T; ++s) {
            float x0, x1, y0, y1;
            ptx::f2_unpack(sum2[s], x0, x1);
            ptx::f2_unpack(sq2[s], y0, y1);
            const float a0 = x0 + x1, a1 = y0 + y1;
            if (k == 0) { v[s][0] = a0; v[s][1] = a1; }
            else if (k == 1) { v[s][0] += a0; v[s][1] += a1; }
            else if (k == 2) { first2[s][0] = a0; first2[s][1] = a1; }
            else { v[s][0] += first2[s][0] + a0; v[s][1] += first2[s][1] + a1; }
          }
        }
        // Sum over the four lanes of a row, halving: a lane hands half of its rows to its partner at each level
        int mine = 0;   // row this lane ends up with
        const bool up2 = (t & 2) != 0, up1 = (t & 1) != 0;
        if constexpr (T == 4) {
#pragma unroll
          for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float send = up2 ? v[s][e] : v[s + 2][e], keep = up2 ? v[s + 2][e] : v[s][e];
              v[s][e] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
            }
          mine = up2 ? 2 : 0;
        } else {
#pragma unroll
          for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int e = 0; e < 2; ++e) v[s][e] += __shfl_xor_sync(0xffffffffu, v[s][e], 2);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float send = up1 ? v[0][e] : v[1][e], keep = up1 ? v[1][e] : v[0][e];
          v[0][e] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
        }
        mine += up1 ? 1 : 0;
        const int tok = r0 + 8 * mine + g;
        if (tok < i1 && (T == 4 || !up2)) {
          const float var = (v[0][1] - v[0][0] * v[0][0] * (1.0f / D)) * inv_dof;
          const float spread = sqrtf(fmaxf(var, 0.f));
          const uint32_t dst = cluster_addr(sel + buf * sel_bytes + ((size_t)z * a.L + tok) * 4, sel_rank);
          asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(spread) : "memory");
        }
      }
    }
    if (want_stats) {
      // over the eight row groups of the warp, then over the four warps of the tensor
#pragma unroll
      for (int o = 16; o >= 4; o >>= 1)
#pragma unroll
        for (int j = 0; j < KC; ++j)
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            mn[j][p] = bmin2(mn[j][p], __shfl_xor_sync(0xffffffffu, mn[j][p], o));
            mx[j][p] = bmax2(mx[j][p], __shfl_xor_sync(0xffffffffu, mx[j][p], o));
          }
      if (g == 0) {
#pragma unroll
        for (int j = 0; j < KC; ++j) {
          *reinterpret_cast<uint4*>(part + (warp * 2 + 0) * D + (t + 4 * j) * 8) = make_uint4(mn[j][0], mn[j][1], mn[j][2], mn[j][3]);
          *reinterpret_cast<uint4*>(part + (warp * 2 + 1) * D + (t + 4 * j) * 8) = make_uint4(mx[j][0], mx[j][1], mx[j][2], mx[j][3]);
        }
      }
      __syncthreads();
      for (int v = tid; v < 2 * D; v += kThreads) {   // pairs of channels: [tensor][min, max][D / 2]
        const int zz = v / D, m = v / (D / 2) & 1, ch = v % (D / 2);
        uint32_t r = *reinterpret_cast<const uint32_t*>(part + (zz * 2 + m) * D + 2 * ch);
#pragma unroll
        for (int k = 1; k < 4; ++k) {
          const uint32_t y = *reinterpret_cast<const uint32_t*>(part + ((2 * k + zz) * 2 + m) * D + 2 * ch);
          r = m ? bmax2(r, y) : bmin2(r, y);
        }
        *reinterpret_cast<uint32_t*>(stat + buf * kStatBytes + v * 4) = r;
      }
    }
    // Every CTA's spreads and statistics of this window are in place.  (A buffer is written again two windows later, behind
    // the barrier of the window between, which a CTA only reaches when it has read the buffer.)
    cluster_sync();
    if (want_stats) {
      for (int v = tid; v < D; v += kThreads) {   // pairs of channels: [tensor][D / 2]
        const int zz = v / (D / 2), ch = v % (D / 2);   // channels 2ch, 2ch + 1
        uint32_t lo = 0x7F807F80u, hi = 0xFF80FF80u;
        for (int r = 0; r < C; ++r) {
          uint32_t x, y;
          const uint32_t src = cluster_addr(stat + buf * kStatBytes + zz * D * 4 + ch * 4, r);
          asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x) : "r"(src) : "memory");
          asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(y) : "r"(src + D * 2) : "memory");
          lo = bmin2(lo, x);
          hi = bmax2(hi, y);
        }
        float f[4];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          // a channel with zero range has zbar = 0, i.e. z' = -1/2
          const float a0 = e ? bf_hi(lo) : bf_lo(lo), a1 = e ? bf_hi(hi) : bf_lo(hi), range = a1 - a0;
          const float inv = range > 0.f ? 1.0f / range : 0.f;
          f[e] = inv;
          f[2 + e] = range > 0.f ? -(0.5f * (a0 + a1)) * inv : -0.5f;
        }
        const int chunk = ch >> 2, p = ch & 3;   // chunk of eight channels: lane chunk % 4, its chunk / 4-th
        sasb[((zz * KC + (chunk >> 2)) * 4 + p) * 4 + (chunk & 3)] = make_float4(f[0], f[1], f[2], f[3]);
      }
    }
    if (scoring && rank == sel_rank)
      select_window(a, bh, seqs.woff[sq] + w, seqs.emit0[sq] + w * a.L, sel + buf * sel_bytes, true);
    __syncthreads();   // scale and offset are in place for the next window
  }
}

// Longest window the one-slice-per-CTA kernel takes: 25 448 tokens, 201 KB of selection scratch.
constexpr int kUnitMaxL = 25448;

template <int D>
constexpr int tok_per_unit() { return kSteps * (kThreads / (D / 8)); }

size_t select_smem_bytes(int L, int d) {
  const size_t phase1 = (size_t)(kThreads / 32) * 4 * d * sizeof(__nv_bfloat16);
  const size_t sel = select_scratch_bytes(L);
  return phase1 > sel ? phase1 : sel;
}

// Polls the one-slice-per-CTA kernel grants its wait for the following window's statistics.  Test hook:
// a negative value makes that wait give up at once (the kernel holds its slice in registers and has no
// copy in flight, so every thread returns after the verdict).
int g_unit_wait_limit = 1 << 21;

struct ScoreWs {
  size_t ready, done, mm, zero_bytes, spread, total;
};
ScoreWs score_ws_layout(const Geom& g) {
  ScoreWs w;
  const size_t BH = (size_t)g.B * g.Hkv;
  size_t off = sizeof(WsHeader);
  w.ready = off; off += align_up(BH * g.W * sizeof(int), 16);
  w.done = off;  off += align_up(BH * g.Wsel * sizeof(int), 16);
  w.mm = off;    off += align_up(BH * g.W * 4 * g.d * sizeof(uint32_t), 256);
  w.zero_bytes = off;   // everything up to here is cleared before the launch
  w.spread = off; off += align_up(BH * g.Wsel * 2 * g.L * sizeof(float), 256);
  w.total = off;
  return w;
}

// Run length and cluster size by the measured cost of a CTA, in tokens streamed (21 ns each at d = 128 with two CTAs an SM):
// (run + 1) windows' parts, 290 for launch, exchange and selection of the first scored window, 550 for every further one (a chain
// of barriers, and half as many loads in flight beside the folded statistics).  At d = 64 a row is half as long and the folded
// form, with two rows of it in flight, streams at two thirds of the other's rate: from windows between 512 and 1000 tokens on that is
// more than it saves, and a CTA takes one window.
// us, run x C: d = 128, 4 heads: 32K tokens in windows of 1024 1x1 23.4, 1x2 22.8, 1x4 30.5, 2x4 28.1; of 256 1x1 26.9, 2x1 25.4; 64K of
// 2048 1x1 56.5, 1x2 48.6, 2x4 49.9; 8 heads: 32K of 512 1x1 48.4, 2x1 43.3; 64K of 512 1x1 88.0, 2x1 90.4, 4x1 79.3; 128K of 512
// 1x1 150.7, 4x1 159.6, 7x1 133.0, 8x1 148.6; 128K of 4096 1x1 167.8, 2x2 160.1, 4x4 171.0; batch 2 of it 2x1 289.9, 4x2 288.9.
// d = 64, 8 heads: 64K of 512 1x1 56.7, 4x1 57.1; of 1000 1x1 55.3, 2x1 61.4; of 2048 1x1 51.4, 2x2 60.5; of 4096 1x2 55.4, 2x4 71.2;
// 128K of 512 1x1 104.4, 7x1 100.7; of 1000 1x1 102.0, 4x1 105.5; of 4096 1x1 97.5, 2x2 117.9; 16K of 333 1x1 32.8, 2x1 25.6.
// (Calls back to back on one set of tensors.)
constexpr int kFoldMaxL64 = 768;
struct ClusterPlan { int run, C; };
ClusterPlan cluster_plan(int BH, int Wsel, int L, int d) {
  ClusterPlan best = {1, 1};
  const ClusterRoom& room = cluster_room();
  double cost = -1;
  for (int C = 1; C <= kClusterMax; C *= 2) {
    const long long slots = room.at_once(2, C);
    for (int r = 1; r <= (d == 64 && L > kFoldMaxL64 ? 1 : Wsel); r = r < 8 ? r + 1 : r * 2) {
      const long long clusters = (long long)BH * ((Wsel + r - 1) / r), waves = (clusters + slots - 1) / slots;
      const double c = waves * ((r + 1.0) * ((L + C - 1) / C) + 290.0 + (r - 1) * 550.0);
      if (cost < 0 || c < cost) { cost = c; best.run = r; best.C = C; }
      if (waves == 1) break;
    }
  }
  return best;
}

}  // namespace

// The cluster kernel uses nothing but the status header; the one-slice-per-CTA kernel needs its counters,
// statistics and spreads.
size_t score_select_ws_bytes(const Geom& g) { return g.L <= kClusterMaxL ? sizeof(WsHeader) : score_ws_layout(g).total; }

void set_unit_wait_limit(int polls) { g_unit_wait_limit = polls; }

bool score_select_clears_status(const Geom& g) { return (g.n_seqs > 0 ? g.Wtot : g.Wsel) > 0 && g.L <= kClusterMaxL; }

static ScoreArgs score_args(const Geom& g, const __nv_bfloat16* K, const __nv_bfloat16* V, int32_t* idx, float* score, void* ws) {
  unsigned char* base = static_cast<unsigned char*>(ws);
  ScoreArgs a = {};
  a.K = K; a.V = V; a.idx = idx; a.score = score;
  a.hdr = reinterpret_cast<WsHeader*>(base);
  a.BH = g.B * g.Hkv; a.N = g.Nrow; a.L = g.L; a.Kk = g.K; a.S = g.S; a.W = g.W; a.Wsel = g.Wsel;
  a.tok0 = g.tok0; a.Wtot = g.Wtot; a.woff = g.woff; a.emit_off = g.emit_off; a.win_stride = g.win_stride;
  a.ddof = g.ddof;
  return a;
}

static int launch_cluster(const Geom* gs, int n_seqs, const __nv_bfloat16* K, const __nv_bfloat16* V, int32_t* idx, float* score,
                          void* ws, cudaStream_t st, bool clear_status) {
  for (int s0 = 0; s0 < n_seqs;) {
    // the next sequences with anything to score
    ScoreSeqs q;
    q.n = 0;
    int windows = 0, s1 = s0;
    for (; s1 < n_seqs && q.n < kScoreSeqs; ++s1)
      if (gs[s1].Wsel > 0) { ++q.n; windows += gs[s1].Wsel; }
    if (q.n == 0) return LRSA_OK;
    const Geom& g = gs[s0];
    ScoreArgs a = score_args(g, K, V, idx, score, ws);
    a.clear_status = clear_status ? 1 : 0;
    const ClusterPlan pl = cluster_plan(a.BH, windows, g.L, g.d);
    q.n = 0;
    q.item0[0] = 0;
    for (int s = s0; s < s1; ++s) {
      const Geom& e = gs[s];
      if (e.Wsel == 0) continue;
      q.runs[q.n] = (e.Wsel + pl.run - 1) / pl.run;
      q.Wsel[q.n] = e.Wsel;
      q.first[q.n] = e.tok0 + e.S;
      q.woff[q.n] = e.woff;
      q.emit0[q.n] = e.emit_off + e.S;
      q.item0[q.n + 1] = q.item0[q.n] + a.BH * q.runs[q.n];
      ++q.n;
    }
    const long long grid = (long long)q.item0[q.n] * pl.C;
    if (grid > 0x7fffffffLL) return LRSA_ERR_UNSUPPORTED;
    const size_t bytes = (size_t)g.d * 16 + 2 * (4 * g.d * 2) + 8 * 2 * g.d * 2 + 2 * select_scratch_bytes(g.L);
    auto kern = g.d == 128 ? (pl.run > 1 ? score_select_cluster_kernel<128, true> : score_select_cluster_kernel<128, false>)
                           : (pl.run > 1 ? score_select_cluster_kernel<64, true> : score_select_cluster_kernel<64, false>);
    if (bytes > 48 * 1024)
      LRSA_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    LRSA_CUDA_CHECK(launch_dependent(kern, dim3((unsigned)grid), dim3(kThreads), bytes, st, pl.C, a, q, pl.run, pl.C));
    launch_counter().n++;
    clear_status = false;
    s0 = s1;
  }
  return LRSA_OK;
}

static int launch_unit(const Geom& g, const __nv_bfloat16* K, const __nv_bfloat16* V, int32_t* idx, float* score, void* ws,
                       cudaStream_t st) {
  if (g.Wsel == 0) return LRSA_OK;  // nothing is scored
  if (g.L > kUnitMaxL) return LRSA_ERR_UNSUPPORTED;
  const ScoreWs lay = score_ws_layout(g);
  unsigned char* base = static_cast<unsigned char*>(ws);
  // The status word (the header) is cleared once per call by the caller; the ticket, the counters and the statistics here.
  LRSA_CUDA_CHECK(cudaMemsetAsync(base + offsetof(WsHeader, ticket), 0, lay.zero_bytes - offsetof(WsHeader, ticket), st));
  launch_counter().n++;
  ScoreArgs a = score_args(g, K, V, idx, score, ws);
  a.ready = reinterpret_cast<int*>(base + lay.ready);
  a.done = reinterpret_cast<int*>(base + lay.done);
  a.mm = reinterpret_cast<uint32_t*>(base + lay.mm);
  a.spread = reinterpret_cast<float*>(base + lay.spread);
  a.unit_wait_limit = g_unit_wait_limit;
  const int tok = g.d == 128 ? tok_per_unit<128>() : tok_per_unit<64>();
  a.n_slices = (g.L + tok - 1) / tok;
  const size_t smem = select_smem_bytes(g.L, g.d);
  const long long units = (long long)a.BH * g.W * a.n_slices;
  if (units > 0x7fffffffLL) return LRSA_ERR_UNSUPPORTED;
  auto kern = g.d == 128 ? score_select_kernel<128> : score_select_kernel<64>;
  LRSA_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  kern<<<(unsigned)units, kThreads, smem, st>>>(a);
  LRSA_CUDA_CHECK(cudaGetLastError());
  launch_counter().n++;
  return LRSA_OK;
}

int launch_score_select(const Geom* gs, int n_seqs, const __nv_bfloat16* K, const __nv_bfloat16* V, int32_t* idx,
                        float* score, void* ws, cudaStream_t st, bool clear_status) {
  const Geom& g = gs[0];   // the shape is the same for all; windows and places differ
  if (g.L <= kClusterMaxL) return launch_cluster(gs, n_seqs, K, V, idx, score, ws, st, clear_status);
  for (int s = 0; s < n_seqs; ++s) {
    const int rc = launch_unit(gs[s], K, V, idx, score, ws, st);
    if (rc != LRSA_OK) return rc;
  }
  return LRSA_OK;
}

}  // namespace lrsa
