// LRSA attention backward, dQ part, on tcgen05 tensor cores.
//
// A CTA owns one 128-row query tile of one (batch, query head) and walks its key list (the same
// row-block decomposition as the forward) in 64-key tiles.  Q and dO are copied once into tensor
// memory, so every product takes its 128-row operand from TMEM and only the K_j / V_j tiles from
// shared memory (with both operands in shared memory the kernel is bound by shared-memory
// bandwidth, not by the tensor core).  As in the forward, a last list tile of at most 16 keys comes
// first and is multiplied 16 wide (whole step 372 -> 370 us at 4K tokens).  Per key tile j:
//   S  = Q K_j^T          (TMEM x smem -> TMEM)      P  = exp2(S*c - LSE*log2e)
//   dP = dO V_j^T         (TMEM x smem -> TMEM)      dS = P * (dP - D)          (bf16, back into TMEM)
//   A += dS K_j           (TMEM x smem -> TMEM)      epilogue: dQ = scale * (A - r * kbar) -> bf16
// S/dP are double-buffered in TMEM (NB = 2; NB = 1, two CTAs per SM: see launch_bwd_dq_sm100), so the
// tensor core computes tile j+1 while tile j is in the softmax; both softmax warpgroups work on every tile (32 key columns each) to keep the latency
// between "S ready" and "dS ready" short.  One warp issues all products, A_j before S_{j+2} and dP_{j+2}, which may then
// overwrite the buffer without a barrier round trip (with a warp for each product and a "buffer free" barrier: whole step
// 372 against 366 us at 4K tokens, 28/4 heads, d = 128; 3.96 against 3.86 ms for 32K tokens in eight sequences).
// Warps: 0 TMA producer, 1 issuer, 4-11 softmax and epilogue.
//
// D_t = sum_j P_tj dP_tj comes from the dK/dV kernel, which runs first and accumulates it in fp32
// (rowsum(dO * O) of the bf16 O is not accurate enough: its error is multiplied by the
// softmax-averaged key, which is large when a few salient keys dominate a row).
// Rows of the exact dS sum to zero; after bf16 rounding they sum to r_t, which multiplies whatever
// constant vector the keys of a head share (outlier channels).  The epilogue subtracts r_t * kbar,
// kbar the mean key of the KV head; in exact arithmetic this subtracts zero.
#include "attn_bwd_sm100.h"

namespace lrsa {
namespace {

using namespace ptx;

constexpr int kKeys = 64;   // keys per tile in this kernel
constexpr int kShort = 16;

template <int D, int NB>
struct DqCfg {
  static constexpr int kSub = D / 64;
  static constexpr int kQSubBytes = kTile * 128;           // 128 query rows x 128 bytes
  static constexpr int kQTileBytes = kSub * kQSubBytes;    // the Q or the dO tile
  static constexpr int kKSubBytes = kKeys * 128;           // 64 key rows x 128 bytes
  static constexpr int kKTileBytes = kSub * kKSubBytes;    // one K or V tile
  static constexpr int kStages = D == 128 ? 9 : 8 * NB;    // ring slots, K and V tiles alternate
  static constexpr int kSmem = 2 * kQTileBytes + kStages * kKTileBytes + 1024;
  static constexpr int kThreads = 384;
  static constexpr int kPerSm = 3 - NB, kCols = 256 * NB;   // resident CTAs, TMEM columns
  // TMEM columns: Q and dO as packed bf16 (D/2 columns each), accumulator A at D, then buffer b with
  // S at 128 NB + 128 b and dP 64 columns further
  static constexpr uint32_t kColQ = 0, kColdO = D / 2, kColA = D, kColBuf = 128 * NB, kColP = 64;
};

template <int NSEQ>
struct DqMaps { CUtensorMap q[NSEQ], dO[NSEQ], k[NSEQ], v[NSEQ], kc[NSEQ], vc[NSEQ]; };

template <int NSEQ>
struct DqArgs {
  BlockPlan plan[NSEQ];
  int tok0[NSEQ];          // first token of the sequence
  int block0[NSEQ + 1];    // blocks of the sequences before, per (batch, head)
  int n_seqs;
  int BH, Hq, Hkv, G, N;   // N: tokens per (batch, head) row of stats, Dacc and dQ (the row stride)
  const float2* stats;   // per query row: (-LSE*log2e, D~); only the first component is used here
  const float* Dacc;     // per query row: D = sum_j P dP
  const float* kbar;     // [B*Hkv][D] mean key
  __nv_bfloat16* dQ;
  float scale, scale_log2;
  int* status;
};

struct DqBars {
  uint64_t q_full, qt_ready, acc_done;
  uint64_t kv_full[16], kv_empty[16];
  uint64_t s_full[2], p_full[2];
};

template <int D, int NSEQ, int NB>
__global__ void __launch_bounds__(DqCfg<D, NB>::kThreads, DqCfg<D, NB>::kPerSm)
lrsa_bwd_dq_kernel(const __grid_constant__ DqMaps<NSEQ> maps, const __grid_constant__ DqArgs<NSEQ> a) {
  using Cfg = DqCfg<D, NB>;
  constexpr int NS = Cfg::kStages;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) DqBars bars;
  __shared__ float red_s[2][kTile];   // [column half][row] sums of the rounded dS
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = smem0, sdO = smem0 + Cfg::kQTileBytes, sRing = smem0 + 2 * Cfg::kQTileBytes;

  const int bh = blockIdx.x % a.BH;
  int blk = blockIdx.x / a.BH, sq = 0;
  if constexpr (NSEQ > 1) {
    while (sq + 1 < a.n_seqs && blk >= a.block0[sq + 1]) ++sq;
    blk -= a.block0[sq];
  }
  const RowBlock rb = decode_block(a.plan[sq], blk);
  const size_t row0 = (size_t)bh * a.N + a.tok0[sq];   // the sequence's first row of stats, Dacc and dQ
  const int bh_kv = (bh / a.Hq) * a.Hkv + (bh % a.Hq) / a.G;
  const int n_ct = (rb.n_front + kKeys - 1) / kKeys;
  const int n = n_ct + (rb.q_end - 1 - rb.dense_start) / kKeys + 1;   // key tiles of this block (>= 1)
  // the list's last tile comes first when it holds no more than kShort keys: its products are that wide only
  const int sh = n_ct > 0 && rb.n_front - (n_ct - 1) * kKeys <= kShort ? 1 : 0;

  // K or V tile `it` of the order K_0, V_0, K_1, ... into its ring slot
  auto load_tile = [&](int it) {
    const int j = it >> 1, which = it & 1, slot = it % NS;
    const uint32_t full = smem_u32(&bars.kv_full[slot]);
    mbar_expect_tx(full, Cfg::kKTileBytes);
    const bool compact = j < n_ct;
    const CUtensorMap* map = compact ? (which ? &maps.vc[sq] : &maps.kc[sq]) : (which ? &maps.v[sq] : &maps.k[sq]);
    const int row = compact ? (j < sh ? n_ct - 1 : j - sh) * kKeys : rb.dense_start + (j - n_ct) * kKeys;
    for (int h = 0; h < Cfg::kSub; ++h)
      tma_load_3d(sRing + slot * Cfg::kKTileBytes + h * Cfg::kKSubBytes, map, h * 64, row, bh_kv, full);
  };
  if (tid == 0) {
    prefetch_tensormap(&maps.q[sq]); prefetch_tensormap(&maps.dO[sq]); prefetch_tensormap(&maps.k[sq]);
    prefetch_tensormap(&maps.v[sq]); prefetch_tensormap(&maps.kc[sq]); prefetch_tensormap(&maps.vc[sq]);
    abort_s = 0;
    mbar_init(smem_u32(&bars.q_full), 1);
    mbar_init(smem_u32(&bars.qt_ready), 256);
    mbar_init(smem_u32(&bars.acc_done), 1);
    for (int i = 0; i < NS; ++i) { mbar_init(smem_u32(&bars.kv_full[i]), 1); mbar_init(smem_u32(&bars.kv_empty[i]), 1); }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars.s_full[b]), 1);
      mbar_init(smem_u32(&bars.p_full[b]), 256);    // every softmax thread
    }
    fence_barrier_init();
    // The first loads, while the other warps get their tensor memory.  No more than what the first products need: the block waits for this
    // thread, and with the whole ring here a CTA starts 1.5 us later (32K tokens, 28/4 heads, d = 128: 2885 us, with two tiles 2801, with
    // all loads behind the barrier 2807; 8K 317 | 305 | 306; 1777 60.1 | 57.5 | 57.9; 4K, 8/8 heads, d = 64 37.6 | 35.5 | 36.0).
    asm volatile("griddepcontrol.wait;" ::: "memory");   // started before the kernel in front of it has ended
    mbar_expect_tx(smem_u32(&bars.q_full), 2 * Cfg::kQTileBytes);
    for (int h = 0; h < Cfg::kSub; ++h) {
      tma_load_3d(sQ + h * Cfg::kQSubBytes, &maps.q[sq], h * 64, rb.q0, bh, smem_u32(&bars.q_full));
      tma_load_3d(sdO + h * Cfg::kQSubBytes, &maps.dO[sq], h * 64, rb.q0, bh, smem_u32(&bars.q_full));
    }
    load_tile(0);
    load_tile(1);
  }
  if (warp == 1) { tmem_alloc(smem_u32(&tmem_base_s), Cfg::kCols); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_s;
  volatile int* abort = &abort_s;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      int it = 2;   // the first two tiles are on their way
      bool ok = true;
      for (; it < 2 * n; ++it) {
        if (it >= NS) ok = mbar_wait(smem_u32(&bars.kv_empty[it % NS]), (it / NS - 1) & 1, abort);
        if (!ok) break;
        load_tile(it);
      }
      if (!ok) {
        // give loads already in flight a bounded chance to land before the CTA's smem is released
        for (int back = 1; back <= NS && back <= it; ++back) {
          const int i2 = it - back;
          const long long t0 = clock64();
          while (!mbar_try_wait(smem_u32(&bars.kv_full[i2 % NS]), (i2 / NS) & 1) && clock64() - t0 < 2000000) {}
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- issuer: S_j, dP_j NB tiles ahead of A += dS_j K_j ----------------
    // One thread issues everything, and the tensor core runs its products in this order (sm100_ptx.h): S_{j+NB} may
    // overwrite dS_j, and dP_{j+NB} dP_j, without waiting for the product that reads dS_j.
    constexpr uint32_t idesc_full = make_idesc_bf16(kTile, kKeys, 0, 0), idesc_short = make_idesc_bf16(kTile, kShort, 0, 0);
    constexpr uint32_t idesc_a = make_idesc_bf16(kTile, D, 0, 1);       // 128 x D, B = K_j MN-major
    const uint64_t descR = make_smem_desc_sw128(sRing, 16, 1024);       // K-major K_j / V_j
    const uint64_t descRmn = make_smem_desc_sw128(sRing, Cfg::kKSubBytes, 1024);
    const uint32_t leader = elect_one();
    int slot = 0, ph = 0, slot_a = 0;   // ring order K_0, V_0, K_1, V_1, ...: the next tile to multiply with, K_j of A
    auto scores = [&](uint32_t d_tmem, uint32_t a_tmem, uint32_t idesc_s) {
      if (!mbar_wait_warp(smem_u32(&bars.kv_full[slot]), ph, abort)) return false;
      const uint64_t dT = desc_advance(descR, slot * Cfg::kKTileBytes);
#pragma unroll
      for (int h = 0; h < Cfg::kSub; ++h)
        umma_ts4<8, 16, 24, 32>(d_tmem, a_tmem + h * 32, desc_advance(dT, h * Cfg::kKSubBytes), idesc_s, h > 0 ? 1u : 0u, leader);
      return true;
    };
    bool ok = mbar_wait_warp(smem_u32(&bars.qt_ready), 0, abort);   // Q and dO are in tensor memory
    tc_fence_after_sync();
    for (int j = -NB; j < n && ok; ++j) {
      const int b = j & (NB - 1);
      const uint32_t buf = tmem + Cfg::kColBuf + b * 128;
      if (j >= 0) {
        ok = mbar_wait_warp(smem_u32(&bars.p_full[b]), (j >> (NB - 1)) & 1, abort);
        if (!ok) break;
        tc_fence_after_sync();
        // packed dS: keys [0,32) in columns [0,16) of the S region, keys [32,64) in columns [32,48)
        const uint64_t dKj = desc_advance(descRmn, slot_a * Cfg::kKTileBytes);
        if (j < sh) umma_ts1(tmem + Cfg::kColA, buf, dKj, idesc_a, 0u, leader);
        else umma_ts4<8, 32, 40, 2048>(tmem + Cfg::kColA, buf, dKj, idesc_a, j > 0 ? 1u : 0u, leader);
        umma_commit(smem_u32(&bars.kv_empty[slot_a]), leader);   // K_j: S (before the softmax) and A are done
        slot_a += 2;
        if (slot_a >= NS) slot_a -= NS;
      }
      if (j + NB < n) {
        const uint32_t idesc_s = j + NB < sh ? idesc_short : idesc_full;
        ok = scores(buf, tmem + Cfg::kColQ, idesc_s);
        if (++slot == NS) { slot = 0; ph ^= 1; }
        if (ok) ok = scores(buf + Cfg::kColP, tmem + Cfg::kColdO, idesc_s);
        if (!ok) break;
        umma_commit(smem_u32(&bars.s_full[b]), leader);
        umma_commit(smem_u32(&bars.kv_empty[slot]), leader);   // V_j is used by dP only
        if (++slot == NS) { slot = 0; ph ^= 1; }
      }
    }
    if (ok) umma_commit(smem_u32(&bars.acc_done), leader);
  } else if (warp >= 4) {
    // ---------------- softmax warps: warpgroup `half` takes key columns [32*half, 32*half+32) ----------------
    const int half = (warp - 4) >> 2, quad = warp & 3;
    const int row = quad * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const int qpos = rb.q0 + row;
    const bool live = qpos < rb.q_end;
    const float c = a.scale_log2;
    // rows outside the block get lse = +inf so that P = 0
    const float nl2 = live ? a.stats[row0 + qpos].x : -INFINITY;
    const float Dt = live ? a.Dacc[row0 + qpos] : 0.f;
    float rsum = 0.f;
    // copy this thread's row of Q (warpgroup 0) or dO (warpgroup 1) from the swizzled shared-memory
    // tile into tensor memory: 16-byte chunk c of row r of a 64-column sub-tile sits at chunk c ^ (r & 7)
    // (A lane whose wait gave up goes on with the others, on whatever is there: the verdicts are voted on every 16 tiles and before the
    // output.  With a vote for every tile the whole backward takes 0.5 % longer: 4K tokens, 8 heads, d = 64, 82.6 | 83.2 us.)
    bool ok = mbar_wait_lanes(smem_u32(&bars.q_full), 0, abort);
    {
      const unsigned char* src = smem_raw + ((half == 0 ? sQ : sdO) - smem_u32(smem_raw)) + row * 128;
      const uint32_t dst = tmem + lane_addr + (half == 0 ? Cfg::kColQ : Cfg::kColdO);
#pragma unroll
      for (int h = 0; h < Cfg::kSub; ++h) {
        uint32_t v[32];
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
          const uint4 x = *reinterpret_cast<const uint4*>(src + h * Cfg::kQSubBytes + ((ch ^ (row & 7)) << 4));
          v[4 * ch] = x.x; v[4 * ch + 1] = x.y; v[4 * ch + 2] = x.z; v[4 * ch + 3] = x.w;
        }
        tmem_st32(dst + h * 32, v);
      }
      tmem_wait_st();
    }
    tc_fence_before_sync();
    mbar_arrive(smem_u32(&bars.qt_ready));   // also when the wait gave up: the issuers then see abort
    const int list_end = rb.n_front + sh * kKeys;   // keys of list tile j: the first list_end - 64 j
    if (sh) {
      ok &= mbar_wait_lanes(smem_u32(&bars.s_full[0]), 0, abort);
      if (half == 0) {   // only the first kShort columns hold scores
        tc_fence_after_sync();
        const uint32_t S_addr = tmem + lane_addr + Cfg::kColBuf;
        const int limit = rb.n_front - (n_ct - 1) * kKeys;
        uint32_t s[32], dp[32], ds[kShort / 2];
        tmem_ld32(S_addr, s);
        tmem_ld32(S_addr + Cfg::kColP, dp);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < kShort / 2; ++i) {
          const float p0 = 2 * i < limit ? ex2(fmaf(__uint_as_float(s[2 * i]), c, nl2)) : 0.f;
          const float p1 = 2 * i + 1 < limit ? ex2(fmaf(__uint_as_float(s[2 * i + 1]), c, nl2)) : 0.f;
          ds[i] = pack_bf16(p0 * (__uint_as_float(dp[2 * i]) - Dt), p1 * (__uint_as_float(dp[2 * i + 1]) - Dt));
          rsum += __uint_as_float(ds[i] << 16) + __uint_as_float(ds[i] & 0xffff0000u);
        }
        tmem_st8(S_addr, ds);
        tmem_wait_st();
        tc_fence_before_sync();
      }
      mbar_arrive(smem_u32(&bars.p_full[0]));
    }
    for (int j = sh; j < n; ++j) {
      if ((j & 15) == 15 && !__all_sync(0xffffffffu, ok)) break;
      const int b = j & (NB - 1);
      ok &= mbar_wait_lanes(smem_u32(&bars.s_full[b]), (j >> (NB - 1)) & 1, abort);
      tc_fence_after_sync();
      const uint32_t S_addr = tmem + lane_addr + Cfg::kColBuf + b * 128 + half * 32;
      uint32_t s[32], dp[32];
      tmem_ld32(S_addr, s);
      tmem_ld32(S_addr + Cfg::kColP, dp);
      tmem_wait_ld();
      const int limit = (j < n_ct ? list_end - j * kKeys : qpos - (rb.dense_start + (j - n_ct) * kKeys) + 1) - half * 32;
      if (limit < 32) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i >= limit) s[i] = 0xff800000u;
      }
      uint32_t ds[16];
      float r0, r1;
      {
        // packed fp32 pairs: one issue slot for two elements of the scale-and-shift, of dP - D, of the
        // product and of the row sum of the rounded dS
        const uint64_t c2 = f2_pack(c, c), nl22 = f2_pack(nl2, nl2), nD2 = f2_pack(-Dt, -Dt);
        uint64_t r2 = f2_pack(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          float x0, x1, d0, d1;
          f2_unpack(f2_fma(f2_pack(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), c2, nl22), x0, x1);
          const float p0 = ex2(x0), p1 = ex2(x1);
          const uint64_t g2 = f2_add(f2_pack(__uint_as_float(dp[2 * i]), __uint_as_float(dp[2 * i + 1])), nD2);
          f2_unpack(f2_mul(f2_pack(p0, p1), g2), d0, d1);
          ds[i] = pack_bf16(d0, d1);
          r2 = f2_add(r2, f2_pack(__uint_as_float(ds[i] << 16), __uint_as_float(ds[i] & 0xffff0000u)));
        }
        f2_unpack(r2, r0, r1);
      }
      rsum += r0 + r1;
      tmem_st16(S_addr, ds);   // over the first half of this warpgroup's own S columns
      tmem_wait_st();
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&bars.p_full[b]));
    }
    red_s[half][row] = rsum;
    asm volatile("bar.sync 1, 256;" ::: "memory");   // the eight softmax warps, whether or not a wait gave up
    ok = __all_sync(0xffffffffu, ok);
    if (ok) ok = mbar_wait_warp(smem_u32(&bars.acc_done), 0, abort);
    // The dQ rows go through shared memory (the Q and dO tiles are idle since their copy into tensor
    // memory), so that a warp writes whole half rows: per-thread 16-byte stores to rows 256 bytes apart cost
    // a transaction each.  Rows are padded by 16 bytes so that a warp's stores spread over the banks.
    // (With a bulk copy per row a CTA waits for the copies to have read them before it may end.)
    constexpr int kRowBytes = D * 2, kStageStride = kRowBytes + 16;
    unsigned char* stage_out = smem_raw + (sQ - smem_u32(smem_raw));
    if (ok) {
      tc_fence_after_sync();
      const float r = red_s[0][row] + red_s[1][row];
      constexpr int CH = D / 2;   // output columns of this warpgroup
      const uint32_t A_addr = tmem + lane_addr + Cfg::kColA + half * CH;
      const float* kb = a.kbar + (size_t)bh_kv * D + half * CH;
      unsigned char* srow = stage_out + row * kStageStride + half * (kRowBytes / 2);
#pragma unroll
      for (int q = 0; q < CH / 32; ++q) {
        uint32_t o[32];
        tmem_ld32(A_addr + q * 32, o);
        tmem_wait_ld();
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          float f[8];
#pragma unroll
          for (int e = 0; e < 8; ++e)
            f[e] = fmaf(-r, kb[q * 32 + 8 * v + e], __uint_as_float(o[8 * v + e])) * a.scale;
          uint4 w;
          w.x = pack_bf16(f[0], f[1]); w.y = pack_bf16(f[2], f[3]);
          w.z = pack_bf16(f[4], f[5]); w.w = pack_bf16(f[6], f[7]);
          *reinterpret_cast<uint4*>(srow + (q * 4 + v) * 16) = w;
        }
      }
      __syncwarp();
      if (!*abort) {
        const int q = rb.q0 + quad * 32;   // the warp's first row
        store_rows<D>(stage_out + quad * 32 * kStageStride + half * D, kStageStride,
                      reinterpret_cast<unsigned char*>(a.dQ + (row0 + q) * D) + half * D, kRowBytes, rb.q_end - q, lane);
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, Cfg::kCols);
  if (tid == 0 && abort_s) atomicExch(a.status, (int)LRSA_ERR_TIMEOUT);
}

}  // namespace

template <int D, int NSEQ, int NB>
static int launch_dq_t(const Geom& whole, const SeqBatch& b, const BwdPtrs& p, cudaStream_t st) {
  using Cfg = DqCfg<D, NB>;
  DqMaps<NSEQ> m;
  DqArgs<NSEQ> a;
  const long long BHq = (long long)whole.B * whole.Hq, BHkv = (long long)whole.B * whole.Hkv;
  a.block0[0] = 0;
  for (int s = 0; s < b.n; ++s) {
    const Geom& g = b.g[s];
    const long long rc = g.Rc > 0 ? g.Rc : 1;
    // the sequence starts at token tok0 of rows of Nrow tokens: shifted bases, rows beyond its end read as zero
    const size_t sh = (size_t)g.tok0 * D, csh = g.Rc > 0 ? (size_t)b.row0[s] * D : 0;
    int r = make_tmap_bf16(&m.q[s], p.Q + sh, D, g.N, BHq, kTile, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.dO[s], p.dO + sh, D, g.N, BHq, kTile, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.k[s], p.K + sh, D, g.N, BHkv, kKeys, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.v[s], p.V + sh, D, g.N, BHkv, kKeys, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.kc[s], p.Kc + csh, D, rc, BHkv, kKeys);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.vc[s], p.Vc + csh, D, rc, BHkv, kKeys);
    if (r != LRSA_OK) return r;
    a.plan[s] = make_plan(g, kTile);
    a.tok0[s] = g.tok0;
    a.block0[s + 1] = a.block0[s] + a.plan[s].total;
  }
  a.n_seqs = b.n;
  a.BH = (int)BHq; a.Hq = whole.Hq; a.Hkv = whole.Hkv; a.G = whole.G; a.N = whole.Nrow;
  a.stats = p.stats; a.Dacc = p.Dacc; a.kbar = p.kbar; a.dQ = p.dQ;
  a.scale = whole.scale; a.scale_log2 = whole.scale * 1.4426950408889634f;
  a.status = p.status;
  const long long grid = (long long)a.block0[b.n] * a.BH;
  if (grid > 0x7fffffffLL) return LRSA_ERR_UNSUPPORTED;
  auto kern = lrsa_bwd_dq_kernel<D, NSEQ, NB>;
  LRSA_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmem));
  LRSA_CUDA_CHECK(launch_dependent(kern, dim3((unsigned)grid), dim3(Cfg::kThreads), Cfg::kSmem, st, 1, m, a));
  launch_counter().n++;
  return LRSA_OK;
}

int launch_bwd_dq_sm100(const Geom& whole, const SeqBatch& b, const BwdPtrs& p, cudaStream_t st) {
  // d = 64: one S/dP buffer per CTA and two CTAs per SM, which start and end at different times, once every SM has more than
  // two CTAs to run; otherwise two buffers, the shorter chain of a CTA alone.  Whole backward, us, with one | two buffers (windows of 512): 8/8
  // heads: 2K tokens (136 CTAs) 62.3 | 52.5, 3K (200) 65.7 | 60.2, 4K (264) 85.6 | 81.1, 5K (328) 100.8 | 100.7, 8K (520) 181.0 | 186.8,
  // 8 x 2000 221.5 | 229.6; 16/2 heads: 2K (272) 62.9 | 60.3, 3K (400) 91.6 | 93.4, 5K (656) 168.0 | 172.5.
  long long ctas = 0;
  for (int s = 0; s < b.n; ++s) ctas += (long long)make_plan(b.g[s], kTile).total * whole.B * whole.Hq;
  const auto dq = whole.d == 128   ? (b.n == 1 ? launch_dq_t<128, 1, 2> : launch_dq_t<128, kMaxSeqs, 2>)
                  : ctas > 2 * kSms ? (b.n == 1 ? launch_dq_t<64, 1, 1> : launch_dq_t<64, kMaxSeqs, 1>)
                                   : (b.n == 1 ? launch_dq_t<64, 1, 2> : launch_dq_t<64, kMaxSeqs, 2>);
  return dq(whole, b, p, st);
}

}  // namespace lrsa
