// LRSA attention forward on tcgen05 tensor cores (Section 3.1 Eq. 3 under the chunked mask of
// Section 3.2).
//
// A CTA owns one or two 128-row query tiles of one (batch, query head) and one query chunk, which share a key list, and
// walks the list (first n_front rows of the compact sinks+kept buffer, then a contiguous range of original positions up to
// the diagonal) in 128-key tiles.  Two tiles (TQ = 2, one CTA per SM): every K_j / V_j tile in shared memory serves both.
// One tile (TQ = 1, two CTAs per SM): small grids and short lists, see one_tile().  The list's last tile often holds only as
// many keys as there are sinks: with at most 16 it comes first, and its products and exponentials are 16 wide (1777 tokens
// 45.8 -> 43.1 us, 4K 92.6 -> 88.0, 32K in eight sequences 870 -> 842, with few sinks and 28 heads).  Roles:
//   warp 0      TMA producer: the Q tiles once, then K_j, V_j tiles through a ring of shared-memory slots
//   warp 1      issues all products, per key tile and query tile  O_t += P_t V_j (P_t from tensor memory), then
//               S_t = Q_t K_{j+1}^T (both operands in shared memory); owns the TMEM allocation
//   warps 4-7   softmax of query tile 0, warps 8-11 of query tile 1 (TQ = 2): one thread per row, S from TMEM, online
//               softmax in fp32 with the maximum only raised when it grew by more than 2^8 (then O_t is
//               rescaled in TMEM), P written back over S as packed bf16
// The two tiles take turns on the tensor core: while one tile's scores are in its softmax warpgroup the
// products of the other run.  A row belongs to one thread from its scores to its output, so the softmax
// threads exchange nothing, and its 128 scores are held in registers at once (setmaxnreg: 216 for these threads).
// What bounds it: the chain of a tile from S_t over its exponentials (one MUFU result per two clocks and thread, 1024
// cycles a tile) to O_t and the next S_t, and the 1000 W power limit, under which the clock settles near 1.65 GHz.
// At 32K tokens, 28/4 heads, d = 128, one kept token in four: 1.97 ms alone and uncapped (1.50 at the measured bf16 rate;
// tensor pipe 63 % active); 2.14 ms under the power limit, 8.6 at 64K with its selection.  With an issuing warp for S and one for O += P V,
// a barrier round trip between a tile's products and P handed over in one piece it takes 2.75 and 9.5 ms.  Measured on the way
// (2.44 ms then) and not taken: sixteen softmax warps (16 rows x 128 columns each, 256-bit loads) 2.66; exponentials started with the
// previous maximum, the tile taken again when it was raised, 2.47; a share of them on the FMA pipe, no gain at 1/8, 2.63 at 1/4.
// All mbarrier waits are bounded; on expiry the CTA records LRSA_ERR_TIMEOUT in the workspace header and leaves.
#include <algorithm>

#include "attn_common_sm100.h"

namespace lrsa {
namespace {

using namespace ptx;

template <int D, int TQ>
struct FwdCfg {
  static constexpr int kSub = D / 64;                 // 64-column (128-byte) sub-tiles per tile
  static constexpr int kSubBytes = kTile * 128;       // 16 KB
  static constexpr int kTileBytes = kSub * kSubBytes; // one Q / K / V tile
  // A Q tile is followed by 2 KB so that the output rows of the tile can be staged there with 16 bytes of
  // padding per row (128 rows x (2D + 16) bytes = tile + 2 KB); the next tile stays 1024-byte aligned.
  static constexpr int kQRegion = kTileBytes + 2048;
  static constexpr int kPerSm = 3 - TQ;                          // resident CTAs
  static constexpr int kStages = D == 64 ? 5 : 4 / kPerSm;       // K/V ring slots
  static_assert(D == 128 || TQ == 1, "d = 64 runs with one tile per CTA");
  static constexpr int kSmem = TQ * kQRegion + kStages * kTileBytes + 1024;
  static constexpr int kThreads = 128 + 128 * TQ;
  // Loaded ahead of the block's barrier: Q, at d = 64 (half as many copies) also K_0 and V_0, with Q into L2 before that.  Every warp waits for the
  // thread that issues them.  us, Q only | all of them: d = 128, 28/4 heads: 32K tokens in eight sequences (kernel alone) 782 | 811, 1777 29.6 | 29.8,
  // 32K 2136 | 2155; 32/8, sixteen sequences of 2048 (kernel alone) 518 | 530; d = 64: 1777 tokens (8/8) 18.4 | 18.1, 4K 27.3 | 27.0, (16/2) 41.0 | 40.8.
  static constexpr bool kFirstTiles = D == 64;
  // TMEM columns: accumulator O of query tile t at 128t, its S (and, packed over it, P) behind the accumulators
  static constexpr uint32_t kColO = 0, kColS = TQ * 128, kCols = 2 * TQ * 128;
};

template <int NSEQ>
struct FwdMaps { CUtensorMap q[NSEQ], k[NSEQ], v[NSEQ], kc[NSEQ], vc[NSEQ]; };

template <int NSEQ>
struct FwdArgs {
  BlockPlan plan[NSEQ];    // blocks of up to 256 query rows (two tiles)
  int tok0[NSEQ];          // first token of the sequence
  int block0[NSEQ + 1];    // blocks of the sequences before, per (batch, head)
  int n_seqs;
  int BH, Hq, Hkv, G, N;   // N: tokens per (batch, head) row of O and LSE (the row stride)
  __nv_bfloat16* O;
  __nv_bfloat16* Olo;        // optional: receives bf16(O_fp32 - O), the part of the output the bf16 O cannot hold
  float* LSE;
  float scale, scale_log2;   // softmax scale, and scale * log2(e)
  int* status;
};

constexpr int kShort = 16;    // keys of a tile of the short form
constexpr int kPParts = 2;   // P_t is handed to the tensor core in two halves (64 keys each)

struct FwdBars {
  uint64_t q_full;
  uint64_t kv_full[5], kv_empty[5];
  uint64_t s_full[2], pv_done[2];   // per query tile
  uint64_t p_full[2][kPParts];      // per query tile: the parts of P_t (128 / kPParts keys each) are stored
};

template <int D, int NSEQ, int TQ>
__global__ void __launch_bounds__(FwdCfg<D, TQ>::kThreads, FwdCfg<D, TQ>::kPerSm)
lrsa_fwd_kernel(const __grid_constant__ FwdMaps<NSEQ> maps, const __grid_constant__ FwdArgs<NSEQ> a) {
  using Cfg = FwdCfg<D, TQ>;
  constexpr int NS = Cfg::kStages;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) FwdBars bars;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = smem0, sRing = smem0 + TQ * Cfg::kQRegion;

  const int bh = blockIdx.x % a.BH;
  int blk = blockIdx.x / a.BH, sq = 0;
  if constexpr (NSEQ > 1) {
    while (sq + 1 < a.n_seqs && blk >= a.block0[sq + 1]) ++sq;
    blk -= a.block0[sq];
  }
  const RowBlock rb = decode_block(a.plan[sq], blk);
  const int bh_kv = (bh / a.Hq) * a.Hkv + (bh % a.Hq) / a.G;
  const int n_ct = (rb.n_front + kTile - 1) / kTile;
  // key tiles of query tile t: the list, then the dense range up to the tile's last row (0: the tile is empty)
  const int n0 = n_ct + (min(rb.q_end, rb.q0 + kTile) - 1 - rb.dense_start) / kTile + 1;
  const int n1 = TQ == 2 && rb.q0 + kTile < rb.q_end ? n_ct + (rb.q_end - 1 - rb.dense_start) / kTile + 1 : 0;
  const int n = max(n0, n1);
  // the list's last tile comes first when it holds no more than kShort keys: its products and exponentials are that wide
  const int sh = n_ct > 0 && rb.n_front - (n_ct - 1) * kTile <= kShort ? 1 : 0;

  // K or V tile `it` of the order K_0, V_0, K_1, ... into its ring slot
  auto load_tile = [&](int it) {
    const int j = it >> 1, which = it & 1, slot = it % NS;
    const uint32_t full = smem_u32(&bars.kv_full[slot]);
    mbar_expect_tx(full, Cfg::kTileBytes);
    const bool compact = j < n_ct;
    const CUtensorMap* map = compact ? (which ? &maps.vc[sq] : &maps.kc[sq]) : (which ? &maps.v[sq] : &maps.k[sq]);
    const int row = compact ? (j < sh ? n_ct - 1 : j - sh) * kTile : rb.dense_start + (j - n_ct) * kTile;
    for (int h = 0; h < Cfg::kSub; ++h)
      tma_load_3d(sRing + slot * Cfg::kTileBytes + h * Cfg::kSubBytes, map, h * 64, row, bh_kv, full);
  };
  if (tid == 0) {
    prefetch_tensormap(&maps.q[sq]); prefetch_tensormap(&maps.k[sq]); prefetch_tensormap(&maps.v[sq]);
    prefetch_tensormap(&maps.kc[sq]); prefetch_tensormap(&maps.vc[sq]);
    abort_s = 0;
    mbar_init(smem_u32(&bars.q_full), 1);
    for (int i = 0; i < NS; ++i) { mbar_init(smem_u32(&bars.kv_full[i]), 1); mbar_init(smem_u32(&bars.kv_empty[i]), 1); }
    for (int t = 0; t < 2; ++t) {
      mbar_init(smem_u32(&bars.s_full[t]), 1);
      for (int i = 0; i < kPParts; ++i) mbar_init(smem_u32(&bars.p_full[t][i]), 4);   // one arrival per softmax warp
      mbar_init(smem_u32(&bars.pv_done[t]), 1);
    }
    fence_barrier_init();
    // the first loads, while the other warps get their tensor memory
    if constexpr (Cfg::kFirstTiles) tma_prefetch_3d(&maps.q[sq], 0, rb.q0, bh);   // while the kernel in front ends
    asm volatile("griddepcontrol.wait;" ::: "memory");   // started before the kernel in front of it has ended
    mbar_expect_tx(smem_u32(&bars.q_full), (n1 > 0 ? 2 : 1) * Cfg::kTileBytes);
    for (int t = 0; t < (n1 > 0 ? 2 : 1); ++t)
      for (int h = 0; h < Cfg::kSub; ++h)
        tma_load_3d(sQ + t * Cfg::kQRegion + h * Cfg::kSubBytes, &maps.q[sq], h * 64, rb.q0 + t * kTile, bh, smem_u32(&bars.q_full));
    if constexpr (Cfg::kFirstTiles) { load_tile(0); load_tile(1); }
  }
  if (warp == 1) { tmem_alloc(smem_u32(&tmem_base_s), Cfg::kCols); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_s;
  volatile int* abort = &abort_s;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // The softmax threads hold a row of 128 scores: they take the registers the other warps do not need
  // (128 x 72 + 256 x 216 = 384 x 168, 128 x 48 + 128 x 208 = 256 x 128: what the CTA was launched with).
  if (warp < 4) {
    if constexpr (TQ == 2) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      int it = Cfg::kFirstTiles ? 2 : 0;
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
    // ---------------- issuer: per key tile j and query tile t  O_t += P_t V_j, then S_t = Q_t K_{j+1}^T ----------------
    // One thread issues everything, and the tensor core runs its products in this order (sm100_ptx.h): S_t of the next
    // key tile may overwrite P_t without waiting for the product that reads it.
    constexpr uint32_t idesc_qk = make_idesc_bf16(kTile, kTile, 0, 0);
    constexpr uint32_t idesc_pv = make_idesc_bf16(kTile, D, 0, 1);
    const uint64_t descK0 = make_smem_desc_sw128(sRing, 16, 1024);
    const uint64_t descV0 = make_smem_desc_sw128(sRing, Cfg::kSubBytes, 1024);   // V_j MN-major
    const uint64_t descQ0 = make_smem_desc_sw128(sQ, 16, 1024);
    const uint32_t leader = elect_one();
    bool ok = mbar_wait_warp(smem_u32(&bars.q_full), 0, abort);
    int slot_v = 0, ph_v = 0, slot_k = 0, ph_k = 0;   // ring order: K_0, V_0, K_1, V_1, ...
    auto next = [](int& slot, int& ph) { if (++slot == NS) { slot = 0; ph ^= 1; } };
    auto scores = [&](int t, uint64_t dK, uint32_t idesc) {
      const uint64_t dQ = desc_advance(descQ0, t * Cfg::kQRegion);
#pragma unroll
      for (int h = 0; h < Cfg::kSub; ++h)
        umma_ss4(tmem + Cfg::kColS + t * kTile, desc_advance(dQ, h * Cfg::kSubBytes), desc_advance(dK, h * Cfg::kSubBytes),
                 idesc, h > 0 ? 1u : 0u, leader);
      umma_commit(smem_u32(&bars.s_full[t]), leader);
    };
    if (sh) {
      // the short tile (key tile 0), apart from the loop: with the choices inside it the two-tile form takes 253 instead of
      // 244 us at 8K tokens (28 heads, d = 128)
      constexpr uint32_t idesc_short = make_idesc_bf16(kTile, kShort, 0, 0);
      if (ok) ok = mbar_wait_warp(smem_u32(&bars.kv_full[0]), 0, abort);
      if (ok) {
        tc_fence_after_sync();
        scores(0, descK0, idesc_short);
        if (n1 > 0) scores(1, descK0, idesc_short);
        umma_commit(smem_u32(&bars.kv_empty[0]), leader);
      }
      next(slot_v, ph_v);                                   // V_0
      next(slot_k, ph_k); next(slot_k, ph_k);               // K_1 (there is one: the dense range is never empty)
      if (ok) ok = mbar_wait_warp(smem_u32(&bars.kv_full[slot_v]), ph_v, abort);
      for (int t = 0; t < TQ && ok; ++t) {
        if (t == 1 && n1 == 0) break;
        for (int part = 0; part < kPParts; ++part)
          if (ok) ok = mbar_wait_warp(smem_u32(&bars.p_full[t][part]), 0, abort);
        if (!ok) break;
        tc_fence_after_sync();
        umma_ts1(tmem + Cfg::kColO + t * kTile, tmem + Cfg::kColS + t * kTile, desc_advance(descV0, slot_v * Cfg::kTileBytes),
                  idesc_pv, 0u, leader);
        umma_commit(smem_u32(&bars.pv_done[t]), leader);
        if (t == 0) ok = mbar_wait_warp(smem_u32(&bars.kv_full[slot_k]), ph_k, abort);
        if (!ok) break;
        tc_fence_after_sync();
        scores(t, desc_advance(descK0, slot_k * Cfg::kTileBytes), idesc_qk);
      }
      if (ok) {
        umma_commit(smem_u32(&bars.kv_empty[slot_v]), leader);
        umma_commit(smem_u32(&bars.kv_empty[slot_k]), leader);
      }
      next(slot_v, ph_v); next(slot_v, ph_v);
      next(slot_k, ph_k); next(slot_k, ph_k);
    }
    for (int j = sh ? 1 : -1; j < n && ok; ++j) {
      uint64_t dV = 0, dK = 0;
      if (j >= 0) {
        ok = mbar_wait_warp(smem_u32(&bars.kv_full[slot_v]), ph_v, abort);
        if (!ok) break;
        dV = desc_advance(descV0, slot_v * Cfg::kTileBytes);
      }
      bool k_here = false;
      for (int t = 0; t < TQ && ok; ++t) {
        const int nt = t == 0 ? n0 : n1;
        if (j >= 0 && j < nt) {
          // packed P_t: keys [16k, 16k+16) in columns [8k, 8k+8) of the tile's S region
#pragma unroll
          for (int part = 0; part < kPParts; ++part) {
            if (ok) ok = mbar_wait_warp(smem_u32(&bars.p_full[t][part]), j & 1, abort);
            if (!ok) break;
            tc_fence_after_sync();
            umma_ts4<8, 16, 24, 2048>(tmem + Cfg::kColO + t * kTile, tmem + Cfg::kColS + t * kTile + part * 32,
                                     desc_advance(dV, part * 4 * 2048), idesc_pv, (part > 0 || j > 0) ? 1u : 0u, leader);
          }
          if (!ok) break;
          umma_commit(smem_u32(&bars.pv_done[t]), leader);     // phase j: O_t holds key tiles 0..j
          if (TQ == 1) umma_commit(smem_u32(&bars.kv_empty[slot_v]), leader);
        }
        if (j + 1 < nt) {
          if (!k_here) {
            ok = mbar_wait_warp(smem_u32(&bars.kv_full[slot_k]), ph_k, abort);
            if (!ok) break;
            dK = desc_advance(descK0, slot_k * Cfg::kTileBytes);
            k_here = true;
          }
          tc_fence_after_sync();
          scores(t, dK, idesc_qk);
        }
      }
      if (!ok) break;
      if (TQ == 2 && j >= 0) umma_commit(smem_u32(&bars.kv_empty[slot_v]), leader);
      if (j + 1 < n) umma_commit(smem_u32(&bars.kv_empty[slot_k]), leader);
      next(slot_v, ph_v);
      if (j >= 0) next(slot_v, ph_v);
      next(slot_k, ph_k);
      next(slot_k, ph_k);
    }
  }
  } else {
    if constexpr (TQ == 2) asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    else asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    // ---------------- softmax + epilogue: warpgroup t owns query tile t, one thread per row ----------------
    const int t = (warp - 4) >> 2, quad = warp & 3;
    const int row = quad * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t S_addr = tmem + lane_addr + Cfg::kColS + t * kTile;
    const uint32_t O_addr = tmem + lane_addr + Cfg::kColO + t * kTile;
    const int nt = t == 0 ? n0 : n1;
    // keys of tile j this row may see: the first list_end - 128 j of a list tile, dense_end - 128 j of a dense one
    const int list_end = rb.n_front + sh * kTile, dense_end = rb.q0 + t * kTile + row + 1 - rb.dense_start + n_ct * kTile;
    const float c = a.scale_log2;
    float m = 0.f, l = 0.f;
    bool ok = true;
    if (sh && nt > 0) {
      ok = mbar_wait_warp(smem_u32(&bars.s_full[t]), 0, abort);
      if (ok) {
        tc_fence_after_sync();
        const int limit = rb.n_front - (n_ct - 1) * kTile;
        uint32_t s[32], pk[kShort / 2];   // only the first kShort columns hold scores
        tmem_ld32(S_addr, s);
        tmem_wait_ld();
        m = __uint_as_float(s[0]);
#pragma unroll
        for (int i = 1; i < kShort; ++i) {
          if (i >= limit) s[i] = 0xff800000u;
          m = fmaxf(m, __uint_as_float(s[i]));
        }
        if (m == -INFINITY) m = 0.f;   // no key of the tile counts: P = 0, as in the full tiles below
#pragma unroll
        for (int i = 0; i < kShort / 2; ++i) {
          const float p0 = ex2(fmaf(__uint_as_float(s[2 * i]), c, -m * c)), p1 = ex2(fmaf(__uint_as_float(s[2 * i + 1]), c, -m * c));
          l += p0 + p1;
          pk[i] = pack_bf16(p0, p1);
        }
        tmem_st8(S_addr, pk);
        tmem_wait_st();
        tc_fence_before_sync();
        __syncwarp();
        if (lane < kPParts) mbar_arrive(smem_u32(&bars.p_full[t][lane]));
      }
    }
    for (int j = sh; j < nt && ok; ++j) {
      ok = mbar_wait_warp(smem_u32(&bars.s_full[t]), j & 1, abort);
      if (!ok) break;
      tc_fence_after_sync();
      const int limit = (j < n_ct ? list_end : dense_end) - j * kTile;
      // the row's 128 scores and their maximum
      uint32_t s[kTile];
#pragma unroll
      for (int h = 0; h < 4; ++h) tmem_ld32(S_addr + h * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[h * 32]));
      tmem_wait_ld();
      if (limit < kTile) {
#pragma unroll
        for (int i = 0; i < kTile; ++i)
          if (i >= limit) s[i] = 0xff800000u;  // -inf
      }
      float mx4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) mx4[e] = __uint_as_float(s[e]);
#pragma unroll
      for (int i = 4; i + 8 <= kTile; i += 8)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          mx4[e] = fmaxf(fmaxf(mx4[e], __uint_as_float(s[i + e])), __uint_as_float(s[i + 4 + e]));
#pragma unroll
      for (int e = 0; e < 4; ++e) mx4[e] = fmaxf(mx4[e], __uint_as_float(s[kTile - 4 + e]));
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      if (j == 0) {
        m = mx == -INFINITY ? 0.f : mx;
      } else {
        // the maximum is only raised when it grew by more than 2^8 (then O is rescaled in tensor memory)
        const bool need = (mx - m) * c > 8.f;
        if (__any_sync(0xffffffffu, need)) {
          // O must hold every earlier tile before it is rescaled; the O issuer cannot start tile j before
          // this thread has arrived on p_full, so the rescale cannot race with it
          ok = mbar_wait_warp(smem_u32(&bars.pv_done[t]), (j - 1) & 1, abort);
          if (!ok) break;
          tc_fence_after_sync();
          const float f = need ? ex2((m - mx) * c) : 1.f;
#pragma unroll
          for (int q = 0; q < D / 32; ++q) {
            uint32_t o[32];
            tmem_ld32(O_addr + q * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
            tmem_st32(O_addr + q * 32, o);
          }
          tmem_wait_st();
          l *= f;
          if (need) m = mx;
        }
      }
      const float nmc = -m * c;
      const uint64_t c2 = f2_pack(c, c), nmc2 = f2_pack(nmc, nmc);
      uint64_t sum2 = f2_pack(0.f, 0.f);
      // exponentials: scale and shift as packed pairs (one issue slot for two elements).  P as packed bf16 over the
      // first 64 columns of the tile's S (this thread's own lane: nobody else reads it), in two halves: the tensor core
      // starts O_t += P_t V_j on the first while the second is formed (in four parts, with twice the waits for
      // stores: 2.86 ms instead of 2.51 at the sizes of the file's head).  The steps are written a few elements ahead of
      // the ones that take their results and kept in that order: one warp per scheduler is in this phase at a time, and
      // nothing else hides the latencies (2.51 -> 2.44 ms).
      constexpr int kPairs = kTile / 2 / kPParts, kLag = 4;
      uint64_t sum2b = f2_pack(0.f, 0.f);
      uint32_t pk[kPairs];
#pragma unroll
      for (int part = 0; part < kPParts; ++part) {
#pragma unroll
        for (int ii = 0; ii < kPairs + kLag; ++ii) {
          if (ii < kPairs) {
            const int i = part * kPairs + ii;
            float x0, x1;
            f2_unpack(f2_fma(f2_pack(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), c2, nmc2), x0, x1);
            s[2 * i] = __float_as_uint(ex2_ordered(x0));
            s[2 * i + 1] = __float_as_uint(ex2_ordered(x1));
          }
          if (ii >= kLag) {
            const int i = part * kPairs + ii - kLag;
            const float p0 = __uint_as_float(s[2 * i]), p1 = __uint_as_float(s[2 * i + 1]);
            if (i & 1) sum2 = f2_add(sum2, f2_pack(p0, p1)); else sum2b = f2_add(sum2b, f2_pack(p0, p1));
            pk[ii - kLag] = pack_bf16(p0, p1);
          }
        }
        tmem_st32(S_addr + part * kPairs, pk);
        tmem_wait_st();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.p_full[t][part]));
      }
      sum2 = f2_add(sum2, sum2b);
      float sum0, sum1;
      f2_unpack(sum2, sum0, sum1);
      l += sum0 + sum1;
    }
    // The output rows go through shared memory (the tile's Q region, idle once its last S product is done,
    // which pv_done implies), so that a warp writes whole rows: per-thread 16-byte stores to rows 256 bytes
    // apart cost a transaction each.  Rows are padded by 16 bytes so that a warp's stores spread over the banks.
    // (With a bulk copy per row a CTA waits for the copies to have read them before it may end: 1777 tokens, 28 heads, 31.0 -> 30.5 us, and
    // 30.2 with the first loads ahead of tensor memory.)
    constexpr int kRowBytes = D * 2, kStageStride = kRowBytes + 16;
    static_assert(kTile * kStageStride <= Cfg::kQRegion, "staging fits the Q region");
    if (ok && nt > 0) {
      // (where the rows lie is formed here again, from the thread and block numbers: kept through the loop it costs registers
      // that the scores need)
      int blk = blockIdx.x, thread = threadIdx.x;
      asm volatile("" : "+r"(blk), "+r"(thread));
      const int bh = blk % a.BH, w = thread >> 5, t = (w - 4) >> 2, row0_w = (w & 3) * 32, lane = thread & 31;   // row0_w: the warp's first row
      blk /= a.BH;
      int sq = 0;
      if constexpr (NSEQ > 1) {
        while (sq + 1 < a.n_seqs && blk >= a.block0[sq + 1]) ++sq;
        blk -= a.block0[sq];
      }
      const RowBlock rb = decode_block(a.plan[sq], blk);
      const int q = rb.q0 + t * kTile + row0_w, left = rb.q_end - q;   // first query of the warp, rows from there on
      const size_t row0 = (size_t)bh * a.N + a.tok0[sq] + q;           // its row of O and LSE
      unsigned char* stage = smem_raw + (smem0 - smem_u32(smem_raw)) + t * Cfg::kQRegion + row0_w * kStageStride;
      if (mbar_wait_warp(smem_u32(&bars.pv_done[t]), (nt - 1) & 1, abort)) {
        tc_fence_after_sync();
        const float inv = 1.0f / l;
        unsigned char* srow = stage + lane * kStageStride;
        // the remainder goes straight to global memory (contiguous bytes per thread, written once)
        __nv_bfloat16* lo_row = a.Olo && lane < left ? a.Olo + (row0 + lane) * D : nullptr;
#pragma unroll
        for (int q = 0; q < D / 32; ++q) {
          uint32_t o[32];
          tmem_ld32(O_addr + q * 32, o);
          tmem_wait_ld();
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(o[8 * v + e]) * inv;
            uint4 w;
            w.x = pack_bf16(f[0], f[1]); w.y = pack_bf16(f[2], f[3]);
            w.z = pack_bf16(f[4], f[5]); w.w = pack_bf16(f[6], f[7]);
            *reinterpret_cast<uint4*>(srow + (q * 4 + v) * 16) = w;
            if (lo_row) {
              const uint32_t hw[4] = {w.x, w.y, w.z, w.w};
              uint32_t lw[4];
#pragma unroll
              for (int e = 0; e < 4; ++e)
                lw[e] = pack_bf16(f[2 * e] - __uint_as_float(hw[e] << 16), f[2 * e + 1] - __uint_as_float(hw[e] & 0xffff0000u));
              *reinterpret_cast<uint4*>(lo_row + q * 32 + v * 8) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
            }
          }
        }
        if (lane < left) a.LSE[row0 + lane] = m * a.scale + logf(l);
        __syncwarp();
        if (!*abort) store_rows<kRowBytes>(stage, kStageStride, reinterpret_cast<unsigned char*>(a.O + row0 * D), kRowBytes, left, lane);
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, Cfg::kCols);
  if (tid == 0 && abort_s) atomicExch(a.status, (int)LRSA_ERR_TIMEOUT);
}

__global__ void __launch_bounds__(256) compact_kv_kernel(const __grid_constant__ CompactArgs c) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (c.status && blockIdx.x == 0 && threadIdx.x == 0) *c.status = 0;
  compact_rows(c, blockIdx.x);
}

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                             const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                             CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) p = nullptr;
    return reinterpret_cast<EncodeFn>(p);
  }();
  return fn;
}

struct FwdWs {
  size_t kc, vc, total;
};
FwdWs fwd_ws_layout(const Geom& g, long long rows) {
  FwdWs w;
  const size_t bytes = align_up((size_t)g.B * g.Hkv * rows * g.d * sizeof(__nv_bfloat16), 1024);
  w.kc = 1024;
  w.vc = w.kc + bytes;
  w.total = w.vc + bytes;
  return w;
}

}  // namespace

int make_tmap_bf16(CUtensorMap* map, const void* base, int d, long long rows, long long outer, int box_rows,
                   long long row_stride) {
  EncodeFn fn = encode_fn();
  if (!fn) return LRSA_ERR_CUDA;
  if (row_stride <= 0) row_stride = rows;
  cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)outer};
  cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)d * 2 * (cuuint64_t)row_stride};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? LRSA_OK : LRSA_ERR_CUDA;
}

int make_tmap_bf16_rows(CUtensorMap* map, const void* base, int d, long long rows) {
  EncodeFn fn = encode_fn();
  if (!fn) return LRSA_ERR_CUDA;
  cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  cuuint32_t box[2] = {64, 1};
  cuuint32_t es[2] = {1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? LRSA_OK : LRSA_ERR_CUDA;
}

size_t attn_fwd_ws_bytes(const Geom& g) { return fwd_ws_layout(g, compact_rows_used(g)).total; }
size_t attn_fwd_ws_bound(const Geom& g) { return fwd_ws_layout(g, compact_rows_bound(g)).total; }

template <int D, int NSEQ, int TQ>
static int launch_fwd_t(const Geom& whole, const SeqBatch& b, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                        const __nv_bfloat16* V, const __nv_bfloat16* Kc, const __nv_bfloat16* Vc, __nv_bfloat16* O,
                        __nv_bfloat16* Olo, float* LSE, int* status, cudaStream_t st) {
  using Cfg = FwdCfg<D, TQ>;
  FwdMaps<NSEQ> m;
  FwdArgs<NSEQ> a;
  const long long BHq = (long long)whole.B * whole.Hq, BHkv = (long long)whole.B * whole.Hkv;
  a.block0[0] = 0;
  for (int s = 0; s < b.n; ++s) {
    const Geom& g = b.g[s];
    const long long rc = g.Rc > 0 ? g.Rc : 1;
    // the sequence starts at token tok0 of rows of Nrow tokens: shifted bases, rows beyond its end read as zero
    const size_t sh = (size_t)g.tok0 * D, csh = g.Rc > 0 ? (size_t)b.row0[s] * D : 0;
    int r = make_tmap_bf16(&m.q[s], Q + sh, D, g.N, BHq, kTile, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.k[s], K + sh, D, g.N, BHkv, kTile, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.v[s], V + sh, D, g.N, BHkv, kTile, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.kc[s], Kc + csh, D, rc, BHkv, kTile);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.vc[s], Vc + csh, D, rc, BHkv, kTile);
    if (r != LRSA_OK) return r;
    a.plan[s] = make_plan(g, TQ * kTile);
    a.tok0[s] = g.tok0;
    a.block0[s + 1] = a.block0[s] + a.plan[s].total;
  }
  a.n_seqs = b.n;
  a.BH = (int)BHq; a.Hq = whole.Hq; a.Hkv = whole.Hkv; a.G = whole.G; a.N = whole.Nrow;
  a.O = O; a.Olo = Olo; a.LSE = LSE; a.scale = whole.scale; a.scale_log2 = whole.scale * 1.4426950408889634f;
  a.status = status;
  const long long grid = (long long)a.block0[b.n] * a.BH;
  if (grid > 0x7fffffffLL) return LRSA_ERR_UNSUPPORTED;
  auto kern = lrsa_fwd_kernel<D, NSEQ, TQ>;
  LRSA_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmem));
  LRSA_CUDA_CHECK(launch_dependent(kern, dim3((unsigned)grid), dim3(Cfg::kThreads), Cfg::kSmem, st, 1, m, a));
  launch_counter().n++;
  return LRSA_OK;
}

// One query tile per CTA and two CTAs per SM, or two tiles that share the K/V tiles in one CTA (d = 128)?  Two CTAs start and
// end at different times and split a small grid more finely, but load K and V twice.  28 heads, us with one | two tiles:
// few CTAs (windows of 512): 1777 tokens 29.9 | 31.8, 3K 53.6 | 56.7, 4K 77.3 | 76.4, 5K 107.0 | 103.7, 6K 138 | 136, 8K 214 | 205, of 1024
// 265 | 251, 32K of 1024 2329 | 2190; short lists: 16 x 600 tokens (of 256) 100 | 128, 8 x 1300 149 | 158, 8 x 1777 207 | 204, 4 x 3000 (8 tiles) 209 | 206.
// d = 64 (always one tile): 4K 37.1 | 41.1, 16K 166 | 178, 64K 1904 | 2084: its K/V tiles cost half as much to load.
static bool one_tile(const Geom& whole, const SeqBatch& b) {
  long long ctas = 0, keys = 0, tokens = 0;
  for (int s = 0; s < b.n; ++s) {
    const Geom& g = b.g[s];
    ctas += (long long)make_plan(g, 2 * kTile).total * whole.B * whole.Hq;
    // about the mean number of keys of a query: half of the history's kept tokens, the dense windows
    const long long hist = g.C > 1 + g.ndp ? (long long)(g.C - 1 - g.ndp) * g.K / 2 : 0;
    const long long dense = std::min<long long>(g.N / 2, g.L * g.ndp + g.L / 2);
    keys += g.N * (g.S + hist + dense);
    tokens += g.N;
  }
  return ctas <= 4 * kSms || 2 * keys <= 15 * kTile * tokens;   // 7.5 tiles
}

int launch_attn_fwd_sm100(const lrsa_params_t* params, const Geom& g, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                          const __nv_bfloat16* V, const int32_t* idx, __nv_bfloat16* O, float* LSE, void* ws,
                          cudaStream_t st) {
  const FwdWs lay = fwd_ws_layout(g, compact_rows_used(g));
  unsigned char* base = static_cast<unsigned char*>(ws);
  __nv_bfloat16* Kc = reinterpret_cast<__nv_bfloat16*>(base + lay.kc);
  __nv_bfloat16* Vc = reinterpret_cast<__nv_bfloat16*>(base + lay.vc);
  int* status = &reinterpret_cast<WsHeader*>(base)->status;
  __nv_bfloat16* Olo = static_cast<__nv_bfloat16*>(params->o_residual);
  SeqBatches batches(g);
  SeqBatch b;
  for (bool first = true; batches.next(&b); first = false) {
    const CompactArgs c = compact_args(g, b, K, V, idx, Kc, Vc, first ? status : nullptr);
    const int blocks = c.blocks();
    if (blocks > 0 || first) {
      LRSA_CUDA_CHECK(launch_dependent(compact_kv_kernel, dim3(blocks > 0 ? blocks : 1), dim3(256), 0, st, 1, c));
      launch_counter().n++;
    }
    const auto fwd = g.d == 64         ? (b.n == 1 ? launch_fwd_t<64, 1, 1> : launch_fwd_t<64, kMaxSeqs, 1>)
                     : one_tile(g, b) ? (b.n == 1 ? launch_fwd_t<128, 1, 1> : launch_fwd_t<128, kMaxSeqs, 1>)
                                      : (b.n == 1 ? launch_fwd_t<128, 1, 2> : launch_fwd_t<128, kMaxSeqs, 2>);
    const int rc = fwd(g, b, Q, K, V, Kc, Vc, O, Olo, LSE, status, st);
    if (rc != LRSA_OK) return rc;
  }
  return LRSA_OK;
}

}  // namespace lrsa
