// LRSA attention backward, dK / dV part, on tcgen05 tensor cores (key-outer).
//
// The keys of one (batch, KV head) are cut into 128-row tiles of two kinds:
//   compact tiles : 128 consecutive entries of the sinks + kept-positions list (the condensed KV cache
//                   of Section 3.2, gathered from K and V by position when the CTA starts); seen by
//                   every query of the chunks that see those windows compressed
//   dense tiles   : original positions of one window (or of the sink region / the tail); seen
//                   causally by the queries from the diagonal to the end of the last chunk that
//                   still sees that window uncompressed
// A CTA takes one tile and a segment of its (128-row query tile, query head of the group) list:
//   S^T  = K_j Q_i^T     (smem x smem -> TMEM, keys on lanes)     P^T  = exp2(S^T*c - LSE_i*log2e)
//   dP^T = V_j dO_i^T    (smem x smem -> TMEM)                    dS^T = P^T * (dP^T - D_i)
//   dV  += P^T dO_i      (TMEM x smem -> TMEM)
//   dK  += dS^T Q_i      (TMEM x smem -> TMEM)
// P^T and dS^T are written back over S^T and dP^T as packed bf16.  One warp issues all products, in the order
// dV(i), S^T(i+1), dK(i), dP^T(i+1): they run in that order, so single buffers for S^T and dP^T (all that tensor
// memory has left beside the two D-wide accumulators) suffice, and the exponentials of step i+1 run while dK(i) and
// dP^T(i+1) are computed, the rest of the softmax while dV and S^T are.  128 x 128 steps instead of 128 x 64 read
// K_j and V_j half as often from shared memory (the tensor core's operands, 192 KB a step, are what bounds the
// kernel together with the exponentials) and pay for half as many hand-offs.  At 32K tokens, 28/4 heads, d = 128, one kept
// token in four: 3.84 ms alone and uncapped, tensor pipe 74 % active (when it was 4.02: 128 x 64 steps 5.23; these with a branch around each
// product and the waits for Q and dO between two products: 4.58).  Warps: 0 TMA producer, 1 issuer, 3 row statistics, 4-19 softmax and
// epilogue.  A softmax warpgroup takes 32 query columns of every step: four warps per scheduler hide the latency
// of one another's exponentials and tensor-memory accesses (two warps with 64 columns each: 4.71 ms), and P^T is
// handed over in two halves so that dV starts on the first (in one piece: 4.90 ms).  The softmax warps also sum
// P^T * dP^T over the keys (through their own dP^T columns and a transposing load shape) and add it to a
// per-query-row accumulator: D_i = sum_j P_ij dP_ij, the accurate replacement of rowsum(dO * O) that the dQ kernel
// (which runs afterwards) needs.  The list of a tile runs from the last query tile backwards with the heads
// innermost, and compact tiles are launched segment by segment, so that the CTAs resident at one time
// read the same Q_i / dO_i tiles (L2 hits instead of one DRAM pass per key tile).  At the end
// the accumulators are added (fp32 atomics) to a zeroed workspace indexed by original position: a
// row of a compact tile goes to the position it was gathered from, so a kept key's compressed and
// uncompressed contributions meet in one row.  A small kernel then converts to bf16.
#include "attn_bwd_sm100.h"

namespace lrsa {
namespace {

using namespace ptx;

template <int D>
struct DkvCfg {
  static constexpr int kSub = D / 64;
  static constexpr int kSubBytes = kTile * 128;             // 128 rows x 128 bytes (kQRows == kTile)
  static constexpr int kTileBytes = kSub * kSubBytes;       // K_j, V_j, Q_i or dO_i
  // Q_i is used by S^T(i) and, a whole step later, by dK(i); dO_i by dP^T(i) and dV(i), which follow each other:
  // one slot more for Q_i keeps both prefetched by about a step.
  static constexpr int kStQ = D == 128 ? 3 : 4;
  static constexpr int kStO = D == 128 ? 2 : 3;
  // K_j, V_j, the two rings, then per-row statistics (two slots of 128 x (-LSE*log2e, D)) and the barriers.
  // At D = 128 this is all the shared memory a CTA can have, so nothing is static and nothing is padded.
  static constexpr int kOffRingQ = 2 * kTileBytes;
  static constexpr int kOffRingO = kOffRingQ + kStQ * kTileBytes;
  static constexpr int kOffStats = kOffRingO + kStO * kTileBytes;
  static constexpr int kOffCtl = kOffStats + 2 * 2 * kQRows * 4;
  static constexpr int kSmem = kOffCtl + 512;
  static constexpr int kSoftWarps = 16;  // four warpgroups, each 32 query columns of every step
  static constexpr int kThreads = 128 + 32 * kSoftWarps;   // TMA producer, MMA issuer, (idle), statistics; softmax
  static constexpr uint32_t kColS = 0, kColP = 128, kColK = 256, kColV = 256 + D;
};

template <int NSEQ>
struct DkvMaps { CUtensorMap q[NSEQ], dO[NSEQ], k[NSEQ], v[NSEQ], kg[NSEQ], vg[NSEQ]; };   // kg, vg: row gathers

template <int NSEQ>
struct DkvArgs {
  DkvPlan plan[NSEQ];
  int tok0[NSEQ];        // first token of the sequence
  int kept_off[NSEQ];    // its first entry of idx, per (batch, KV head)
  int map0[NSEQ];        // its part of seg_map
  int seg0[NSEQ + 1];    // (tile, segment) pairs of the sequences before
  int n_seqs;
  int BHkv, Hq, Hkv;
  const int32_t* idx;    // kept positions: head bh at idx + bh * kept_stride
  int kept_stride;       // Wtot * K entries per (batch, KV head)
  int Nrow;              // tokens per (batch, head) row (the stride of every tensor)
  const float* kpart;    // when not null: partial sums of the mean key (splits of them), to be finished
  int splits;
  float* kbar;
  const float2* stats;   // per query row: (-LSE * log2(e), D~ = rowsum(dO * O) from the bf16 O)
  float* Dacc;           // [B*Hq][N], zeroed: receives sum_j P_tj dP_tj, the accurate D for the dQ kernel
  const int2* seg_map;   // launch order: (tile, segment of the tile)
  float* dKf;   // [BHkv][N][D] fp32, zeroed
  float* dVf;
  float scale, scale_log2;
  int* status;
};

// Barriers and per-step words, behind the statistics in shared memory.
struct DkvCtl {
  uint64_t kv_full, acc_done;
  uint64_t q_full[4], q_empty[4], o_full[3], o_empty[3];
  uint64_t s_full[2];            // S^T of the step is in tensor memory and its statistics are staged (slot = step & 1)
  uint64_t dp_full;              // dP^T of the step is in tensor memory
  uint64_t p_full[2];            // halves of P^T: the first / last 16 query columns of every warpgroup
  uint64_t ds_full[2];           // dS^T of the step is stored (slot = step & 1; also frees the statistics slot)
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(DkvCtl) <= 512, "control block fits");

__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

template <int D, int NSEQ>
__global__ void __launch_bounds__(DkvCfg<D>::kThreads, 1)
lrsa_bwd_dkv_kernel(const __grid_constant__ DkvMaps<NSEQ> maps, const __grid_constant__ DkvArgs<NSEQ> a) {
  using Cfg = DkvCfg<D>;
  constexpr int NQ = Cfg::kStQ, NO = Cfg::kStO;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t smem0 = smem_u32(smem_raw);
  float* st_nl2 = reinterpret_cast<float*>(smem_raw + Cfg::kOffStats);   // [2][kQRows] -LSE*log2(e) (-inf: not seen)
  float* st_D = st_nl2 + 2 * kQRows;                                     // [2][kQRows]
  DkvCtl& ctl = *reinterpret_cast<DkvCtl*>(smem_raw + Cfg::kOffCtl);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sK = smem0, sV = smem0 + Cfg::kTileBytes;
  const uint32_t sQ = smem0 + Cfg::kOffRingQ, sO = smem0 + Cfg::kOffRingO;

  if (smem0 & 1023u) {   // the swizzled tiles need it; dynamic shared memory starts there when nothing is static
    if (tid == 0) atomicExch(a.status, (int)LRSA_ERR_TIMEOUT);
    return;
  }
  if (tid == 0) {
    ctl.abort = 0;
    mbar_init(smem_u32(&ctl.kv_full), 1);
    mbar_init(smem_u32(&ctl.acc_done), 1);
    for (int i = 0; i < NQ; ++i) { mbar_init(smem_u32(&ctl.q_full[i]), 1); mbar_init(smem_u32(&ctl.q_empty[i]), 1); }
    for (int i = 0; i < NO; ++i) { mbar_init(smem_u32(&ctl.o_full[i]), 1); mbar_init(smem_u32(&ctl.o_empty[i]), 1); }
    mbar_init(smem_u32(&ctl.dp_full), 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&ctl.p_full[b]), 32 * Cfg::kSoftWarps);   // every softmax thread (a lane per warp: 0.6 % slower)
      mbar_init(smem_u32(&ctl.s_full[b]), 2);   // the product and the statistics
      mbar_init(smem_u32(&ctl.ds_full[b]), 32 * Cfg::kSoftWarps);
    }
    fence_barrier_init();
  }
  if (warp == 1) { tmem_alloc(smem_u32(&ctl.tmem_base), 512); tmem_relinquish(); }

  // ---- which tile, which segment ----
  const int bh_kv = blockIdx.x % a.BHkv;
  int seg = blockIdx.x / a.BHkv, sq = 0;
  if constexpr (NSEQ > 1) {
    while (sq + 1 < a.n_seqs && seg >= a.seg0[sq + 1]) ++sq;
    seg -= a.seg0[sq];
  }
  const DkvPlan& p = a.plan[sq];
  if (tid == 0) {
    prefetch_tensormap(&maps.q[sq]); prefetch_tensormap(&maps.dO[sq]); prefetch_tensormap(&maps.k[sq]);
    prefetch_tensormap(&maps.v[sq]); prefetch_tensormap(&maps.kg[sq]); prefetch_tensormap(&maps.vg[sq]);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");   // started before the kernel in front of it has ended
  const int tok0 = a.tok0[sq];
  const int32_t* kept = a.idx + (size_t)bh_kv * a.kept_stride + a.kept_off[sq];   // this head's, this sequence's windows
  const int2 ts = a.seg_map[a.map0[sq] + seg];
  const KvTile kt = describe_tile(p, ts.x);
  const int seg_len = segment_length(p, p.G * kt.nq), it_begin = ts.y * seg_len;
  const int n = min(seg_len, p.G * kt.nq - it_begin);
  const int hq0 = (bh_kv / a.Hkv) * a.Hq + (bh_kv % a.Hkv) * p.G;   // first query head of the group

  // iteration gi of the tile: query tile nq-1 - gi/G (from the last query backwards) of head gi % G
  const int qt0 = kt.nq - 1 - it_begin / p.G, hd0 = it_begin % p.G;

  // TMA producer's loads of the step with query tile qt of head hd (of the group)
  auto load_q = [&](int slot, int qt, int hd) {
    const uint32_t full = smem_u32(&ctl.q_full[slot]);
    mbar_expect_tx(full, Cfg::kTileBytes);
    for (int h = 0; h < Cfg::kSub; ++h)
      tma_load_3d(sQ + slot * Cfg::kTileBytes + h * Cfg::kSubBytes, &maps.q[sq], h * 64, kt.qb + qt * kQRows, hq0 + hd, full);
  };
  auto load_o = [&](int slot, int qt, int hd) {
    const uint32_t full = smem_u32(&ctl.o_full[slot]);
    mbar_expect_tx(full, Cfg::kTileBytes);
    for (int h = 0; h < Cfg::kSub; ++h)
      tma_load_3d(sO + slot * Cfg::kTileBytes + h * Cfg::kSubBytes, &maps.dO[sq], h * 64, kt.qb + qt * kQRows, hq0 + hd, full);
  };
  if (warp == 0) {
    // K_j, V_j and the first Q and dO are fetched while the other warps get their tensor memory
    if (lane == 0) mbar_expect_tx(smem_u32(&ctl.kv_full), 2 * Cfg::kTileBytes);
    __syncwarp();
    if (kt.kind == 0) {
      // every lane gathers four rows of the list tile from their positions in K and V
      int pos[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        pos[i] = bh_kv * a.Nrow + compact_row_pos(kept, p.S, p.Rc, kt.row0 + 4 * lane + i, tok0);
      for (int h = 0; h < Cfg::kSub; ++h) {
        tma_gather4_2d(sK + h * Cfg::kSubBytes + lane * 512, &maps.kg[sq], h * 64, pos[0], pos[1], pos[2], pos[3], smem_u32(&ctl.kv_full));
        tma_gather4_2d(sV + h * Cfg::kSubBytes + lane * 512, &maps.vg[sq], h * 64, pos[0], pos[1], pos[2], pos[3], smem_u32(&ctl.kv_full));
      }
    } else if (lane == 0) {
      for (int h = 0; h < Cfg::kSub; ++h) {
        tma_load_3d(sK + h * Cfg::kSubBytes, &maps.k[sq], h * 64, kt.row0, bh_kv, smem_u32(&ctl.kv_full));
        tma_load_3d(sV + h * Cfg::kSubBytes, &maps.v[sq], h * 64, kt.row0, bh_kv, smem_u32(&ctl.kv_full));
      }
    }
    if (lane == 0) { load_q(0, qt0, hd0); load_o(0, qt0, hd0); }
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort = &ctl.abort;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // ---------------- TMA producer: the other steps ----------------
    if (lane == 0) {
      int qt = qt0, hd = hd0, slq = 1, slo = 1, phq = 0, pho = 0;
      int nq_issued = 1, no_issued = 1;
      bool ok = true;
      for (int it = 1; it < n; ++it) {
        if (++hd == p.G) { hd = 0; --qt; }
        if (it >= NQ) ok = mbar_wait(smem_u32(&ctl.q_empty[slq]), phq ^ 1, abort);
        if (!ok) break;
        load_q(slq, qt, hd);
        ++nq_issued;
        if (it >= NO) ok = mbar_wait(smem_u32(&ctl.o_empty[slo]), pho ^ 1, abort);
        if (!ok) break;
        load_o(slo, qt, hd);
        ++no_issued;
        if (++slq == NQ) { slq = 0; phq ^= 1; }
        if (++slo == NO) { slo = 0; pho ^= 1; }
      }
      if (!ok) {
        // give loads already in flight a bounded chance to land before the CTA's smem is released
        auto drain = [](uint64_t* bars, int slots, int issued) {
          for (int back = 1; back <= slots && back <= issued; ++back) {
            const int i2 = issued - back;
            const long long t0 = clock64();
            while (!mbar_try_wait(smem_u32(&bars[i2 % slots]), (i2 / slots) & 1) && clock64() - t0 < 2000000) {}
          }
        };
        drain(ctl.q_full, NQ, nq_issued);
        drain(ctl.o_full, NO, no_issued);
        drain(&ctl.kv_full, 1, 1);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: dV(i), S^T(i+1), dK(i), dP^T(i+1), ... ----------------
    // One thread issues everything, and the tensor core runs its products in this order (sm100_ptx.h): S^T(i+1) may
    // overwrite P^T(i) and dP^T(i+1) may overwrite dS^T(i) without waiting for the products that read them.  The loop runs
    // with all lanes (uniform control flow, descriptors computed once); one lane issues, by predicate.
    constexpr uint32_t idesc_s = make_idesc_bf16(kTile, kQRows, 0, 0);  // 128 keys x 128 queries
    constexpr uint32_t idesc_a = make_idesc_bf16(kTile, D, 0, 1);       // 128 keys x D
    const uint64_t descK = make_smem_desc_sw128(sK, 16, 1024), descV = make_smem_desc_sw128(sV, 16, 1024);
    const uint64_t descQ = make_smem_desc_sw128(sQ, 16, 1024), descO = make_smem_desc_sw128(sO, 16, 1024);   // K-major
    const uint64_t descQm = make_smem_desc_sw128(sQ, Cfg::kSubBytes, 1024);                                   // MN-major
    const uint64_t descOm = make_smem_desc_sw128(sO, Cfg::kSubBytes, 1024);
    const uint32_t leader = elect_one();
    auto scores = [&](uint64_t dA, uint64_t dB, uint32_t d_tmem, uint64_t* bar) {
#pragma unroll
      for (int h = 0; h < Cfg::kSub; ++h)
        umma_ss4(d_tmem, desc_advance(dA, h * Cfg::kSubBytes), desc_advance(dB, h * Cfg::kSubBytes), idesc_s, h > 0 ? 1u : 0u, leader);
      umma_commit(smem_u32(bar), leader);
    };
    bool ok = mbar_wait_warp(smem_u32(&ctl.kv_full), 0, abort);
    if (ok) ok = mbar_wait_warp(smem_u32(&ctl.q_full[0]), 0, abort);
    if (ok) {
      scores(descK, descQ, tmem + Cfg::kColS, &ctl.s_full[0]);
      ok = mbar_wait_warp(smem_u32(&ctl.o_full[0]), 0, abort);
    }
    if (ok) scores(descV, descO, tmem + Cfg::kColP, &ctl.dp_full);
    int slq = 0, slo = 0, phq = 0, pho = 0;   // slots of step `it` and the phases of the slots of step it+1
    for (int it = 0; it < n && ok; ++it) {
      const int nslq = slq + 1 == NQ ? 0 : slq + 1, nslo = slo + 1 == NO ? 0 : slo + 1;
      if (nslq == 0) phq ^= 1;
      if (nslo == 0) pho ^= 1;
      const uint32_t acc0 = it > 0 ? 1u : 0u;
      // (the next Q and dO are long here: waited for ahead of the softmax warps, not between two products)
      if (it + 1 < n) ok = mbar_wait_warp(smem_u32(&ctl.q_full[nslq]), phq, abort);
      // packed P^T / dS^T: the 32 query columns of warpgroup w in columns [32w, 32w+16) of the region
      {
        const uint64_t dB = desc_advance(descOm, slo * Cfg::kTileBytes);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          if (ok) ok = mbar_wait_warp(smem_u32(&ctl.p_full[half]), it & 1, abort);
          if (!ok) break;
          tc_fence_after_sync();
          umma_ts4<32, 64, 96, 4096>(tmem + Cfg::kColV, tmem + Cfg::kColS + half * 8, desc_advance(dB, half * 2048), idesc_a,
                                     half > 0 ? 1u : acc0, leader);
        }
        if (!ok) break;
      }
      if (it + 1 < n) {
        scores(descK, desc_advance(descQ, nslq * Cfg::kTileBytes), tmem + Cfg::kColS, &ctl.s_full[(it + 1) & 1]);
      }
      umma_commit(smem_u32(&ctl.o_empty[slo]), leader);
      if (it + 1 < n) ok = mbar_wait_warp(smem_u32(&ctl.o_full[nslo]), pho, abort);
      if (ok) ok = mbar_wait_warp(smem_u32(&ctl.ds_full[it & 1]), (it >> 1) & 1, abort);
      if (!ok) break;
      tc_fence_after_sync();
      {
        const uint64_t dB = desc_advance(descQm, slq * Cfg::kTileBytes);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          umma_ts4<8, 32, 40, 2048>(tmem + Cfg::kColK, tmem + Cfg::kColP + h * 64, desc_advance(dB, h * 4 * 2048), idesc_a,
                                    h > 0 ? 1u : acc0, leader);
      }
      if (it + 1 < n) scores(descV, desc_advance(descO, nslo * Cfg::kTileBytes), tmem + Cfg::kColP, &ctl.dp_full);
      umma_commit(smem_u32(&ctl.q_empty[slq]), leader);
      slq = nslq; slo = nslo;
    }
    if (ok) umma_commit(smem_u32(&ctl.acc_done), leader);
  } else if (warp == 2) {
    // the mean key of head blockIdx.x from its partial sums, for the dQ kernel
    if (a.kpart && blockIdx.x < a.BHkv) {
      for (int ch = lane * 4; ch < D; ch += 128) {
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int i = 0; i < a.splits; ++i) {
          const float4 x = *reinterpret_cast<const float4*>(a.kpart + ((size_t)i * a.BHkv + blockIdx.x) * D + ch);
          sum.x += x.x; sum.y += x.y; sum.z += x.z; sum.w += x.w;
        }
        *reinterpret_cast<float4*>(a.kbar + (size_t)blockIdx.x * D + ch) = sum;
      }
    }
  } else if (warp == 3) {
    // ---------------- per-row statistics of every step, fetched one step ahead ----------------
    int qt = qt0, hd = hd0;
    auto fetch = [&](int qt_, int hd_, float2 (&v)[kQRows / 32]) {
      const int hq = hq0 + hd_, q0 = kt.qb + qt_ * kQRows;
#pragma unroll
      for (int k = 0; k < kQRows / 32; ++k) {
        const int q = q0 + lane + 32 * k;
        v[k] = q < kt.qend ? a.stats[(size_t)hq * a.Nrow + tok0 + q] : make_float2(-INFINITY, 0.f);
      }
    };
    float2 cur[kQRows / 32], nxt[kQRows / 32];
    bool ok = true;
    fetch(qt, hd, cur);
    for (int it = 0; it < n; ++it) {
      const int b = it & 1;
      int qt_n = qt, hd_n = hd + 1;
      if (hd_n == p.G) { hd_n = 0; --qt_n; }
      if (it + 1 < n) fetch(qt_n, hd_n, nxt);
      if (it >= 2) ok = mbar_wait_warp(smem_u32(&ctl.ds_full[b]), ((it >> 1) - 1) & 1, abort);
      if (!ok) break;
#pragma unroll
      for (int k = 0; k < kQRows / 32; ++k) {
        st_nl2[b * kQRows + lane + 32 * k] = cur[k].x;
        st_D[b * kQRows + lane + 32 * k] = cur[k].y;
        cur[k] = nxt[k];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl.s_full[b]));
      qt = qt_n; hd = hd_n;
    }
  } else if (warp >= 4) {
    // ---------------- P^T / dS^T: warpgroup `wg` takes query columns [32*wg, 32*wg+32) of every step ----------------
    const int wg = (warp - 4) >> 2, quad = warp & 3;
    const int r = quad * 32 + lane;            // key row of this thread inside the tile
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t S_addr = tmem + lane_addr + Cfg::kColS + wg * 32;
    const uint32_t P_addr = tmem + lane_addr + Cfg::kColP + wg * 32;
    const float c = a.scale_log2;
    const bool key_ok = kt.row0 + r < kt.key_end;
    // First query position that sees this thread's key: its own (dense), or the start of the first chunk that sees
    // its window compressed (list row; sinks: the first position after them).  Every later query sees it too.
    int q_first = kt.row0 + r;
    if (kt.kind == 0)
      q_first = p.S + (q_first < p.S ? 0 : first_compressed_chunk((q_first - p.S) / p.K, p.ndp, p.Wsel, p.C) * p.L);
    if (!key_ok) q_first = 0x40000000;
    int q0 = kt.qb + qt0 * kQRows, hd = hd0;   // first query row and head (of the group) of the step
    const int col = wg * 32 + 16 * ((lane >> 4) & 1) + 8 * ((lane >> 3) & 1) + 2 * (lane & 3) + ((lane >> 2) & 1);
    bool ok = true;
    for (int it = 0; it < n; ++it) {
      const int b = it & 1;
      const int lo = q_first - q0 - wg * 32;     // columns below it do not see the key
      const float4* nl2v = reinterpret_cast<const float4*>(st_nl2 + b * kQRows + wg * 32);
      const float4* Dv = reinterpret_cast<const float4*>(st_D + b * kQRows + wg * 32);
      ok = mbar_wait_warp(smem_u32(&ctl.s_full[b]), (it >> 1) & 1, abort);
      if (!ok) break;
      tc_fence_after_sync();
      // P^T in halves of 16 columns: the tensor core starts dV on the first halves while the second are formed
      float pr[32];
      {
        uint32_t s[32];
        tmem_ld32(S_addr, s);
        tmem_wait_ld();
        if (lo > 0) {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (i < lo) s[i] = 0xff800000u;
        }
        const uint64_t c2 = f2_pack(c, c);   // packed fp32 pairs: one issue slot for two elements
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t pp[8];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const int e = 16 * h + 4 * v;
            const float4 nl = nl2v[4 * h + v];
            float a0, a1, a2, a3;
            f2_unpack(f2_fma(f2_pack(__uint_as_float(s[e]), __uint_as_float(s[e + 1])), c2, f2_pack(nl.x, nl.y)), a0, a1);
            f2_unpack(f2_fma(f2_pack(__uint_as_float(s[e + 2]), __uint_as_float(s[e + 3])), c2, f2_pack(nl.z, nl.w)), a2, a3);
            pr[e] = ex2(a0); pr[e + 1] = ex2(a1); pr[e + 2] = ex2(a2); pr[e + 3] = ex2(a3);
            pp[2 * v] = pack_bf16(pr[e], pr[e + 1]);
            pp[2 * v + 1] = pack_bf16(pr[e + 2], pr[e + 3]);
          }
          tmem_st8(S_addr + 8 * h, pp);   // over the first half of this warpgroup's own columns, already loaded
          tmem_wait_st();
          tc_fence_before_sync();
          mbar_arrive(smem_u32(&ctl.p_full[h]));
        }
      }
      ok = mbar_wait_warp(smem_u32(&ctl.dp_full), it & 1, abort);
      if (!ok) break;
      tc_fence_after_sync();
      // dS^T = P dP - P D; x = P dP (whose sum over the keys is the accurate D of the query column) replaces P
      uint32_t ds[16];
      {
        uint32_t dp[32];
        tmem_ld32(P_addr, dp);
        tmem_wait_ld();
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          const float4 dd = Dv[v];
          float d0, d1, d2, d3;
          const uint64_t p01 = f2_pack(pr[4 * v], pr[4 * v + 1]), p23 = f2_pack(pr[4 * v + 2], pr[4 * v + 3]);
          const uint64_t x01 = f2_mul(p01, f2_pack(__uint_as_float(dp[4 * v + 0]), __uint_as_float(dp[4 * v + 1])));
          const uint64_t x23 = f2_mul(p23, f2_pack(__uint_as_float(dp[4 * v + 2]), __uint_as_float(dp[4 * v + 3])));
          f2_unpack(f2_fma(p01, f2_pack(-dd.x, -dd.y), x01), d0, d1);
          f2_unpack(f2_fma(p23, f2_pack(-dd.z, -dd.w), x23), d2, d3);
          f2_unpack(x01, pr[4 * v], pr[4 * v + 1]);
          f2_unpack(x23, pr[4 * v + 2], pr[4 * v + 3]);
          ds[2 * v] = pack_bf16(d0, d1);
          ds[2 * v + 1] = pack_bf16(d2, d3);
        }
      }
      // Sum of x over the warp's 32 keys: the values go through this warpgroup's own dP^T columns (all loaded, and
      // dS^T is not stored yet: the tensor core is busy with dV and the next S^T meanwhile) and come back with the
      // 16-lane x 256-bit load shape, which hands every thread four key rows of eight query columns; the
      // remaining three levels are register exchanges, after dS^T is on its way.
      tmem_st32(P_addr, *reinterpret_cast<uint32_t(*)[32]>(&pr[0]));
      tmem_wait_st();
      uint32_t ra[16], rb[16];
      tmem_ld_16x256b_x4(P_addr, ra);
      tmem_ld_16x256b_x4(P_addr + (16u << 16), rb);
      tmem_wait_ld();
      tmem_st16(P_addr, ds);
      tmem_wait_st();
      tc_fence_before_sync();
      mbar_arrive(smem_u32(&ctl.ds_full[b]));
      float c8[8];   // index 2j + e: column 8j + 2(lane%4) + e of the warpgroup's 32
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e)
          c8[2 * j + e] = (__uint_as_float(ra[4 * j + e]) + __uint_as_float(ra[4 * j + 2 + e])) +
                          (__uint_as_float(rb[4 * j + e]) + __uint_as_float(rb[4 * j + 2 + e]));
#pragma unroll
      for (int m = 4, bit = 16; m >= 1; m >>= 1, bit >>= 1) {
        const bool up = (lane & bit) != 0;
#pragma unroll
        for (int i = 0; i < m; ++i) {
          const float send = up ? c8[i] : c8[i + m];
          const float keep = up ? c8[i + m] : c8[i];
          c8[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
        }
      }
      if (q0 + col < kt.qend) atomicAdd(a.Dacc + (size_t)(hq0 + hd) * a.Nrow + tok0 + q0 + col, c8[0]);
      if (++hd == p.G) { hd = 0; q0 -= kQRows; }
    }
    if (ok) ok = mbar_wait_warp(smem_u32(&ctl.acc_done), 0, abort);
    if (ok) {
      tc_fence_after_sync();
      // warpgroups 0 and 1 add dK (scaled), 2 and 3 dV, half of the columns each
      constexpr int CH = D / 2;
      const bool is_k = wg < 2;
      const uint32_t acc = tmem + lane_addr + (is_k ? Cfg::kColK : Cfg::kColV) + (wg & 1) * CH;
      const float mul = is_k ? a.scale : 1.0f;
      // A row of a compact tile lands on the position it was gathered from.  The rows go through shared memory (the rings are
      // idle: every product is done), so that a warp adds to whole lines: with every lane on a row of its own the epilogue is bound by
      // the 32 lines that each instruction touches (with the earlier first loads, whole backward: 8K tokens, 8 heads, d = 64, 189 -> 181 us).  Rows are padded by 16 bytes so that a warp's stores spread over the banks.
      const int out_row = !key_ok ? -1 : kt.kind == 0 ? compact_row_pos(kept, p.S, p.Rc, kt.row0 + r, tok0) : kt.row0 + r;
      constexpr int kStride = CH + 4;
      static_assert(Cfg::kSoftWarps * 32 * kStride * 4 <= Cfg::kOffStats - Cfg::kOffRingQ, "the rows of every warp fit the rings");
      float* stage = reinterpret_cast<float*>(smem_raw + Cfg::kOffRingQ) + (warp - 4) * 32 * kStride;
#pragma unroll
      for (int q = 0; q < CH / 32; ++q) {
        uint32_t o[32];
        tmem_ld32(acc + q * 32, o);
        tmem_wait_ld();
#pragma unroll
        for (int v = 0; v < 8; ++v)
          *reinterpret_cast<float4*>(stage + lane * kStride + q * 32 + v * 4) =
              make_float4(__uint_as_float(o[4 * v]) * mul, __uint_as_float(o[4 * v + 1]) * mul,
                          __uint_as_float(o[4 * v + 2]) * mul, __uint_as_float(o[4 * v + 3]) * mul);
      }
      __syncwarp();
      constexpr int kLanes = CH / 4, kRows = 32 / kLanes;   // lanes per row, rows per instruction
      float* dst = (is_k ? a.dKf : a.dVf) + ((size_t)bh_kv * a.Nrow + tok0) * D + (wg & 1) * CH + lane % kLanes * 4;
#pragma unroll 4
      for (int i = 0; i < 32; i += kRows) {
        const int row = i + lane / kLanes, to = __shfl_sync(0xffffffffu, out_row, row);
        const float4 x = *reinterpret_cast<const float4*>(stage + row * kStride + lane % kLanes * 4);
        if (to >= 0) red_add_v4(dst + (size_t)to * D, x.x, x.y, x.z, x.w);
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
  if (tid == 0 && ctl.abort) atomicExch(a.status, (int)LRSA_ERR_TIMEOUT);
}

}  // namespace

template <int D, int NSEQ>
static int launch_dkv_t(const Geom& whole, const SeqBatch& b, const DkvBatch& db, const BwdPtrs& p, bool mean, cudaStream_t st) {
  using Cfg = DkvCfg<D>;
  DkvMaps<NSEQ> m;
  DkvArgs<NSEQ> a;
  const long long BHq = (long long)whole.B * whole.Hq, BHkv = (long long)whole.B * whole.Hkv;
  a.seg0[0] = 0;
  for (int s = 0; s < b.n; ++s) {
    const Geom& g = b.g[s];
    const size_t sh = (size_t)g.tok0 * D;
    int r = make_tmap_bf16(&m.q[s], p.Q + sh, D, g.N, BHq, kQRows, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.dO[s], p.dO + sh, D, g.N, BHq, kQRows, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.k[s], p.K + sh, D, g.N, BHkv, kTile, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16(&m.v[s], p.V + sh, D, g.N, BHkv, kTile, g.Nrow);
    if (r == LRSA_OK) r = make_tmap_bf16_rows(&m.kg[s], p.K + sh, D, BHkv * g.Nrow - g.tok0);
    if (r == LRSA_OK) r = make_tmap_bf16_rows(&m.vg[s], p.V + sh, D, BHkv * g.Nrow - g.tok0);
    if (r != LRSA_OK) return r;
    a.plan[s] = db.plan[s];
    a.tok0[s] = g.tok0;
    a.kept_off[s] = g.woff * g.K;
    a.map0[s] = db.map0[s];
    a.seg0[s + 1] = a.seg0[s] + db.segs[s];
  }
  a.n_seqs = b.n;
  a.BHkv = (int)BHkv; a.Hq = whole.Hq; a.Hkv = whole.Hkv;
  a.idx = p.idx; a.kept_stride = whole.Wtot * whole.K; a.Nrow = whole.Nrow;
  a.kpart = mean ? p.kpart : nullptr; a.kbar = p.kbar; a.splits = mean_splits(whole.Nrow);
  a.stats = p.stats; a.Dacc = p.Dacc; a.seg_map = p.seg_map; a.dKf = p.dKf; a.dVf = p.dVf;
  a.scale = whole.scale; a.scale_log2 = whole.scale * 1.4426950408889634f; a.status = p.status;
  auto kern = lrsa_bwd_dkv_kernel<D, NSEQ>;
  LRSA_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmem));
  const long long grid = (long long)a.seg0[b.n] * a.BHkv;
  if (grid > 0x7fffffffLL) return LRSA_ERR_UNSUPPORTED;
  LRSA_CUDA_CHECK(launch_dependent(kern, dim3((unsigned)grid), dim3(Cfg::kThreads), Cfg::kSmem, st, 1, m, a));
  launch_counter().n++;
  return LRSA_OK;
}

int launch_bwd_dkv_sm100(const Geom& whole, const SeqBatch& b, const DkvBatch& db, const BwdPtrs& p, bool mean, cudaStream_t st) {
  if (whole.d == 128)
    return b.n == 1 ? launch_dkv_t<128, 1>(whole, b, db, p, mean, st) : launch_dkv_t<128, kMaxSeqs>(whole, b, db, p, mean, st);
  return b.n == 1 ? launch_dkv_t<64, 1>(whole, b, db, p, mean, st) : launch_dkv_t<64, kMaxSeqs>(whole, b, db, p, mean, st);
}

}  // namespace lrsa
