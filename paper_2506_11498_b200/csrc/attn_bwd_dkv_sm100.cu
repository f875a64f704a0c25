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
// kernel together with the exponentials) and pay for half as many hand-offs: 5.23 -> 4.58 ms at 32K tokens, 28/4
// heads, d = 128, one kept token in four.  Warps: 0 TMA producer, 1 issuer, 3 row statistics, 4-19 softmax and
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
#include "attn_common_sm100.h"

namespace lrsa {
namespace {

using namespace ptx;

constexpr int kQRows = 128;   // query rows per inner tile
constexpr int kSeg = 128;     // inner iterations per CTA at most

struct DkvPlan {
  int S, L, K, N, W, T, C, Wsel, ndp, Rc, G;
  int n_cmp;       // compact tiles
  int n_sink;      // dense tiles of the sink region
  int per_win;     // dense tiles per full window
  int per_tail;    // dense tiles of the tail
  int n_tiles;
};

struct KvTile {
  int kind;      // 0 compact, 1 dense
  int row0;      // first compact row / first key position
  int key_end;   // rows at or beyond this are not part of the tile
  int qb, qend;  // query positions [qb, qend) see (part of) the tile
  int nq;        // query tiles (kQRows rows) per head
};

inline DkvPlan make_dkv_plan(const Geom& g) {
  DkvPlan p;
  p.S = g.S; p.L = g.L; p.K = g.K; p.N = g.N; p.W = g.W; p.T = g.T; p.C = g.C; p.Wsel = g.Wsel;
  p.ndp = g.ndp; p.Rc = g.Rc; p.G = g.G;
  p.n_cmp = (g.Rc + kTile - 1) / kTile;
  p.n_sink = (g.S + kTile - 1) / kTile;
  p.per_win = (g.L + kTile - 1) / kTile;
  p.per_tail = (g.T + kTile - 1) / kTile;
  p.n_tiles = p.n_cmp + p.n_sink + g.W * p.per_win + p.per_tail;
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
  return (p.G * t.nq + kSeg - 1) / kSeg;
}

// Launch order of the (tile, segment) pairs (one block).  Iteration i of a tile is query tile
// nq-1 - i/G (counted from the last query) of head i%G, so segment s of every compact tile covers the
// same queries of the same heads.  Compact tiles are therefore issued segment-major: the CTAs that run at
// the same time then stream the same Q_i / dO_i tiles and share them through L2 instead of fetching
// them from DRAM once per key tile.  Dense tiles (short lists, neighbours already overlap) follow in
// position order.  seg_cnt: scratch of n_tiles + 1 ints; seg_map[x] = (tile, segment of the tile).
constexpr int kMaxSegsPerTile = 2048;
__global__ void dkv_setup_kernel(const DkvPlan p, int* seg_cnt, int2* seg_map) {
  __shared__ int off[kMaxSegsPerTile + 1];   // off[s] = pairs of compact tiles with a segment index below s
  __shared__ int s_mode, s_cmp_total;
  __shared__ int run_sum[256];   // blockDim.x = 256
  for (int i = threadIdx.x; i < p.n_tiles; i += blockDim.x) seg_cnt[i] = tile_segments(p, describe_tile(p, i));
  __syncthreads();
  if (threadIdx.x == 0) {
    // segment-major order needs the compact tiles' segment counts to be non-increasing (later rows are
    // seen by later chunks only) and few enough for the table; otherwise keep tile-major order
    bool mono = p.n_cmp > 0 && seg_cnt[0] <= kMaxSegsPerTile;
    for (int c = 1; c < p.n_cmp && mono; ++c) mono = seg_cnt[c] <= seg_cnt[c - 1];
    int total = 0;
    if (mono) {
      int c = p.n_cmp;   // tiles [0, c) have more than s segments
      const int maxs = seg_cnt[0];
      for (int sgm = 0; sgm < maxs; ++sgm) {
        while (c > 0 && seg_cnt[c - 1] <= sgm) --c;
        off[sgm] = total;
        total += c;
      }
    } else {
      for (int c = 0; c < p.n_cmp; ++c) {
        for (int sgm = 0; sgm < seg_cnt[c]; ++sgm) seg_map[total + sgm] = make_int2(c, sgm);
        total += seg_cnt[c];
      }
    }
    s_mode = mono ? 1 : 0;
    s_cmp_total = total;
  }
  // dense tiles, position order: every thread takes a run of consecutive tiles
  const int nd = p.n_tiles - p.n_cmp, per = (nd + (int)blockDim.x - 1) / (int)blockDim.x;
  const int d_lo = min(p.n_tiles, p.n_cmp + (int)threadIdx.x * per), d_hi = min(p.n_tiles, d_lo + per);
  int mine = 0;
  for (int t = d_lo; t < d_hi; ++t) mine += seg_cnt[t];
  run_sum[threadIdx.x] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = s_cmp_total;
    for (int i = 0; i < (int)blockDim.x; ++i) { const int v = run_sum[i]; run_sum[i] = acc; acc += v; }
  }
  __syncthreads();
  {
    int pos = run_sum[threadIdx.x];
    for (int t = d_lo; t < d_hi; ++t) {
      for (int sgm = 0; sgm < seg_cnt[t]; ++sgm) seg_map[pos + sgm] = make_int2(t, sgm);
      pos += seg_cnt[t];
    }
  }
  if (s_mode) {
    for (int c = threadIdx.x; c < p.n_cmp; c += blockDim.x)
      for (int sgm = 0; sgm < seg_cnt[c]; ++sgm) seg_map[off[sgm] + c] = make_int2(c, sgm);
  }
}

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

struct DkvArgs {
  DkvPlan plan;
  int BHkv, Hq, Hkv, total_segs;
  const int32_t* idx;    // kept positions of this sequence's windows: head bh at idx + bh * kept_stride
  int kept_stride;       // Wtot * K entries per (batch, KV head)
  int Nrow, tok0;        // tokens per (batch, head) row (the stride of every tensor); first token of the sequence
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
  uint64_t s_full, dp_full;      // S^T / dP^T of the step are in tensor memory
  uint64_t p_full[2];            // halves of P^T: the first / last 16 query columns of every warpgroup
  uint64_t st_full[2];           // statistics of the step (slot = step & 1) are staged
  uint64_t ds_full[2];           // dS^T of the step is stored (slot = step & 1; also frees the statistics slot)
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(DkvCtl) <= 512, "control block fits");

__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

template <int D>
__global__ void __launch_bounds__(DkvCfg<D>::kThreads, 1)
lrsa_bwd_dkv_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapdO,
                    const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV,
                    const __grid_constant__ CUtensorMap mapKg, const __grid_constant__ CUtensorMap mapVg,
                    const DkvArgs a) {
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

  // ---- which tile, which segment ----
  const DkvPlan& p = a.plan;
  const int bh_kv = blockIdx.x % a.BHkv, seg = blockIdx.x / a.BHkv;
  const int2 ts = a.seg_map[seg];
  const KvTile kt = describe_tile(p, ts.x);
  const int it_begin = ts.y * kSeg;
  const int n = min(kSeg, p.G * kt.nq - it_begin);
  const int hq0 = (bh_kv / a.Hkv) * a.Hq + (bh_kv % a.Hkv) * p.G;   // first query head of the group

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
    mbar_init(smem_u32(&ctl.s_full), 1);
    mbar_init(smem_u32(&ctl.dp_full), 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&ctl.p_full[b]), Cfg::kSoftWarps);   // one arrival per softmax warp
      mbar_init(smem_u32(&ctl.st_full[b]), 1);
      mbar_init(smem_u32(&ctl.ds_full[b]), Cfg::kSoftWarps);
    }
    fence_barrier_init();
  }
  if (warp == 1) { tmem_alloc(smem_u32(&ctl.tmem_base), 512); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort = &ctl.abort;
  // iteration gi of the tile: query tile nq-1 - gi/G (from the last query backwards) of head gi % G
  const int qt0 = kt.nq - 1 - it_begin / p.G, hd0 = it_begin % p.G;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      prefetch_tensormap(&mapQ); prefetch_tensormap(&mapdO);
      mbar_expect_tx(smem_u32(&ctl.kv_full), 2 * Cfg::kTileBytes);
    }
    __syncwarp();
    if (kt.kind == 0) {
      // every lane gathers four rows of the list tile from their positions in K and V
      const int32_t* kept = a.idx + (size_t)bh_kv * a.kept_stride;
      int pos[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        pos[i] = bh_kv * a.Nrow + compact_row_pos(kept, p.S, p.Rc, kt.row0 + 4 * lane + i, a.tok0);
      for (int h = 0; h < Cfg::kSub; ++h) {
        tma_gather4_2d(sK + h * Cfg::kSubBytes + lane * 512, &mapKg, h * 64, pos[0], pos[1], pos[2], pos[3], smem_u32(&ctl.kv_full));
        tma_gather4_2d(sV + h * Cfg::kSubBytes + lane * 512, &mapVg, h * 64, pos[0], pos[1], pos[2], pos[3], smem_u32(&ctl.kv_full));
      }
    } else if (lane == 0) {
      for (int h = 0; h < Cfg::kSub; ++h) {
        tma_load_3d(sK + h * Cfg::kSubBytes, &mapK, h * 64, kt.row0, bh_kv, smem_u32(&ctl.kv_full));
        tma_load_3d(sV + h * Cfg::kSubBytes, &mapV, h * 64, kt.row0, bh_kv, smem_u32(&ctl.kv_full));
      }
    }
    if (lane == 0) {
      int qt = qt0, hd = hd0, slq = 0, slo = 0, phq = 0, pho = 0;
      int nq_issued = 0, no_issued = 0;
      bool ok = true;
      for (int it = 0; it < n; ++it) {
        const int hq = hq0 + hd, q0 = kt.qb + qt * kQRows;
        if (it >= NQ) ok = mbar_wait(smem_u32(&ctl.q_empty[slq]), phq ^ 1, abort);
        if (!ok) break;
        const uint32_t qf = smem_u32(&ctl.q_full[slq]);
        mbar_expect_tx(qf, Cfg::kTileBytes);
        for (int h = 0; h < Cfg::kSub; ++h)
          tma_load_3d(sQ + slq * Cfg::kTileBytes + h * Cfg::kSubBytes, &mapQ, h * 64, q0, hq, qf);
        ++nq_issued;
        if (it >= NO) ok = mbar_wait(smem_u32(&ctl.o_empty[slo]), pho ^ 1, abort);
        if (!ok) break;
        const uint32_t of = smem_u32(&ctl.o_full[slo]);
        mbar_expect_tx(of, Cfg::kTileBytes);
        for (int h = 0; h < Cfg::kSub; ++h)
          tma_load_3d(sO + slo * Cfg::kTileBytes + h * Cfg::kSubBytes, &mapdO, h * 64, q0, hq, of);
        ++no_issued;
        if (++slq == NQ) { slq = 0; phq ^= 1; }
        if (++slo == NO) { slo = 0; pho ^= 1; }
        if (++hd == p.G) { hd = 0; --qt; }
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
    // One warp issues everything, so the products run in this order on the tensor core: S^T(i+1) may overwrite
    // P^T(i) and dP^T(i+1) may overwrite dS^T(i) without waiting for the products that read them.  The loop runs
    // with all lanes (uniform control flow, descriptors computed once) and elects one lane per instruction.
    constexpr uint32_t idesc_s = make_idesc_bf16(kTile, kQRows, 0, 0);  // 128 keys x 128 queries
    constexpr uint32_t idesc_a = make_idesc_bf16(kTile, D, 0, 1);       // 128 keys x D
    const uint64_t descK = make_smem_desc_sw128(sK, 16, 1024), descV = make_smem_desc_sw128(sV, 16, 1024);
    const uint64_t descQ = make_smem_desc_sw128(sQ, 16, 1024), descO = make_smem_desc_sw128(sO, 16, 1024);   // K-major
    const uint64_t descQm = make_smem_desc_sw128(sQ, Cfg::kSubBytes, 1024);                                   // MN-major
    const uint64_t descOm = make_smem_desc_sw128(sO, Cfg::kSubBytes, 1024);
    auto scores = [&](uint64_t dA, uint64_t dB, uint32_t d_tmem, uint64_t* bar) {
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t off = (kk >> 2) * Cfg::kSubBytes + (kk & 3) * 32;
        const uint64_t ad = desc_advance(dA, off), bd = desc_advance(dB, off);
        if (elect_one()) umma_ss(d_tmem, ad, bd, idesc_s, kk > 0 ? 1u : 0u);
      }
      if (elect_one()) umma_commit(smem_u32(bar));
      __syncwarp();
    };
    bool ok = mbar_wait_warp(smem_u32(&ctl.kv_full), 0, abort);
    if (ok) ok = mbar_wait_warp(smem_u32(&ctl.q_full[0]), 0, abort);
    if (ok) {
      scores(descK, descQ, tmem + Cfg::kColS, &ctl.s_full);
      ok = mbar_wait_warp(smem_u32(&ctl.o_full[0]), 0, abort);
    }
    if (ok) scores(descV, descO, tmem + Cfg::kColP, &ctl.dp_full);
    int slq = 0, slo = 0, phq = 0, pho = 0;   // slots of step `it` and the phases of the slots of step it+1
    for (int it = 0; it < n && ok; ++it) {
      const int nslq = slq + 1 == NQ ? 0 : slq + 1, nslo = slo + 1 == NO ? 0 : slo + 1;
      if (nslq == 0) phq ^= 1;
      if (nslo == 0) pho ^= 1;
      const uint32_t acc0 = it > 0 ? 1u : 0u;
      // packed P^T / dS^T: the 32 query columns of warpgroup w in columns [32w, 32w+16) of the region
      {
        const uint64_t dB = desc_advance(descOm, slo * Cfg::kTileBytes);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          if (ok) ok = mbar_wait_warp(smem_u32(&ctl.p_full[half]), it & 1, abort);
          if (!ok) break;
          tc_fence_after_sync();
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4) {
            const int kk = 2 * k4 + half;
            const uint64_t bd = desc_advance(dB, kk * 2048);
            if (elect_one())
              umma_ts(tmem + Cfg::kColV, tmem + Cfg::kColS + (kk >> 1) * 32 + (kk & 1) * 8, bd, idesc_a,
                      kk > 0 ? 1u : acc0);
          }
        }
        if (!ok) break;
        if (elect_one()) umma_commit(smem_u32(&ctl.o_empty[slo]));
        __syncwarp();
      }
      if (it + 1 < n) {
        ok = mbar_wait_warp(smem_u32(&ctl.q_full[nslq]), phq, abort);
        if (!ok) break;
        scores(descK, desc_advance(descQ, nslq * Cfg::kTileBytes), tmem + Cfg::kColS, &ctl.s_full);
      }
      ok = mbar_wait_warp(smem_u32(&ctl.ds_full[it & 1]), (it >> 1) & 1, abort);
      if (!ok) break;
      tc_fence_after_sync();
      {
        const uint64_t dB = desc_advance(descQm, slq * Cfg::kTileBytes);
#pragma unroll
        for (int kk = 0; kk < kQRows / 16; ++kk) {
          const uint64_t bd = desc_advance(dB, kk * 2048);
          if (elect_one())
            umma_ts(tmem + Cfg::kColK, tmem + Cfg::kColP + (kk >> 1) * 32 + (kk & 1) * 8, bd, idesc_a, kk > 0 ? 1u : acc0);
        }
        if (elect_one()) umma_commit(smem_u32(&ctl.q_empty[slq]));
        __syncwarp();
      }
      if (it + 1 < n) {
        ok = mbar_wait_warp(smem_u32(&ctl.o_full[nslo]), pho, abort);
        if (!ok) break;
        scores(descV, desc_advance(descO, nslo * Cfg::kTileBytes), tmem + Cfg::kColP, &ctl.dp_full);
      }
      slq = nslq; slo = nslo;
    }
    if (ok && elect_one()) umma_commit(smem_u32(&ctl.acc_done));
    __syncwarp();
  } else if (warp == 3) {
    // ---------------- per-row statistics of every step, fetched one step ahead ----------------
    int qt = qt0, hd = hd0;
    auto fetch = [&](int qt_, int hd_, float2 (&v)[kQRows / 32]) {
      const int hq = hq0 + hd_, q0 = kt.qb + qt_ * kQRows;
#pragma unroll
      for (int k = 0; k < kQRows / 32; ++k) {
        const int q = q0 + lane + 32 * k;
        v[k] = q < kt.qend ? __ldg(a.stats + (size_t)hq * a.Nrow + q) : make_float2(-INFINITY, 0.f);
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
      if (lane == 0) mbar_arrive(smem_u32(&ctl.st_full[b]));
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
      ok = mbar_wait_warp(smem_u32(&ctl.st_full[b]), (it >> 1) & 1, abort);
      if (!ok) break;
      const float4* nl2v = reinterpret_cast<const float4*>(st_nl2 + b * kQRows + wg * 32);
      const float4* Dv = reinterpret_cast<const float4*>(st_D + b * kQRows + wg * 32);
      ok = mbar_wait_warp(smem_u32(&ctl.s_full), it & 1, abort);
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
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&ctl.p_full[h]));
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
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl.ds_full[b]));
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
      if (q0 + col < kt.qend) atomicAdd(a.Dacc + (size_t)(hq0 + hd) * a.Nrow + q0 + col, c8[0]);
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
      // a row of a compact tile lands on the position it was gathered from
      const int out_row = kt.kind == 0
                              ? compact_row_pos(a.idx + (size_t)bh_kv * a.kept_stride, p.S, p.Rc, kt.row0 + r, a.tok0)
                              : kt.row0 + r;
      float* dst = (is_k ? a.dKf : a.dVf) + ((size_t)bh_kv * a.Nrow + out_row) * D + (wg & 1) * CH;
#pragma unroll
      for (int q = 0; q < CH / 32; ++q) {
        uint32_t o[32];
        tmem_ld32(acc + q * 32, o);
        tmem_wait_ld();
        if (key_ok) {
#pragma unroll
          for (int v = 0; v < 8; ++v)
            red_add_v4(dst + q * 32 + v * 4, __uint_as_float(o[4 * v]) * mul, __uint_as_float(o[4 * v + 1]) * mul,
                       __uint_as_float(o[4 * v + 2]) * mul, __uint_as_float(o[4 * v + 3]) * mul);
        }
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
  if (tid == 0 && ctl.abort) atomicExch(a.status, (int)LRSA_ERR_TIMEOUT);
}

// bf16 outputs from the fp32 accumulators [BHkv][N][d]; n4 = number of float4 groups
__global__ void convert_dkv_kernel(const float* __restrict__ dKf, const float* __restrict__ dVf,
                                   __nv_bfloat16* __restrict__ dK, __nv_bfloat16* __restrict__ dV, long long n4) {
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

}  // namespace

static int dkv_total_segs(const DkvPlan& p) {
  int total = 0;
  for (int i = 0; i < p.n_tiles; ++i) total += tile_segments(p, describe_tile(p, i));
  return total;
}

// Layout: [segment counts: n_tiles + 1 ints][launch order: total_segs int2][dK fp32][dV fp32]
size_t dkv_ws_bytes(const Geom& g, size_t* prefix_bytes) {
  const DkvPlan p = make_dkv_plan(g);
  const size_t cnt = align_up((size_t)(p.n_tiles + 1) * sizeof(int), 1024);
  const size_t pre = cnt + align_up((size_t)(dkv_total_segs(p) + 1) * sizeof(int2), 1024);
  if (prefix_bytes) *prefix_bytes = pre;
  const size_t acc = align_up((size_t)g.B * g.Hkv * g.Nrow * g.d * sizeof(float), 1024);
  return pre + 2 * acc;
}

template <int D>
static int launch_dkv_t(const Geom& g, const DkvArgs& a, const CUtensorMap* m, cudaStream_t st) {
  using Cfg = DkvCfg<D>;
  auto kern = lrsa_bwd_dkv_kernel<D>;
  LRSA_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmem));
  const long long grid = (long long)a.total_segs * a.BHkv;
  if (grid > 0x7fffffffLL) return LRSA_ERR_UNSUPPORTED;
  if (grid == 0) return LRSA_OK;
  kern<<<(unsigned)grid, Cfg::kThreads, Cfg::kSmem, st>>>(m[0], m[1], m[2], m[3], m[4], m[5], a);
  LRSA_CUDA_CHECK(cudaGetLastError());
  launch_counter().n++;
  return LRSA_OK;
}

// ws_dkv: region of dkv_ws_bytes(whole row) bytes.  Three steps: dkv_zero clears the fp32 accumulators of
// the whole row, launch_bwd_dkv_sm100 runs the tile kernel of one sequence (its launch-order table is
// rebuilt in the region's prefix, in stream order), dkv_convert writes bf16 dK, dV.
static void dkv_regions(const Geom& whole, void* ws_dkv, int** seg_cnt, int2** seg_map, float** dKf, float** dVf,
                        size_t* acc_bytes) {
  size_t pre = 0;
  const size_t total = dkv_ws_bytes(whole, &pre);
  unsigned char* base = static_cast<unsigned char*>(ws_dkv);
  const DkvPlan p = make_dkv_plan(whole);
  *acc_bytes = (total - pre) / 2;
  *seg_cnt = reinterpret_cast<int*>(base);
  *seg_map = reinterpret_cast<int2*>(base + align_up((size_t)(p.n_tiles + 1) * sizeof(int), 1024));
  *dKf = reinterpret_cast<float*>(base + pre);
  *dVf = reinterpret_cast<float*>(base + pre + *acc_bytes);
}

int dkv_zero(const Geom& whole, void* ws_dkv, cudaStream_t st) {
  int* seg_cnt; int2* seg_map; float *dKf, *dVf; size_t acc;
  dkv_regions(whole, ws_dkv, &seg_cnt, &seg_map, &dKf, &dVf, &acc);
  LRSA_CUDA_CHECK(cudaMemsetAsync(dKf, 0, 2 * acc, st));
  launch_counter().n++;
  return LRSA_OK;
}

int dkv_convert(const Geom& whole, void* ws_dkv, __nv_bfloat16* dK, __nv_bfloat16* dV, cudaStream_t st) {
  int* seg_cnt; int2* seg_map; float *dKf, *dVf; size_t acc;
  dkv_regions(whole, ws_dkv, &seg_cnt, &seg_map, &dKf, &dVf, &acc);
  const long long n4 = (long long)whole.B * whole.Hkv * whole.Nrow * whole.d / 4;
  convert_dkv_kernel<<<(unsigned)((n4 + 255) / 256), 256, 0, st>>>(dKf, dVf, dK, dV, n4);
  LRSA_CUDA_CHECK(cudaGetLastError());
  launch_counter().n++;
  return LRSA_OK;
}

// `whole`: the geometry of the whole row (workspace layout); `g`: the sequence to process.
int launch_bwd_dkv_sm100(const Geom& whole, const Geom& g, const __nv_bfloat16* Q, const __nv_bfloat16* dO,
                         const __nv_bfloat16* K, const __nv_bfloat16* V, const float2* stats, float* Dacc,
                         const int32_t* idx, void* ws_dkv, int* status, cudaStream_t st) {
  const DkvPlan p = make_dkv_plan(g);
  int* seg_cnt; int2* seg_map; float *dKf, *dVf; size_t acc;
  dkv_regions(whole, ws_dkv, &seg_cnt, &seg_map, &dKf, &dVf, &acc);
  // a part of a row never needs more than the whole row; checked all the same
  if (p.n_tiles > make_dkv_plan(whole).n_tiles || dkv_total_segs(p) > dkv_total_segs(make_dkv_plan(whole)))
    return LRSA_ERR_WORKSPACE_TOO_SMALL;
  dkv_setup_kernel<<<1, 256, 0, st>>>(p, seg_cnt, seg_map);
  LRSA_CUDA_CHECK(cudaGetLastError());
  launch_counter().n++;
  const int total_segs = dkv_total_segs(p);

  CUtensorMap m[6];
  const size_t sh = (size_t)g.tok0 * g.d;
  int r = make_tmap_bf16(&m[0], Q + sh, g.d, g.N, (long long)g.B * g.Hq, kQRows, g.Nrow);
  if (r == LRSA_OK) r = make_tmap_bf16(&m[1], dO + sh, g.d, g.N, (long long)g.B * g.Hq, kQRows, g.Nrow);
  if (r == LRSA_OK) r = make_tmap_bf16(&m[2], K + sh, g.d, g.N, (long long)g.B * g.Hkv, kTile, g.Nrow);
  if (r == LRSA_OK) r = make_tmap_bf16(&m[3], V + sh, g.d, g.N, (long long)g.B * g.Hkv, kTile, g.Nrow);
  if (r == LRSA_OK) r = make_tmap_bf16_rows(&m[4], K + sh, g.d, (long long)g.B * g.Hkv * g.Nrow - g.tok0);
  if (r == LRSA_OK) r = make_tmap_bf16_rows(&m[5], V + sh, g.d, (long long)g.B * g.Hkv * g.Nrow - g.tok0);
  if (r != LRSA_OK) return r;
  DkvArgs a;
  a.plan = p; a.BHkv = g.B * g.Hkv; a.Hq = g.Hq; a.Hkv = g.Hkv; a.total_segs = total_segs;
  a.idx = idx + (size_t)g.woff * g.K; a.kept_stride = g.Wtot * g.K; a.Nrow = g.Nrow; a.tok0 = g.tok0;
  a.stats = stats + g.tok0; a.Dacc = Dacc + g.tok0; a.seg_map = seg_map; a.dKf = dKf + sh; a.dVf = dVf + sh;
  a.scale = g.scale; a.scale_log2 = g.scale * 1.4426950408889634f; a.status = status;
  return g.d == 128 ? launch_dkv_t<128>(g, a, m, st) : launch_dkv_t<64>(g, a, m, st);
}

}  // namespace lrsa
