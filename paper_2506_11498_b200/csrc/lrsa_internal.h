// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <nvtx3/nvToolsExt.h>

#include "../../include/lrsa.h"

namespace lrsa {

// Problem geometry derived from lrsa_params_t (Section 3.2: sink of size S, windows of lag L).
struct Geom {
  int B, Hq, Hkv, G, N, d, L, K, S, ndp, ddof;
  float scale;
  int W;     // full windows
  int T;     // tail tokens
  int C;     // query chunks = W + [T > 0]
  int Wsel;  // scored windows = max(W - 1, 0)
  int Rc;    // rows of the compact (sinks + kept) K/V buffer per KV head = S + Wsel*K
  // Packed batches: this Geom describes ONE sequence of N tokens that starts at token `tok0` of rows
  // that hold Nrow tokens per (batch, head); its scored windows are windows [woff, woff + Wsel) of the
  // Wtot windows of the whole row.  Single sequence: Nrow = N, tok0 = 0, Wtot = Wsel, woff = 0.
  // The launchers shift every tensor pointer by tok0 tokens and use Nrow as the row stride, so the
  // kernels see an ordinary sequence; kept positions (idx) stay positions in the whole row.
  int Nrow, tok0, Wtot, woff;
  // Scoring only: value added to the positions written to idx (tok0 unless the rows are a ring buffer)
  // and distance in tokens from window w to window w+1 (L unless the rows are a ring buffer).
  int emit_off, win_stride;
  // Packed batches, host only: the boundaries (valid during the call) and number of sequences (0: one sequence).
  const int32_t* cu;
  int n_seqs;
  int has_o_res;   // the caller gave a buffer for the rounding remainder of O (lrsa_params_t::o_residual)
};

// Sequence s of a packed batch (cu = boundaries, n_seqs + 1 entries) as a Geom of its own.
void seq_geom(const Geom& whole, const int32_t* cu, int n_seqs, int s, int woff, Geom* out);

// Validates `p` and fills `g`. Returns an lrsa_status.
int make_geom(const lrsa_params_t* p, Geom* g);

constexpr int kSms = 148;   // of a B200; used in the rules that choose between forms (what a cluster finds room in is asked: ClusterRoom)

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Workspace header (first 256 bytes of every workspace).
struct WsHeader {
  int status;   // lrsa_status written by kernels (0 or LRSA_ERR_TIMEOUT)
  int ticket;   // dynamic work counter of the scoring kernel
  int pad[62];
};
static_assert(sizeof(WsHeader) == 256, "header is 256 bytes");

// Number of leading windows that query chunk c sees only through their kept tokens.
__host__ __device__ inline int n_hist_windows(int c, int ndp, int Wsel) {
  int n = c - ndp;
  if (n < 0) n = 0;
  return n < Wsel ? n : Wsel;
}

// First chunk that sees window w compressed (C if none): smallest c with n_hist_windows(c) > w.
__host__ __device__ inline int first_compressed_chunk(int w, int ndp, int Wsel, int C) {
  if (w >= Wsel) return C;
  int c = w + 1 + ndp;
  return c < C ? c : C;
}

// NVTX range around an entry point (visible in a timeline profiler; free when no tool is attached).
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

struct LaunchCounter {
  int n = 0;
};
LaunchCounter& launch_counter();

// lrsa_api.cu : scores and selects every sequence of the row; the status word of `ws` is cleared by the first launch.
int run_score_select(const Geom& whole, const __nv_bfloat16* K, const __nv_bfloat16* V,
                     int32_t* idx, float* score, void* ws, cudaStream_t st);

// score_select.cu : scores and selects the windows of n sequences of a packed row (or one sequence).  The status header of
// `ws` is cleared by the caller, or (clear_status) by the kernel.
size_t score_select_ws_bytes(const Geom& g);
int launch_score_select(const Geom* gs, int n, const __nv_bfloat16* K, const __nv_bfloat16* V, int32_t* idx,
                        float* score, void* ws, cudaStream_t st, bool clear_status);
// True when the kernel that scores `g` can clear the status word itself (clear_status above).
bool score_select_clears_status(const Geom& g);
void set_unit_wait_limit(int polls);

// attn_ref.cu : CUDA-core reference kernels (one warp per row), used for validation.
size_t attn_ref_fwd_ws_bytes(const Geom& g);
size_t attn_ref_bwd_ws_bytes(const Geom& g);
int launch_attn_ref_fwd(const Geom& g, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                        const __nv_bfloat16* V, const int32_t* idx, __nv_bfloat16* O, float* LSE,
                        void* ws, cudaStream_t st);
int launch_attn_ref_bwd(const Geom& g, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                        const __nv_bfloat16* V, const __nv_bfloat16* O, const __nv_bfloat16* dO,
                        const float* LSE, const int32_t* idx, __nv_bfloat16* dQ, __nv_bfloat16* dK,
                        __nv_bfloat16* dV, void* ws, cudaStream_t st);

// attn_fwd_sm100.cu : tcgen05 / TMEM forward (workspace: header + compact K/V).
// (*_ws_bytes: what a call of this geometry uses; *_ws_bound: enough for every packing of rows of this shape)
size_t attn_fwd_ws_bytes(const Geom& g);
size_t attn_fwd_ws_bound(const Geom& g);
int launch_attn_fwd_sm100(const lrsa_params_t* params, const Geom& g, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                          const __nv_bfloat16* V, const int32_t* idx, __nv_bfloat16* O, float* LSE,
                          void* ws, cudaStream_t st);

// attn_bwd_*_sm100.cu : tcgen05 / TMEM backward.
size_t attn_bwd_ws_bytes(const Geom& g);
size_t attn_bwd_ws_bound(const Geom& g);
int launch_attn_bwd_sm100(const lrsa_params_t* params, const Geom& g, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                          const __nv_bfloat16* V, const __nv_bfloat16* O, const __nv_bfloat16* dO,
                          const float* LSE, const int32_t* idx, __nv_bfloat16* dQ, __nv_bfloat16* dK,
                          __nv_bfloat16* dV, void* ws, cudaStream_t st);
// Launch (in clusters of `cluster` CTAs) that may start before the kernel in front of it has ended: the kernel itself waits
// for that (griddepcontrol.wait) before it reads or writes memory; in front of that it may at most bring lines that it will read into
// L2 (a hint: they are read behind the wait, from L2 where all writes meet).  Memory that the kernel in front may have written is not read-only for
// such a kernel's lifetime: plain loads (or __ldcg), no __ldg and no __restrict__, which the compiler may also move ahead of the wait.
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// lrsa_api.cu : clusters of 2^c CTAs that the device runs at a time with 2^p CTAs on an SM, n[p][c].
struct ClusterRoom {
  int n[3][5];
  int at_once(int per_sm, int cluster) const {
    int p = 0, c = 0;
    while ((1 << p) < per_sm) ++p;
    while ((1 << c) < cluster) ++c;
    return n[p][c];
  }
};
const ClusterRoom& cluster_room();

#define LRSA_CUDA_CHECK(expr)                                 \
  do {                                                        \
    cudaError_t _e = (expr);                                  \
    if (_e != cudaSuccess) return (int)LRSA_ERR_CUDA;         \
  } while (0)

}  // namespace lrsa
