// Stateless operator entry points of include/atspeed.h (GEMM, SwiGLU GEMM, RMSNorm, tree attention)
// on caller-owned device buffers.  Used by the parity tests and by callers composing their own loop.
#include <cuda.h>
#include <cuda_runtime.h>

#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "atspeed.h"
#include "attention.cuh"
#include "gemm.cuh"
#include "common.cuh"
#include "kernels.cuh"

using namespace atspeed;

namespace {

int current_grid() {
  int dev = 0;
  cudaGetDevice(&dev);
  return gemm_grid_size(dev);
}

GemmScratch scratch_from(void* ws, int G) {
  GemmScratch s;
  s.ws = static_cast<float*>(ws);
  s.ws_bytes = gemm_ws_bytes(G);
  s.counters = reinterpret_cast<int*>(static_cast<char*>(ws) + s.ws_bytes);
  s.max_tiles = gemm_max_tiles();
  s.err = reinterpret_cast<unsigned int*>(static_cast<char*>(ws) + s.ws_bytes + (size_t)s.max_tiles * 4);
  return s;
}

// gemm_launch result -> status: a refused shape is E_SHAPE, an operand the tensor-map encoder
// refuses (misaligned base address) is E_ARG, any other launch failure is E_CUDA.
atspeed_status gemm_status(cudaError_t e) {
  if (e == cudaSuccess) return ATSPEED_OK;
  if (e == cudaErrorInvalidValue) return ATSPEED_E_SHAPE;
  if (e == kGemmMapError) return ATSPEED_E_ARG;
  return ATSPEED_E_CUDA;
}

atspeed_status run_gemm(cudaStream_t st, const GemmArgs& a, void* ws) {
  if (!ws) return ATSPEED_E_ARG;
  char eb[256];
  const int grid = current_grid();
  const GemmScratch s = scratch_from(ws, grid);
  if (gemm_cluster_fits(a, grid)) return gemm_status(gemm_cluster_launch(a, s.err, grid, st, eb, sizeof eb));
  return gemm_status(gemm_pair_launch(a, s, grid, st, eb, sizeof eb));
}

// CTAs (prefix splits) per (query tile, head) of the attention operator, 1, 2 or 4, and the pages of a split.
//
// Up to 256 tokens, where a row of the GEMMs does not depend on the call's other tokens, a query's result does
// not either: the splits' boundaries come from the prefix, the number of heads and whether there are path keys.
// As many as run at once (three CTAs per SM) for 128 queries, of a short prefix for 256.  One CTA without path
// keys writes its rows directly, so a short prefix is not split then.  us of kernel, 1 / 2 / 4 CTAs, 32 heads of
// 128 with path keys: 128 queries, 2 pages 13.4 / 10.3 / -, 4 pages - / 11.9 / 13.1, 8 pages 21.8 / 14.4 / 14.6; 10
// queries, 8 pages - / 14.9 / 11.0; 200 queries, 4 pages - / 14.7 / 21.2, 8 pages - / 18.5 / 25.4 (the boundaries of 128
// queries cost most there); 4 heads of 32, 4 pages, 120 queries - / 8.5 / 6.2; no path keys: 250 queries, 4 pages
// 9.3 / 13.3 / 22.4.
//
// More tokens: as many as run at once and leave each CTA pages enough, the pages each tile sees balanced over
// them (pages = 0).  us, 1 / 2 / 4 CTAs, 128-wide heads: 256 pairs of 8 pages with path keys 26.6 / 32.7 / 42.0,
// causal without 17.5 / 22.2 / 36.8; 64-wide heads: 72 of 6 8.6 / 8.5 / 8.0, 192 of 16 19.6 / 16.9 / 19.5.
struct AttnSplits {
  int n, pages;
};
AttnSplits attention_splits(int T, int n_heads, int pages, bool paths, int sms) {
  const long long room = 3LL * sms;
  if (T <= 256) {
    int n = pages > 4 || (pages > 2 && 16LL * n_heads <= room) ? 4 : pages > 1 ? 2 : 1;
    if (!paths && pages < 8) n = 1;
    while (n > 1 && 2LL * n * n_heads > room) n /= 2;
    return {n, std::max(1, (pages + n - 1) / n)};
  }
  const long long pairs = (long long)((T + ATT_QTILE - 1) / ATT_QTILE) * n_heads;
  const int least4 = paths ? (8 * pairs <= room ? 4 : 8) : 4 * pairs <= sms ? 4 : 6;
  if (4 * pairs <= room && pages >= least4) return {4, 0};
  return {2 * pairs <= room && pages >= (paths ? 2 : 8) ? 2 : 1, 0};
}

// ---------------------------------------------------------------------------------------------
// Allocation-free GEMM: its split-K scratch lives in a fixed device array of this library.
// ---------------------------------------------------------------------------------------------
constexpr int kNoAllocGrid = 32;        // CTAs of the persistent grid (caps the workspace)
constexpr int kNoAllocTiles = 4096;     // output tiles (128 weight rows x up to 256 tokens)
constexpr size_t kNoAllocWsBytes = (size_t)2 * kNoAllocGrid * 256 * 128 * sizeof(float);  // 8 MiB
constexpr size_t kNoAllocBytes = kNoAllocWsBytes + (size_t)kNoAllocTiles * sizeof(int) + 256;

// One copy per GPU that loads the library, held until the process exits.  Host code must not use
// this name as an address: the device address comes from cudaGetSymbolAddress (per device).
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

std::mutex g_noalloc_mu;
void* g_noalloc_ptr[64] = {nullptr};

// Device address of the allocation-free scratch on the current device, looked up on first use.
void* noalloc_base() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return nullptr;
    g_noalloc_ptr[dev] = ptr;
  }
  return g_noalloc_ptr[dev];
}

unsigned int* noalloc_err_word(void* base) {
  return reinterpret_cast<unsigned int*>(static_cast<char*>(base) + kNoAllocWsBytes + (size_t)kNoAllocTiles * 4);
}

}  // namespace

extern "C" {

size_t atspeed_op_workspace_bytes(void) {
  return gemm_ws_bytes(current_grid()) + (size_t)gemm_max_tiles() * 4 + 256;
}

atspeed_status atspeed_op_gemm(atspeed_stream stream, const void* d_W, const void* d_X, int M, int K, int T, int x_rows,
                               float* d_Y, int ldy, int accumulate, void* d_ws) {
  if (!d_W || !d_X || !d_Y || M <= 0 || K <= 0 || T <= 0 || ldy < M) return ATSPEED_E_ARG;
  GemmArgs a = {};
  a.epi = accumulate ? EPI_RESID : EPI_F32;
  a.W = static_cast<const __nv_bfloat16*>(d_W);
  a.X = static_cast<const __nv_bfloat16*>(d_X);
  a.M = M;
  a.K = K;
  a.T = T;
  a.X_rows = x_rows;
  a.out_f32 = d_Y;
  a.ldo = ldy;
  return run_gemm((cudaStream_t)stream, a, d_ws);
}

atspeed_status atspeed_op_gemm_swiglu(atspeed_stream stream, const void* d_W, const void* d_X, int F, int K, int T,
                                      int x_rows, void* d_out, int ldo, void* d_ws) {
  // the epilogue stores two adjacent bf16 outputs at once: ldo even, d_out 4-byte aligned
  if (!d_W || !d_X || !d_out || F <= 0 || K <= 0 || T <= 0 || ldo < F || (ldo & 1) ||
      (reinterpret_cast<uintptr_t>(d_out) & 3))
    return ATSPEED_E_ARG;
  GemmArgs a = {};
  a.epi = EPI_SWIGLU;
  a.W = static_cast<const __nv_bfloat16*>(d_W);
  a.X = static_cast<const __nv_bfloat16*>(d_X);
  a.M = 2 * F;
  a.K = K;
  a.T = T;
  a.X_rows = x_rows;
  a.out_bf16 = static_cast<__nv_bfloat16*>(d_out);
  a.ldo = ldo;
  return run_gemm((cudaStream_t)stream, a, d_ws);
}

atspeed_status atspeed_op_rmsnorm(atspeed_stream stream, const float* d_h, const void* d_g, int T, int d, float eps,
                                  void* d_x, int ldx) {
  if (!d_h || !d_g || !d_x || T <= 0 || d <= 0 || ldx < d) return ATSPEED_E_ARG;
  const cudaError_t e = rmsnorm_launch(d_h, static_cast<const __nv_bfloat16*>(d_g), T, d, eps,
                                       static_cast<__nv_bfloat16*>(d_x), ldx, (cudaStream_t)stream);
  return e == cudaSuccess ? ATSPEED_OK : ATSPEED_E_CUDA;
}

size_t atspeed_op_attention_scratch(int T, int n_heads, int head_dim, int P) {
  (void)n_heads;
  (void)head_dim;
  AttnArgs a = {};   // the call's tables (used where they are more than kernel parameters hold)
  a.T = T;
  a.n_qtiles = (T + ATT_QTILE - 1) / ATT_QTILE;
  a.max_pages = std::max(1, (P + ATT_PAGE - 1) / ATT_PAGE);
  return attn_tables(a, nullptr, true) * sizeof(int);
}

atspeed_status atspeed_op_attention(atspeed_stream stream, const void* d_q, const void* d_kcache, const void* d_vcache,
                                    int cache_rows, int T, int n_heads, int head_dim, int P, const int32_t* h_pages,
                                    const int32_t* h_vis, const int32_t* h_path_rows, const int32_t* h_n_path,
                                    void* d_out, void* d_part) {
  if (!d_q || !d_kcache || !d_vcache || !d_out || !d_part || !h_pages || !h_vis || T <= 0 || P < 0 ||
      cache_rows <= 0)
    return ATSPEED_E_ARG;
  if (head_dim != 32 && head_dim != 64 && head_dim != 128) return ATSPEED_E_SHAPE;
  cudaStream_t st = (cudaStream_t)stream;
  const int pages = (P + ATT_PAGE - 1) / ATT_PAGE;
  const int nqt = (T + ATT_QTILE - 1) / ATT_QTILE;
  for (int p = 0; p < pages; ++p)
    if (h_pages[p] < 0 || (h_pages[p] + 1) * ATT_PAGE > cache_rows) return ATSPEED_E_ARG;
  for (int t = 0; t < T; ++t) {
    if (h_vis[t] < 0 || h_vis[t] > P) return ATSPEED_E_ARG;
    const int np = h_n_path ? h_n_path[t] : 0;
    if (np < 0 || np > ATT_MAX_ANC || (np > 0 && !h_path_rows)) return ATSPEED_E_ARG;
    for (int j = 0; j < np; ++j)
      if (h_path_rows[t * 4 + j] < 0 || h_path_rows[t * 4 + j] >= cache_rows) return ATSPEED_E_ARG;
  }
  bool paths = false;
  for (int t = 0; h_n_path && t < T; ++t) paths |= h_n_path[t] > 0;
  const AttnSplits splits = attention_splits(T, n_heads, pages, paths, current_grid());
  const int S = splits.n;
  const int d = n_heads * head_dim;
  CUtensorMap mk, mv;
  char eb[256];
  if (!attn_make_maps(static_cast<const __nv_bfloat16*>(d_kcache), static_cast<const __half*>(d_vcache),
                      cache_rows, d, head_dim, &mk, &mv, eb, sizeof eb))
    return ATSPEED_E_CUDA;
  AttnArgs a = {};
  a.T = T;
  a.n_heads = n_heads;
  a.head_dim = head_dim;
  a.q = static_cast<const __nv_bfloat16*>(d_q);
  a.k_cache = static_cast<const __nv_bfloat16*>(d_kcache);
  a.v_cache = static_cast<const __half*>(d_vcache);
  a.kv_rows = cache_rows;
  a.n_qtiles = nqt;
  a.max_pages = std::max(1, pages);
  a.chunks_per_split = splits.pages;
  a.max_splits = S;
  a.out = static_cast<__nv_bfloat16*>(d_out);
  a.direct = S == 1 && !paths;
  std::vector<int> host(attn_tables(a, nullptr, paths), 0);
  AttnArgs at = a;
  attn_tables(at, host.data(), paths);
  auto put = [](const int* p) { return const_cast<int*>(p); };
  for (int i = 0; i < nqt; ++i) {
    put(at.qt_t0)[i] = i * ATT_QTILE;
    put(at.qt_n)[i] = std::min(ATT_QTILE, T - i * ATT_QTILE);
  }
  *put(at.user_splits) = S;
  for (int p = 0; p < pages; ++p) put(at.page_table)[p] = h_pages[p];
  for (int t = 0; t < T; ++t) {
    put(at.tok_vis)[t] = h_vis[t];
    put(at.qt_vis)[t / ATT_QTILE] = std::max(put(at.qt_vis)[t / ATT_QTILE], h_vis[t]);
    if (!paths) continue;
    const int na = h_n_path[t];
    put(at.anc_n)[t] = na;
    for (int j = 0; j < na; ++j) put(at.anc_row)[t * 4 + j] = h_path_rows[t * 4 + j];
  }
  const cudaError_t e = attn_cluster_launch(a, mk, mv, S, host.data(), host.size(), paths, static_cast<int*>(d_part), st);
  return e == cudaSuccess ? ATSPEED_OK : ATSPEED_E_CUDA;
}

/* See include/atspeed.h.  The device address of the scratch array is looked up once per device, on
 * that device's first call (so the first call on a device should come before any stream capture). */
atspeed_status atspeed_op_gemm_noalloc(atspeed_stream stream, const void* d_W, const void* d_X, int M, int K, int T,
                                       int x_rows, float* d_Y, int ldy, int accumulate) {
  if (!d_W || !d_X || !d_Y || M <= 0 || K <= 0 || T <= 0 || ldy < M) return ATSPEED_E_ARG;
  const int BN = T <= 128 ? 128 : 256;
  const long long tiles = (long long)((M + 127) / 128) * ((T + BN - 1) / BN);
  if (tiles > kNoAllocTiles || K % 64 != 0 || K / 64 > 256) return ATSPEED_E_SHAPE;
  void* base = noalloc_base();
  if (!base) return ATSPEED_E_CUDA;
  GemmScratch s;
  s.ws = static_cast<float*>(base);
  s.ws_bytes = kNoAllocWsBytes;
  s.counters = reinterpret_cast<int*>(static_cast<char*>(base) + kNoAllocWsBytes);
  s.max_tiles = kNoAllocTiles;
  s.err = noalloc_err_word(base);
  // the tile counters must start at zero (a call that failed part-way could have left some set);
  // the error word after them is left alone: it is sticky until atspeed_op_status reads it
  if (cudaMemsetAsync(s.counters, 0, (size_t)kNoAllocTiles * sizeof(int), (cudaStream_t)stream) != cudaSuccess)
    return ATSPEED_E_CUDA;
  GemmArgs a = {};
  a.epi = accumulate ? EPI_RESID : EPI_F32;
  a.W = static_cast<const __nv_bfloat16*>(d_W);
  a.X = static_cast<const __nv_bfloat16*>(d_X);
  a.M = M;
  a.K = K;
  a.T = T;
  a.X_rows = x_rows;
  a.out_f32 = d_Y;
  a.ldo = ldy;
  char eb[256];
  return gemm_status(gemm_launch(a, s, kNoAllocGrid, kNoAllocGrid, (cudaStream_t)stream, false, eb, sizeof eb));
}

/* See include/atspeed.h.  Reads (and clears) the error words that the operators' bounded waits set. */
atspeed_status atspeed_op_status(atspeed_stream stream, void* d_ws) {
  unsigned int* words[2] = {nullptr, nullptr};
  if (d_ws) {
    words[0] = scratch_from(d_ws, current_grid()).err;
  } else {
    void* base = noalloc_base();
    words[1] = attn_err_word();
    if (!base || !words[1]) return ATSPEED_E_CUDA;
    words[0] = noalloc_err_word(base);
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaStreamSynchronize(st) != cudaSuccess) return ATSPEED_E_CUDA;
  unsigned int all = 0;
  for (unsigned int* word : words) {
    unsigned int v = 0;
    if (!word) continue;
    if (cudaMemcpy(&v, word, sizeof v, cudaMemcpyDeviceToHost) != cudaSuccess) return ATSPEED_E_CUDA;
    if (v != 0 && cudaMemset(word, 0, sizeof v) != cudaSuccess) return ATSPEED_E_CUDA;
    all |= v;
  }
  if (all == 0) return ATSPEED_OK;
  return (all & ATSPEED_DEV_ERR_TIMEOUT) ? ATSPEED_E_TIMEOUT : ATSPEED_E_CUDA;
}

}  // extern "C"
