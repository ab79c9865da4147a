// Embedding gather and RMSNorm (LLaMA pre-norm).  (The decoder forward uses embed_rows for layer 0 and
// folds every other norm into its GEMMs; rmsnorm serves the operator API.)
//   h[t] = embed[token[t]]                      (fp32 residual stream; the table is bf16)
//   x[t] = bf16( h[t] / sqrt(mean(h[t]^2) + eps) * g )
#include "common.cuh"
#include "kernels.cuh"
#include "norm_core.cuh"

namespace atspeed {

// RMSNorm of T rows, TPR threads per row (one warp, or the whole CTA of 256), each holding up to NV
// float4 of the row in registers, so a row is read once and written once.
// Bound: HBM (6 bytes per element, read 4 + write 2).  With two passes over the row (the second through
// L2) and 2-byte stores, 2501 rows of 4096 took 21.4 us (2.9 TB/s); one pass with 16-byte loads and
// 8-byte stores: 12.4 us (5.0 TB/s).
template <int TPR, int NV>
__global__ void __launch_bounds__(256) rmsnorm_kernel(const float* __restrict__ h, const __nv_bfloat16* __restrict__ g,
                                                      int T, int d, float eps, __nv_bfloat16* __restrict__ x, int ldx) {
  static_assert(TPR == 32 || TPR == 256, "a row is one warp's or one CTA's");
  const int t = TPR == 32 ? blockIdx.x * 8 + (threadIdx.x >> 5) : blockIdx.x;
  if (t >= T) return;
  const int tid = threadIdx.x & (TPR - 1), nc = d >> 2;
  const float4* h4 = reinterpret_cast<const float4*>(h + (size_t)t * d);
  float4 v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int c = tid + TPR * k;
    v[k] = c < nc ? __ldcs(h4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < NV; ++k) ss += (v[k].x * v[k].x + v[k].y * v[k].y) + (v[k].z * v[k].z + v[k].w * v[k].w);
  ss = warp_sum(ss);
  if constexpr (TPR > 32) {
    __shared__ float red[8];
    if ((tid & 31) == 0) red[tid >> 5] = ss;
    __syncthreads();
    ss = rms_total(red);
  }
  const float r = 1.0f / sqrtf(ss / (float)d + eps);
  __nv_bfloat16* xr = x + (size_t)t * ldx;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int c = tid + TPR * k;
    if (c >= nc) break;
    const uint2 graw = __ldg(reinterpret_cast<const uint2*>(g) + c);
    const __nv_bfloat162* gb = reinterpret_cast<const __nv_bfloat162*>(&graw);
    const float2 g0 = __bfloat1622float2(gb[0]), g1 = __bfloat1622float2(gb[1]);
    __nv_bfloat162 o[2];
    o[0] = __floats2bfloat162_rn(v[k].x * r * g0.x, v[k].y * r * g0.y);
    o[1] = __floats2bfloat162_rn(v[k].z * r * g1.x, v[k].w * r * g1.y);
    *reinterpret_cast<uint2*>(xr + 4 * c) = *reinterpret_cast<const uint2*>(o);
  }
}

// Any width and alignment: two passes over the row, one value at a time.
__global__ void __launch_bounds__(256) rmsnorm_any_kernel(const float* __restrict__ h,
                                                          const __nv_bfloat16* __restrict__ g, int d, float eps,
                                                          __nv_bfloat16* __restrict__ x, int ldx) {
  const float* hr = h + (size_t)blockIdx.x * d;
  __shared__ float red[8];
  float ss = 0.f;
  for (int i = threadIdx.x; i < d; i += 256) ss += hr[i] * hr[i];
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  const float r = 1.0f / sqrtf(rms_total(red) / (float)d + eps);
  for (int i = threadIdx.x; i < d; i += 256)
    x[(size_t)blockIdx.x * ldx + i] = __float2bfloat16_rn(hr[i] * r * __bfloat162float(g[i]));
}

// Layer 0's input rows: h[t] = embed[token[t]], xg[t] = bf16(g * h[t]) and the partial sums of
// squares per 128-row tile (the first norm's scale is applied by the QKV epilogue).
__global__ void __launch_bounds__(256) embed_rows_kernel(const int* __restrict__ tokens,
                                                         const __nv_bfloat16* __restrict__ embed,
                                                         const __nv_bfloat16* __restrict__ g, float* __restrict__ h,
                                                         __nv_bfloat16* __restrict__ xg, float* __restrict__ ssq,
                                                         int ld, int d) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x;
  embed_row(embed + (size_t)tokens[t] * d, g, h + (size_t)t * d, xg + (size_t)t * d, ssq, ld, t, d, threadIdx.x,
            blockDim.x);
}

cudaError_t embed_rows_launch(const int* tokens, const __nv_bfloat16* embed, const __nv_bfloat16* g, float* h,
                              __nv_bfloat16* xg, float* ssq, int ld, int T, int d, cudaStream_t st, bool pdl) {
  if (T <= 0) return cudaSuccess;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(T);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, embed_rows_kernel, tokens, embed, g, h, xg, ssq, ld, d);
}

cudaError_t rmsnorm_launch(const float* h, const __nv_bfloat16* g, int T, int d, float eps, __nv_bfloat16* x, int ldx,
                           cudaStream_t st) {
  if (T <= 0) return cudaSuccess;
  const auto aligned = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; };
  // (launch failures come back from the launch itself)
  const auto launch = [&](auto kernel, int blocks, auto... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
  };
  // The one-pass kernels move four values at once and hold a row in at most 8 float4 per thread; other
  // widths and alignments take the general kernel.
  if (d % 4 || ldx % 4 || d > 8192 || !aligned(h, 16) || !aligned(g, 8) || !aligned(x, 8))
    return launch(rmsnorm_any_kernel, T, h, g, d, eps, x, ldx);
  // one warp per row while the row fits its registers (1024 values), else one CTA per row
  const int rows8 = T / 8 + (T % 8 != 0);
  if (d <= 256) return launch(rmsnorm_kernel<32, 2>, rows8, h, g, T, d, eps, x, ldx);
  if (d <= 1024) return launch(rmsnorm_kernel<32, 8>, rows8, h, g, T, d, eps, x, ldx);
  if (d <= 4096) return launch(rmsnorm_kernel<256, 4>, T, h, g, T, d, eps, x, ldx);
  return launch(rmsnorm_kernel<256, 8>, T, h, g, T, d, eps, x, ldx);
}

}  // namespace atspeed
