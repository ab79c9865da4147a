// Shared-prefix tree attention: TMA-staged K/V pages, tensor cores (mma.sync m16n8k16: bf16 Q K^T; P V in
// fp16, with P rounded to fp16 once, 2^-11 of a weight, and V exact) with an fp32 online softmax, prefix split
// across CTAs.  The one-kernel-per-op schedule's prefix kernel leaves the splits to a combine kernel, which
// merges them with each node's path keys (ancestors + self, at most 4); the operator's kernel does both, with
// the splits of a tile in one cluster.
#include <cudaTypedefs.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "attention.cuh"
#include "attn_core.cuh"
#include "common.cuh"

namespace atspeed {

namespace {

constexpr int ATT_OP_BUFS = 3;   // K/V buffers of an item

template <int HD>
__global__ void __launch_bounds__(128)
    attn_prefix_kernel(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                       const AttnArgs a) {
  using C = AttCfg<HD, ATT_OP_BUFS>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::SMEM_BODY);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) {
    for (int b = 0; b < ATT_OP_BUFS; ++b) mbar_init(&bars[b], 1);
    fence_mbar_init();
    tma_prefetch_desc(&mk);
    tma_prefetch_desc(&mv);
  }
  __syncthreads();
  uint32_t par = 0;
  attn_item<HD, ATT_OP_BUFS>(a, &mk, &mv, blockIdx.x, blockIdx.y, blockIdx.z, smem, bars, par, threadIdx.x, 1);
}

// One CTA of 128 threads per (query tile, head, group of 16 queries): merge the prefix splits with
// the path keys.
template <int HD>
__global__ void __launch_bounds__(128) attn_combine_kernel(const AttnArgs a) {
  pdl_launch_dependents();
  pdl_wait();
  attn_combine_group<HD>(a, blockIdx.x, blockIdx.y, blockIdx.z, threadIdx.x, []() { return true; });
}

// ---- the operator's attention: one kernel, the prefix splits of a (query tile, head) in one cluster
// S CTAs (1, 2 or 4) share the prefix's pages (ranges that do not depend on the tile, or the tile's visible pages
// evenly: chunks_per_split); their partials (o, m, l) meet in distributed shared memory -- 16-query group g
// belongs to CTA g mod S, every CTA stores its rows of the group there -- and the owner merges them with the
// queries' path keys.  Against the two kernels above (partials through global memory, splits of two pages, most
// of them empty for the early tiles of a causal prefill): causal 1000 tokens x 32 heads of 128 61 + 30 us
// before, 38 now, the call 106 -> 40 us; a tree of 120 tokens over 512 keys 65 -> 36 us a call (host-bound: the
// kernel takes 14.6).
// Bound: latency for few queries (Q, K/V and path-key round trips); for many, a step's shared-memory
// reads (every warp reads the whole K/V tile through ldmatrix) and its MMAs, which take about as long.
template <int HD>
struct AttClusterCfg {
  static constexpr int LD = HD + 4;                          // floats per query row of a slot
  static constexpr int SLOT = ATT_CQ * LD + 2 * ATT_CQ;      // o rows, then (m, l)
  static constexpr int RING = AttCfg<HD, ATT_OP_BUFS>::SMEM_BODY;
  static constexpr int BODY = 4 * SLOT * 4 > RING ? 4 * SLOT * 4 : RING;
  static constexpr int SMEM = 1024 + BODY + 64;
};

template <int HD>
struct AttClusterSink {
  static constexpr bool kCustom = true;
  uint8_t* smem;
  int S, rank, tid;
  __device__ __forceinline__ void operator()(const float (&o)[HD / 8][4], float m_a, float l_a, float m_b,
                                             float l_b) const {
    using CC = AttClusterCfg<HD>;
    if (S > 1)
      cluster_sync();   // every CTA's K/V ring is idle: it may receive partials
    else
      __syncthreads();
    const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
    // warp w holds group w: its owner's slot (group's index there, this CTA)
    float* slot = reinterpret_cast<float*>(smem) + (size_t)((warp / S) * S + rank) * CC::SLOT;
    const uint32_t dst = S > 1 ? mapa_u32(slot, (uint32_t)(warp % S)) : smem_u32(slot);
#pragma unroll
    for (int j = 0; j < HD / 8; ++j) {
      const int col = j * 8 + tq * 2;
      st2(dst + (uint32_t)(g * CC::LD + col) * 4, o[j][0], o[j][1]);
      st2(dst + (uint32_t)((g + 8) * CC::LD + col) * 4, o[j][2], o[j][3]);
    }
    if (tq == 0) {
      st2(dst + (uint32_t)(ATT_CQ * CC::LD + 2 * g) * 4, m_a, l_a);
      st2(dst + (uint32_t)(ATT_CQ * CC::LD + 2 * (g + 8)) * 4, m_b, l_b);
    }
  }
  static __device__ __forceinline__ void st2(uint32_t addr, float a, float b) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
  }
};

// Set by a bounded wait of the operator's kernel that gave up; sticky until atspeed_op_status reads it.
__device__ unsigned int g_attn_err;

// The call's tables in the kernel's parameters (NTAB ints), or in memory (NTAB = 0).
template <int NTAB>
struct AttTables {
  int v[NTAB > 0 ? NTAB : 1];
};

template <int HD, int NTAB>
__global__ void __launch_bounds__(128, 3)
    attn_cluster_kernel(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                        const AttnArgs args, const int S, const int paths, const __grid_constant__ AttTables<NTAB> tab) {
  AttnArgs a = args;
  a.err = &g_attn_err;
  if constexpr (NTAB > 0) attn_tables(a, tab.v, paths);
  using CC = AttClusterCfg<HD>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + CC::BODY);
  const int tid = threadIdx.x, rank = S > 1 ? (int)cluster_ctarank() : 0;
  // the last tiles first: in a causal prefill they see the most keys
  const int pair = blockIdx.x / S, h = pair % a.n_heads, tile = a.n_qtiles - 1 - pair / a.n_heads;
  if (tid == 0) {
    for (int b = 0; b < ATT_OP_BUFS; ++b) mbar_init(&bars[b], 1);
    fence_mbar_init();
    tma_prefetch_desc(&mk);
    tma_prefetch_desc(&mv);
  }
  __syncthreads();
  uint32_t par = 0;
  if (a.direct) {   // one split, no path keys: straight to the output
    attn_item<HD, ATT_OP_BUFS>(a, &mk, &mv, tile, h, 0, smem, bars, par, tid, 1);
    return;
  }
  const AttClusterSink<HD> sink{smem, S, rank, tid};
  const bool ok =
      attn_item<HD, ATT_OP_BUFS, AttClusterSink<HD>>(a, &mk, &mv, tile, h, rank, smem, bars, par, tid, 1, nullptr, 0, sink);
  if (!ok && S > 1) cluster_sync();   // (a failed wait: the sink's barrier still has to be met)
  if (S > 1)
    cluster_sync();   // the partials are in place
  else
    __syncthreads();
  if (!ok) return;

  // merge: eight threads per query, HD / 8 consecutive dimensions each
  constexpr int DH = HD / 8;
  const int part = tid & 7, d = a.n_heads * HD, dim0 = h * HD + part * DH;
  const float scale = kLog2e / sqrtf((float)HD);
  const int t0 = a.qt_t0[tile], nq = a.qt_n[tile];
  for (int g = rank; g * ATT_CQ < nq; g += S) {
    const int ql = tid >> 3, t = t0 + g * ATT_CQ + ql;
    const bool active = g * ATT_CQ + ql < nq;
    const int tc = active ? t : t0;
    const int na = a.anc_n && active ? a.anc_n[tc] : 0;
    int arow[ATT_MAX_ANC];
#pragma unroll
    for (int j = 0; j < ATT_MAX_ANC; ++j) arow[j] = na > 0 ? a.anc_row[tc * ATT_MAX_ANC + j] : 0;
    __nv_bfloat16 qb[DH], kb[ATT_MAX_ANC][DH];
    __half vb[ATT_MAX_ANC][DH];
#pragma unroll
    for (int i = 0; i < DH; i += 4) *reinterpret_cast<uint2*>(qb + i) = *reinterpret_cast<const uint2*>(a.q + (size_t)tc * d + dim0 + i);
#pragma unroll
    for (int j = 0; j < ATT_MAX_ANC; ++j)
      if (j < na) {
#pragma unroll
        for (int i = 0; i < DH; i += 4) {
          *reinterpret_cast<uint2*>(kb[j] + i) = *reinterpret_cast<const uint2*>(a.k_cache + (size_t)arow[j] * d + dim0 + i);
          *reinterpret_cast<uint2*>(vb[j] + i) = *reinterpret_cast<const uint2*>(a.v_cache + (size_t)arow[j] * d + dim0 + i);
        }
      }
    const float* slots = reinterpret_cast<const float*>(smem) + (size_t)(g / S) * S * CC::SLOT;
    float M = -INFINITY, sa[ATT_MAX_ANC];
    for (int s = 0; s < S; ++s) M = fmaxf(M, slots[s * CC::SLOT + ATT_CQ * CC::LD + 2 * ql]);
#pragma unroll
    for (int j = 0; j < ATT_MAX_ANC; ++j) {
      float pd = 0.f;
      if (j < na) {
#pragma unroll
        for (int i = 0; i < DH; ++i) pd += __bfloat162float(qb[i]) * __bfloat162float(kb[j][i]);
      }
      pd += __shfl_xor_sync(0xffffffffu, pd, 1);
      pd += __shfl_xor_sync(0xffffffffu, pd, 2);
      pd += __shfl_xor_sync(0xffffffffu, pd, 4);
      sa[j] = pd * scale;
      if (j < na) M = fmaxf(M, sa[j]);
    }
    const float Mu = (M == -INFINITY) ? 0.f : M;
    float L = 0.f, o[DH];
#pragma unroll
    for (int i = 0; i < DH; ++i) o[i] = 0.f;
    for (int s = 0; s < S; ++s) {
      const float* sl = slots + s * CC::SLOT;
      const float w = exp2f(sl[ATT_CQ * CC::LD + 2 * ql] - Mu);
      L += sl[ATT_CQ * CC::LD + 2 * ql + 1] * w;
      const float4* po = reinterpret_cast<const float4*>(sl + ql * CC::LD + part * DH);
#pragma unroll
      for (int i = 0; i < DH / 4; ++i) {
        const float4 v = po[i];
        o[4 * i] += v.x * w;
        o[4 * i + 1] += v.y * w;
        o[4 * i + 2] += v.z * w;
        o[4 * i + 3] += v.w * w;
      }
    }
#pragma unroll
    for (int j = 0; j < ATT_MAX_ANC; ++j)
      if (j < na) {
        const float w = exp2f(sa[j] - Mu);
        L += w;
#pragma unroll
        for (int i = 0; i < DH; ++i) o[i] += w * __half2float(vb[j][i]);
      }
    if (!active) continue;
    const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
    for (int i = 0; i < DH; i += 2)
      *reinterpret_cast<__nv_bfloat162*>(a.out + (size_t)t * d + dim0 + i) =
          __floats2bfloat162_rn(o[i] * inv, o[i + 1] * inv);
  }
}

template <int HD, int NTAB>
cudaError_t launch_cluster(AttnArgs& a, const CUtensorMap& mk, const CUtensorMap& mv, int S, const int* tables,
                           size_t n, bool paths, int* d_tables, cudaStream_t st) {
  using CC = AttClusterCfg<HD>;
  static std::atomic<unsigned long long> attr_done{0};
  cudaError_t e = smem_attr_once(attr_done, attn_cluster_kernel<HD, NTAB>, CC::SMEM);
  if (e != cudaSuccess) return e;
  AttTables<NTAB> tab;
  if constexpr (NTAB > 0) {
    memcpy(tab.v, tables, n * sizeof(int));
  } else {
    e = cudaMemcpyAsync(d_tables, tables, n * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    attn_tables(a, d_tables, paths);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.n_qtiles * a.n_heads * S));
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = CC::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)S;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = S > 1 ? 1 : 0;
  int with_paths = paths;
  void* kargs[] = {const_cast<CUtensorMap*>(&mk), const_cast<CUtensorMap*>(&mv), &a, &S, &with_paths, &tab};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(attn_cluster_kernel<HD, NTAB>), kargs);
}

template <int HD>
cudaError_t launch_cluster_hd(AttnArgs& a, const CUtensorMap& mk, const CUtensorMap& mv, int S, const int* tables,
                              size_t n, bool paths, int* d_tables, cudaStream_t st) {
  // Tables as kernel parameters (32,764 bytes at most): no copy ahead of the kernel.  Two sizes, since the
  // whole parameter block is copied at the launch.  120 tree tokens of 32 heads (740 ints), us per call:
  // through memory 39, 7680 ints 38, 1984 ints 34-36; 1000 prefill tokens (1081 ints): 44 -> 39.
  if (n <= 1984) return launch_cluster<HD, 1984>(a, mk, mv, S, tables, n, paths, d_tables, st);
  if (n <= 7680) return launch_cluster<HD, 7680>(a, mk, mv, S, tables, n, paths, d_tables, st);
  return launch_cluster<HD, 0>(a, mk, mv, S, tables, n, paths, d_tables, st);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn_att() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  }
  return fn;
}

template <int HD>
cudaError_t launch_hd(const AttnArgs& a, const CUtensorMap& mk, const CUtensorMap& mv, cudaStream_t st, bool pdl) {
  using C = AttCfg<HD, ATT_OP_BUFS>;
  static std::atomic<unsigned long long> attr_done{0};
  {
    const cudaError_t e = smem_attr_once(attr_done, attn_prefix_kernel<HD>, C::SMEM);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.n_qtiles, a.n_heads, a.max_splits);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaError_t e = cudaLaunchKernelEx(&cfg, attn_prefix_kernel<HD>, mk, mv, a);
  if (e != cudaSuccess || a.direct) return e;
  cudaLaunchConfig_t c2 = {};
  c2.gridDim = dim3(a.n_qtiles, a.n_heads, ATT_QTILE / ATT_CQ);
  c2.blockDim = dim3(128);
  c2.stream = st;
  c2.attrs = at;
  c2.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&c2, attn_combine_kernel<HD>, a);
}

}  // namespace

bool attn_make_maps(const __nv_bfloat16* k_cache, const __half* v_cache, int rows, int d_model, int head_dim,
                    CUtensorMap* mk, CUtensorMap* mv, char* eb, size_t el) {
  auto fn = encode_fn_att();
  if (!fn) {
    snprintf(eb, el, "cuTensorMapEncodeTiled unavailable");
    return false;
  }
  const int boxw = head_dim >= 64 ? 64 : head_dim;
  cuuint64_t dims[2] = {(cuuint64_t)d_model, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)d_model * 2};
  cuuint32_t box[2] = {(cuuint32_t)boxw, (cuuint32_t)ATT_SUB};
  cuuint32_t es[2] = {1, 1};
  const CUtensorMapSwizzle sw = head_dim >= 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE;
  for (int i = 0; i < 2; ++i) {
    CUresult r = fn(i == 0 ? mk : mv, i == 0 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                    i == 0 ? (void*)k_cache : (void*)v_cache, dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      snprintf(eb, el, "attention tensor map failed (%d)", (int)r);
      return false;
    }
  }
  return true;
}

cudaError_t attn_launch(const AttnArgs& a, const CUtensorMap& mk, const CUtensorMap& mv, cudaStream_t st, bool pdl) {
  switch (a.head_dim) {
    case 32: return launch_hd<32>(a, mk, mv, st, pdl);
    case 64: return launch_hd<64>(a, mk, mv, st, pdl);
    case 128: return launch_hd<128>(a, mk, mv, st, pdl);
  }
  return cudaErrorInvalidValue;
}

cudaError_t attn_cluster_launch(AttnArgs a, const CUtensorMap& mk, const CUtensorMap& mv, int S, const int* tables,
                                size_t n, bool paths, int* d_tables, cudaStream_t st) {
  switch (a.head_dim) {
    case 32: return launch_cluster_hd<32>(a, mk, mv, S, tables, n, paths, d_tables, st);
    case 64: return launch_cluster_hd<64>(a, mk, mv, S, tables, n, paths, d_tables, st);
    case 128: return launch_cluster_hd<128>(a, mk, mv, S, tables, n, paths, d_tables, st);
  }
  return cudaErrorInvalidValue;
}

unsigned int* attn_err_word() {
  void* p = nullptr;
  return cudaGetSymbolAddress(&p, g_attn_err) == cudaSuccess ? static_cast<unsigned int*>(p) : nullptr;
}

}  // namespace atspeed
