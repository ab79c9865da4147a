// Cluster split-K GEMM for sm_103a: the operators' GEMM when there are few output tiles (decode and
// small prefill shapes).  Same product and operands as gemm.cu (weight rows are the MMA's M, tokens
// its N), another decomposition:
//
//   * one cluster of C CTAs (C <= 8) per tile of 128 weight rows x BN tokens; CTA r streams the r-th
//     share of the k-blocks through its TMA ring into its own TMEM accumulator;
//   * the partial sums meet in distributed shared memory: the tile's 16-token groups are dealt out to
//     the CTAs, every CTA stores its partial of a group straight into the owner's shared memory (the
//     ring, idle by then), and the owner adds the C partials in CTA order and runs the epilogue.
//
// So a split tile costs two cluster barriers and one shared-memory exchange, where the stream-K
// kernel publishes parts to global memory and leaves the last CTA to add them all; no CTA waits for
// one that may not be resident, nothing needs a workspace, and the sums' order is fixed.  C depends
// on the weight shape and the number of token tiles alone, so a token's result does not depend on the
// other tokens of the call (one token tile up to 256 tokens).
//
// Measured against the stream-K kernel (us, GB300): [12288 x 4096] x 120 tokens 32.1 -> 24.4 (4.4 TB/s),
// [4096 x 11008] x 120 31.4 -> 24.7, [4096 x 4096] x 120 23.3 -> 16.4, [768 x 768] x 10 9.4 -> 6.6,
// [4096 x 11008] x 512 56.6 -> 45.8, [4096 x 11008] x 960 90.2 -> 72.6.
//
// A CTA takes at most half an SM's shared memory (96 KB ring, two CTAs per SM), so up to 304 CTAs
// stream at once and one CTA's exchange overlaps the other's stream.
// Bound: HBM up to ~256 tokens (weights once), the tensor pipe and the ring's fill rate above.
//
// Roles (320 threads): warp 0 = TMA producer, warp 1 = TMEM + MMA issue, warps 2-9 = two epilogue
// warpgroups (TMEM lane quadrant = warp % 4), which alternate the groups they own.
#include <stdio.h>

#include <algorithm>

#include "common.cuh"
#include "gemm.cuh"
#include "gemm_core.cuh"

namespace atspeed {

namespace {

constexpr int THREADS = 320;
constexpr int GROUP = 16;                            // tokens of an exchange group
constexpr int GROUP_FLOATS = GROUP * GEMM_BM;        // one CTA's partial of a group: [token/4][row][4]
constexpr int ROUND = 128;                           // tokens exchanged at once (bounds the receive area)
constexpr int STG_LD = GEMM_BM + 4;                  // staging row of one token (SwiGLU), floats
constexpr int MAX_CLUSTER = 8;

template <int BN>
struct KCfg {
  static constexpr int A_BYTES = GEMM_BM * 128;
  static constexpr int B_BYTES = BN * 128;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = BN >= 256 ? 2 : BN >= 128 ? 3 : BN >= 64 ? 4 : 5;
  static constexpr int RING = STAGES * STAGE_BYTES;
  // after the last MMA: receive area (a CTA owns at most ceil(8 / C) groups of a round, each with
  // C - 1 received partials), then a staging buffer per warpgroup
  static constexpr int RECV_GROUPS = 10;
  static constexpr int STG_OFF = RECV_GROUPS * GROUP_FLOATS * 4;
  static constexpr int STG_BYTES = 16 * STG_LD * 4;
  static constexpr int BODY = STG_OFF + 2 * STG_BYTES > RING ? STG_OFF + 2 * STG_BYTES : RING;
  static constexpr int SMEM = 1024 + BODY + 256;
  static_assert(SMEM <= 113 * 1024, "two CTAs per SM");
};

struct KcParams {
  GemmArgs a;
  int m_tiles, n_tiles, kb, C, up_row0;
  unsigned int* err;
};

__device__ __forceinline__ void st_cluster_f4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

template <int BN, int EPI>
__global__ void __launch_bounds__(THREADS, 2)
    gemm_cluster_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const KcParams p) {
  using C = KCfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BODY);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tfull = empty + C::STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull + 1);
  int* failed = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nc = p.C, rank = nc > 1 ? (int)cluster_ctarank() : 0;
  const int tile = blockIdx.x / nc;
  const int m_tile = tile / p.n_tiles, n_tile = tile % p.n_tiles;
  const int k0 = rank * p.kb / nc, k1 = (rank + 1) * p.kb / nc;   // this CTA's k-blocks (never empty: C <= kb)

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    *failed = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, BN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ------------------------------------------------------------------ TMA producer
      // weights read by one token tile alone are streamed past the cache
      const uint64_t pol_w = p.n_tiles == 1 ? policy_evict_first() : policy_evict_last();
      const uint64_t pol_x = policy_evict_last();
      int r0, r1;
      if (EPI == EPI_SWIGLU) {
        r0 = m_tile * 64;
        r1 = p.up_row0 + m_tile * 64;
      } else {
        r0 = m_tile * GEMM_BM;
        r1 = r0 + 64;
      }
      int stage = 0;
      uint32_t phase = 0;
      for (int k = k0; k < k1; ++k) {
        if (!mbar_wait(&empty[stage], phase ^ 1u, p.err)) {
          *failed = 1;
          break;
        }
        uint8_t* sa = smem + stage * C::STAGE_BYTES;
        mbar_arrive_expect_tx(&full[stage], C::STAGE_BYTES);
        tma_load_2d(sa, &tmA, &full[stage], k * GEMM_BK, r0, pol_w);
        tma_load_2d(sa + 8192, &tmA, &full[stage], k * GEMM_BK, r1, pol_w);
        tma_load_2d(sa + C::A_BYTES, &tmB, &full[stage], k * GEMM_BK, n_tile * BN, pol_x);
        if (++stage == C::STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ------------------------------------------------------------------ MMA issuer
      constexpr uint32_t idesc = idesc_bf16_f32(GEMM_BM, BN);
      int stage = 0;
      uint32_t phase = 0;
      for (int k = k0; k < k1; ++k) {
        if (!mbar_wait(&full[stage], phase, p.err)) {
          *failed = 1;
          break;
        }
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + stage * C::STAGE_BYTES);
        const uint64_t ad = smem_desc_sw128(sa), bd = smem_desc_sw128(sa + C::A_BYTES);
#pragma unroll
        for (int kk = 0; kk < GEMM_BK / 16; ++kk)
          tc_mma_bf16(tmem_base, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc, (k > k0 || kk > 0) ? 1u : 0u);
        tc_commit(&empty[stage]);
        if (++stage == C::STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
      tc_commit(tfull);   // (also after a failure: nothing may run when TMEM is released)
    }
  }
  __syncwarp();   // (the other lanes of the role warps do not poll beside their lane 0)
  // Every thread waits for the accumulator: all of this CTA's MMAs are done, so all of its ring's
  // copies have landed and been read (after a failure: those of the stages that were consumed).
  if (!mbar_wait(tfull, 0, p.err)) *failed = 1;
  tc_fence_after();
  __syncthreads();
  if (*failed) {
    // copies still in flight must land before the shared memory is reused or released
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < kDrainNs) __nanosleep(1000);
  }

  const GemmArgs& a = p.a;
  const int ep = (int)threadIdx.x - 64, wg = ep >> 7, wt = ep & 127;   // epilogue warpgroup, its thread
  const int m = (warp & 3) * 32 + lane;                               // TMEM lane = row of the tile
  const uint32_t tb = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
  float* recv = reinterpret_cast<float*>(smem);
  float* stg = reinterpret_cast<float*>(smem + C::STG_OFF + (wg & 1) * C::STG_BYTES);
  const int nvalid = min(BN, a.T - n_tile * BN);
  if (nc > 1) cluster_sync();   // every CTA's ring is idle: it may receive partials
#pragma unroll 1
  for (int t0 = 0; t0 < nvalid; t0 += ROUND) {
    const int ng = (min(ROUND, nvalid - t0) + GROUP - 1) / GROUP;   // groups of this round: owner = group % C
    if (nc > 1) {
      if (warp >= 2) {
#pragma unroll 1
        for (int g = wg; g < ng; g += 2) {
          const int owner = g % nc;
          if (owner == rank) continue;
          uint32_t r[16];
          tmem_ld_32x32b_x16(tb + t0 + g * GROUP, r);
          tmem_ld_wait();
          // slot of (group, source) in the owner's receive area
          const int slot = (g / nc) * (nc - 1) + (rank < owner ? rank : rank - 1);
          const uint32_t dst = mapa_u32(recv + slot * GROUP_FLOATS + m * 4, (uint32_t)owner);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            st_cluster_f4(dst + j * (GEMM_BM * 16), r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        }
      }
      cluster_sync();   // the partials of every group are in place
    }
    if (warp >= 2) {
#pragma unroll 1
      for (int g = rank + wg * nc; g < ng; g += 2 * nc) {
        const int tok0 = n_tile * BN + t0 + g * GROUP, nv = min(GROUP, a.T - tok0);
        const int row = m_tile * GEMM_BM + m;
        float old[16];
        if constexpr (EPI == EPI_RESID) {
#pragma unroll
          for (int n = 0; n < GROUP; ++n)
            old[n] = row < a.M && n < nv ? __ldcg(a.out_f32 + (size_t)(tok0 + n) * a.ldo + row) : 0.f;
        }
        uint32_t own[16];
        tmem_ld_32x32b_x16(tb + t0 + g * GROUP, own);
        tmem_ld_wait();
        float acc[16];
#pragma unroll
        for (int n = 0; n < GROUP; ++n) acc[n] = rank == 0 ? __uint_as_float(own[n]) : 0.f;
#pragma unroll 1
        for (int src = 0; src < nc; ++src) {   // CTA order
          if (src == rank) {
            if (rank > 0) {
#pragma unroll
              for (int n = 0; n < GROUP; ++n) acc[n] += __uint_as_float(own[n]);
            }
            continue;
          }
          const int slot = (g / nc) * (nc - 1) + (src < rank ? src : src - 1);
          const float4* q = reinterpret_cast<const float4*>(recv + slot * GROUP_FLOATS) + m;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 v = q[j * GEMM_BM];
            acc[4 * j] += v.x;
            acc[4 * j + 1] += v.y;
            acc[4 * j + 2] += v.z;
            acc[4 * j + 3] += v.w;
          }
        }
        if constexpr (EPI == EPI_F32 || EPI == EPI_RESID) {
          if (row < a.M) {
            float* o = a.out_f32 + (size_t)tok0 * a.ldo + row;
#pragma unroll
            for (int n = 0; n < GROUP; ++n)
              if (n < nv) o[(size_t)n * a.ldo] = EPI == EPI_RESID ? old[n] + acc[n] : acc[n];
          }
          continue;
        }
        named_bar_sync(1 + wg, 128);   // the previous group's rows have been read
#pragma unroll
        for (int n = 0; n < GROUP; ++n) stg[n * STG_LD + m] = acc[n];
        named_bar_sync(1 + wg, 128);
        if constexpr (EPI == EPI_LSE) {
          // (max, sum of exp(y - max)) of each token over the tile's rows: eight threads per token, 16 rows
          // each (four at a time), then combined in a fixed order
          const int j = wt >> 3, sub = wt & 7;
          const int valid = min(GEMM_BM, a.M - m_tile * GEMM_BM) - sub * 16;
          const float4* s4 = reinterpret_cast<const float4*>(stg + j * STG_LD + sub * 16);
          float x[16];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 v = s4[i];
            x[4 * i] = v.x;
            x[4 * i + 1] = v.y;
            x[4 * i + 2] = v.z;
            x[4 * i + 3] = v.w;
          }
          float mx = -INFINITY, sm = 0.f;
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (i < valid) mx = fmaxf(mx, x[i]);
          if (mx != -INFINITY) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (i < valid) sm += expf(x[i] - mx);
          }
          lse_pair<4>(mx, sm);
          if (sub == 0 && j < nv) a.lse_part[(size_t)m_tile * a.lse_ld + tok0 + j] = make_float2(mx, sm);
        } else {   // EPI_SWIGLU: rows 0-63 of the tile are gates, 64-127 the matching ups
          const int f = wt & 31, n0 = wt >> 5;   // two adjacent features, every fourth token
          __nv_bfloat16* out = a.out_bf16 + m_tile * 64 + 2 * f;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int n = n0 + 4 * k;
            if (n < nv) {
              const float2 gv = *reinterpret_cast<const float2*>(stg + n * STG_LD + 2 * f);
              const float2 uv = *reinterpret_cast<const float2*>(stg + n * STG_LD + 64 + 2 * f);
              *reinterpret_cast<__nv_bfloat162*>(out + (size_t)(tok0 + n) * a.ldo) =
                  __floats2bfloat162_rn(swiglu(gv.x, uv.x), swiglu(gv.y, uv.y));
            }
          }
        }
      }
    }
    // (a further round overwrites the receive areas that this one reads)
    if (nc > 1 && t0 + ROUND < nvalid) cluster_sync();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, BN);
  }
}

template <int BN, int EPI>
cudaError_t launch_t(const CUtensorMap& ma, const CUtensorMap& mb, const KcParams& kp, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(attr_done, gemm_cluster_kernel<BN, EPI>, KCfg<BN>::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(kp.m_tiles * kp.n_tiles * kp.C));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = KCfg<BN>::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)kp.C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = kp.C > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gemm_cluster_kernel<BN, EPI>, ma, mb, kp);
}

template <int BN>
cudaError_t launch_bn(EpiKind e, const CUtensorMap& ma, const CUtensorMap& mb, const KcParams& kp, cudaStream_t st) {
  switch (e) {
    case EPI_F32: return launch_t<BN, EPI_F32>(ma, mb, kp, st);
    case EPI_RESID: return launch_t<BN, EPI_RESID>(ma, mb, kp, st);
    case EPI_SWIGLU: return launch_t<BN, EPI_SWIGLU>(ma, mb, kp, st);
    case EPI_LSE: return launch_t<BN, EPI_LSE>(ma, mb, kp, st);
    default: return cudaErrorInvalidValue;
  }
}

// CTAs of a tile's cluster: as many as keep every CTA of the grid resident at once (two per SM), one
// k-block at least each.  (Not 7: its receive area would not fit.)
int cluster_size(long long tiles, int kb, int sms) {
  long long c = std::max<long long>(1, 2LL * sms / tiles);
  c = std::min<long long>(c, std::min(kb, MAX_CLUSTER));
  return c == 7 ? 6 : (int)c;
}

}  // namespace

bool gemm_cluster_fits(const GemmArgs& a, int sms) {
  if (a.epi != EPI_F32 && a.epi != EPI_RESID && a.epi != EPI_SWIGLU && a.epi != EPI_LSE) return false;
  // One token tile: always (so that up to 256 tokens the k-split does not depend on the token count).
  // More: while the grid cannot give every SM a whole tile.  At the line (us, cluster / stream-K):
  // 172 weight tiles x 120 tokens 37.5 / 39.2 and x 200 tokens 52.0 / 49.5; 96 tiles x 2 token tiles
  // (192 in all) 51.4 / 50.9, 32 x 4 (128) 72.6 / 90.2.
  if (a.T <= 256) return true;
  const long long m_tiles = a.epi == EPI_SWIGLU ? a.M / 128 : ((long long)a.M + 127) / 128;
  return m_tiles * ((a.T + 255) / 256) <= sms;
}

cudaError_t gemm_cluster_launch(const GemmArgs& a, unsigned int* err, int sms, cudaStream_t stream, char* eb,
                                size_t el) {
  const cudaError_t ce = gemm_check(a, gemm_max_tiles(), eb, el);
  if (ce != cudaSuccess) return ce;
  const int BN = a.T <= 32 ? 32 : a.T <= 64 ? 64 : a.T <= 128 ? 128 : 256;
  KcParams kp;
  kp.a = a;
  kp.n_tiles = (a.T + BN - 1) / BN;
  kp.m_tiles = a.epi == EPI_SWIGLU ? a.M / 128 : (a.M + GEMM_BM - 1) / GEMM_BM;
  kp.up_row0 = a.epi == EPI_SWIGLU ? a.M / 2 : 0;
  kp.kb = a.K / GEMM_BK;
  kp.C = cluster_size((long long)kp.m_tiles * kp.n_tiles, kp.kb, sms);
  kp.err = err;
  CUtensorMap ma, mb;
  if (!gemm_make_map(&ma, a.W, a.K, a.M, 64, eb, el)) return kGemmMapError;
  if (!gemm_make_map(&mb, a.X, a.K, a.X_rows, BN, eb, el)) return kGemmMapError;
  switch (BN) {
    case 32: return launch_bn<32>(a.epi, ma, mb, kp, stream);
    case 64: return launch_bn<64>(a.epi, ma, mb, kp, stream);
    case 128: return launch_bn<128>(a.epi, ma, mb, kp, stream);
    default: return launch_bn<256>(a.epi, ma, mb, kp, stream);
  }
}

}  // namespace atspeed
