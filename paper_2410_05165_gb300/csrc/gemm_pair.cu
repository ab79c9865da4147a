// CTA-pair GEMM for sm_103a: the operators' GEMM (and FULL normalisation's LM head) with many output
// tiles, where the tensor pipe binds.  Same product and operands as gemm.cu; a cluster of two CTAs runs
// one tcgen05.mma (cta_group::2) over 256 weight rows x 256 tokens: each CTA loads its 128 weight rows and
// half of the tokens, and its TMEM holds its rows' accumulator for all 256 tokens.  A k-block costs a
// CTA 32 KB of copies instead of 48 KB (the rate at which an SM takes copies in, ~64 bytes per clock, binds
// the one-CTA tile of 128 x 256), and the ring holds six of them.
//
// Decomposition: 76 pairs on 152 SMs take whole tiles round robin after the stream-K shares of the
// remainder (WorkSplit over pairs, gemm_core.cuh); split tiles are summed by the last pair to publish,
// each CTA its 128 rows, in k order, while the whole tiles' MMAs run.  No CTA waits for another pair.
//
// Measured (GB300, us, one-CTA stream-K kernel / this one): [22016 x 4096] x 3840 tokens 419 / 369, and 355
// (1.95 PFLOP/s, tensor pipe 91% active) with the converged producer and issuer (elect_one);
// [19456 x 4096] x 1024 tokens 113 / 94, x 1024 (K) x 3840 tokens 141 / 112.
//
// Roles (320 threads): warp 0 = TMA producer, warp 1 = TMEM + MMA issue (CTA 0's issues for both), warps
// 2-9 = two epilogue warpgroups (TMEM lane quadrant = warp % 4), alternate 32-token chunks each.
#include <stdio.h>

#include "common.cuh"
#include "gemm.cuh"
#include "gemm_core.cuh"

namespace atspeed {

namespace {

constexpr int BN = 256;
constexpr int STAGES = 6;
constexpr int A_BYTES = GEMM_BM * 128;
constexpr int B_BYTES = BN / 2 * 128;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int STG_OFF = STAGES * STAGE_BYTES;             // one [32][128] fp32 chunk per warpgroup
constexpr int BAR_OFF = STG_OFF + 2 * 32 * GEMM_BM * 4;
constexpr int SMEM = 1024 + BAR_OFF + 1536;               // barriers, flags, split-part slots
constexpr int TMEM_COLS = 2 * BN;
constexpr int THREADS = 320;
static_assert(SMEM <= 232448, "shared memory of a CTA");

struct PairParams {
  GemmArgs a;
  int m_tiles, n_tiles, kb;
  WorkSplit w;   // over CTA pairs
  float* ws;
  int* counters;
  unsigned int* err;
};

template <int EPI>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const PairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + BAR_OFF);   // (CTA 0's count both CTAs' copies)
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + 2;                                   // (CTA 0's: the issuer waits there)
  uint64_t* mma_done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  int* flag = reinterpret_cast<int*>(tmem_slot + 1);
  int* failed = flag + 1;
  int* last_fill = failed + 1;          // [STAGES] parity of the last fill issued, -1: none
  int* part_slot = last_fill + STAGES;  // [<= 256] workspace slots of a split tile's parts

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pr = blockIdx.x >> 1, rank = (int)cluster_ctarank();
  const int kb = p.kb;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      last_fill[s] = -1;
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 16);   // one arrival per epilogue warp of both CTAs
    }
    mbar_init(mma_done, 1);
    *failed = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc<2>(tmem_slot, TMEM_COLS);
    tmem_relinquish<2>();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // the other CTA's barriers are initialised too
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    {
      // ------------------------------------------------------------------ TMA producer (converged, one elected thread)
      const uint32_t lead_t = elect_one();
      tma_prefetch_desc(&tmA);
      tma_prefetch_desc(&tmB);
      const uint64_t pol_w = policy_evict_first(), pol_x = policy_evict_last();
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      SegIter it;
      it.init(p.w, pr);
      int tile, k0, k1;
      while (ok && it.next(p.w, tile, k0, k1)) {
        const int mt = 2 * (tile / p.n_tiles) + rank, brow = tile % p.n_tiles * BN + rank * (BN / 2);
        for (int k = k0; k < k1; ++k) {
          if (!__all_sync(0xffffffffu, mbar_wait(&empty[stage], phase ^ 1u, p.err))) {
            ok = false;
            break;
          }
          uint8_t* sa = smem + stage * STAGE_BYTES;
          const uint32_t fb = mapa_u32(&full[stage], 0);
          if (rank == 0) mbar_expect_tx_lead(lead_t, &full[stage], 2 * STAGE_BYTES);
          last_fill[stage] = (int)phase;
          if constexpr (EPI == EPI_SWIGLU)   // 64 gate rows and the matching 64 up rows
            tma_load_3d_cg<2>(lead_t, sa, &tmA, fb, k * GEMM_BK, mt * 64, 0, pol_w);
          else
            tma_load_2d_cg<2>(lead_t, sa, &tmA, fb, k * GEMM_BK, mt * GEMM_BM, pol_w);
          tma_load_2d_cg<2>(lead_t, sa + A_BYTES, &tmB, fb, k * GEMM_BK, brow, pol_x);
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) *failed = 1;
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ------------------------------------------------------------------ MMA issuer (converged, one elected thread)
      const uint32_t lead_t = elect_one();
      constexpr uint32_t idesc = idesc_bf16_f32(2 * GEMM_BM, BN);
      int stage = 0, si = 0;
      uint32_t phase = 0;
      bool ok = true;
      SegIter it;
      it.init(p.w, pr);
      int tile, k0, k1;
      for (; ok && it.next(p.w, tile, k0, k1); ++si) {
        const int acc = si & 1, use = si >> 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&tempty[acc], (uint32_t)(use & 1) ^ 1u, p.err))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t dt = tmem_base + (uint32_t)(acc * BN);
        for (int k = k0; k < k1; ++k) {
          if (!__all_sync(0xffffffffu, mbar_wait(&full[stage], phase, p.err))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * STAGE_BYTES);
          const uint64_t ad = smem_desc_sw128(sa), bd = smem_desc_sw128(sa + A_BYTES);
          tc_mma_kblock<2>(lead_t, dt, ad, bd, idesc, k > k0 ? 1u : 0u);
          tc_commit_lead<2>(lead_t, &empty[stage]);
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        tc_commit_lead<2>(lead_t, &tfull[acc]);
      }
      if (!ok) *failed = 1;
      // no MMA may still be running when TMEM is released: both CTAs wait for this commit at the end
      tc_commit_lead<2>(lead_t, mma_done);
    }
  } else {
    // -------------------------------------------------------------------- epilogue
    const int ep = threadIdx.x - 64, wg = ep >> 7, wt = ep & 127, bar = 2 + wg;
    const int q = warp & 3, m = q * 32 + lane;
    float* staging = reinterpret_cast<float*>(smem + STG_OFF) + wg * (32 * GEMM_BM);
    int si = 0;
    SegIter it;
    it.init(p.w, pr);
    int tile, k0, k1;
    for (; it.next(p.w, tile, k0, k1); ++si) {
      const int acc = si & 1, use = si >> 1;
      const bool got = named_bar_and(1, 256, mbar_wait(&tfull[acc], (uint32_t)(use & 1), p.err));
      if (!got) {
        *failed = 1;
        break;
      }
      tc_fence_after();
      const int m_tile = 2 * (tile / p.n_tiles) + rank, n_tile = tile % p.n_tiles;
      const uint32_t tb = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
      // 32-token chunks with valid tokens; none past the last weight tile (CTA 1's with an odd count)
      const int nch = m_tile < p.m_tiles ? min(BN / 32, (p.a.T - n_tile * BN + 31) / 32) : 0;
      auto release = [&]() {
        tc_fence_before();
        if (lane == 0) mbar_arrive_cluster(mapa_u32(&tempty[acc], 0));
      };
      if (k0 == 0 && k1 == kb) {
        for (int ch = wg; ch < nch; ch += 2) {
          uint32_t r[32];
          tmem_ld_32x32b_x32(tb + ch * 32, r);
          tmem_ld_wait();
          if constexpr (EPI == EPI_F32 || EPI == EPI_RESID) {   // a thread's row of the tile: no exchange
            epi_rows<EPI>(p.a, r, m_tile * GEMM_BM + m, n_tile * BN + ch * 32);
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) staging[j * GEMM_BM + m] = __uint_as_float(r[j]);
            named_bar_sync(bar, 128);
            epi_chunk<BN, EPI>(p.a, staging, m_tile, n_tile, ch, wt, nullptr, nullptr);
            named_bar_sync(bar, 128);
          }
        }
        release();
        continue;
      }
      // a part of a split tile: publish it; the last pair's CTAs sum
      const int slot = (2 * pr + rank) * 2 + (si == 0 ? 0 : 1);
      ws_store_partial(p.ws + (size_t)slot * GEMM_WS_SLOT_FLOATS, tb, nch, m, wg, 2);
      release();
      __threadfence();
      named_bar_sync(1, 256);
      const int tu0 = tile * kb;
      const int c_first = sk_owner(p.w, tu0), parts = sk_owner(p.w, tu0 + kb - 1) - c_first + 1;
      if (ep == 0) {
        int* cnt = &p.counters[2 * tile + rank];
        const int last = atomicAdd(cnt, 1) == parts - 1;
        if (last) {
          *cnt = 0;
          __threadfence();
        }
        *flag = last;
      }
      for (int pi = ep; pi < parts; pi += 256) {
        const int cc = c_first + pi;
        part_slot[pi] = (2 * cc + rank) * 2 + (sk_start(p.w, cc) >= tu0 ? 0 : 1);
      }
      named_bar_sync(1, 256);
      if (*flag) {
        for (int ch = wg; ch < nch; ch += 2) {
          ws_reduce_chunk<2>(p.ws, part_slot, parts, ch, m, staging);
          named_bar_sync(bar, 128);
          epi_chunk<BN, EPI>(p.a, staging, m_tile, n_tile, ch, wt, nullptr, nullptr);
          named_bar_sync(bar, 128);
        }
      }
      named_bar_sync(1, 256);   // flag and part_slot are reused
    }
  }

  __syncthreads();
  cluster_sync();   // neither CTA issues copies or MMAs any more
  if (threadIdx.x == 0) {
    // the issuer's last commit arrives in both CTAs once every MMA (and its arrivals) is done
    mbar_wait(mma_done, 0, p.err);
    if (*failed) {
      // copies in flight: CTA 0's barriers count them; a fill that only one CTA issued never completes
      // its phase, so these waits are short, and long enough for any copy to land
      if (rank == 0)
        for (int s = 0; s < STAGES; ++s)
          if (last_fill[s] >= 0) mbar_wait(&full[s], (uint32_t)last_fill[s], nullptr, kDrainNs);
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < kDrainNs) __nanosleep(1000);
    }
  }
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc<2>(tmem_base, TMEM_COLS);
  }
}

template <int EPI>
cudaError_t launch_t(const CUtensorMap& ma, const CUtensorMap& mb, const PairParams& kp, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(attr_done, gemm_pair_kernel<EPI>, SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * kp.w.Gw));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, gemm_pair_kernel<EPI>, ma, mb, kp);
}

}  // namespace

cudaError_t gemm_pair_launch(const GemmArgs& a, const GemmScratch& s, int grid, cudaStream_t stream, char* eb,
                             size_t el) {
  const cudaError_t ce = gemm_check(a, s.max_tiles, eb, el);
  if (ce != cudaSuccess) return ce;
  PairParams kp;
  kp.a = a;
  kp.n_tiles = (a.T + BN - 1) / BN;
  kp.m_tiles = (a.M + GEMM_BM - 1) / GEMM_BM;
  kp.kb = a.K / GEMM_BK;
  kp.w = work_split((kp.m_tiles + 1) / 2 * kp.n_tiles, kp.kb, grid / 2, grid / 2);
  kp.ws = s.ws;
  kp.counters = s.counters;
  kp.err = s.err;
  CUtensorMap ma, mb;
  const bool mapped = a.epi == EPI_SWIGLU ? gemm_make_map_pairs(&ma, a.W, a.K, a.M / 2, eb, el)
                                          : gemm_make_map(&ma, a.W, a.K, a.M, GEMM_BM, eb, el);
  if (!mapped || !gemm_make_map(&mb, a.X, a.K, a.X_rows, BN / 2, eb, el)) return kGemmMapError;
  switch (a.epi) {
    case EPI_F32: return launch_t<EPI_F32>(ma, mb, kp, stream);
    case EPI_RESID: return launch_t<EPI_RESID>(ma, mb, kp, stream);
    case EPI_SWIGLU: return launch_t<EPI_SWIGLU>(ma, mb, kp, stream);
    case EPI_LSE: return launch_t<EPI_LSE>(ma, mb, kp, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace atspeed
