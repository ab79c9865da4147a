// Cluster split-K GEMM for sm_103a: the operators' GEMM when there are few output tiles (decode and
// small prefill shapes).  Same product and operands as gemm.cu (weight rows are the MMA's M, tokens
// its N), another decomposition:
//
//   * one cluster of C CTAs (C <= 8; or CTA pairs) per tile of 128 weight rows x BN tokens; CTA r streams the
//     r-th share of the k-blocks through its TMA ring into two TMEM accumulators, half of the share each, or into more
//     (below);
//   * the partial sums meet in distributed shared memory: the tile's 16-token groups are dealt out to
//     the CTAs, every CTA stores its partial of a group straight into the owner's shared memory (the
//     ring, idle by then), and the owner adds the C partials in CTA order and runs the epilogue.
//
// So a split tile costs two cluster barriers and one shared-memory exchange, where the stream-K
// kernel publishes parts to global memory and leaves the last CTA to add them all; no CTA waits for
// one that may not be resident, nothing needs a workspace, and the sums' order is fixed.  C and the
// accumulations depend on the weight shape and the number of token tiles alone, so a token's result does
// not depend on the other tokens of the call (one token tile up to 256 tokens).
//
// Accumulations ("chains").  The tensor core rounds towards zero, so the error grows with the length of an
// accumulation.  Where the two halves of a CTA's share would be longer than what the stream-K kernel (the k-blocks
// of all tiles over all SMs) accumulates, the share is cut into more chains, which take the two accumulators in
// turn while the epilogue warps add the finished ones up in registers (CHAINS).  Relative error against fp64,
// stream-K kernel / two halves everywhere / here: [768 x 768] 9.4e-8 / 1.14e-7 / 8.5e-8, [768 x 3072] 1.48e-7 /
// 1.82e-7 / 9.9e-8, [256 x 11008] 2.1e-7 / 6.5e-7 / 1.2e-7, [11264 x 2048] 9.8e-7 / 1.0e-6 / 6.5e-7; two halves: [4096 x
// 11008] 2.3e-6 / 1.4e-6, [12288 x 4096] 2.2e-6 / 2.1e-6, [22016 x 4096] 4.2e-6 / 2.1e-6.  What the third chain costs
// (us, two halves / here): [768 x 768] x 10 5.7 / 6.2, x 120 6.9 / 7.5, [768 x 3072] x 120 8.6 / 9.8, [256 x 11008] x 120
// (22 chains of a k-block) 11.2 / 15.4, [11264 x 2048] x 200 16.3 / 17.5.
//
// A CTA takes a whole SM (220 KB ring: 7 k-blocks in flight at 128 tokens), one wave.  Only where the tiles
// alone are more than the SMs (C = 1) do two share one (NARROW: 96 KB ring), so that the second wave's CTAs
// run beside the first's; 256-token tiles, whose two accumulators fill an SM's TMEM, then go round robin over a
// fixed grid of pairs (gemm_tiles_kernel).  Two CTAs per SM and larger clusters were slower where one wave is
// enough: half the copies in flight per CTA and more partials to exchange.
//
// Long shares run as CTA pairs (CG = 2): two CTAs of 128 weight rows each and half of the tokens' operand
// issue one tcgen05.mma of 256 rows.  The order of every sum is the same; the tokens' operand is written
// to and read from shared memory once per pair, where its 128 bytes a clock bind the 256-token tile (48 KB in
// and 48 KB out per k-block of 512 clocks of MMA), and the ring is half as deep again (us, 256-token tiles:
// [4096 x 11008] x 512 40.4 -> 34.4, x 960 66.9 -> 55.3, [12288 x 4096] x 200 29.4 -> 24.6; 128: [19456 x 4096] x 120
// 29.9 -> 28.6).
//
// Measured against the stream-K kernel (us, GB300): [12288 x 4096] x 120 tokens 30.9 -> 20.2 (5.0 TB/s), x 200 40.4 ->
// 25.4, x 10 24.3 -> 18.8, [4096 x 11008] x 120 31.1 -> 19.9, x 200 43.5 -> 25.3, [4096 x 4096] x 120 23.1 -> 11.7,
// [768 x 768] x 10 9.1 -> 6.2, [4096 x 11008] x 512 56.3 -> 35.1, [256 x 11008] x 10 23.8 -> 13.3, [22016 x 4096] x 10 32.8 ->
// 29.0, x 120 39.0 -> 33.2, x 200 50.5 -> 48.7.
//
// Bound: HBM and the SM's intake up to ~256 tokens (weights once), the tensor pipe and the ring's fill
// rate above.
//
// Roles (320 threads): warp 0 = TMA producer, warp 1 = TMEM + MMA issue, warps 2-9 = two epilogue
// warpgroups (TMEM lane quadrant = warp % 4), which alternate the groups they own.
#include <stdio.h>

#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "gemm.cuh"
#include "gemm_core.cuh"

namespace atspeed {

namespace {

constexpr int THREADS = 320;
constexpr int GROUP = 16;                            // tokens of an exchange group
constexpr int GROUP_FLOATS = GROUP * GEMM_BM;        // one CTA's partial of a group: [token/4][row][4]
constexpr int STG_LD = GEMM_BM + 4;                  // staging row of one token (SwiGLU), floats

// NARROW: two CTAs per SM.  WIDE: one.  CHAINS: one, and more than two accumulations, added up as they end.
enum KForm { NARROW, WIDE, CHAINS };

template <int BN, int CG, int FORM>
struct KCfg {
  static constexpr int A_BYTES = GEMM_BM * 128;
  static constexpr int B_BYTES = BN / CG * 128;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  // copies in flight
  static constexpr int STAGES =
      FORM != NARROW ? (232448 - 1024 - 256) / STAGE_BYTES : CG == 2 ? 4 : BN >= 128 ? 3 : BN >= 64 ? 4 : 5;
  // after the last MMA: (one CTA per SM) receive area, a CTA owns at most ceil(groups / C) groups, each with C - 1
  // received partials; then a staging buffer per warpgroup
  static constexpr int RECV_GROUPS = BN >= 256 ? 15 : 10;
  static constexpr int STG_BYTES = 16 * STG_LD * 4;
  static constexpr int STG_OFF = FORM != NARROW ? RECV_GROUPS * GROUP_FLOATS * 4 : 0;
  static constexpr int RING = STAGES * STAGE_BYTES, EXCHANGE = STG_OFF + 2 * STG_BYTES;
  static constexpr int BODY = RING > EXCHANGE ? RING : EXCHANGE;
  static constexpr int SMEM = 1024 + BODY + 256;   // barriers, flags
  static_assert(FORM != NARROW ? SMEM <= 232448 && SMEM > 117 * 1024 : SMEM <= 113 * 1024, "one or two CTAs per SM");
  static_assert(2 * BN <= (FORM != NARROW ? 512 : 256), "two accumulators");
  static_assert((2 * STAGES + 5) * 8 + 8 <= 256, "barriers");
};

struct KcParams {
  GemmArgs a;
  int m_tiles, n_tiles, kb, C, up_row0;
  int chain;   // longest accumulation in k-blocks; 0: two of half the CTA's share
  unsigned int* err;
};

__device__ __forceinline__ void st_cluster_f4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// A CTA's partial of 16 tokens of its TMEM lane's row: the sum of its accumulators (the second's
// `second` columns on, 0: none).
__device__ __forceinline__ void ld_group(uint32_t addr, uint32_t second, float (&v)[16]) {
  uint32_t r[16];
  tmem_ld_32x32b_x16(addr, r);
  tmem_ld_wait();
#pragma unroll
  for (int n = 0; n < 16; ++n) v[n] = __uint_as_float(r[n]);
  if (second) {
    tmem_ld_32x32b_x16(addr + second, r);
    tmem_ld_wait();
#pragma unroll
    for (int n = 0; n < 16; ++n) v[n] += __uint_as_float(r[n]);
  }
}

// The residual of a group's tokens in this thread's row (EPI_RESID).
template <int EPI>
__device__ __forceinline__ void load_old(const GemmArgs& a, int row, int tok0, int nv, float (&old)[GROUP]) {
  if constexpr (EPI == EPI_RESID) {
#pragma unroll
    for (int n = 0; n < GROUP; ++n)
      old[n] = row < a.M && n < nv ? __ldcg(a.out_f32 + (size_t)(tok0 + n) * a.ldo + row) : 0.f;
  }
}

// Epilogue of a group's nv tokens from tok0: acc, this thread's row m of the weight tile.  A warpgroup (thread
// wt) and its staging buffer and named barrier.
template <int EPI>
__device__ __forceinline__ void store_group(const GemmArgs& a, const float* acc, const float (&old)[GROUP], int m_tile,
                                            int m, int tok0, int nv, float* stg, int bar, int wt) {
  const int row = m_tile * GEMM_BM + m;
  if constexpr (EPI == EPI_F32 || EPI == EPI_RESID) {
    if (row < a.M) {
      float* o = a.out_f32 + (size_t)tok0 * a.ldo + row;
#pragma unroll
      for (int n = 0; n < GROUP; ++n)
        if (n < nv) o[(size_t)n * a.ldo] = EPI == EPI_RESID ? old[n] + acc[n] : acc[n];
    }
    return;
  }
  named_bar_sync(bar, 128);   // the previous group's rows have been read
#pragma unroll
  for (int n = 0; n < GROUP; ++n) stg[n * STG_LD + m] = acc[n];
  named_bar_sync(bar, 128);
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

// The epilogue warps' part while more than two chains run: each chain's accumulator is added, in order, to a
// sum in registers (rounded to nearest), and the sum goes to the first accumulator's columns.  Warpgroup wg
// takes half of the columns.
template <int BN, int CG>
__device__ __forceinline__ void sum_chains(int nch, uint64_t* cfull, uint64_t* cempty, uint32_t lead, uint32_t tmem_base,
                                           int warp, int lane, int* failed, unsigned int* err) {
  constexpr int NC = BN / 2;
  const uint32_t tb = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp - 2) >> 2) * NC;
  float acc[NC];
#pragma unroll
  for (int n = 0; n < NC; ++n) acc[n] = 0.f;
#pragma unroll 1
  for (int ch = 0; ch < nch; ++ch) {
    if (!__all_sync(0xffffffffu, mbar_wait(&cfull[ch & 1], (uint32_t)((ch >> 1) & 1), err))) {
      *failed = 1;
      return;
    }
    tc_fence_after();
#pragma unroll
    for (int n = 0; n < NC; n += 16) {
      uint32_t r[16];
      tmem_ld_32x32b_x16(tb + (uint32_t)((ch & 1) * BN + n), r);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[n + i] += __uint_as_float(r[i]);
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
      if constexpr (CG == 2)
        mbar_arrive_cluster(mapa_u32(&cempty[ch & 1], lead));
      else
        mbar_arrive(&cempty[ch & 1]);
    }
  }
#pragma unroll
  for (int n = 0; n < NC; n += 16) tmem_st_32x32b_x16(tb + n, acc + n);
  tmem_st_wait();
}

template <int BN, int EPI, int CG, int FORM>
__global__ void __launch_bounds__(THREADS, FORM == NARROW ? 2 : 1)
    gemm_cluster_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const KcParams p) {
  using C = KCfg<BN, CG, FORM>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int stages = C::STAGES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BODY);
  uint64_t* empty = full + stages;
  uint64_t* tfull = empty + stages;
  uint64_t* cfull = tfull + 1;    // [2] a chain is complete in its accumulator (chains added up as they end)
  uint64_t* cempty = cfull + 2;   // [2] it has been read (the issuing CTA's)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(cempty + 2);
  int* failed = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // rank: the k-share; half: the CTA of a pair (CG = 2), whose 128 of the pair's 256 weight rows it takes
  const int nc = p.C, crank = nc * CG > 1 ? (int)cluster_ctarank() : 0, rank = crank / CG, half = crank % CG;
  const int lead = crank - half;   // cluster rank of the pair's issuing CTA
  const int tile = blockIdx.x / (nc * CG);
  const int m_tile = tile / p.n_tiles * CG + half, n_tile = tile % p.n_tiles;
  const int k0 = rank * p.kb / nc, k1 = (rank + 1) * p.kb / nc;   // this CTA's k-blocks (never empty: C <= kb)
  // its chains of cl k-blocks: one or two, each in an accumulator, or more, added up as they end
  const int want = FORM == CHAINS ? max(2, (k1 - k0 + p.chain - 1) / p.chain) : 2;
  const int cl = (k1 - k0 + want - 1) / want, nch = (k1 - k0 + cl - 1) / cl;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&cfull[i], 1);
      mbar_init(&cempty[i], 8 * CG);   // one arrival per epilogue warp (of both CTAs of a pair)
    }
    *failed = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc<CG>(tmem_slot, 2 * BN);
    tmem_relinquish<CG>();
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();   // the other CTA's barriers are initialised too
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    {
      // ------------------------------------------------------------------ TMA producer (converged, one elected thread)
      const uint32_t lead_t = elect_one();
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
        if (!__all_sync(0xffffffffu, mbar_wait(&empty[stage], phase ^ 1u, p.err))) {
          *failed = 1;
          break;
        }
        uint8_t* sa = smem + stage * C::STAGE_BYTES;
        // (a pair's copies all count on the issuing CTA's barrier)
        const uint32_t fb = CG == 2 ? mapa_u32(&full[stage], (uint32_t)lead) : smem_u32(&full[stage]);
        if (half == 0) mbar_expect_tx_lead(lead_t, &full[stage], CG * C::STAGE_BYTES);
        tma_load_2d_cg<CG>(lead_t, sa, &tmA, fb, k * GEMM_BK, r0, pol_w);
        tma_load_2d_cg<CG>(lead_t, sa + 8192, &tmA, fb, k * GEMM_BK, r1, pol_w);
        tma_load_2d_cg<CG>(lead_t, sa + C::A_BYTES, &tmB, fb, k * GEMM_BK, n_tile * BN + half * (BN / CG), pol_x);
        if (++stage == stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
  } else if (warp == 1) {
    if (half == 0) {
      // ------------------------------------------------------------------ MMA issuer (converged, one elected thread)
      const uint32_t lead_t = elect_one();
      constexpr uint32_t idesc = idesc_bf16_f32(CG * GEMM_BM, BN);
      const uint16_t pair = (uint16_t)(3u << lead);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int ch = 0; ch < nch && ok; ++ch) {
        // (more than two chains: the accumulator's last one has been read)
        if (FORM == CHAINS && ch >= 2 &&
            !__all_sync(0xffffffffu, mbar_wait(&cempty[ch & 1], (uint32_t)((ch >> 1) & 1) ^ 1u, p.err))) {
          ok = false;
          break;
        }
        const uint32_t dt = tmem_base + (uint32_t)((ch & 1) * BN);
        const int kc = k0 + ch * cl, ke = min(k1, kc + cl);
        for (int k = kc; k < ke; ++k) {
          if (!__all_sync(0xffffffffu, mbar_wait(&full[stage], phase, p.err))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * C::STAGE_BYTES);
          const uint64_t ad = smem_desc_sw128(sa), bd = smem_desc_sw128(sa + C::A_BYTES);
          tc_mma_kblock<CG>(lead_t, dt, ad, bd, idesc, k != kc ? 1u : 0u);
          tc_commit_lead<CG>(lead_t, &empty[stage], pair);
          if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (FORM == CHAINS && nch > 2) tc_commit_lead<CG>(lead_t, &cfull[ch & 1], pair);
      }
      if (!ok) *failed = 1;
      tc_commit_lead<CG>(lead_t, tfull, pair);   // (also after a failure: nothing may run when TMEM is released)
    }
  }
  if constexpr (FORM == CHAINS) {
    if (warp >= 2 && nch > 2) sum_chains<BN, CG>(nch, cfull, cempty, (uint32_t)lead, tmem_base, warp, lane, failed, p.err);
  }
  __syncwarp();
  // Every thread waits for the accumulator: all of this CTA's MMAs are done, so all of its ring's
  // copies have landed and been read (after a failure: those of the stages that were consumed).
  if (!mbar_wait(tfull, 0, p.err)) *failed = 1;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
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
  // (an odd last weight tile leaves a pair's second CTA without rows)
  const int nvalid = CG == 1 || m_tile < p.m_tiles ? min(BN, a.T - n_tile * BN) : 0;
  const uint32_t second = nch == 2 ? BN : 0;   // the second accumulator's columns
  if (nc > 1) cluster_sync();   // every CTA's ring is idle: it may receive partials
  const int ng = (nvalid + GROUP - 1) / GROUP;   // groups: owner = group % C
  if (nc > 1) {
    if (warp >= 2) {
#pragma unroll 1
      for (int g = wg; g < ng; g += 2) {
        const int owner = g % nc;
        if (owner == rank) continue;
        float r[16];
        ld_group(tb + g * GROUP, second, r);
        // slot of (group, source) in the owner's receive area
        const int slot = (g / nc) * (nc - 1) + (rank < owner ? rank : rank - 1);
        const uint32_t dst = mapa_u32(recv + slot * GROUP_FLOATS + m * 4, (uint32_t)(owner * CG + half));
#pragma unroll
        for (int j = 0; j < 4; ++j)
          st_cluster_f4(dst + j * (GEMM_BM * 16), make_float4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]));
      }
    }
    cluster_sync();   // the partials of every group are in place
  }
  if (warp >= 2) {
#pragma unroll 1
    for (int g = rank + wg * nc; g < ng; g += 2 * nc) {
      const int tok0 = n_tile * BN + g * GROUP, nv = min(GROUP, a.T - tok0);
      const int row = m_tile * GEMM_BM + m;
      float old[GROUP];
      load_old<EPI>(a, row, tok0, nv, old);
      float own[GROUP], acc[GROUP];
      ld_group(tb + g * GROUP, second, own);
#pragma unroll
      for (int n = 0; n < GROUP; ++n) acc[n] = rank == 0 ? own[n] : 0.f;
#pragma unroll 1
      for (int src = 0; src < nc; ++src) {   // CTA order
        if (src == rank) {
          if (rank > 0) {
#pragma unroll
            for (int n = 0; n < GROUP; ++n) acc[n] += own[n];
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
      store_group<EPI>(a, acc, old, m_tile, m, tok0, nv, stg, 1 + wg, wt);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();   // neither CTA of a pair leaves before the other is done
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<CG>(tmem_base, 2 * BN);
  }
}

// More tiles of one 256-token tile than SMs: CTA pairs on a fixed grid, pair after pair of weight tiles.  A tile's
// two accumulations (the halves of its k-blocks, as above) take the two accumulators in turn; the epilogue
// warps add them up in registers, so the next tile's MMAs run while this one's results are stored.
// us, the one-accumulation NARROW form that it replaces (4% to 19% further off than the stream-K kernel) / NARROW's
// 256-token tiles as single CTAs with two accumulations, one per SM / here: [22016 x 4096] x 200 44.7 / 53.9 / 48.7,
// [33024 x 4096] 51.9 / 55.5 / 50.5, [22016 x 512] 13.3 / 18.2 / 14.6; the stream-K kernel 50.5, 64, 34.
struct TCfg {
  static constexpr int BN = 256, STAGES = 6;
  static constexpr int A_BYTES = GEMM_BM * 128, STAGE_BYTES = A_BYTES + BN / 2 * 128;
  static constexpr int STG_BYTES = 16 * STG_LD * 4, STG_OFF = STAGES * STAGE_BYTES;
  static constexpr int BODY = STG_OFF + 2 * STG_BYTES;
  static constexpr int SMEM = 1024 + BODY + 256;
  static_assert(SMEM <= 232448, "one CTA per SM");
};

template <int EPI>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_tiles_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const KcParams p) {
  using C = TCfg;
  constexpr int BN = C::BN, NC = BN / 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BODY);
  uint64_t* empty = full + C::STAGES;
  uint64_t* cfull = empty + C::STAGES;   // [2] a chain is complete in its accumulator
  uint64_t* cempty = cfull + 2;          // [2] it has been read (CTA 0's)
  uint64_t* mma_done = cempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  int* failed = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half = (int)cluster_ctarank(), pairs = (p.m_tiles + 1) / 2, step = gridDim.x / 2;
  const int kh = (p.kb + 1) / 2;   // k-blocks of the first chain
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&cfull[i], 1);
      mbar_init(&cempty[i], 16);   // one arrival per epilogue warp of both CTAs
    }
    mbar_init(mma_done, 1);
    *failed = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc<2>(tmem_slot, 2 * BN);
    tmem_relinquish<2>();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // the other CTA's barriers are initialised too
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    const uint32_t lead_t = elect_one();
    const uint64_t pol_w = policy_evict_first(), pol_x = policy_evict_last();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int t = blockIdx.x / 2; t < pairs && ok; t += step) {
      const int m_tile = 2 * t + half;
      const int r0 = EPI == EPI_SWIGLU ? m_tile * 64 : m_tile * GEMM_BM;
      const int r1 = EPI == EPI_SWIGLU ? p.up_row0 + m_tile * 64 : r0 + 64;
      for (int k = 0; k < p.kb; ++k) {
        if (!__all_sync(0xffffffffu, mbar_wait(&empty[stage], phase ^ 1u, p.err))) {
          ok = false;
          break;
        }
        uint8_t* sa = smem + stage * C::STAGE_BYTES;
        const uint32_t fb = mapa_u32(&full[stage], 0);
        if (half == 0) mbar_expect_tx_lead(lead_t, &full[stage], 2 * C::STAGE_BYTES);
        tma_load_2d_cg<2>(lead_t, sa, &tmA, fb, k * GEMM_BK, r0, pol_w);
        tma_load_2d_cg<2>(lead_t, sa + 8192, &tmA, fb, k * GEMM_BK, r1, pol_w);
        tma_load_2d_cg<2>(lead_t, sa + C::A_BYTES, &tmB, fb, k * GEMM_BK, half * (BN / 2), pol_x);
        if (++stage == C::STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) *failed = 1;
  } else if (warp == 1) {
    if (half == 0) {
      const uint32_t lead_t = elect_one();
      constexpr uint32_t idesc = idesc_bf16_f32(2 * GEMM_BM, BN);
      int stage = 0, ch = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int t = blockIdx.x / 2; t < pairs && ok; t += step) {
        for (int kc = 0; kc < p.kb && ok; kc += kh, ++ch) {
          if (!__all_sync(0xffffffffu, mbar_wait(&cempty[ch & 1], (uint32_t)((ch >> 1) & 1) ^ 1u, p.err))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dt = tmem_base + (uint32_t)((ch & 1) * BN);
          const int ke = min(p.kb, kc + kh);
          for (int k = kc; k < ke; ++k) {
            if (!__all_sync(0xffffffffu, mbar_wait(&full[stage], phase, p.err))) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + stage * C::STAGE_BYTES);
            const uint64_t ad = smem_desc_sw128(sa), bd = smem_desc_sw128(sa + C::A_BYTES);
            tc_mma_kblock<2>(lead_t, dt, ad, bd, idesc, k > kc ? 1u : 0u);
            tc_commit_lead<2>(lead_t, &empty[stage]);
            if (++stage == C::STAGES) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (ok) tc_commit_lead<2>(lead_t, &cfull[ch & 1]);
        }
      }
      if (!ok) *failed = 1;
      tc_commit_lead<2>(lead_t, mma_done);   // nothing may run when TMEM is released
    }
  } else {
    const GemmArgs& a = p.a;
    const int ep = (int)threadIdx.x - 64, wg = ep >> 7, wt = ep & 127, m = (warp & 3) * 32 + lane;
    const uint32_t tb = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(wg * NC);
    float* stg = reinterpret_cast<float*>(smem + C::STG_OFF + wg * C::STG_BYTES);
    int ch = 0;
    bool ok = true;
    for (int t = blockIdx.x / 2; t < pairs && ok; t += step) {
      const int m_tile = 2 * t + half;
      // this warpgroup's tokens (none past the last weight tile)
      const int nt = m_tile < p.m_tiles ? min(NC, a.T - wg * NC) : 0;
      float acc[NC];
#pragma unroll
      for (int n = 0; n < NC; ++n) acc[n] = 0.f;
#pragma unroll 1
      for (int kc = 0; kc < p.kb; kc += kh, ++ch) {
        if (!named_bar_and(3, 256, mbar_wait(&cfull[ch & 1], (uint32_t)((ch >> 1) & 1), p.err))) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int n = 0; n < NC; n += 16) {
          if (n < nt) {
            uint32_t r[16];
            tmem_ld_32x32b_x16(tb + (uint32_t)((ch & 1) * BN + n), r);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[n + i] += __uint_as_float(r[i]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa_u32(&cempty[ch & 1], 0));
      }
      if (!ok) break;
#pragma unroll
      for (int n = 0; n < NC; n += GROUP) {
        if (n < nt) {
          const int tok0 = wg * NC + n, nv = min(GROUP, nt - n);
          float old[GROUP];
          load_old<EPI>(a, m_tile * GEMM_BM + m, tok0, nv, old);
          store_group<EPI>(a, acc + n, old, m_tile, m, tok0, nv, stg, 1 + wg, wt);
        }
      }
    }
    if (!ok) *failed = 1;
  }
  __syncwarp();
  __syncthreads();
  cluster_sync();   // neither CTA issues copies or MMAs any more
  if (threadIdx.x == 0) {
    mbar_wait(mma_done, 0, p.err);
    if (*failed) {   // copies still in flight must land before the shared memory is released
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < kDrainNs) __nanosleep(1000);
    }
  }
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<2>(tmem_base, 2 * BN);
  }
}

template <int BN, int EPI, int CG, int FORM>
cudaError_t launch_t(const CUtensorMap& ma, const CUtensorMap& mb, const KcParams& kp, cudaStream_t st) {
  using C = KCfg<BN, CG, FORM>;
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(attr_done, gemm_cluster_kernel<BN, EPI, CG, FORM>, C::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((kp.m_tiles + CG - 1) / CG * kp.n_tiles * kp.C * CG));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)(kp.C * CG);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = kp.C * CG > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gemm_cluster_kernel<BN, EPI, CG, FORM>, ma, mb, kp);
}

template <int BN, int CG, int FORM>
cudaError_t launch_bn(EpiKind e, const CUtensorMap& ma, const CUtensorMap& mb, const KcParams& kp, cudaStream_t st) {
  switch (e) {
    case EPI_F32: return launch_t<BN, EPI_F32, CG, FORM>(ma, mb, kp, st);
    case EPI_RESID: return launch_t<BN, EPI_RESID, CG, FORM>(ma, mb, kp, st);
    case EPI_SWIGLU: return launch_t<BN, EPI_SWIGLU, CG, FORM>(ma, mb, kp, st);
    case EPI_LSE: return launch_t<BN, EPI_LSE, CG, FORM>(ma, mb, kp, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int BN, int CG>
cudaError_t launch_form(int form, EpiKind e, const CUtensorMap& ma, const CUtensorMap& mb, const KcParams& kp, cudaStream_t st) {
  if (form == WIDE) return launch_bn<BN, CG, WIDE>(e, ma, mb, kp, st);
  if (form == CHAINS) return launch_bn<BN, CG, CHAINS>(e, ma, mb, kp, st);
  if constexpr (BN <= 128) return launch_bn<BN, CG, NARROW>(e, ma, mb, kp, st);
  return cudaErrorInvalidValue;
}

template <int EPI>
cudaError_t launch_tiles_t(const CUtensorMap& ma, const CUtensorMap& mb, const KcParams& kp, int sms, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(attr_done, gemm_tiles_kernel<EPI>, TCfg::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * std::min(sms / 2, (kp.m_tiles + 1) / 2)));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = TCfg::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, gemm_tiles_kernel<EPI>, ma, mb, kp);
}

cudaError_t launch_tiles(EpiKind e, const CUtensorMap& ma, const CUtensorMap& mb, const KcParams& kp, int sms, cudaStream_t st) {
  switch (e) {
    case EPI_F32: return launch_tiles_t<EPI_F32>(ma, mb, kp, sms, st);
    case EPI_RESID: return launch_tiles_t<EPI_RESID>(ma, mb, kp, sms, st);
    case EPI_SWIGLU: return launch_tiles_t<EPI_SWIGLU>(ma, mb, kp, sms, st);
    case EPI_LSE: return launch_tiles_t<EPI_LSE>(ma, mb, kp, sms, st);
    default: return cudaErrorInvalidValue;
  }
}

// CTAs of a tile's cluster: as many as can all run at once, one per SM, with three k-blocks each at
// least.  On 152 SMs there is room for 76 clusters of two, 46 of three, 36 of four, 23 of six, 15 of eight;
// a cluster that has to wait costs a second wave (us, 120 tokens, C = 3 / 4 / 6 / 8: 24 weight tiles x 64
// k-blocks 13.1 / 11.6 / 20.4 / 15.2, 19 x 64 13.0 / 11.4 / 11.4 / 20.1), and eight are better than six only
// where six would leave most SMs idle (12 x 64: 10.5 with six, 11.0 with eight; 2 x 172, 10 tokens: 13.6,
// 12.3).  Small K: 6 x 12, C = 2 / 3 / 4 / 6 / 8: 6.1 / 6.2 / 6.1 / 6.4 / 6.9.
int cluster_size(long long tiles, int kb, int sms) {
  auto fits = [&](int c, int room) { return tiles * c <= room && kb >= 3 * c; };
  if (fits(8, sms / 2)) return 8;
  for (int c : {6, 4, 3})
    if (fits(c, sms * 9 / 10)) return c;
  return fits(2, sms) ? 2 : 1;
}

}  // namespace

bool gemm_cluster_fits(const GemmArgs& a, int sms) {
  if (a.epi != EPI_F32 && a.epi != EPI_RESID && a.epi != EPI_SWIGLU && a.epi != EPI_LSE) return false;
  // One token tile: always (so that up to 256 tokens the k-split does not depend on the token count).
  // More: while every tile has an SM of its own.  At the line (us, here / gemm_pair.cu, K = 4096): 128 tiles
  // ([8192] x 512 tokens) 26.0 / 41.2, 152 ([9728] x 512) 27.5 / 27.7, 192 ([12288] x 512) 56.5 / 41.9.
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
  const long long tiles = (long long)kp.m_tiles * kp.n_tiles;
  // The longest accumulation where two halves of the CTA's share would exceed it: 0.8 of an SM's share of all
  // k-blocks (a stream-K piece is that long, less where a tile ends: with 1.0, 16 k-blocks at [11264 x 2048] were
  // 2% further off than its pieces of up to 18).
  const double longest = 0.8 * (double)tiles * kp.kb / sms;
  const int share = (kp.kb + kp.C - 1) / kp.C;
  kp.chain = tiles <= sms && (share + 1) / 2 > longest ? std::max(1, (int)longest) : 0;
  kp.err = err;
  CUtensorMap ma, mb;
  if (!gemm_make_map(&ma, a.W, a.K, a.M, 64, eb, el)) return kGemmMapError;
  // CTA pairs (the same sums) for long shares, while all clusters of 2 C CTAs still run at once.  At the
  // lines (us, one CTA / pair): 256 tokens, C = 2 of 40 k-blocks 14.3 / 14.8 as C = 3, 1 of 4 7.2 / 7.7, 1 of 12
  // 16.9 / 16.3, 1 of 64 30.1 / 25.5; 120 tokens, C = 1 of 12 k-blocks 11.5 / 12.6, of 32 14.1 / 14.5, of 64 with
  // 128 weight tiles 27.7 / 26.4, 160 35.8 / 34.6, 258 47.5 / 48.1.
  const long long pair_ctas = 2LL * ((kp.m_tiles + 1) / 2) * kp.n_tiles * kp.C;
  const bool room = tiles > sms || pair_ctas <= (kp.C == 1 ? sms : sms * 9 / 10);
  const bool pairs = BN == 256 ? tiles > sms || (kp.C <= 2 && kp.kb >= 8 * kp.C && room)
                               : BN == 128 && kp.C == 1 && kp.kb >= 48 && 2 * tiles <= 3 * sms && room;
  if (!gemm_make_map(&mb, a.X, a.K, a.X_rows, pairs ? BN / 2 : BN, eb, el)) return kGemmMapError;
  if (BN == 256 && tiles > sms) return launch_tiles(a.epi, ma, mb, kp, sms, stream);
  const int form = tiles > sms ? NARROW : kp.chain > 0 ? CHAINS : WIDE;
  if (BN == 256) return pairs ? launch_form<256, 2>(form, a.epi, ma, mb, kp, stream) : launch_form<256, 1>(form, a.epi, ma, mb, kp, stream);
  if (pairs) return launch_form<128, 2>(form, a.epi, ma, mb, kp, stream);
  switch (BN) {
    case 32: return launch_form<32, 1>(form, a.epi, ma, mb, kp, stream);
    case 64: return launch_form<64, 1>(form, a.epi, ma, mb, kp, stream);
    default: return launch_form<128, 1>(form, a.epi, ma, mb, kp, stream);
  }
}

}  // namespace atspeed
