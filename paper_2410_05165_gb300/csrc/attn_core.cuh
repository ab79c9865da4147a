// Device functions of the shared-prefix tree attention, used by the standalone kernels
// (attention.cu) and by the persistent forward kernel (fwd.cu).
#pragma once
#include <cuda.h>
#include <math.h>

#include "attention.cuh"
#include "common.cuh"

namespace atspeed {

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// 2^x with the hardware's approximation (results below the smallest normal number flush to zero: such a
// weight, against the row maximum's 1, changes no sum)
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// K and V tiles of ATT_SUB rows as written by TMA.  HD >= 64: boxes of 64 columns (128-byte rows),
// 128-byte swizzle: 16-byte chunk c of row r sits at chunk c ^ (r & 7).  HD == 32: one box of 64-byte
// rows, no swizzle.
// frag_base: address of (row, chunk b) with b in {0, 1}; frag_addr: from it, that of (row + 16 rows16,
// chunk + b) with an even `chunk` (only bits 4-6 of the swizzled address depend on it: one xor).
template <int HD>
__device__ __forceinline__ uint32_t frag_base(uint32_t tile, int row, int b) {
  if constexpr (HD >= 64)
    return tile + (uint32_t)(row * 128 + ((b ^ (row & 7)) << 4));
  else
    return tile + (uint32_t)(row * (HD * 2) + (b << 4));
}
template <int HD>
__device__ __forceinline__ uint32_t frag_addr(uint32_t base, int chunk, int rows16) {
  if constexpr (HD >= 64)
    return (base ^ (uint32_t)((chunk & 7) << 4)) + (uint32_t)((chunk >> 3) * (ATT_SUB * 128) + rows16 * 16 * 128);
  else
    return base + (uint32_t)((chunk << 4) + rows16 * 16 * (HD * 2));
}

// Physical 16-byte chunk of logical chunk c of Q row r (conflict-free ldmatrix without padding).
template <int HD>
__device__ __forceinline__ int q_chunk(int r, int c) {
  return c ^ (r & ((HD / 8 < 8 ? HD / 8 : 8) - 1));
}

template <int HD, int D>
struct AttCfg {
  // SMEM_BODY: bytes from the 1024-aligned base: the ring of D K/V buffers (half pages of ATT_SUB
  // keys); the Q tile (rows of HD bf16, 16-byte chunks XOR-swizzled by row) is staged in the last
  // buffer before its first K/V copy (Q lives in registers from then on)
  static constexpr int Q_BYTES = ATT_QTILE * HD * 2;
  static constexpr int KV_BYTES = ATT_SUB * HD * 2;          // one K (or V) half-page tile
  static constexpr int BUF_BYTES = 2 * KV_BYTES;             // K + V
  static constexpr int SMEM_BODY = D * BUF_BYTES;
  static_assert(Q_BYTES <= BUF_BYTES, "the Q tile must fit in one K/V buffer");
  static constexpr int SMEM = 1024 + SMEM_BODY + 64;
};

// One work item (query tile, head, prefix split) with 128 threads (4 warps, 16 queries each).
// smem: 1024-aligned, AttCfg<HD, D>::SMEM_BODY bytes; bars: D mbarriers initialised by the caller
// (count 1); par: bit b is the parity of buffer b's next fill (zero at first), kept identically by
// every thread from item to item.  Writes the normalised output (a.direct) or the split's
// unnormalised partials.  Returns false if a bounded wait timed out.
// Sink::kCustom: the partials go to sink(o, m, l of the thread's two rows) instead, and with chunks_per_split = 0
// the tile's visible pages are balanced over user_splits.
// D - 1 copies are in flight ahead of the arithmetic: a step of 32 keys takes ~0.5 us of tensor and
// softmax work, a copy 1.5 - 2 us (more from DRAM), so two buffers left the warps waiting for copies.
struct AttGlobalSink {
  static constexpr bool kCustom = false;
};
template <int HD, int D, class Sink = AttGlobalSink>
__device__ bool attn_item(const AttnArgs& a, const CUtensorMap* mk, const CUtensorMap* mv, int tile, int h, int split,
                          uint8_t* smem, uint64_t* bars, uint32_t& par, int tid, int bar_id,
                          unsigned long long* tr = nullptr, size_t trs = 0, const Sink& sink = Sink()) {
#define ATT_TR(k) do { if (tr && tid == 0) tr[(size_t)(k) * trs] = globaltimer_ns(); } while (0)
  using C = AttCfg<HD, D>;
  constexpr int NDT = HD / 8;    // dim n-tiles of O
  constexpr int NKS = HD / 16;   // k-steps of Q K^T
  uint8_t* kvbuf = smem;                                             // [D][K | V]
  __nv_bfloat16* qs = reinterpret_cast<__nv_bfloat16*>(smem + (D - 1) * C::BUF_BYTES);   // last buffer, until its copy
  const int warp = tid >> 5, lane = tid & 31;
  const int d = a.n_heads * HD;
  const int u = a.qt_user[tile];
  const int t0 = a.qt_t0[tile];
  const int nq = a.qt_n[tile];
  const int S_u = a.user_splits[u];
  if (split >= S_u) return true;

  // this item's prefix pages [c0, c1): the split's share of the pages the tile's queries see
  const int* ptab = a.page_table + (size_t)u * a.max_pages;
  constexpr int NBOX = HD >= 64 ? HD / 64 : 1;
  constexpr int BOXW = HD >= 64 ? 64 : HD;
  const int nch = (a.qt_vis[tile] + ATT_PAGE - 1) / ATT_PAGE;
  int c0 = 0, c1 = nch;
  if (a.chunks_per_split > 0) {
    c0 = min(nch, split * a.chunks_per_split);
    c1 = min(nch, c0 + a.chunks_per_split);
  } else if constexpr (Sink::kCustom) {
    c0 = split * nch / S_u;
    c1 = (split + 1) * nch / S_u;
  }
  ATT_TR(0);
  constexpr int SUBS = ATT_PAGE / ATT_SUB;
  static_assert(SUBS == 2, "copies alternate between a page's halves");
  const int nst = (c1 - c0) * SUBS;   // steps: half pages
  // copies are issued in order by thread 0: half page `is` of the item next, page ids read a page ahead
  int is = 0, page = 0, page_next = 0;
  auto issue = [&](int buf) {
    if ((is & 1) == 0) {
      page = page_next;
      const int pn = c0 + is / SUBS + 1;
      if (pn < c1) page_next = ptab[pn];
    }
    const int row0 = page * ATT_PAGE + (is & 1) * ATT_SUB;
    ++is;
    uint8_t* kb = kvbuf + buf * C::BUF_BYTES;
    mbar_arrive_expect_tx(&bars[buf], C::BUF_BYTES);
    const uint64_t pol = policy_evict_last();
    for (int b = 0; b < NBOX; ++b) {
      tma_load_2d(kb + b * (ATT_SUB * BOXW * 2), mk, &bars[buf], h * HD + b * BOXW, row0, pol);
      tma_load_2d(kb + C::KV_BYTES + b * (ATT_SUB * BOXW * 2), mv, &bars[buf], h * HD + b * BOXW, row0, pol);
    }
  };
  // the first K / V half pages do not depend on Q: start their copies now
  if (tid == 0 && nst > 0) {
    page_next = ptab[c0];
    for (int b = 0; b < D - 1 && b < nst; ++b) issue(b);
  }
  // Q tile -> shared memory (rows >= nq are zero); all of a thread's loads are issued first
  {
    constexpr int NQL = ATT_QTILE * (HD / 8) / 128;
    uint4 v[NQL];
#pragma unroll
    for (int k = 0; k < NQL; ++k) {
      const int i = tid + 128 * k;
      const int r = i / (HD / 8), c = i % (HD / 8);
      v[k] = r < nq ? __ldcg(reinterpret_cast<const uint4*>(a.q + (size_t)(t0 + r) * d + h * HD + c * 8))
                    : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int k = 0; k < NQL; ++k) {
      const int i = tid + 128 * k;
      const int r = i / (HD / 8), c = i % (HD / 8);
      *reinterpret_cast<uint4*>(qs + r * HD + q_chunk<HD>(r, c) * 8) = v[k];
    }
  }
  named_bar_sync(bar_id, 128);
  ATT_TR(1);

  // Q fragments (A operand) for this warp's 16 rows
  uint32_t qf[NKS][4];
  {
    const uint32_t qbase = smem_u32(qs);
    const int r = warp * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
    const int cofs = lane >> 4;   // 16-byte chunk within the 16-column k-step
#pragma unroll
    for (int kk = 0; kk < NKS; ++kk)
      ldsm_x4(qbase + (uint32_t)((r * HD + q_chunk<HD>(r, kk * 2 + cofs) * 8) * 2), qf[kk][0], qf[kk][1], qf[kk][2],
              qf[kk][3]);
  }
  // The vote at the first step lets thread 0 copy K/V over the Q tile.  A barrier alone does not order the
  // fragment loads before that copy (another proxy): without the fence a warp that ran late had K/V rows for Q
  // (heads of 32, many CTAs per SM).  The same goes for the K/V fragments of each step, below.  (Both fences
  // together: operator kernels +1.4% on average, no change of a forward.)
  fence_proxy_async_shared();
  const int g = lane >> 2, tq = lane & 3;
  const int row_a = warp * 16 + g, row_b = row_a + 8;
  const int vis_a = row_a < nq ? a.tok_vis[t0 + row_a] : 0;
  const int vis_b = row_b < nq ? a.tok_vis[t0 + row_b] : 0;
  const float scale = kLog2e / sqrtf((float)HD);
  // keys below vis_full are visible to every query of the warp (rows past the tile's last query are
  // not stored and do not count)
  int vis_full = min(row_a < nq ? vis_a : 0x7fffffff, row_b < nq ? vis_b : 0x7fffffff);
#pragma unroll
  for (int i = 16; i > 0; i >>= 1) vis_full = min(vis_full, __shfl_xor_sync(0xffffffffu, vis_full, i));
  // ldmatrix rows of this lane in buffer 0: K (keys (lane & 7) + 8 (lane / 16), 8-dimension halves by lane
  // bit 3), V (keys (lane & 7) + 8 (lane bit 3), halves by lane / 16)
  const uint32_t kf0 = frag_base<HD>(smem_u32(kvbuf), (lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1);
  const uint32_t vf0 = frag_base<HD>(smem_u32(kvbuf) + C::KV_BYTES, (lane & 7) + (((lane >> 3) & 1) << 3), lane >> 4);

  float o[NDT][4];
#pragma unroll
  for (int j = 0; j < NDT; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
  float m_a = -INFINITY, m_b = -INFINITY, l_a = 0.f, l_b = 0.f;
  bool ok = true;

  int buf = 0;
  for (int st = 0; st < nst; ++st) {
    // (the vote is also the barrier after which every warp has read the previous step's buffer -- at
    // the first step the Q tile --, which the next copy fills)
    const bool got = named_bar_and(bar_id, 128, mbar_wait(&bars[buf], (par >> buf) & 1u, a.err));
    if (st < 2) ATT_TR(2 + 2 * st);
    if (!got) {
      ok = false;
      break;
    }
    par ^= 1u << buf;
    if (tid == 0 && is < nst) issue(buf == 0 ? D - 1 : buf - 1);
    const int sc = c0 * SUBS + st;
    const uint32_t koff = kf0 + (uint32_t)(buf * C::BUF_BYTES), voff = vf0 + (uint32_t)(buf * C::BUF_BYTES);
    {
      float s[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
      // Q K^T and P V in batches of four fragment loads, each batch's loads issued before the previous
      // batch's MMAs; the four score accumulators (sixteen output ones) are independent chains
      uint32_t f[2][4][4];
      auto load_k = [&](int b) {   // fragments of k-steps 2 b, 2 b + 1: keys 0 .. 15 and 16 .. 31
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int kk = 2 * b + (i >> 1), jj = i & 1;
          uint32_t(&r)[4] = f[b & 1][i];
          ldsm_x4(frag_addr<HD>(koff, kk * 2, jj), r[0], r[1], r[2], r[3]);
        }
      };
      auto load_v = [&](int b) {   // fragments 4 b .. 4 b + 3 of (16 keys, 16 dimensions)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int n = 4 * b + i, kk = n / (NDT / 2), dd = n % (NDT / 2);
          uint32_t(&r)[4] = f[b & 1][i];
          ldsm_x4_t(frag_addr<HD>(voff, dd * 2, kk), r[0], r[1], r[2], r[3]);
        }
      };
      constexpr int NKB = NKS / 2, NVB = NDT / 4;   // batches
      load_k(0);
#pragma unroll
      for (int b = 0; b < NKB; ++b) {
        if (b + 1 < NKB) load_k(b + 1);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int kk = 2 * b + (i >> 1), jj = i & 1;
          const uint32_t(&r)[4] = f[b & 1][i];
          mma_bf16_16816(s[2 * jj], qf[kk], r[0], r[1]);
          mma_bf16_16816(s[2 * jj + 1], qf[kk], r[2], r[3]);
        }
      }
      load_v(0);   // (in flight during the softmax)
      // scale, mask, online softmax (base 2)
      const int kbase_idx = sc * ATT_SUB;
      if (kbase_idx + ATT_SUB > vis_full) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int k0 = kbase_idx + j * 8 + tq * 2;
          s[j][0] = (k0 < vis_a) ? s[j][0] * scale : -INFINITY;
          s[j][1] = (k0 + 1 < vis_a) ? s[j][1] * scale : -INFINITY;
          s[j][2] = (k0 < vis_b) ? s[j][2] * scale : -INFINITY;
          s[j][3] = (k0 + 1 < vis_b) ? s[j][3] * scale : -INFINITY;
        }
      } else {   // every key is visible to every query of the warp
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s[j][0] *= scale;
          s[j][1] *= scale;
          s[j][2] *= scale;
          s[j][3] *= scale;
        }
      }
      float mx_a = m_a, mx_b = m_b;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        mx_a = fmaxf(mx_a, fmaxf(s[j][0], s[j][1]));
        mx_b = fmaxf(mx_b, fmaxf(s[j][2], s[j][3]));
      }
      mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, 1));
      mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, 2));
      mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, 1));
      mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, 2));
      const float ua = (mx_a == -INFINITY) ? 0.f : mx_a;
      const float ub = (mx_b == -INFINITY) ? 0.f : mx_b;
      const float alpha_a = ex2(m_a - ua), alpha_b = ex2(m_b - ub);
      m_a = mx_a;
      m_b = mx_b;
      l_a *= alpha_a;
      l_b *= alpha_b;
#pragma unroll
      for (int j = 0; j < NDT; ++j) {
        o[j][0] *= alpha_a;
        o[j][1] *= alpha_a;
        o[j][2] *= alpha_b;
        o[j][3] *= alpha_b;
      }
      uint32_t ph[2][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p0 = ex2(s[j][0] - ua), p1 = ex2(s[j][1] - ua);
        const float p2 = ex2(s[j][2] - ub), p3 = ex2(s[j][3] - ub);
        l_a += p0 + p1;
        l_b += p2 + p3;
        const int kk = j >> 1, r = (j & 1) * 2;
        const __half2 h01 = __floats2half2_rn(p0, p1), h23 = __floats2half2_rn(p2, p3);
        ph[kk][r] = *reinterpret_cast<const uint32_t*>(&h01);
        ph[kk][r + 1] = *reinterpret_cast<const uint32_t*>(&h23);
      }
      // O += P V with P in fp16 (11 significant bits; the row sum l uses the fp32 values) and V fp16
      // (exactly the bf16-rounded values)
#pragma unroll
      for (int b = 0; b < NVB; ++b) {
        if (b + 1 < NVB) load_v(b + 1);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int n = 4 * b + i, kk = n / (NDT / 2), dd = n % (NDT / 2);
          const uint32_t(&r)[4] = f[b & 1][i];
          mma_f16_16816(o[2 * dd], ph[kk], r[0], r[1]);
          mma_f16_16816(o[2 * dd + 1], ph[kk], r[2], r[3]);
        }
      }
    }
    fence_proxy_async_shared();   // (the next step's vote hands this buffer to a copy)
    if (++buf == D) buf = 0;
    if (st < 2) ATT_TR(3 + 2 * st);
  }
  if (!ok) {
    // copies ahead of the failed step may still be in flight: wait for them (bounded; a buffer that
    // has none runs into its limit) before returning
    if (tid == 0) {
      for (int b = 0; b < D; ++b) mbar_wait(&bars[b], (par >> b) & 1u, nullptr, kDrainNs);
    }
    named_bar_sync(bar_id, 128);
    return false;
  }
  // the next item's copies and Q tile overwrite the buffers: every warp is done with the last ones
  named_bar_sync(bar_id, 128);
  l_a += __shfl_xor_sync(0xffffffffu, l_a, 1);
  l_a += __shfl_xor_sync(0xffffffffu, l_a, 2);
  l_b += __shfl_xor_sync(0xffffffffu, l_b, 1);
  l_b += __shfl_xor_sync(0xffffffffu, l_b, 2);

  if constexpr (Sink::kCustom) {
    sink(o, m_a, l_a, m_b, l_b);
    return true;
  }
  if (a.direct) {
    const float ia = l_a > 0.f ? 1.f / l_a : 0.f, ib = l_b > 0.f ? 1.f / l_b : 0.f;
#pragma unroll
    for (int j = 0; j < NDT; ++j) {
      const int col = h * HD + j * 8 + tq * 2;
      if (row_a < nq)
        *reinterpret_cast<__nv_bfloat162*>(a.out + (size_t)(t0 + row_a) * d + col) =
            __floats2bfloat162_rn(o[j][0] * ia, o[j][1] * ia);
      if (row_b < nq)
        *reinterpret_cast<__nv_bfloat162*>(a.out + (size_t)(t0 + row_b) * d + col) =
            __floats2bfloat162_rn(o[j][2] * ib, o[j][3] * ib);
    }
  } else {
    const size_t base = (size_t)split * a.T;
#pragma unroll
    for (int j = 0; j < NDT; ++j) {
      const int col = j * 8 + tq * 2;
      if (row_a < nq)
        *reinterpret_cast<float2*>(a.part_o + ((base + t0 + row_a) * a.n_heads + h) * HD + col) =
            make_float2(o[j][0], o[j][1]);
      if (row_b < nq)
        *reinterpret_cast<float2*>(a.part_o + ((base + t0 + row_b) * a.n_heads + h) * HD + col) =
            make_float2(o[j][2], o[j][3]);
    }
    if (tq == 0) {
      if (row_a < nq)
        *reinterpret_cast<float2*>(a.part_ml + ((base + t0 + row_a) * a.n_heads + h) * 2) = make_float2(m_a, l_a);
      if (row_b < nq)
        *reinterpret_cast<float2*>(a.part_ml + ((base + t0 + row_b) * a.n_heads + h) * 2) = make_float2(m_b, l_b);
    }
  }
  ATT_TR(6);
#undef ATT_TR
  return true;
}

// Queries per combine group: the merge of one (query tile, head) is split into ATT_QTILE / 16
// groups of 16 queries, each handled by 128 threads (8 per query).
constexpr int ATT_CQ = 16;

// 128 threads: merge the prefix splits of 16 queries (group qg of the tile) of one head with each
// query's path keys and write the normalised bf16 output.  Eight threads per query, each owning
// HD / 8 consecutive dimensions; a path-key dot product adds the eight partial sums by a butterfly
// over the eight lanes (exact in any lane, as fp32 addition commutes), so the result does not
// depend on the schedule that calls it.
// wait(): called once the path-key scores, which need nothing from the splits, are there; returns whether
// every split's partials are published (false: give up).
template <int HD, class Wait>
__device__ __forceinline__ bool attn_combine_group(const AttnArgs& a, int tile, int h, int qg, int ctid, Wait wait) {
  constexpr int TPQ = 8, DH = HD / TPQ;
  const int ql = qg * ATT_CQ + (ctid >> 3), part = ctid & 7;
  const int t0 = a.qt_t0[tile], nq = a.qt_n[tile];
  const bool active = ql < nq;
  const int t = t0 + (active ? ql : 0);
  const int d = a.n_heads * HD;
  const int S = a.user_splits[a.qt_user[tile]];
  const float scale = kLog2e / sqrtf((float)HD);
  const int dim0 = h * HD + part * DH;
  // loads that do not depend on each other first: q, the path rows, the split statistics
  float qv[DH];
  {
    __nv_bfloat16 qb[DH];
#pragma unroll
    for (int i = 0; i < DH; i += 4) *reinterpret_cast<uint2*>(qb + i) = __ldcg(reinterpret_cast<const uint2*>(a.q + (size_t)t * d + dim0 + i));
#pragma unroll
    for (int i = 0; i < DH; ++i) qv[i] = __bfloat162float(qb[i]);
  }
  const int na = (a.anc_n && active) ? a.anc_n[t] : 0;
  int arow[ATT_MAX_ANC];
#pragma unroll
  for (int j = 0; j < ATT_MAX_ANC; ++j) arow[j] = j < na ? a.anc_row[t * ATT_MAX_ANC + j] : 0;
  // path keys (rows written earlier in this forward; cached loads, queries share ancestors)
  float sa[ATT_MAX_ANC];
  __nv_bfloat16 kb[ATT_MAX_ANC][DH];
#pragma unroll
  for (int j = 0; j < ATT_MAX_ANC; ++j)
#pragma unroll
    for (int i = 0; i < DH; i += 4)
      *reinterpret_cast<uint2*>(kb[j] + i) = *reinterpret_cast<const uint2*>(a.k_cache + (size_t)arow[j] * d + dim0 + i);
#pragma unroll
  for (int j = 0; j < ATT_MAX_ANC; ++j) {
    float pd = 0.f;
#pragma unroll
    for (int i = 0; i < DH; ++i) pd += qv[i] * __bfloat162float(kb[j][i]);
    pd += __shfl_xor_sync(0xffffffffu, pd, 1);
    pd += __shfl_xor_sync(0xffffffffu, pd, 2);
    pd += __shfl_xor_sync(0xffffffffu, pd, 4);
    sa[j] = pd * scale;
  }
  if (!wait()) return false;
  float M = -INFINITY;
  for (int s0 = 0; s0 < S; s0 += 4) {
    float mv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      mv[i] = s0 + i < S ? __ldcg(a.part_ml + (((size_t)(s0 + i) * a.T + t) * a.n_heads + h) * 2) : -INFINITY;
#pragma unroll
    for (int i = 0; i < 4; ++i) M = fmaxf(M, mv[i]);
  }
#pragma unroll
  for (int j = 0; j < ATT_MAX_ANC; ++j)
    if (j < na) M = fmaxf(M, sa[j]);
  const float Mu = (M == -INFINITY) ? 0.f : M;
  float L = 0.f, o[DH];
#pragma unroll
  for (int i = 0; i < DH; ++i) o[i] = 0.f;
  const size_t bs = (size_t)a.T * a.n_heads;
  float2 ml_n;
  float4 pv_n[DH / 4];
  auto load_part = [&](int s) {
    const size_t b = (size_t)s * bs + (size_t)t * a.n_heads + h;
    ml_n = __ldcg(reinterpret_cast<const float2*>(a.part_ml + b * 2));
#pragma unroll
    for (int i = 0; i < DH / 4; ++i) pv_n[i] = __ldcg(reinterpret_cast<const float4*>(a.part_o + b * HD + part * DH) + i);
  };
  load_part(0);
  for (int s = 0; s < S; ++s) {
    const float2 ml = ml_n;
    float4 pv[DH / 4];
#pragma unroll
    for (int i = 0; i < DH / 4; ++i) pv[i] = pv_n[i];
    if (s + 1 < S) load_part(s + 1);
    const float w = exp2f(ml.x - Mu);
    L += ml.y * w;
#pragma unroll
    for (int i = 0; i < DH; i += 4) {
      o[i] += pv[i / 4].x * w;
      o[i + 1] += pv[i / 4].y * w;
      o[i + 2] += pv[i / 4].z * w;
      o[i + 3] += pv[i / 4].w * w;
    }
  }
  __half vb[ATT_MAX_ANC][DH];
#pragma unroll
  for (int j = 0; j < ATT_MAX_ANC; ++j)
#pragma unroll
    for (int i = 0; i < DH; i += 4)
      *reinterpret_cast<uint2*>(vb[j] + i) = *reinterpret_cast<const uint2*>(a.v_cache + (size_t)arow[j] * d + dim0 + i);
#pragma unroll
  for (int j = 0; j < ATT_MAX_ANC; ++j) {
    if (j >= na) continue;
    const float w = exp2f(sa[j] - Mu);
    L += w;
#pragma unroll
    for (int i = 0; i < DH; ++i) o[i] += w * __half2float(vb[j][i]);
  }
  if (!active) return true;
  const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
  for (int i = 0; i < DH; i += 2)
    *reinterpret_cast<__nv_bfloat162*>(a.out + (size_t)t * d + dim0 + i) = __floats2bfloat162_rn(o[i] * inv, o[i + 1] * inv);
  return true;
}

}  // namespace atspeed
