// Block-causal attention of the q block rows against the KV cache (flash decoding).
//
// In one block forward, row j of sequence s attends to the committed slots
// [0, len[s]) and to block rows 0..j (slots len[s] .. len[s]+j), which the QKV
// epilogue has just written; this is how Eq. 1-2 evaluate every appended
// position of the block in one pass.  A tree block (Sec. 2.1.2) replaces the
// rows 0..j by row j's ancestors and itself, given as one bit mask per row.
// (Prefill attention, many query rows per sequence, is prefill_attention.cu.)
// The bytes are the K and V rows (bf16, hd*2 bytes each), read once per
// (sequence, head) for all q rows together.
//
// Work: the grid is nclusters thread-block clusters of cs CTAs, all resident
// at once (launch_attention picks the largest cs <= ATT_CS_MAX for which one
// cluster per (sequence, head) pair fits on the GPU with room to spare; else
// cs = 1 and each CTA takes several pairs).  Three CTAs fit on an SM.  Cluster c
// takes the pairs c, c + nclusters, ...; the nu units of ATT_UNIT = 64
// consecutive slots of a pair are split over the cluster's CTAs as
// [r*nu/cs, (r+1)*nu/cs) for CTA rank r.  One thread keeps a
// two-stage ring of K and V tiles (TMA, boxes of 64 dims x 64 rows, 128-byte
// swizzle) full, walking the CTA's units pair by pair; tiles made of committed
// slots only are requested before the QKV projection has finished, and the
// next ATT_PREFETCH tiles (one for long slices) are kept on their way into L2.  Per unit, on the
// tensor cores (mma.sync m16n8k16) in transposed form, so that the q <= 8
// block rows fill an N = 8 tile instead of padding an M = 16 one: S^T = K Q^T
// with each warp on 16 keys, an online-softmax update of the running row max
// and exp-sum (reductions over the warp's lanes, then the warps via shared
// memory), then O^T = O^T * alpha + V^T P^T with each warp on hd/4
// dimensions.  Q and P enter as bf16 hi + lo pairs (two MMAs each), K and V
// are the cache's own bf16 values, accumulation is fp32.
//
// Each CTA's run over its units of a pair ends in a partial result (row max,
// exp-sum, unnormalised output) that it leaves in its own shared memory; after
// a cluster barrier every CTA merges its share of the pair's output elements
// from the cs partials through distributed shared memory, in a fixed order with
// the usual log-sum-exp rescaling (deterministic), and writes them in fp32 and
// as the O projection's bf16 hi + lo operand.  A second cluster barrier keeps
// the partials in place until every CTA of the cluster has read them.
#include <algorithm>
#include <cstdlib>

#include "common.cuh"
#include "internal.h"

namespace sdsat {

constexpr int ATT_STAGES = 2;
constexpr int ATT_PREFETCH = 4;   // units past the ring requested into L2 ahead of their loads
// ... but only one for a CTA whose slice has at least this many units.  Thread 0 issues the
// window before the dependency wait, and the TMA unit works through the requests of the SM's
// three CTAs in order: with long slices (13B at context 4096: 7-8 units) thread 0 reached the
// wait 2.8 us after the QKV projection ended with a window of 4 (1.0 us with 1; 13B forward
// 5.303 -> 5.256 ms), while shorter slices (batch 4 at context 1024: 5-6 units) lose more from
// the later units' missed L2 hits than they gain (attention 13.7 -> 15.1 us with 1)
constexpr int ATT_LONG_SLICE = 7;
constexpr size_t ATT_TWO_PER_SM = 96 * 1024;   // dynamic shared memory of which only two fit on an SM
constexpr int ATT_MERGE = 6;            // partials that one lane merges, at most
constexpr int ATT_SPARE_CLUSTERS = 8;   // room left for this many more clusters (measured: 7B/13B shapes, b = 1, 4)

template <int HD, int QT = 2>
struct AttCfg {
  static constexpr int ROWS = QT * 8;                    // query rows the tiles hold
  static constexpr int HALVES = HD / 64;                 // 64-dim column boxes per row
  static constexpr int HALF_BYTES = ATT_UNIT * 128;      // one box: 64 rows x 64 dims bf16
  static constexpr int TILE = HALF_BYTES * HALVES;       // K (or V) of one unit
  static constexpr int STAGE = 2 * TILE;                 // K then V
  static constexpr int QSTRIDE = HD * 2 + 16;            // bytes per row of the bf16 Q tiles (padded)
  static constexpr int PSTRIDE = ATT_UNIT * 2 + 16;      // bytes per row of the bf16 P tiles (padded)
  // Q hi + lo tiles; once the CTA's units of a pair are done, its partial output [ROWS][HD] fp32
  static constexpr size_t OFF_Q = (size_t)ATT_STAGES * STAGE;
  // P hi + lo tiles in their own area; with two query tiles of 128 dimensions over the unit's K
  // tile, whose last reader has passed the barrier before P is written, so that three CTAs fit
  // on an SM (75.9 KB instead of 81.5): 32 heads, 11 rows, context 16384 67.8 -> 58.5 us, three
  // sequences of 16 rows, context 8000 111 -> 76, 11 rows, context 2048 14.5 -> 13.6.  (Three CTAs
  // leave 168 registers a thread, at which this instance spills 32 bytes; at two, 254 and no spill.)
  static constexpr bool P_OVER_K = QT == 2 && HD == 128;
  static constexpr size_t OFF_P = OFF_Q + 2 * ROWS * QSTRIDE;
  static constexpr size_t OFF_RED = OFF_P + (P_OVER_K ? 0 : 2 * ROWS * PSTRIDE);   // unit row max, sums; partial stats
  static constexpr size_t OFF_SEQ = OFF_RED + (128 + 2 * 16) * 4;                   // len, units [64]
  static constexpr size_t OFF_ANC = OFF_SEQ + (64 + 64) * 4;                        // [16] visible block rows per row
  static constexpr size_t OFF_BAR = (OFF_ANC + 16 * 4 + 7) / 8 * 8;
  static constexpr size_t SMEM = 1024 + OFF_BAR + ATT_STAGES * 8 + 16;
  static_assert(ROWS * HD * 4 <= 2 * ROWS * QSTRIDE, "the partial output fits in the Q tiles");
};

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
// D (16x8 fp32) += A (16x16 bf16, row) * B (16x8 bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo_elem, float hi_elem) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo_elem)) |
         ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi_elem)) << 16);
}

// QT: tiles of 8 query rows (1 for q <= 8, 2 for q <= 16)
template <int HD, int QT>
__global__ void __launch_bounds__(128, 3) attention_kernel(const __grid_constant__ AttnParams p) {
  using C = AttCfg<HD, QT>;
  constexpr int KSTEPS = HD / 16;          // MMA k-steps over the head dimension
  constexpr int MT = HD / 64;              // 16-dimension tiles per warp in V^T P^T
  constexpr int D4 = HD / 4;               // float4 columns of an output row
  constexpr int QI = QT * 8 * (HD / 2) / 128;   // (row, 2 dims) items of the q tiles per thread
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* Qh = smem + C::OFF_Q;                    // bf16 [ROWS][HD] (scaled q, hi part), padded rows
  uint8_t* Ql = Qh + C::ROWS * C::QSTRIDE;          // lo part
  float* po = reinterpret_cast<float*>(smem + C::OFF_Q);        // [ROWS][HD] partial output (after the units)
  float* red = reinterpret_cast<float*>(smem + C::OFF_RED);     // row-reduction scratch [4][16] max, [4][16] sums
  float* pml = red + 128;                                       // [ROWS][2] partial row max, exp-sum (after the units)
  int* len_seq = reinterpret_cast<int*>(smem + C::OFF_SEQ);     // [64] committed length of each sequence
  int* nu_seq = len_seq + 64;                                   // [64] units per head of each sequence
  uint32_t* anc_s = reinterpret_cast<uint32_t*>(smem + C::OFF_ANC);   // [16] block rows row j sees (bit i)
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);   // [ATT_STAGES] K and V of the stage landed
  volatile int* abort_flag = reinterpret_cast<volatile int*>(full + ATT_STAGES);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tig = lane & 3;
  const int mi = lane >> 3, r8 = lane & 7;        // ldmatrix: this thread's matrix and row
  const int q = p.q, H = p.H;
  const int CS = p.cs, NC = p.nclusters;
  const int rank = (int)cluster_ctarank(), cl = (int)blockIdx.x / CS;
  const unsigned long long t_entry = p.trace.rec ? globaltimer_ns() : 0;
  // In a forward the O projection starts beside this kernel.  A launch by itself lets nothing
  // start early: the clusters that a next attention launch could place beside this grid's (4 of 32
  // with 32 heads) leave the others to enter late.  32 heads, calls in a row, us, with an early
  // start -> without: 6 rows, context 500 6.9 -> 6.5, 1000 11.0 -> 8.7, 2048 13.4 -> 11.3; 16 rows,
  // 2048 15.1 -> 13.9, 4096 24.8 -> 22.4; 40 heads, 4096 21.1 -> 21.4; 16384 the same.
  if (!p.op) pdl_trigger();
  if (tid == 64) {   // the tensor maps into the TMA unit while the lengths are read
    tma_prefetch_desc(&p.kmap);
    tma_prefetch_desc(&p.vmap);
  }

  // In a block forward the committed lengths are final before this kernel can start: the
  // forward's first kernel (RMSNorm) lets its dependents launch only after every earlier kernel
  // has completed.  Slots below them are not written during this forward either.  Launched by
  // itself there is no such kernel in front: whatever precedes it (a commit, which lets its
  // dependents launch before it writes the lengths, a compaction of rows, the caller's own
  // kernels) has to complete before a length or a row is read.
  if (p.op) pdl_wait();
  if (tid < p.nb) {
    const int len = __ldcg(p.len + p.seq0 + tid);
    len_seq[tid] = len;
    nu_seq[tid] = (min(len + q, p.cap) + ATT_UNIT - 1) / ATT_UNIT;
  }
  if (tid == 0) {
    for (int s = 0; s < ATT_STAGES; ++s) mbar_init(&full[s], 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  const int npairs = p.nb * H;

  // this CTA's units [cb, ce) of pair pi (sequence pi / H, head pi % H)
  auto slice = [&](int pi, int& cb, int& ce) {
    const int nu = nu_seq[pi / H];
    cb = nu * rank / CS;
    ce = nu * (rank + 1) / CS;
  };
  // a position in the CTA's sequence of units: unit c of pair pi, its slice ending at ce
  struct Cursor {
    int pi, c, ce;
  };
  auto seek = [&](Cursor& u, int pi) {   // the first unit of the CTA's slices from pair pi on
    for (; pi < npairs; pi += NC) {
      int cb, ce;
      slice(pi, cb, ce);
      if (cb < ce) {
        u.pi = pi;
        u.c = cb;
        u.ce = ce;
        return;
      }
    }
    u.pi = npairs;
    u.c = u.ce = 0;
  };
  auto advance = [&](Cursor& u) {
    if (++u.c == u.ce) seek(u, u.pi + NC);
  };
  // first cache row of the cursor's unit, and whether all of its slots are committed
  auto unit_row = [&](const Cursor& u, bool& committed) {
    const int s = u.pi / H, hh = u.pi - s * H;
    committed = (u.c + 1) * ATT_UNIT <= len_seq[s];
    return p.row0 + ((p.seq0 + s) * H + hh) * p.cap + u.c * ATT_UNIT;
  };
  uint64_t pol = 0;
  auto issue = [&](int k, int row) {   // the CTA's unit k into stage k % ATT_STAGES
    uint8_t* st = smem + (size_t)(k % ATT_STAGES) * C::STAGE;
    uint64_t* bar = &full[k % ATT_STAGES];
    mbar_arrive_expect_tx(bar, C::STAGE);
#pragma unroll
    for (int hh = 0; hh < C::HALVES; ++hh) tma_load_2d(st + hh * C::HALF_BYTES, &p.kmap, bar, hh * 64, row, pol);
#pragma unroll
    for (int hh = 0; hh < C::HALVES; ++hh)
      tma_load_2d(st + C::TILE + hh * C::HALF_BYTES, &p.vmap, bar, hh * 64, row, pol);
  };
  auto prefetch = [&](int row) {   // a unit's K and V tiles into L2
#pragma unroll
    for (int hh = 0; hh < C::HALVES; ++hh) {
      tma_prefetch_l2_2d(&p.kmap, hh * 64, row);
      tma_prefetch_l2_2d(&p.vmap, hh * 64, row);
    }
  };
  // thread 0: units whose loads were issued, the next unit to load (isu) and the next
  // to prefetch into L2 (pfc, ATT_PREFETCH units past the ring)
  int issued = 0;
  Cursor isu{npairs, 0, 0}, pfc{npairs, 0, 0};
  if (tid == 0) {
    pol = l2_policy_evict_first();
    // Tiles of committed slots do not depend on the QKV projection: the first ones go
    // to the ring now, the next ATT_PREFETCH into L2 (and one more each time the ring is
    // refilled), so that the ring's loads are L2 hits instead of HBM round trips.
    seek(isu, cl);
    for (; issued < ATT_STAGES && isu.pi < npairs; ++issued) {
      bool committed;
      const int row = unit_row(isu, committed);
      if (!committed) break;
      issue(issued, row);
      advance(isu);
    }
    pfc = isu;
    for (int k = issued; k < ATT_STAGES && pfc.pi < npairs; ++k) advance(pfc);
    int cb0 = 0, ce0 = 0;
    if (cl < npairs) slice(cl, cb0, ce0);
    const int window = ce0 - cb0 >= ATT_LONG_SLICE ? 1 : ATT_PREFETCH;
    for (int k = 0; k < window && pfc.pi < npairs; ++k) {
      bool committed;
      const int row = unit_row(pfc, committed);
      if (committed) prefetch(row);
      advance(pfc);
    }
  }
  pdl_wait();   // q and this forward's new K/V rows come from the QKV projection
  const unsigned long long t_wait = p.trace.rec ? globaltimer_ns() : 0;
  if (tid == 0) {
    for (; issued < ATT_STAGES && isu.pi < npairs; ++issued) {
      bool committed;
      issue(issued, unit_row(isu, committed));
      advance(isu);
    }
  }
  unsigned long long t_k = 0, t_part = 0, t_merge = 0;
  unsigned pairs_done = 0;

  const float scale = rsqrtf((float)HD);
  const int kb = warp * 16;                       // first key (within the unit) of this warp's scores
  const int db = warp * (HD / 4);                 // first dimension of this warp's outputs
  // O^T of this warp's HD/4 dimensions (MT tiles of 16) x the query tiles, products with the
  // hi and with the lo part of P (summed when published); this thread holds query rows
  // t*8 + 2*tig + {0, 1} and keeps their running max and exp-sum in registers
  float O[MT][QT][4], Ol[MT][QT][4];
  float mr[QT][2], lr[QT][2];
  int k = 0;                                      // units of this CTA consumed (ring position)
  for (int pi = cl; pi < npairs; pi += NC) {
    const int sl = pi / H, h = pi - sl * H;
    int cb, ce;
    slice(pi, cb, ce);
#pragma unroll
    for (int t = 0; t < QT; ++t) mr[t][0] = mr[t][1] = -INFINITY, lr[t][0] = lr[t][1] = 0.f;
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int t = 0; t < QT; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) O[mt][t][e] = Ol[mt][t][e] = 0.f;
    if (cb < ce) {
      // ---- the rows' visible block rows (causal: 0..j; tree: the ancestors and the row
      // itself), q (scaled by 1/sqrt(hd)) as bf16 hi + lo, rows >= q zero; every load first
      if (tid < 16) anc_s[tid] = (p.anc && tid < q) ? __ldcg(p.anc + sl * q + tid) : (2u << tid) - 1u;
      float2 qv[QI];
#pragma unroll
      for (int r = 0; r < QI; ++r) {
        const int i = tid + 128 * r, j = i / (HD / 2), d = (i % (HD / 2)) * 2;
        qv[r] = j < q ? __ldcg(reinterpret_cast<const float2*>(p.Q + (size_t)(sl * q + j) * p.q_ld + h * HD + d))
                      : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int r = 0; r < QI; ++r) {
        const int i = tid + 128 * r, j = i / (HD / 2), d = (i % (HD / 2)) * 2;
        const float x0 = qv[r].x * scale, x1 = qv[r].y * scale;
        const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
        *reinterpret_cast<uint32_t*>(Qh + j * C::QSTRIDE + d * 2) =
            (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        *reinterpret_cast<uint32_t*>(Ql + j * C::QSTRIDE + d * 2) =
            pack_bf16(x0 - __bfloat162float(h0), x1 - __bfloat162float(h1));
      }
      __syncthreads();
    }
    const int len = len_seq[sl];
    const int nkeys = min(len + q, p.cap);
    for (int c = cb; c < ce; ++c, ++k) {
      const int c0 = c * ATT_UNIT;                  // slot of the unit's first key
      const uint8_t* Kt = smem + (size_t)(k % ATT_STAGES) * C::STAGE;
      const uint8_t* Vt = Kt + C::TILE;
      uint8_t* Ph = C::P_OVER_K ? const_cast<uint8_t*>(Kt) : smem + C::OFF_P;
      uint8_t* Pl = Ph + C::ROWS * C::PSTRIDE;
      // one decision per warp (mma.sync needs every lane; a wait can run out for some only)
      const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&full[k % ATT_STAGES], (k / ATT_STAGES) & 1,
                                                              abort_flag, p.err));
      if (k == 0 && p.trace.rec) t_k = globaltimer_ns();

      // ---- S^T = K Q^T for this warp's 16 keys: m16n8k16 with A = K (16 keys x 16 dims) and
      // B = Q^T (16 dims x 8 query rows), so up to 8 block rows fill one N = 8 tile
      float St[QT][4], Sl[QT][4];   // products with the hi and the lo part of q
#pragma unroll
      for (int t = 0; t < QT; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) St[t][e] = Sl[t][e] = 0.f;
      if (ok) {
#pragma unroll
        for (int kk = 0; kk < KSTEPS; ++kk) {
          const int hh = kk >> 2, cg = 2 * (kk & 3);  // 64-dim half and first 16-byte granule
          const int key = kb + r8 + 8 * (mi & 1), cc = cg + (mi >> 1);
          uint32_t a0, a1, a2, a3;
          ldsm_x4(smem_u32(Kt + hh * C::HALF_BYTES + key * 128 + ((cc ^ (key & 7)) << 4)), a0, a1, a2, a3);
#pragma unroll
          for (int t = 0; t < QT; ++t) {
            uint32_t bh0, bh1, bl0, bl1;   // q rows t*8 .. t*8+7: hi (matrices 0, 1), lo (2, 3)
            const uint8_t* qsrc = (mi >> 1) ? Ql : Qh;
            ldsm_x4(smem_u32(qsrc + (t * 8 + r8) * C::QSTRIDE + (kk * 16 + 8 * (mi & 1)) * 2), bh0, bh1, bl0, bl1);
            mma_bf16_16816(St[t], a0, a1, a2, a3, bh0, bh1);
            mma_bf16_16816(Sl[t], a0, a1, a2, a3, bl0, bl1);
          }
        }
#pragma unroll
        for (int t = 0; t < QT; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) St[t][e] += Sl[t][e];
      }
      // St[t][e] is the score of key kb + g + 8*(e >> 1) for query row t*8 + 2*tig + (e & 1).
      // mask: row j sees key slot kp iff kp < len, or kp = len + i for a block row i that
      // anc_s[j] marks (and kp < nkeys, j < q)
      // (a unit of committed slots only is seen whole by every row; rows j >= q are never
      // merged, so their unmasked scores of zero do no harm)
      if (!ok || c0 + ATT_UNIT > len) {
#pragma unroll
        for (int t = 0; t < QT; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = t * 8 + 2 * tig + (e & 1);
            const int kp = c0 + kb + g + 8 * (e >> 1);
            if (!ok || j >= q || kp >= nkeys || (kp >= len && !((anc_s[j] >> (kp - len)) & 1u))) St[t][e] = -INFINITY;
          }
      }
      // ---- the unit's row maxima: over the warp's lanes holding other keys (g), then the four
      // warps through shared memory; the running statistics stay in registers
      float* redm = red;          // [4 warps][16 rows] unit row maxima
      float* redl = red + 64;     // [4 warps][16 rows] unit row exp-sums
      float mx[QT][2];
#pragma unroll
      for (int t = 0; t < QT; ++t) {
        mx[t][0] = fmaxf(St[t][0], St[t][2]);
        mx[t][1] = fmaxf(St[t][1], St[t][3]);
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          mx[t][0] = fmaxf(mx[t][0], __shfl_xor_sync(0xffffffffu, mx[t][0], o));
          mx[t][1] = fmaxf(mx[t][1], __shfl_xor_sync(0xffffffffu, mx[t][1], o));
        }
        if (g == 0) {
          redm[warp * 16 + t * 8 + 2 * tig] = mx[t][0];
          redm[warp * 16 + t * 8 + 2 * tig + 1] = mx[t][1];
        }
      }
      __syncthreads();   // every warp is also done with the previous unit (its stage, P, red)
      if (tid == 0 && k >= 1 && isu.pi < npairs && !*abort_flag) {
        // refill the previous unit's stage with unit k + 1, extend the L2 window
        if (C::P_OVER_K) fence_proxy_async_smem();   // the load overwrites P, written by every thread
        bool committed;
        issue(issued, unit_row(isu, committed));
        advance(isu);
        ++issued;
        if (pfc.pi < npairs) {
          prefetch(unit_row(pfc, committed));
          advance(pfc);
        }
      }
      float al[QT][2];   // rescale of what the units before contributed
#pragma unroll
      for (int t = 0; t < QT; ++t)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int j = t * 8 + 2 * tig + i;
          const float mc = fmaxf(fmaxf(redm[j], redm[16 + j]), fmaxf(redm[32 + j], redm[48 + j]));
          const float mn = fmaxf(mr[t][i], mc);
          al[t][i] = (mn == -INFINITY) ? 1.f : __expf(mr[t][i] - mn);
          mr[t][i] = mn;
        }
      // ---- P^T = exp(S^T - m) as bf16 hi + lo, stored as P [query row][key], and its row sums
      float rs[QT][2];   // this thread's part of the unit row sums
#pragma unroll
      for (int t = 0; t < QT; ++t) {
        rs[t][0] = rs[t][1] = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int i = e & 1, j = t * 8 + 2 * tig + i, key = kb + g + 8 * (e >> 1);
          const float pv = (St[t][e] == -INFINITY) ? 0.f : __expf(St[t][e] - mr[t][i]);
          rs[t][i] += pv;
          const __nv_bfloat16 hi = __float2bfloat16_rn(pv);
          *reinterpret_cast<__nv_bfloat16*>(Ph + j * C::PSTRIDE + key * 2) = hi;
          *reinterpret_cast<__nv_bfloat16*>(Pl + j * C::PSTRIDE + key * 2) = __float2bfloat16_rn(pv - __bfloat162float(hi));
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          rs[t][0] += __shfl_xor_sync(0xffffffffu, rs[t][0], o);
          rs[t][1] += __shfl_xor_sync(0xffffffffu, rs[t][1], o);
        }
        if (g == 0) {
          redl[warp * 16 + t * 8 + 2 * tig] = rs[t][0];
          redl[warp * 16 + t * 8 + 2 * tig + 1] = rs[t][1];
        }
      }
      __syncthreads();   // P tiles and the row sums are complete
#pragma unroll
      for (int t = 0; t < QT; ++t)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int j = t * 8 + 2 * tig + i;
          lr[t][i] = lr[t][i] * al[t][i] + ((redl[j] + redl[16 + j]) + (redl[32 + j] + redl[48 + j]));
        }
      // ---- O^T = O^T * alpha + V^T P^T: A = V^T (16 dims x 16 keys, transposed loads of the V
      // tile), B = P^T (16 keys x 8 query rows), for this warp's dimensions and every query tile
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int t = 0; t < QT; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            O[mt][t][e] *= al[t][e & 1];
            Ol[mt][t][e] *= al[t][e & 1];
          }
      if (ok) {
#pragma unroll
        for (int kk = 0; kk < ATT_UNIT / 16; ++kk) {
          uint32_t va[MT][4];
#pragma unroll
          for (int mt = 0; mt < MT; ++mt) {
            const int key = kk * 16 + r8 + 8 * (mi >> 1);
            const int dim = db + 16 * mt + 8 * (mi & 1);
            const int hh = dim >> 6, cc = (dim & 63) >> 3;
            ldsm_x4_t(smem_u32(Vt + hh * C::HALF_BYTES + key * 128 + ((cc ^ (key & 7)) << 4)), va[mt][0], va[mt][1],
                      va[mt][2], va[mt][3]);
          }
#pragma unroll
          for (int t = 0; t < QT; ++t) {
            uint32_t ph0, ph1, pl0, pl1;   // P rows t*8 .. t*8+7, keys kk*16 ..: hi (0, 1), lo (2, 3)
            const uint8_t* psrc = (mi >> 1) ? Pl : Ph;
            ldsm_x4(smem_u32(psrc + (t * 8 + r8) * C::PSTRIDE + (kk * 16 + 8 * (mi & 1)) * 2), ph0, ph1, pl0, pl1);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
              mma_bf16_16816(O[mt][t], va[mt][0], va[mt][1], va[mt][2], va[mt][3], ph0, ph1);
              mma_bf16_16816(Ol[mt][t], va[mt][0], va[mt][1], va[mt][2], va[mt][3], pl0, pl1);
            }
          }
        }
      }
    }

    // ---- this CTA's partial for the pair into its own shared memory (the output over the
    // Q tiles, which no warp reads any more; the statistics beside the row-reduction
    // scratch): O^T[mt][t][e] is dimension db + 16*mt + g + 8*(e >> 1) of query row
    // t*8 + 2*tig + (e & 1); a CTA without units of the pair leaves (-inf, 0, 0)
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int t = 0; t < QT; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          po[(t * 8 + 2 * tig + (e & 1)) * HD + db + 16 * mt + g + 8 * (e >> 1)] = O[mt][t][e] + Ol[mt][t][e];
    if (warp == 0 && g == 0) {
#pragma unroll
      for (int t = 0; t < QT; ++t)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          pml[(t * 8 + 2 * tig + i) * 2] = mr[t][i];
          pml[(t * 8 + 2 * tig + i) * 2 + 1] = lr[t][i];
        }
    }
    if (p.trace.rec) t_part = globaltimer_ns();
    cluster_sync_all();   // the cluster's cs partials of the pair are complete
    // ---- merge this CTA's share of the pair's (row, 4 dimensions) outputs over the cs
    // partials, read from the cluster's shared memory: w_r = exp(m_r - max m),
    // L = sum_r w_r l_r, O = (sum_r w_r o_r) / L.  The second cluster barrier only keeps the
    // partials in place until every CTA has read them, so each thread arrives at it right
    // after its last remote loads and waits only at the end: the barrier's round trip
    // overlaps the merge arithmetic and the output stores.
    // Few threads have an item (18 of 128 with 11 CTAs), and this code runs once per launch and is
    // fetched cold, so G lanes share an item, each with at most six of the cs partials: one
    // thread with an unrolled loop over 16 took 1.5 us from the loads to the stores with 11 CTAs.
    // With 9 to 12 CTAs and more than 32 items (10 rows and up) two lanes and one pass instead of
    // four lanes and two: 16 rows, context 2048 14.8 -> 13.9 us (7B, four layers: 432.8 -> 430.8).
    bool arrived = false;
    {
      const int items = q * D4, i0 = items * rank / CS, i1 = items * (rank + 1) / CS;
      const int G = CS <= 4 ? 1 : (CS <= 8 || (CS <= 2 * ATT_MERGE && i1 - i0 > 32) ? 2 : 4), gl = tid & (G - 1), per = 128 / G;
      const int passes = (i1 - i0 + per - 1) / per;
#pragma unroll 1
      for (int pass = 0; pass < passes; ++pass) {
        const int mine = i0 + pass * per + tid / G, it = min(mine, i1 - 1);   // (every lane shuffles)
        const int j = it / D4, d4 = it - j * D4;
        const uint32_t a_ml = smem_u32(pml + 2 * j), a_o = smem_u32(po + j * HD + 4 * d4);
        float2 ml[ATT_MERGE];
        float4 ov[ATT_MERGE];
#pragma unroll
        for (int u = 0; u < ATT_MERGE; ++u) {
          const int r = gl + u * G;
          ml[u] = make_float2(-INFINITY, 0.f);
          ov[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (r < CS) {
            ml[u] = ld_dsmem_f2(mapa_shared(a_ml, r));
            ov[u] = ld_dsmem_f4(mapa_shared(a_o, r));
          }
        }
        if (pass + 1 == passes) {   // this thread's reads of the partials are done
          cluster_arrive_thread();
          arrived = true;
        }
        float mx = ml[0].x;
#pragma unroll
        for (int u = 1; u < ATT_MERGE; ++u) mx = fmaxf(mx, ml[u].x);
        for (int o = 1; o < G; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float L = 0.f;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < ATT_MERGE; ++u) {
          const float w = (ml[u].x == -INFINITY) ? 0.f : __expf(ml[u].x - mx);
          L += w * ml[u].y;
          a.x += w * ov[u].x;
          a.y += w * ov[u].y;
          a.z += w * ov[u].z;
          a.w += w * ov[u].w;
        }
        for (int o = 1; o < G; o <<= 1) {
          L += __shfl_xor_sync(0xffffffffu, L, o);
          a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
          a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
          a.z += __shfl_xor_sync(0xffffffffu, a.z, o);
          a.w += __shfl_xor_sync(0xffffffffu, a.w, o);
        }
        if (gl || mine >= i1) continue;
        const float iv = 1.0f / L;
        const float4 o = make_float4(a.x * iv, a.y * iv, a.z * iv, a.w * iv);
        const size_t idx = (size_t)(sl * q + j) * p.out_ld + h * HD + 4 * d4;
        *reinterpret_cast<float4*>(p.out + idx) = o;
        const __nv_bfloat16 h0 = __float2bfloat16_rn(o.x), h1 = __float2bfloat16_rn(o.y);
        const __nv_bfloat16 h2 = __float2bfloat16_rn(o.z), h3 = __float2bfloat16_rn(o.w);
        uint2 hi, lo;
        hi.x = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        hi.y = (uint32_t)__bfloat16_as_ushort(h2) | ((uint32_t)__bfloat16_as_ushort(h3) << 16);
        lo.x = pack_bf16(o.x - __bfloat162float(h0), o.y - __bfloat162float(h1));
        lo.y = pack_bf16(o.z - __bfloat162float(h2), o.w - __bfloat162float(h3));
        *reinterpret_cast<uint2*>(p.out_hi + idx) = hi;
        *reinterpret_cast<uint2*>(p.out_lo + idx) = lo;
      }
    }
    if (p.trace.rec) t_merge = globaltimer_ns();
    ++pairs_done;
    if (!arrived) cluster_arrive_thread();   // a thread without an item to merge
    cluster_wait_thread();   // every CTA of the cluster has read this CTA's partial
  }
  if (*abort_flag && tid == 0) {   // let the copies in flight land before the CTA exits
    for (int i = max(0, issued - ATT_STAGES); i < issued; ++i) {
      const uint64_t t0 = globaltimer_ns();
      while (!mbar_try_wait(&full[i % ATT_STAGES], (i / ATT_STAGES) & 1))
        if (globaltimer_ns() - t0 > WAIT_LIMIT_NS) break;
    }
  }
  if (tid == 0 && p.trace.rec)
    trace_write(p.trace, pairs_done | ((unsigned)k << 8), t_entry, t_wait, t_k, t_part, t_merge, globaltimer_ns());
}

size_t attention_smem_bytes(int hd, int q) {
  if (hd == 64) return q <= 8 ? AttCfg<64, 1>::SMEM : AttCfg<64, 2>::SMEM;
  return q <= 8 ? AttCfg<128, 1>::SMEM : AttCfg<128, 2>::SMEM;
}

namespace {
// most clusters of cs CTAs resident at once, per decode kernel instance (hd 64 / 128,
// one or two query tiles) and cs = 1 .. ATT_CS_MAX; 0 = that cluster size cannot launch
int g_att_clusters[2][2][ATT_CS_MAX + 1];
bool g_att_clusters_known = false;
int g_att_cs_cap = ATT_CS_MAX;   // SDSAT_ATT_CLUSTER_MAX: the largest cluster size launch_attention may pick

template <int HD, int QT>
cudaError_t prepare_decode_kernel(int (&maxc)[ATT_CS_MAX + 1]) {
  cudaError_t e;
  if ((e = prefer_shared(attention_kernel<HD, QT>)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(attention_kernel<HD, QT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)std::max<size_t>(AttCfg<HD, QT>::SMEM, ATT_TWO_PER_SM))) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(attention_kernel<HD, QT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) !=
      cudaSuccess)
    return e;
  for (int cs = 1; cs <= ATT_CS_MAX; ++cs) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs * 64);
    cfg.blockDim = dim3(128);
    cfg.dynamicSmemBytes = AttCfg<HD, QT>::SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, attention_kernel<HD, QT>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();   // this cluster size is not available: never chosen
      n = 0;
    }
    maxc[cs] = n;
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t attention_prepare() {
  cudaError_t e;
  if (!g_att_clusters_known) {
    const char* cap = std::getenv("SDSAT_ATT_CLUSTER_MAX");
    if (cap && cap[0]) g_att_cs_cap = std::max(1, std::min(ATT_CS_MAX, std::atoi(cap)));
    if ((e = prepare_decode_kernel<64, 1>(g_att_clusters[0][0])) != cudaSuccess) return e;
    if ((e = prepare_decode_kernel<64, 2>(g_att_clusters[0][1])) != cudaSuccess) return e;
    if ((e = prepare_decode_kernel<128, 1>(g_att_clusters[1][0])) != cudaSuccess) return e;
    if ((e = prepare_decode_kernel<128, 2>(g_att_clusters[1][1])) != cudaSuccess) return e;
    g_att_clusters_known = true;
  }
  return cudaSuccess;
}

void attention_grid(int pairs, const int* maxc, int cs_cap, int num_sms, int* cs, int* nclusters) {
  // One cluster per (sequence, head) pair, of the largest size cs that leaves room for
  // ATT_SPARE_CLUSTERS more clusters among the CTAs resident at once: clusters are placed
  // whole within one GPC, and grids that filled the GPU left some clusters waiting for
  // a second wave.  If not even pairs of CTAs fit, single CTAs (as many as are resident
  // at once) take several pairs each.
  const int resident = maxc[1] > 0 ? maxc[1] : 2 * num_sms;
  auto largest = [&](int cap) {
    for (int c = std::min(cap, ATT_CS_MAX); c >= 2; --c)
      if (maxc[c] >= pairs && c * (pairs + ATT_SPARE_CLUSTERS) <= resident) return c;
    return 1;
  };
  *cs = largest(cs_cap);
  // A tenth more clusters than pairs have to fit: 80 pairs (13B, two sequences) need nearly every
  // place that the QKV projection's CTAs leave for clusters of 5 (87 fit), and some of them enter
  // late.  13B, four layers, 5 CTAs -> 4: 6 rows, context 1024 589.6 -> 571.7 us, 8 rows, 3000 662.9
  // -> 627.3, 14 rows, 1000 691 -> 654.5.  (32, 40, 64, 96, 120 and 128 pairs: 12 to 23 % more fit,
  // and smaller clusters are no faster; with 32, 36 clusters of 11 fit, context 2048: 386.8 us for
  // four 7B layers against 391.3 with 10.)
  if (*cs > 2 && 10 * maxc[*cs] < 11 * pairs) *cs = largest(*cs - 1);
  *nclusters = *cs > 1 ? pairs : std::max(1, std::min(pairs, resident));
}

cudaError_t launch_attention(const AttnParams& p0, int num_sms, cudaStream_t st, bool pdl) {
  AttnParams p = p0;
  // No more CTAs per pair than the cache has units: the others only widened the merge (one
  // sequence, 32 heads, 6 rows, us: capacity 106 6.5 -> 5.5 a launch, 367 -> 362 for a 7B step of
  // four layers; 506 6.8 -> 6.5).
  const int units = (p.cap + ATT_UNIT - 1) / ATT_UNIT;
  attention_grid(p.nb * p.H, g_att_clusters[p.hd == 128][p.q > 8], std::min(g_att_cs_cap, units), num_sms, &p.cs,
                 &p.nclusters);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.nclusters * p.cs);
  cfg.blockDim = dim3(128);
  // Single CTAs that fit two to an SM: room for no third, or some SMs get three and others one
  // while the QKV projection's CTAs leave (four layers and LM head, us, without -> with: 7B, 7
  // sequences of 4 rows, context 2000 678 -> 665, 13B, 6 of 10 rows, context 1000 762 -> 736).
  cfg.dynamicSmemBytes = attention_smem_bytes(p.hd, p.q);
  if (p.cs == 1 && p.nclusters <= 2 * num_sms)
    cfg.dynamicSmemBytes = std::max<size_t>(cfg.dynamicSmemBytes, ATT_TWO_PER_SM);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  const bool one = p.q <= 8;
  if (p.hd == 64) return one ? cudaLaunchKernelEx(&cfg, attention_kernel<64, 1>, p) : cudaLaunchKernelEx(&cfg, attention_kernel<64, 2>, p);
  return one ? cudaLaunchKernelEx(&cfg, attention_kernel<128, 1>, p) : cudaLaunchKernelEx(&cfg, attention_kernel<128, 2>, p);
}

}  // namespace sdsat
