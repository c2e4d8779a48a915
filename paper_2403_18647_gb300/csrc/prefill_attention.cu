// Causal attention of a prefill chunk over the KV cache: flash attention on tcgen05.
//
// One CTA per (head, NT tiles of 128 chunk positions), heaviest blocks first; blocks of 128
// keys.  Per tile and block, with accumulators and probabilities in TMEM:
//   S = Qhi K^T + Qlo K^T          (A and B from shared memory, 128 x 128 fp32)
//   P = exp2(c S - m), as bf16 hi + lo over S's own columns
//   O += Phi V + Plo V             (A from TMEM, V as the MN-major B operand)
// K and V are the cache's bf16 values, Q and P enter as hi + lo pairs (16 bits), sums are fp32.
//
// What bounds it: the four 128^3 products of a (tile, block), 2048 tensor cycles, against
// about 1200 issue cycles of softmax per warp.  So two tiles take turns (NT = 2): while one
// tile's 128 threads (a row each, no shuffles) work on its scores, the tensor cores run the
// other tile's products.  With few blocks NT = 1 spreads the work over more SMs.  TMEM: S and
// O of two tiles are all 512 columns, so P has to take S's place; the next S is issued after
// the P V product that reads it, in order, by the same thread.
//
// O is rescaled only when a row's maximum has grown by more than 2^8 since the last time
// (exact: the reference value cancels in the division by the row's sum; P stays below 2^8).
//
// Measured, 32 heads x 128, us per launch: 4095 positions 254 (872 with mma.sync m16n8k16 on
// 64-position blocks, whose K and V fragments each warp read from shared memory again), 2047
// 81 (256), 512 23 (43), 99 12.3 (20); at 4095 1.08 PFLOP/s executed.
//
// Warps 0-3: TMA (warp 0), MMA issue and TMEM (warp 1), two idle; warps 4-7 and 8-11: softmax
// and output of tile 0 and 1.  Shared memory: Q 64 KB per tile, a ring of three 32 KB slots in
// which K and V blocks alternate (hd 128).
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sdsat {

constexpr int PA_ROWS = 128;      // chunk positions per tile, and keys per block
constexpr int PA_SLOTS = 3;
constexpr int PA_THREADS = 384;
constexpr float PA_LAZY = 8.0f;   // log2 of the growth of a row maximum that is left unscaled

template <int HD>
struct PaCfg {
  static constexpr int HALVES = HD / 64;
  static constexpr int BOX = 64 * 128;                      // one TMA box of K or V: 64 keys x 64 dims
  static constexpr int HALF = PA_ROWS * 128;                // 128 rows x 64 dims, 128-byte swizzle
  static constexpr int TILE = HALVES * HALF;                // Q hi, Q lo, K or V: 128 rows
  static constexpr size_t OFF_RING = 2 * 2 * (size_t)TILE;  // after Q hi + lo of two tiles
  static constexpr size_t OFF_BAR = OFF_RING + (size_t)PA_SLOTS * TILE;
  static constexpr int NBAR = 2 * PA_SLOTS + 2 * 4 + 1;
  static constexpr size_t SMEM = 1024 + OFF_BAR + NBAR * 8 + 16;
  static_assert(SMEM <= 232448, "shared memory of one CTA");
};

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// D[tmem] (+)= A[tmem] * B[smem]: A's rows on the lanes, two bf16 of K per column
__device__ __forceinline__ void umma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// MN-major operand in the 128-byte swizzle layout: atoms of 64 dims (128 bytes) x 8 keys;
// `lead` bytes to the next 64 dims, 1024 to the next 8 keys
__device__ __forceinline__ uint64_t sdesc_sw128_mn(uint32_t saddr, uint32_t lead) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(lead >> 4) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// (a, b) as packed bf16 hi parts and packed bf16 lo parts (a in the low half)
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
  const float ra = a - __uint_as_float(hi << 16), rb = b - __uint_as_float(hi & 0xFFFF0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(rb), "f"(ra));
}

template <int HD>
__global__ void __launch_bounds__(PA_THREADS, 1) prefill_attention_kernel(const __grid_constant__ PfAttnParams p) {
  using C = PaCfg<HD>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* ring = smem + C::OFF_RING;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);   // [PA_SLOTS] K or V block landed
  uint64_t* empty = full + PA_SLOTS;      // [PA_SLOTS] its products are done
  uint64_t* q_full = empty + PA_SLOTS;    // [2] per tile: Q landed
  uint64_t* s_full = q_full + 2;          // [2] S of a block is complete (and everything issued before it)
  uint64_t* p_full = s_full + 2;          // [2] P is in TMEM, O is rescaled (128 threads)
  uint64_t* o_full = p_full + 2;          // [2] the last product is complete
  uint64_t* drain = o_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rows = p.tiles * PA_ROWS, nqb = (p.M + rows - 1) / rows;
  const int q0 = (nqb - 1 - (int)blockIdx.x / p.H) * rows, h = (int)blockIdx.x % p.H;
  const int nt = p.tiles == 2 && q0 + PA_ROWS < p.M ? 2 : 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < PA_SLOTS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&q_full[t], 1);
      mbar_init(&s_full[t], 1);
      mbar_init(&p_full[t], 128);
      mbar_init(&o_full[t], 1);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&p.kmap);
    tma_prefetch_desc(&p.vmap);
    tma_prefetch_desc(&p.qmap[0]);
    tma_prefetch_desc(&p.qmap[1]);
  }
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;   // S of tile t at column 128 t, O at 256 + 128 t
  pdl_trigger();
  pdl_wait();   // q and this chunk's K / V rows come from the QKV projection
  const int len = __ldcg(p.len + p.seq);
  // keys tile t's positions may see, and their blocks (tile 1 sees at least as many as tile 0)
  auto keys = [&](int t) { return len + min(q0 + (t + 1) * PA_ROWS, p.M); };
  auto blocks = [&](int t) { return (keys(t) + PA_ROWS - 1) / PA_ROWS; };
  const int nb = blocks(nt - 1);

  if (warp == 0) {
    if (lane == 0) {
      const uint64_t pol = l2_policy_evict_last();   // K and V are read by every block of positions
      const int rowbase = p.row0 + (p.seq * p.H + h) * p.cap;
      for (int t = 0; t < nt; ++t) {
        mbar_arrive_expect_tx(&q_full[t], 2 * C::TILE);
        for (int part = 0; part < 2; ++part)
          for (int hh = 0; hh < C::HALVES; ++hh)
            tma_load_2d(smem + (size_t)(2 * t + part) * C::TILE + hh * C::HALF, &p.qmap[part], &q_full[t],
                        h * HD + hh * 64, q0 + t * PA_ROWS, pol);
      }
      int it = 0;
      for (; it < 2 * nb; ++it) {   // K of block 0, V of block 0, K of block 1, ...
        const int s = it % PA_SLOTS;
        if (!mbar_wait_bounded(&empty[s], ((it / PA_SLOTS) & 1) ^ 1, abort_flag, p.err)) break;
        mbar_arrive_expect_tx(&full[s], C::TILE);
        const CUtensorMap* map = (it & 1) ? &p.vmap : &p.kmap;
        const int row = rowbase + (it >> 1) * PA_ROWS;
        for (int hh = 0; hh < C::HALVES; ++hh)
          for (int b = 0; b < 2; ++b)
            tma_load_2d(ring + (size_t)s * C::TILE + hh * C::HALF + b * C::BOX, map, &full[s], hh * 64, row + b * 64,
                        pol);
      }
      if (*abort_flag) {   // let the copies in flight land before the CTA exits
        auto land = [&](uint64_t* bar, uint32_t parity) {
          const uint64_t t0 = globaltimer_ns();
          while (!mbar_try_wait(bar, parity))
            if (globaltimer_ns() - t0 > WAIT_LIMIT_NS) break;
        };
        for (int t = 0; t < nt; ++t) land(&q_full[t], 0);
        for (int i = max(0, it - PA_SLOTS); i < it; ++i) land(&full[i % PA_SLOTS], (i / PA_SLOTS) & 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc_s = idesc_bf16_f32(128, PA_ROWS);
      constexpr uint32_t idesc_o = idesc_bf16_f32(128, HD) | (1u << 16);   // B is MN-major
      bool ok = true;
      auto wait = [&](uint64_t* bar, uint32_t parity) {
        ok = ok && mbar_wait_bounded(bar, parity, abort_flag, p.err);
        if (ok) tc_fence_after();
        return ok;
      };
      auto qk = [&](int t, int j) {
        const uint32_t k = smem_u32(ring + (size_t)((2 * j) % PA_SLOTS) * C::TILE);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const uint32_t q = smem_u32(smem + (size_t)(2 * t + part) * C::TILE);
#pragma unroll
          for (int kk = 0; kk < HD / 16; ++kk) {
            const uint32_t o = (kk >> 2) * C::HALF + (kk & 3) * 32;
            umma_bf16(tmem + 128 * t, sdesc_sw128(q + o), sdesc_sw128(k + o), idesc_s, part | kk ? 1u : 0u);
          }
        }
        umma_commit(&s_full[t]);
      };
      auto pv = [&](int t, int j) {
        const uint32_t v = smem_u32(ring + (size_t)((2 * j + 1) % PA_SLOTS) * C::TILE);
        // the last block stops at the 16 keys that hold the tile's last one
        const int steps = min(PA_ROWS / 16, (keys(t) - j * PA_ROWS + 15) / 16);
        for (int part = 0; part < 2; ++part)
          for (int kk = 0; kk < steps; ++kk)
            umma_bf16_ta(tmem + 256 + 128 * t, tmem + 128 * t + part * 64 + kk * 8,
                         sdesc_sw128_mn(v + kk * 2048, C::HALF), idesc_o, j | part | kk ? 1u : 0u);
        if (j == blocks(t) - 1) umma_commit(&o_full[t]);
      };
      for (int t = 0; t < nt && ok; ++t) wait(&q_full[t], 0);
      // step j: per tile, block j - 1's P V and then block j's S over the P it has read; the last
      // tile has every block, so its products release V of block j - 1 and K of block j
      for (int j = 0; j <= nb && ok; ++j) {
        const int ks = (2 * j) % PA_SLOTS, vs = (2 * j + PA_SLOTS - 1) % PA_SLOTS;
        for (int t = 0; t < nt && ok; ++t) {
          const int n = blocks(t);
          if (j > 0 && j <= n && wait(&full[vs], ((2 * j - 1) / PA_SLOTS) & 1) && wait(&p_full[t], (j - 1) & 1)) {
            pv(t, j - 1);
            if (t == nt - 1) umma_commit(&empty[vs]);
          }
          if (j < n && ok && wait(&full[ks], (2 * j / PA_SLOTS) & 1)) {
            qk(t, j);
            if (t == nt - 1) umma_commit(&empty[ks]);
          }
        }
      }
      if (*abort_flag) {   // wait for issued MMAs before shared memory goes away
        umma_commit(drain);
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(drain, 0))
          if (globaltimer_ns() - t0 > WAIT_LIMIT_NS) break;
      }
    }
  } else if (warp >= 4 && (warp >> 2) - 1 < nt) {
    const int t = (warp >> 2) - 1, e = warp & 3;
    const uint32_t lane_off = (uint32_t)(e * 32) << 16;
    const uint32_t ts = tmem + lane_off + 128 * t, to = tmem + lane_off + 256 + 128 * t;
    const int row = q0 + t * PA_ROWS + e * 32 + lane;     // this thread's chunk position
    const int pos0 = len + q0 + t * PA_ROWS + e * 32;     // position of the warp's first row
    const int n = blocks(t);
    const float c = rsqrtf((float)HD) * 1.4426950408889634f;
    float m = 0.f, l = 0.f;   // reference exponent (log2) and the row's sum relative to it
    bool ok = true;
    for (int j = 0; j < n; ++j) {
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(&s_full[t], j & 1, abort_flag, p.err));
      if (!ok) break;
      tc_fence_after();
      float s[PA_ROWS];
#pragma unroll
      for (int i = 0; i < 4; ++i) tmem_ld32(ts + 32 * i, s + 32 * i);
      tmem_wait_ld();
      if ((j + 1) * PA_ROWS - 1 > pos0) {   // key j*128 + i is visible iff it is at or before the row's position
        const int last = pos0 + lane - j * PA_ROWS;
#pragma unroll
        for (int i = 0; i < PA_ROWS; ++i)
          if (i > last) s[i] = -INFINITY;
      }
      float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
      for (int i = 4; i < PA_ROWS; ++i) mx[i & 3] = fmaxf(mx[i & 3], s[i]);
      const float mb = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * c;
      if (j == 0) {
        m = mb;   // block 0 holds key 0, which every row sees
      } else {
        // the S that is ready was issued after block j - 1's P V product: O holds blocks 0 .. j-1
        const bool grow = mb > m + PA_LAZY;
        if (__any_sync(0xffffffffu, grow)) {
          const float f = grow ? ex2(m - mb) : 1.f;
          l *= f;
          if (grow) m = mb;
#pragma unroll 1
          for (int i = 0; i < HD; i += 16) {
            float o[16];
            uint32_t u[16];
            tmem_ld16(to + i, o);
            tmem_wait_ld();
#pragma unroll
            for (int x = 0; x < 16; ++x) u[x] = __float_as_uint(o[x] * f);
            tmem_st16(to + i, u);
          }
        }
      }
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < PA_ROWS; i += 32) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int x = 0; x < 16; ++x) {
          const float a = ex2(fmaf(s[i + 2 * x], c, -m)), b = ex2(fmaf(s[i + 2 * x + 1], c, -m));
          sum[(2 * x) & 3] += a;
          sum[(2 * x + 1) & 3] += b;
          split2(a, b, hi[x], lo[x]);
        }
        tmem_st16(ts + i / 2, hi);
        tmem_st16(ts + 64 + i / 2, lo);
      }
      l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&p_full[t]);
    }
    ok = ok && mbar_wait_bounded(&o_full[t], 0, abort_flag, p.err);
    if (__all_sync(0xffffffffu, ok)) {
      tc_fence_after();
      const float inv = 1.0f / l;
#pragma unroll 1
      for (int i = 0; i < HD; i += 16) {
        float o[16];
        tmem_ld16(to + i, o);
        tmem_wait_ld();
        if (row < p.M) {
          uint32_t hi[8], lo[8];
#pragma unroll
          for (int x = 0; x < 8; ++x) split2(o[2 * x] * inv, o[2 * x + 1] * inv, hi[x], lo[x]);
          const size_t at = (size_t)row * p.out_ld + h * HD + i;
          uint4* dh = reinterpret_cast<uint4*>(p.out_hi + at);
          uint4* dl = reinterpret_cast<uint4*>(p.out_lo + at);
          dh[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          dh[1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
          dl[0] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          dl[1] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

cudaError_t prefill_attention_prepare() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(prefill_attention_kernel<64>, a, (int)PaCfg<64>::SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prefill_attention_kernel<128>, a, (int)PaCfg<128>::SMEM);
  if (e == cudaSuccess) e = prefer_shared(prefill_attention_kernel<64>);
  if (e == cudaSuccess) e = prefer_shared(prefill_attention_kernel<128>);
  return e;
}

cudaError_t launch_prefill_attention(PfAttnParams& p, int num_sms, cudaStream_t st, bool pdl) {
  // two tiles a CTA once that still gives every SM a CTA
  p.tiles = (p.M + 2 * PA_ROWS - 1) / (2 * PA_ROWS) * p.H >= num_sms ? 2 : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((p.M + p.tiles * PA_ROWS - 1) / (p.tiles * PA_ROWS) * p.H);
  cfg.blockDim = dim3(PA_THREADS);
  cfg.dynamicSmemBytes = p.hd == 64 ? PaCfg<64>::SMEM : PaCfg<128>::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return p.hd == 64 ? cudaLaunchKernelEx(&cfg, prefill_attention_kernel<64>, p)
                    : cudaLaunchKernelEx(&cfg, prefill_attention_kernel<128>, p);
}

}  // namespace sdsat
