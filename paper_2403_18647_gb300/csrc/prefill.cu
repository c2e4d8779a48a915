// Prefill: the prompt's positions through the model in chunks of up to PF_ROWS, before the
// decode loop.  Unlike the decode step (a handful of rows, bound by the weight stream), a
// chunk of hundreds of positions makes every projection a dense contraction, so it runs
// on a tiled tensor-core GEMM:
//
//   Y[m][n] = sum_k X[m][k] W[n][k], one tile = 256 weight rows x TOK positions per CTA pair.
//
// The weight rows are the MMA's A operand (cta_group::2, M = 256: 128 rows from each CTA's
// shared memory), the positions its B operand: the bf16 hi parts of X in rank 0, the lo parts
// in rank 1, together N = 2 TOK, so one tcgen05.mma per 16-wide k-step computes W*Xhi and
// W*Xlo side by side in TMEM and the epilogue adds the two halves (fp32-like activations,
// exact bf16 weights, fp32 accumulation -- the decode path's precision).
//
// What bounds it: with many positions the tensor cores (twice 2 M N K FLOPs because of hi +
// lo); with few the L2 -> SM traffic of weights and positions (about 11 TB/s over the GPU
// when the weights come from HBM).  A tile of one CTA (128 x 128) asked L2 for 96 bytes per
// clock and SM and ran at that limit; a pair shares the positions and asks for 64.  M = 512,
// K = 4096, N = 12288 / 22016: 82.0 / 129.4 us with single CTAs, 63 / 106 us with pairs.
//
// One persistent pair per two SMs: per CTA six 32 KB TMA stages (eight of 24 KB for TOK = 64),
// two TMEM accumulators so that a tile's epilogue overlaps the next tile's MMAs; warp 0
// streams TMA, warp 1 of rank 0 issues the MMAs for the pair, warps 2-9 drain TMEM.  The
// tiles of an incomplete wave are split along K over all the pairs and come first, so that
// their reduction overlaps the whole tiles that follow.
// TOK = 64 for at most 64 positions: half the position traffic and half the split parts.
//
// Epilogues: store; RoPE and the KV append (QKV); residual add (O and down projections), which
// also emits the next RMSNorm's operand h * g and per-tile sums of h^2, as the decode GEMM
// does, so that the consuming GEMM (QKV, gate/up, the LM head) only scales its result by each
// position's factor; SiLU(gate) * up as the down projection's bf16 hi + lo operand.  RMSNorm and
// RoPE as row kernels of their own cost two more passes over the chunk's rows each (2047
// positions: 34 us per RMSNorm, 59 us per RoPE + append).  Attention is prefill_attention.cu.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sdsat {

constexpr int PF_W_BYTES = 128 * 128;                    // a CTA's 128 weight rows x 64 bf16
constexpr int PF_CHUNK = 32;                             // positions per epilogue round
constexpr int PF_EPI_WARPS = 8;                          // two per TMEM lane quarter
constexpr int PF_THREADS = 64 + 32 * PF_EPI_WARPS;
constexpr int PF_STAGING = 2 * 128 * PF_CHUNK;           // fp32 slabs of the two epilogue groups
constexpr int PF_GROUP = 8;                              // position blocks numbered together (16: no better, 32: 4 % slower)
constexpr int PF_TOK = 128;                              // positions per tile, at most
constexpr int PF_SK_MIN = 4;                             // chunks of a split-K share, at least

// TOK: positions per tile, 128 or 64
template <int TOK>
struct PfCfg {
  static constexpr int STAGES = TOK == 128 ? 6 : 8;
  static constexpr int X_BYTES = TOK * 128;              // TOK positions x 64 bf16: hi in rank 0, lo in rank 1
  static constexpr int STAGE = PF_W_BYTES + X_BYTES;     // per CTA: 32 KB (24 KB)
  static constexpr int RING = STAGES * STAGE;
  static constexpr int ACC = 2 * TOK;                    // TMEM columns of one accumulator (hi, lo)
  static constexpr int NBAR = 2 * STAGES + 7;
  static constexpr size_t SMEM = 1024 + (size_t)RING + PF_STAGING * 4 + 2 * TOK * 4 + NBAR * 8 + 64;
  static_assert(SMEM <= 232448, "shared memory of one CTA");
};

__device__ __forceinline__ void pf_tile_half_src(int map_mode, int rows_per_map, int t, int h, int& map, int& row) {
  if (map_mode == MAP_GATEUP) {
    map = h;
    row = 64 * t;
  } else if (map_mode == MAP_QKV3) {
    const int g = 128 * t;
    map = g / rows_per_map;
    row = g % rows_per_map + 64 * h;
  } else {
    map = 0;
    row = 128 * t + 64 * h;
  }
}

// A pair's work in order: its share of the split tiles 0 .. sk_tiles-1 (a flat range of
// (tile, chunk) units, less than one tile's worth, so parts of at most two tiles), then the
// whole tiles sk_tiles + pair, + P, ...  All roles of both CTAs walk the same list.  Splitting
// one more wave (two or three parts a tile instead of up to ten) was no better: M = 256,
// N = 12288 39.5 us against 34.4, M = 512, N = 22016 100.2 against 102.9.
struct PfWalk {
  int u, u1, t, T, P, kc;
  int tile, k0, k1;   // the current segment
  __device__ PfWalk(const PfGemmParams& p, int pair) {
    kc = p.kc;
    T = p.n_pairs_w * p.n_tblocks;
    P = gridDim.x >> 1;
    const int U = p.sk_tiles * kc;
    u = pair < p.sk_pairs ? pair * U / p.sk_pairs : 0;
    u1 = pair < p.sk_pairs ? (pair + 1) * U / p.sk_pairs : 0;
    t = p.sk_tiles + pair;
  }
  __device__ bool done() const { return u >= u1 && t >= T; }   // no segment after the current one
  __device__ bool next() {
    if (u < u1) {
      tile = u / kc;
      k0 = u - tile * kc;
      k1 = min(kc, k0 + u1 - u);
      u += k1 - k0;
      return true;
    }
    if (t >= T) return false;
    tile = t;
    k0 = 0;
    k1 = kc;
    t += P;
    return true;
  }
};

// Tile -> (pair of weight tiles, position block).  Position blocks go in groups of p.group:
// within a group the tiles are numbered weight-major, so the pairs working at the same time
// share a few weight tiles and the group's positions through L2.
__device__ __forceinline__ void pf_tile(const PfGemmParams& p, int tile, int& wp, int& tb) {
  const int per = p.n_pairs_w * p.group, g = tile / per, rem = tile - g * per;
  const int width = min(p.group, p.n_tblocks - g * p.group);
  wp = rem / width;
  tb = g * p.group + rem - wp * width;
}

// two bf16 in a word (a in the low half); four values as bf16 hi + lo at element o (8-byte aligned)
__device__ __forceinline__ uint32_t pf_pack(float a, float b) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
         ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}
__device__ __forceinline__ void pf_store4(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t o, float a, float b, float c,
                                          float d) {
  const uint32_t h0 = pf_pack(a, b), h1 = pf_pack(c, d);
  *reinterpret_cast<uint2*>(hi + o) = make_uint2(h0, h1);
  *reinterpret_cast<uint2*>(lo + o) =
      make_uint2(pf_pack(a - __uint_as_float(h0 << 16), b - __uint_as_float(h0 & 0xFFFF0000u)),
                 pf_pack(c - __uint_as_float(h1 << 16), d - __uint_as_float(h1 & 0xFFFF0000u)));
}

// sequence, cache slot and RoPE position of row m (len0: the length when all rows are of seq0)
struct PfRow {
  int seq, slot, pos;
  __device__ PfRow(const PfGemmParams& p, int m, int len0) {
    const int s = m < p.q ? 0 : m / p.q;
    seq = p.seq0 + s;
    slot = (p.q >= p.M ? len0 : __ldcg(p.len + seq)) + m - s * p.q;
    pos = p.positions ? __ldcg(p.positions + m) : slot;
  }
  __device__ void report(const PfGemmParams& p) const {   // (by one thread of a row)
    if (slot >= p.cap) set_error(p.err, ERR_CAPACITY);
    if (pos < 0 || pos >= p.rope_len) set_error(p.err, ERR_POSITION);
  }
};
// rotate-half RoPE of a head's dimensions i .. i + 3 (a) and i + hd/2 .. (b)
__device__ __forceinline__ void pf_rope4(const PfGemmParams& p, int pos, int i, float4& a, float4& b) {
  const float4* cs =
      reinterpret_cast<const float4*>(p.rope + (size_t)min(max(pos, 0), p.rope_len - 1) * (p.hd >> 1) + i);
  const float4 t0 = __ldg(cs), t1 = __ldg(cs + 1);   // cos, sin of two frequencies each
  const float4 o = a;
  a = make_float4(a.x * t0.x - b.x * t0.y, a.y * t0.z - b.y * t0.w, a.z * t1.x - b.z * t1.y, a.w * t1.z - b.w * t1.w);
  b = make_float4(b.x * t0.x + o.x * t0.y, b.y * t0.z + o.y * t0.w, b.z * t1.x + o.z * t1.y, b.w * t1.z + o.w * t1.w);
}
// features f .. f + 3 (a) and f + hd/2 .. (b) of row m: q in fp32 or as bf16 hi + lo, k and v into
// the row's cache slot when there is one
__device__ __forceinline__ void pf_qkv_store(const PfGemmParams& p, int which, int m, const PfRow& r, int f, int i,
                                             const float4& a, const float4& b) {
  const int half = p.hd >> 1;
  if (which == 0) {
    const size_t o = (size_t)m * p.out_ld + f;
    if (p.out) {
      *reinterpret_cast<float4*>(p.out + o) = a;
      *reinterpret_cast<float4*>(p.out + o + half) = b;
    } else {
      pf_store4(p.out_hi, p.out_lo, o, a.x, a.y, a.z, a.w);
      pf_store4(p.out_hi, p.out_lo, o + half, b.x, b.y, b.z, b.w);
    }
  } else if (r.slot < p.cap) {
    __nv_bfloat16* dst = (which == 1 ? p.k_layer : p.v_layer) +
                         ((size_t)(r.seq * p.H + (f - i) / p.hd) * p.cap + r.slot) * p.hd + i;
    *reinterpret_cast<uint2*>(dst) = make_uint2(pf_pack(a.x, a.y), pf_pack(a.z, a.w));
    *reinterpret_cast<uint2*>(dst + half) = make_uint2(pf_pack(b.x, b.y), pf_pack(b.z, b.w));
  }
}

__device__ __forceinline__ void pf_drain(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity))
    if (globaltimer_ns() - t0 > WAIT_LIMIT_NS) break;
}

template <int TOK>
__global__ void __launch_bounds__(PF_THREADS, 1) prefill_gemm_kernel(const __grid_constant__ PfGemmParams p) {
  using C = PfCfg<TOK>;
  constexpr int S = C::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stages = smem;
  float* staging = reinterpret_cast<float*>(smem + C::RING);
  float* s_inv = staging + PF_STAGING;    // [2][TOK] RMSNorm factors of a tile's positions
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_inv + 2 * TOK);
  uint64_t* full = bars;                  // rank 0: both CTAs' weights and positions landed (TMA)
  uint64_t* empty = bars + S;     // the stage was consumed by the tensor cores
  uint64_t* acc_full = bars + 2 * S;   // [2] accumulator ready
  uint64_t* acc_empty = acc_full + 2;          // [2] rank 0: accumulator drained in both CTAs
  uint64_t* drain = acc_empty + 2;
  uint64_t* red_bar = drain + 1;               // parts of the tile being reduced landed (bulk copies)
  uint64_t* res_bar = red_bar + 1;             // a round's residual rows landed in the slabs
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(res_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* s_last = reinterpret_cast<int*>(tmem_slot + 2);
  // trace marks of the epilogue: after the dependency wait, first and last accumulator, last tile summed
  unsigned long long t_wait = 0, t_acc0 = 0, t_acc1 = 0, t_sum = 0;
  const unsigned long long t_entry = p.trace.rec ? globaltimer_ns() : 0;
  unsigned t_flags = 0;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank(), pair = (int)blockIdx.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * PF_EPI_WARPS);
    }
    mbar_init(drain, 1);
    mbar_init(red_bar, 1);
    mbar_init(res_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (threadIdx.x == 64) {
    const int nmaps = p.map_mode == MAP_QKV3 ? 3 : (p.map_mode == MAP_GATEUP ? 2 : 1);
    for (int i = 0; i < nmaps; ++i) tma_prefetch_desc(&p.tmap[i]);
    tma_prefetch_desc(&p.tmap_x[rank]);
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, 2 * C::ACC);
  tc_fence_before();
  cluster_sync_all();   // both CTAs' barriers are initialised before either signals the other's
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();

  if (warp == 0) {
    // ------------------------------------------------ weight + position stream (TMA)
    if (lane == 0) {
      // A weight tile is read by the pairs of every position block at about the same time.  With
      // few blocks nothing else of it is worth keeping: evicted first, the weights leave the
      // operands and the split parts in L2 (two 7B layers, 99 positions: 315 us against 273; 200:
      // 370 and 355).  With more they are needed again: 500 rows, N = 12288 76.9 us against 79.7.
      const uint64_t pol_w = p.n_tblocks <= 2 ? l2_policy_evict_first() : l2_policy_evict_normal();
      const uint64_t pol_x = l2_policy_evict_last();    // a position block is read by every weight tile
      PfWalk w(p, pair);
      bool more = w.next();
      int kc = w.k0, map0, row0, map1, row1, tb = 0;
      auto src = [&] {   // the CTA's weight tile (past the last one: that one, unused)
        int wp;
        pf_tile(p, w.tile, wp, tb);
        const int wt = min(2 * wp + rank, p.n_wtiles - 1);
        pf_tile_half_src(p.map_mode, p.rows_per_map, wt, 0, map0, row0);
        pf_tile_half_src(p.map_mode, p.rows_per_map, wt, 1, map1, row1);
      };
      auto step = [&] {   // to the next (tile, chunk); true when the tile changed
        if (++kc < w.k1) return false;
        more = w.next();
        kc = w.k0;
        return true;
      };
      auto load_w = [&](int s, uint32_t bar) {
        uint8_t* dst = stages + (size_t)s * C::STAGE;
        tma_load_2d_pair(dst, &p.tmap[map0], bar, kc * 64, row0, pol_w);
        tma_load_2d_pair(dst + 8192, &p.tmap[map1], bar, kc * 64, row1, pol_w);
      };
      auto load_x = [&](int s, uint32_t bar, int k, int tb) {
        tma_load_2d_pair(stages + (size_t)s * C::STAGE + PF_W_BYTES, &p.tmap_x[rank], bar, k * 64, tb * TOK, pol_x);
      };
      // the weights of the first stages do not depend on the previous kernel
      int xk[S], xt[S], npre = 0;
      src();
#pragma unroll
      for (int s = 0; s < S; ++s) {
        xk[s] = kc;
        xt[s] = tb;
        if (!more) continue;
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * C::STAGE);
        load_w(s, mapa_shared(smem_u32(&full[s]), 0));
        npre = s + 1;
        if (step() && more) src();
      }
      pdl_wait();   // the positions are the previous kernel's output
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (s < npre) load_x(s, mapa_shared(smem_u32(&full[s]), 0), xk[s], xt[s]);
      int it = npre, s = it % S;
      uint32_t ph = 0;   // parity of the stage's previous use being consumed
      while (more) {
        if (!mbar_wait_bounded(&empty[s], ph, abort_flag, p.err)) break;
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * C::STAGE);
        const uint32_t bar = mapa_shared(smem_u32(&full[s]), 0);
        load_w(s, bar);
        load_x(s, bar, kc, tb);
        ++it;
        if (++s == S) {
          s = 0;
          ph ^= 1u;
        }
        if (step() && more) src();
      }
      if (!*abort_flag) {
        // the CTA stays until the tensor cores have released its last stages (the commits of
        // rank 0 arrive on this CTA's barriers)
        for (int i = std::max(0, it - S); i < it; ++i)
          if (!mbar_wait_bounded(&empty[i % S], (i / S) & 1, abort_flag, p.err)) break;
      }
      if (*abort_flag) {   // let every copy in flight land before the CTA exits
        if (rank == 0) {
          for (int i = std::max(0, it - S); i < it; ++i) pf_drain(&full[i % S], (i / S) & 1);
        } else {           // counted on rank 0's barriers: 10 ms, far past any copy
          const uint64_t t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 < 10000000ull) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ tensor-core issue, for the pair
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(256, C::ACC);
      int s = 0, seg = 0;
      uint32_t ph = 0;
      bool ok = true;
      PfWalk w(p, pair);
      while (ok && w.next()) {
        const int buf = seg & 1;
        if (!mbar_wait_bounded(&acc_empty[buf], ((seg >> 1) & 1) ^ 1, abort_flag, p.err)) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * C::ACC;
        for (int kc = w.k0; kc < w.k1; ++kc) {
          if (!mbar_wait_bounded(&full[s], ph, abort_flag, p.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t wa = smem_u32(stages + (size_t)s * C::STAGE);
          const uint32_t xb = wa + PF_W_BYTES;   // rows of Xhi here, of Xlo in rank 1
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma_bf16_pair(d, sdesc_sw128(wa + kk * 32), sdesc_sw128(xb + kk * 32), idesc,
                           (kc > w.k0 || kk > 0) ? 1u : 0u);
          umma_commit_pair(&empty[s]);
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        umma_commit_pair(&acc_full[buf]);
        ++seg;
      }
      if (*abort_flag) {   // wait for issued MMAs before shared memory goes away
        umma_commit_pair(drain);
        pf_drain(drain, 0);
      }
    }
  } else {
    // ------------------------------------------------ epilogue (TMEM -> registers -> global)
    const int e = warp & 3;              // TMEM lane quarter this warp may access
    const int grp = (warp - 2) >> 2;     // rounds grp, grp + 2 of 32 positions
    const int r = e * 32 + lane;         // the CTA's weight row
    const int tid = threadIdx.x - 64;
    constexpr int NE = 32 * PF_EPI_WARPS;
    float* slab = staging + grp * 128 * PF_CHUNK;   // [32 positions][128 rows] of the group's round
    const int w8 = ((warp - 2) & 3) * 8;            // this warp finishes the round's positions w8 .. w8 + 7
    const uint32_t acc_empty0 = mapa_shared(smem_u32(acc_empty), 0);
    const int U = p.sk_tiles * p.kc;
    uint32_t res_ph = 0;
    pdl_wait();   // residual rows and outputs belong to the previous kernels' results
    if (p.trace.rec) t_wait = globaltimer_ns();
    const int len0 = p.epi == EPI_QKV ? __ldcg(p.len + p.seq0) : 0;
    int seg = 0;
    PfWalk w(p, pair);
    for (; w.next(); ++seg) {
      int wp, tb;
      pf_tile(p, w.tile, wp, tb);
      const int wt = 2 * wp + rank;
      const int buf = seg & 1;
      const int mt = tb * TOK;   // the tile's first position
      const int vr = min(TOK, p.M - mt);   // the tile's positions
      const bool shared = p.publish || w.k1 - w.k0 < p.kc;
      // EPI_RESID: a round's residual rows (512 bytes a position) go into the slabs by bulk
      // copies, for the first round of a whole tile while the tensor cores work; the values are
      // then added to them there.  Loading them when the sums were ready took 5 us per tile.
      const uint32_t res_bytes = p.epi == EPI_RESID ? 4u * max(0, min(128, p.N - 128 * wt)) : 0u;
      auto load_resid = [&](int b0) {
        const int cnt = min(2 * PF_CHUNK, vr - b0);
        if (tid == 0) mbar_arrive_expect_tx(res_bar, cnt * res_bytes);
        named_bar_sync(1, NE);   // every read of the slabs is done; the bytes are announced
        if (tid < cnt && res_bytes) {
          fence_proxy_async_smem();
          bulk_load_g2s(staging + tid * 128, p.out + (size_t)(mt + b0 + tid) * p.out_ld + 128 * wt, res_bytes, res_bar);
        }
      };
      if (p.epi == EPI_RESID && !shared) load_resid(0);
      const float* inv = s_inv + (seg & 1) * TOK;
      if (p.ssq_in && !p.publish) {
        // RMSNorm factors of the tile's positions while the tensor cores work: eight lanes sum a
        // position's parts, in a fixed order (read after the barrier below)
        for (int c = tid >> 3; c < TOK; c += NE / 8) {
          const float* src = p.ssq_in + (size_t)min(mt + c, p.M - 1) * p.ssq_ld;
          float q = 0.f;
          for (int t = tid & 7; t < p.ssq_ld; t += 8) q += __ldcg(src + t);
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
          if ((tid & 7) == 0) s_inv[(seg & 1) * TOK + c] = 1.0f / sqrtf(q / (float)p.norm_dim + p.norm_eps);
        }
      }
      const bool got = named_bar_and(1, NE, mbar_wait_bounded(&acc_full[buf], (seg >> 1) & 1, abort_flag, p.err));
      if (!got) {
        if (p.epi == EPI_RESID && !shared && tid == 0) pf_drain(res_bar, res_ph);   // copies in flight land
        break;
      }
      tc_fence_after();
      if (p.trace.rec) {
        t_acc1 = globaltimer_ns();
        if (seg == 0) t_acc0 = t_acc1;
      }
      const uint32_t lane_addr = tmem + ((uint32_t)(e * 32) << 16) + buf * C::ACC;
      // hi + lo products of 32 positions; after the warp's last round the accumulator is drained
      auto load_acc = [&](int c0, float (&y)[PF_CHUNK]) {
        float ya[16], yb[16], la[16], lb[16];
        tmem_ld16(lane_addr + c0, ya);
        tmem_ld16(lane_addr + c0 + 16, yb);
        tmem_ld16(lane_addr + TOK + c0, la);
        tmem_ld16(lane_addr + TOK + c0 + 16, lb);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          y[j] = ya[j] + la[j];
          y[16 + j] = yb[j] + lb[j];
        }
      };
      auto drained = [&] {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty0 + buf * 8);
      };
      int lo = 0, hi = 0, batch = 0;
      if (shared) {
        // a split tile: publish this pair's part; the last contributor sums the parts in pair
        // order (deterministic) and runs the epilogue.  A share holds at most one part that
        // starts its tile (slot 1).
        float* mine = p.partials + ((size_t)(pair * 2 + (w.k0 == 0)) * 2 + rank) * PF_TOK * 128 + r;
#pragma unroll 1
        for (int c0 = grp * PF_CHUNK; c0 < vr; c0 += 2 * PF_CHUNK) {
          float y[PF_CHUNK];
          load_acc(c0, y);
#pragma unroll
          for (int j = 0; j < PF_CHUNK; ++j)
            if (c0 + j < vr) __stcg(mine + (c0 + j) * 128, y[j]);
        }
        drained();
        if (p.publish) continue;   // a second kernel sums the parts
        lo = (w.tile * p.kc * p.sk_pairs + p.sk_pairs - 1) / U;
        hi = ((w.tile * p.kc + p.kc - 1) * p.sk_pairs + p.sk_pairs - 1) / U;
        named_bar_sync(1, NE);
        if (tid == 0)
          *s_last = atomic_add_acq_rel_gpu(&p.counters[w.tile * 2 + rank], 1) == hi - lo;
        named_bar_sync(1, NE);
        if (!*s_last) continue;
        if (tid == 0) p.counters[w.tile * 2 + rank] = 0;
        // With no segment after this one the stage ring is idle (every load landed, every MMA
        // that read it completed): the parts come in by bulk copies, `batch` positions of all
        // of them at a time.
        if (w.done()) batch = C::RING / ((hi - lo + 1) * 512) / (2 * PF_CHUNK) * (2 * PF_CHUNK);
      }
      if (p.trace.rec) {
        t_sum = globaltimer_ns();
        t_flags += shared ? 0x101 : 0x100;
      }
      // Rounds of 2 x 32 positions.  This code runs a few times per launch and is fetched cold, so
      // it stays small: rolled rounds, and the values go through shared memory so that a few
      // vector instructions finish a position (a row per thread, 32 positions unrolled, took 16.6 us
      // from the last MMA to the end of the O projection at 99 positions, 12.5 now; QKV 12.1, 8.7).
      bool ok = true;
#pragma unroll 1
      for (int b0 = 0; b0 < vr; b0 += 2 * PF_CHUNK) {
        const int c0 = b0 + grp * PF_CHUNK, m0 = mt + c0;
        const bool fetch = batch && b0 % batch == 0;
        if (p.epi == EPI_RESID && (shared || b0 > 0)) load_resid(b0);
        if (fetch) {
          const uint32_t bytes = (uint32_t)min(batch, vr - b0) * 512;
          const int cnt = hi - lo + 1;
          if (tid == 0) mbar_arrive_expect_tx(red_bar, cnt * bytes);
          named_bar_sync(1, NE);   // the previous batch's reads are done; the bytes are announced
          if (tid < cnt) {
            fence_proxy_async_global();
            bulk_load_g2s(stages + tid * bytes,
                          p.partials + ((size_t)((lo + tid) * 2 + (tid == 0)) * 2 + rank) * PF_TOK * 128 + b0 * 128,
                          bytes, red_bar);
          }
        }
        if (fetch || p.epi == EPI_RESID) {
          const uint32_t ph = batch ? (b0 / batch) & 1 : 0;
          bool in = !fetch || mbar_wait_bounded(red_bar, ph, abort_flag, p.err);
          if (p.epi == EPI_RESID) in = in && mbar_wait_bounded(res_bar, res_ph, abort_flag, p.err);
          ok = named_bar_and(1, NE, in);
          if (!ok) {
            if (tid == 0) {   // copies in flight land before the CTA exits
              if (fetch) pf_drain(red_bar, ph);
              if (p.epi == EPI_RESID) pf_drain(res_bar, res_ph);
            }
            break;
          }
          if (p.epi == EPI_RESID) res_ph ^= 1u;
        }
        if (c0 >= vr) break;   // the second group, in the tile's last round
        // The round's values, position-major, into the slab: from the accumulator each thread
        // writes its row (all positions), from the parts of a split tile each warp sums its own
        // eight positions.
        if (!shared) {
          float y[PF_CHUNK];
          load_acc(c0, y);
          if (b0 + 2 * PF_CHUNK >= TOK || c0 + 2 * PF_CHUNK >= vr) drained();
          if (p.epi == EPI_STORE && !p.ssq_in) {   // nothing to combine: straight to memory, a row per thread
            const int n = 128 * wt + r;
            float* dst = p.out + (size_t)m0 * p.out_ld + n;
            const int cnt = n < p.N ? vr - c0 : 0;
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j)
              if (j < cnt) dst[(size_t)j * p.out_ld] = y[j];
            continue;
          }
          if (p.epi == EPI_RESID) {
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j) y[j] += slab[j * 128 + r];
          } else {
            named_bar_sync(2 + grp, 128);   // the last round's reads of the slab are done
          }
#pragma unroll
          for (int j = 0; j < PF_CHUNK; ++j) slab[j * 128 + r] = y[j];
          named_bar_sync(2 + grp, 128);
        } else {
          // (positions past the tile's last read rows that are not used)
          float4 v[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            v[k] = p.epi == EPI_RESID ? reinterpret_cast<const float4*>(slab + (w8 + k) * 128)[lane]
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
          const int base = batch ? b0 / batch * batch : 0;
          const int rows = min(batch, vr - base);
#pragma unroll 1
          for (int q = lo; q <= hi; ++q) {
            const float* src = batch ? reinterpret_cast<const float*>(stages) + ((q - lo) * rows + c0 - base + w8) * 128
                                     : p.partials + (((size_t)(q * 2 + (q == lo)) * 2 + rank) * PF_TOK + c0 + w8) * 128;
            float4 t[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float4* a = reinterpret_cast<const float4*>(src + k * 128) + lane;
              t[k] = batch ? *a : __ldcg(a);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k].x += t[k].x, v[k].y += t[k].y, v[k].z += t[k].z, v[k].w += t[k].w;
          }
          if (p.epi == EPI_STORE && !p.ssq_in) {
            const int n = 128 * wt + 4 * lane, cnt = vr - c0 - w8;
            float* dst = p.out + (size_t)(m0 + w8) * p.out_ld + n;
            const bool vec = (p.out_ld & 3) == 0 && (reinterpret_cast<uintptr_t>(p.out) & 15u) == 0 && n + 4 <= p.N;
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (k < cnt) {
                float* d = dst + (size_t)k * p.out_ld;
                if (vec) {
                  *reinterpret_cast<float4*>(d) = v[k];
                } else {
                  if (n < p.N) d[0] = v[k].x;
                  if (n + 1 < p.N) d[1] = v[k].y;
                  if (n + 2 < p.N) d[2] = v[k].z;
                  if (n + 3 < p.N) d[3] = v[k].w;
                }
              }
            continue;
          }
          __syncwarp();
#pragma unroll
          for (int k = 0; k < 8; ++k) reinterpret_cast<float4*>(slab + (w8 + k) * 128)[lane] = v[k];
          __syncwarp();
        }
        // Each warp finishes its eight positions, lanes along the rows (features): vector loads
        // and stores, and little code (see above).
        const int left = min(8, vr - c0 - w8);   // (may be <= 0)
        if (p.epi == EPI_SWIGLU) {
          // rows 0-63: gate features 64*wt + .., rows 64-127: the matching up features; half a
          // warp per position
          const int i = 4 * (lane & 15), f = 64 * wt + i;
#pragma unroll 2
          for (int k = lane >> 4; k < left; k += 2) {
            const float* row = slab + (w8 + k) * 128 + i;
            const float4 g = *reinterpret_cast<const float4*>(row), u = *reinterpret_cast<const float4*>(row + 64);
            const float s = p.ssq_in ? inv[c0 + w8 + k] : 1.f;
            auto act = [&](float x, float up) { return x * s / (1.0f + expf(-(x * s))) * (up * s); };
            if (wt < p.n_wtiles && f < p.N) {
              const size_t o = (size_t)(m0 + w8 + k) * p.out_ld + f;
              const float4 a = make_float4(act(g.x, u.x), act(g.y, u.y), act(g.z, u.z), act(g.w, u.w));
              if (p.out) *reinterpret_cast<float4*>(p.out + o) = a;
              pf_store4(p.out_hi, p.out_lo, o, a.x, a.y, a.z, a.w);
            }
          }
        } else if (p.epi == EPI_QKV) {
          // The tile lies in one of q, k, v and holds whole heads.  RoPE (rotate-half) pairs row
          // i of a head with row i + hd/2; position m sits at slot (and position) len + m.  Half
          // a warp per position, four pairs of rows a lane.
          const int R = p.rows_per_map, g0 = 128 * wt, half = p.hd >> 1;
          const int which = (g0 >= R) + (g0 >= 2 * R);
          const int x = 4 * (lane & 15), i = x & (half - 1), r1 = (x - i) * 2 + i;   // rows r1 .. and r1 + half ..
          const int f = g0 - which * R + r1;   // feature of row r1 within its matrix
          if (wt < p.n_wtiles) {
#pragma unroll 2
            for (int k = lane >> 4; k < left; k += 2) {
              const float* row = slab + (w8 + k) * 128 + r1;
              float4 a = *reinterpret_cast<const float4*>(row), b = *reinterpret_cast<const float4*>(row + half);
              const float s = p.ssq_in ? inv[c0 + w8 + k] : 1.f;
              a.x *= s, a.y *= s, a.z *= s, a.w *= s, b.x *= s, b.y *= s, b.z *= s, b.w *= s;
              const int m = m0 + w8 + k;
              const PfRow row_of(p, m, len0);
              if (which < 2) pf_rope4(p, row_of.pos, i, a, b);
              pf_qkv_store(p, which, m, row_of, f, i, a, b);
              if (which == 1 && (lane & 15) == 0) row_of.report(p);
            }
          }
        } else if (p.epi == EPI_STORE) {
          // the LM head whose operand still needs the positions' RMSNorm factors
#pragma unroll 1
          for (int k = 0; k < left; ++k) {
            float* dst = p.out + (size_t)(m0 + w8 + k) * p.out_ld;
            for (int i = lane, n = 128 * wt + lane; i < 128 && n < p.N; i += 32, n += 32)
              dst[n] = slab[(w8 + k) * 128 + i] * inv[c0 + w8 + k];
          }
        } else {
          const int n = 128 * wt + 4 * lane;
          const float* row = slab + w8 * 128 + 4 * lane;
          float* dst = p.out + (size_t)(m0 + w8) * p.out_ld + n;
          {
            // (N and the row stride are multiples of 8.)  The residual row is updated; with gain_next
            // also the next RMSNorm's operand h * g and this weight tile's sum of h^2 per position
            const bool in = n < p.N;
            float g[4] = {0.f, 0.f, 0.f, 0.f};
            if (p.gain_next && in) {
              const uint2 gb = __ldg(reinterpret_cast<const uint2*>(p.gain_next + n));
              g[0] = __uint_as_float(gb.x << 16), g[1] = __uint_as_float(gb.x & 0xFFFF0000u);
              g[2] = __uint_as_float(gb.y << 16), g[3] = __uint_as_float(gb.y & 0xFFFF0000u);
            }
#pragma unroll 1
            for (int k = 0; k < left; k += 4, row += 512, dst += 4 * (size_t)p.out_ld) {
              float4 h[4];
              float sq[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const bool on = in && k + u < left;
                h[u] = *reinterpret_cast<const float4*>(row + u * 128);
                sq[u] = on ? (h[u].x * h[u].x + h[u].y * h[u].y) + (h[u].z * h[u].z + h[u].w * h[u].w) : 0.f;
                if (on) {
                  *reinterpret_cast<float4*>(dst + (size_t)u * p.out_ld) = h[u];
                  if (p.gain_next)
                    pf_store4(p.out_hi, p.out_lo, (size_t)(m0 + w8 + k + u) * p.out_ld + n, h[u].x * g[0],
                              h[u].y * g[1], h[u].z * g[2], h[u].w * g[3]);
                }
              }
              if (p.gain_next) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                  for (int u = 0; u < 4; ++u) sq[u] += __shfl_xor_sync(0xffffffffu, sq[u], o);
                if (lane < 4 && k + lane < left && wt < p.n_wtiles)
                  p.ssq_out[(size_t)(m0 + w8 + k + lane) * p.ssq_ld + wt] =
                      lane == 0 ? sq[0] : (lane == 1 ? sq[1] : (lane == 2 ? sq[2] : sq[3]));
              }
            }
          }
        }
      }
      if (!shared && grp * PF_CHUNK >= vr) drained();   // no round of its own in this tile
      if (!ok) break;
    }
  }

  if (threadIdx.x == 64 && p.trace.rec)
    trace_write(p.trace, t_flags, t_entry, t_wait, t_acc0, t_acc1, t_sum, globaltimer_ns());
  tc_fence_before();
  cluster_sync_all();   // neither CTA leaves while the other may still signal its barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 2 * C::ACC);
  }
}

// ---- the second kernel of a GEMM whose every tile is split -------------------------------
// With fewer tiles than pairs (O and down projections up to some 500 positions, QKV up to 128)
// the last contributors of the tiles, 32 of 152 CTAs at 99 positions, summed the parts and ran
// the epilogue alone: 10 to 12 us after the last MMA, bound by the bytes and latency of one CTA
// each.  Instead all CTAs only publish, and a kernel of one CTA per position (and matrix, for
// QKV) does the rest on every SM (prefill of two 7B layers, 99 positions: 273 -> 239 us, 200:
// 355 -> 337, 512: 609 -> 603).  A position's CTA has its whole row, so RMSNorm is applied here
// and the next GEMM needs no factor.
constexpr int PF_FIN_THREADS = 512;
// a whole row per CTA in one round of loads for up to 4096 features: 512 -> 1024 threads, prefill of
// two 7B layers, 30 positions 221.0 -> 216.3 us, 99 248.6 -> 246.0, 300 475.5 -> 466.0
constexpr int PF_FIN_ROW_THREADS = 1024;
constexpr int PF_FIN_PARTS = 6;   // parts loaded together

// the contributors lo .. hi of (weight tile wt, position block tb), and the start of lo's part of
// row `pos`; the other parts follow from part_of()
struct PfParts {
  int lo, hi;
  const float* base;
  __device__ PfParts(const PfGemmParams& p, int wt, int tb, int pos) {
    const int g = tb / p.group, width = min(p.group, p.n_tblocks - g * p.group);
    const int tile = g * p.n_pairs_w * p.group + (wt >> 1) * width + tb - g * p.group;
    const int U = p.sk_tiles * p.kc;
    lo = (tile * p.kc * p.sk_pairs + p.sk_pairs - 1) / U;
    hi = ((tile * p.kc + p.kc - 1) * p.sk_pairs + p.sk_pairs - 1) / U;
    base = p.partials + (size_t)(wt & 1) * PF_TOK * 128 + pos * 128;
  }
  __device__ const float* part(int q) const { return base + (size_t)(q * 2 + (q == lo)) * 2 * PF_TOK * 128; }
};

__device__ __forceinline__ void pf_add(float4& a, const float4& b) {
  a.x += b.x, a.y += b.y, a.z += b.z, a.w += b.w;
}

// sum of v over the CTA, in a fixed order
__device__ __forceinline__ float pf_block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = (threadIdx.x & 31) < blockDim.x / 32 ? red[threadIdx.x & 31] : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// RMSNorm factor of operand row m (1 when the operand is normalised already)
__device__ __forceinline__ float pf_row_factor(const PfGemmParams& p, int m) {
  if (!p.ssq_in) return 1.f;
  float q = 0.f;
  for (int t = 0; t < p.ssq_ld; ++t) q += __ldcg(p.ssq_in + (size_t)m * p.ssq_ld + t);
  return 1.0f / sqrtf(q / (float)p.norm_dim + p.norm_eps);
}

// h += sum of the parts; with gain_next the next GEMM's operand RMSNorm(h)
__global__ void __launch_bounds__(PF_FIN_ROW_THREADS) prefill_finish_resid_kernel(const __grid_constant__ PfGemmParams p) {
  constexpr int I = 64 * 128 / (4 * PF_FIN_ROW_THREADS);   // float4 of a row per thread: rows of up to 8192
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x, tok = p.tok, tb = m / tok, pos = m - tb * tok;
  float* row = p.out + (size_t)m * p.out_ld;
  float4 h[I];
  float sq = 0.f;
#pragma unroll
  for (int i = 0; i < I; ++i) {
    const int n = 4 * ((int)threadIdx.x + i * PF_FIN_ROW_THREADS);
    h[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n >= p.N) break;
    const PfParts w(p, n >> 7, tb, pos);
    const float4 old = __ldcg(reinterpret_cast<const float4*>(row + n));
    for (int q = w.lo; q <= w.hi; q += PF_FIN_PARTS) {
      float4 t[PF_FIN_PARTS];
#pragma unroll
      for (int u = 0; u < PF_FIN_PARTS; ++u)
        t[u] = q + u <= w.hi ? __ldcg(reinterpret_cast<const float4*>(w.part(q + u) + (n & 127)))
                             : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < PF_FIN_PARTS; ++u) pf_add(h[i], t[u]);
    }
    pf_add(h[i], old);
    *reinterpret_cast<float4*>(row + n) = h[i];
    sq += (h[i].x * h[i].x + h[i].y * h[i].y) + (h[i].z * h[i].z + h[i].w * h[i].w);
  }
  if (!p.gain_next) return;
  const float inv = 1.0f / sqrtf(pf_block_sum(sq, red) / (float)p.norm_dim + p.norm_eps);
#pragma unroll
  for (int i = 0; i < I; ++i) {
    const int n = 4 * ((int)threadIdx.x + i * PF_FIN_ROW_THREADS);
    if (n >= p.N) break;
    const uint2 g = __ldg(reinterpret_cast<const uint2*>(p.gain_next + n));
    pf_store4(p.out_hi, p.out_lo, (size_t)m * p.out_ld + n, h[i].x * inv * __uint_as_float(g.x << 16),
              h[i].y * inv * __uint_as_float(g.x & 0xFFFF0000u), h[i].z * inv * __uint_as_float(g.y << 16),
              h[i].w * inv * __uint_as_float(g.y & 0xFFFF0000u));
  }
}

// out = sum of the parts (SCALED: times the operand row's RMSNorm factor; blockIdx.y: 2048 features)
template <bool SCALED>
__global__ void __launch_bounds__(PF_FIN_THREADS) prefill_finish_store_kernel(const __grid_constant__ PfGemmParams p) {
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x, tb = m / p.tok, n = 4 * ((int)blockIdx.y * PF_FIN_THREADS + (int)threadIdx.x);
  if (n >= p.N) return;
  const PfParts w(p, n >> 7, tb, m - tb * p.tok);
  float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int q = w.lo; q <= w.hi; q += PF_FIN_PARTS) {
    float4 t[PF_FIN_PARTS];
#pragma unroll
    for (int u = 0; u < PF_FIN_PARTS; ++u)
      t[u] = q + u <= w.hi ? __ldcg(reinterpret_cast<const float4*>(w.part(q + u) + (n & 127)))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < PF_FIN_PARTS; ++u) pf_add(y, t[u]);
  }
  if constexpr (SCALED) {
    const float s = pf_row_factor(p, m);
    y.x *= s, y.y *= s, y.z *= s, y.w *= s;
  }
  float* dst = p.out + (size_t)m * p.out_ld + n;
  if (n + 4 <= p.N && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
    *reinterpret_cast<float4*>(dst) = y;
  } else {
    const float v[4] = {y.x, y.y, y.z, y.w};
    for (int e = 0; e < 4 && n + e < p.N; ++e) dst[e] = v[e];
  }
}

// RoPE on the queries and keys of a position, KV append (blockIdx.y: q, k, v)
__global__ void __launch_bounds__(PF_FIN_THREADS) prefill_finish_qkv_kernel(const __grid_constant__ PfGemmParams p) {
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x, which = blockIdx.y, tok = p.tok, tb = m / tok, pos = m - tb * tok;
  const int R = p.rows_per_map, half = p.hd >> 1;
  const PfRow row_of(p, m, __ldcg(p.len + p.seq0));
  const float s = pf_row_factor(p, m);
  if (threadIdx.x == 0 && which == 1) row_of.report(p);
  for (int x = 4 * (int)threadIdx.x; x < R / 2; x += 4 * PF_FIN_THREADS) {
    // four pairs of features: i .. i + 3 of a head and those half a head further
    const int i = x & (half - 1), f = (x - i) * 2 + i;   // head * hd + i
    const PfParts w(p, (which * R + f) >> 7, tb, pos), v(p, (which * R + f + half) >> 7, tb, pos);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    for (int q = w.lo; q <= w.hi; q += PF_FIN_PARTS) {   // (a head lies in one tile: both rows have the same parts)
      float4 t[PF_FIN_PARTS], u4[PF_FIN_PARTS];
#pragma unroll
      for (int u = 0; u < PF_FIN_PARTS; ++u) {
        t[u] = u4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q + u <= w.hi) {
          t[u] = __ldcg(reinterpret_cast<const float4*>(w.part(q + u) + (f & 127)));
          u4[u] = __ldcg(reinterpret_cast<const float4*>(v.part(q + u) + ((f + half) & 127)));
        }
      }
#pragma unroll
      for (int u = 0; u < PF_FIN_PARTS; ++u) pf_add(a, t[u]), pf_add(b, u4[u]);
    }
    a.x *= s, a.y *= s, a.z *= s, a.w *= s, b.x *= s, b.y *= s, b.z *= s, b.w *= s;
    if (which < 2) pf_rope4(p, row_of.pos, i, a, b);
    pf_qkv_store(p, which, m, row_of, f, i, a, b);
  }
}

namespace {
int g_pf_pairs = 0;   // CTA pairs resident at once

cudaLaunchConfig_t pf_config(int tok, int pairs, cudaStream_t st, bool pdl, cudaLaunchAttribute (&attr)[2]) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(PF_THREADS);
  cfg.dynamicSmemBytes = tok == 64 ? PfCfg<64>::SMEM : PfCfg<128>::SMEM;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cfg;
}
}  // namespace

cudaError_t prefill_prepare() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(prefill_gemm_kernel<128>, a, (int)PfCfg<128>::SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prefill_gemm_kernel<64>, a, (int)PfCfg<64>::SMEM);
  if (e == cudaSuccess) e = prefer_shared(prefill_gemm_kernel<128>);
  if (e == cudaSuccess) e = prefer_shared(prefill_gemm_kernel<64>);
  if (e == cudaSuccess) e = prefer_shared(prefill_finish_resid_kernel);
  if (e == cudaSuccess) e = prefer_shared(prefill_finish_qkv_kernel);
  if (e == cudaSuccess) e = prefer_shared(prefill_finish_store_kernel<false>);
  if (e == cudaSuccess) e = prefer_shared(prefill_finish_store_kernel<true>);
  if (e != cudaSuccess || g_pf_pairs > 0) return e;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = pf_config(128, 1, nullptr, false, attr);
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, prefill_gemm_kernel<128>, &cfg);
  if (e == cudaSuccess) g_pf_pairs = n;
  return e;
}

int prefill_tok(int M) { return M <= 64 ? 64 : 128; }

size_t prefill_partials(int num_sms) { return (size_t)(num_sms / 2) * 2 * 2 * PF_TOK * 128; }

void plan_prefill_gemm(PfGemmParams& p, int num_sms) {
  const int tok = prefill_tok(p.M), P = std::max(1, std::min(num_sms / 2, g_pf_pairs));
  p.tok = tok;
  p.n_pairs_w = (p.n_wtiles + 1) / 2;
  p.n_tblocks = (p.M + tok - 1) / tok;
  p.group = std::min(p.n_tblocks, PF_GROUP * (128 / tok));
  const int T = p.n_pairs_w * p.n_tblocks, rem = T % P;
  p.sk_tiles = 0;
  p.sk_pairs = 0;
  // Tiles of an incomplete wave are split where that saves eight chunks or more.  Plain products with
  // few chunks to save would be faster whole (rows, K, N, us, split / whole: 200, 1024, 12288 24.6 / 19.3;
  // 512, 4096, 4096 40.7 / 34.9; 512, 11008, 4096 99 / 84), but less exact: a tile's fp32 sum over all
  // of K loses more than the shorter sums of its parts (error against 64 bits 2.63e-6 / 2.66e-6, 3.70e-6
  // / 5.05e-6, 8.2e-6 / 12.6e-6).
  if (rem && (P - rem) * p.kc >= 8 * P) {
    p.sk_tiles = rem;
    p.sk_pairs = std::max(rem, std::min(P, rem * p.kc / PF_SK_MIN));
    if (p.sk_pairs == rem) p.sk_tiles = p.sk_pairs = 0;   // nothing to split
  }
  p.publish = p.sk_tiles == T && p.epi != EPI_SWIGLU;
}

cudaError_t launch_prefill_gemm(const PfGemmParams& p, cudaStream_t st, bool pdl) {
  const int tok = prefill_tok(p.M), T = p.n_pairs_w * p.n_tblocks;
  const int P = std::max(1, g_pf_pairs);
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = pf_config(tok, std::min(P, std::max(p.sk_pairs, T - p.sk_tiles)), st, pdl, attr);
  const cudaError_t e = tok == 64 ? cudaLaunchKernelEx(&cfg, prefill_gemm_kernel<64>, p)
                                  : cudaLaunchKernelEx(&cfg, prefill_gemm_kernel<128>, p);
  if (e != cudaSuccess || !p.publish) return e;
  cudaLaunchConfig_t fin = {};
  fin.gridDim = p.epi == EPI_RESID ? dim3(p.M)
                                   : dim3(p.M, p.epi == EPI_QKV ? 3 : (p.N + 4 * PF_FIN_THREADS - 1) / (4 * PF_FIN_THREADS));
  fin.blockDim = dim3(p.epi == EPI_RESID ? PF_FIN_ROW_THREADS : PF_FIN_THREADS);
  fin.stream = st;
  attr[0] = attr[1];
  fin.attrs = attr;
  fin.numAttrs = pdl ? 1 : 0;
  return p.epi == EPI_QKV     ? cudaLaunchKernelEx(&fin, prefill_finish_qkv_kernel, p)
         : p.epi == EPI_RESID ? cudaLaunchKernelEx(&fin, prefill_finish_resid_kernel, p)
         : p.ssq_in           ? cudaLaunchKernelEx(&fin, prefill_finish_store_kernel<true>, p)
                              : cudaLaunchKernelEx(&fin, prefill_finish_store_kernel<false>, p);
}

}  // namespace sdsat
