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
// Epilogues: store (q, k, v before RoPE), residual add (O and down projections), and
// SiLU(gate) * up written as the down projection's bf16 hi + lo operand.  RMSNorm and
// RoPE + the KV append are small row kernels here (the decode path folds them into the
// GEMMs); attention is the causal flash-attention kernel at the end of attention.cu.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sdsat {

constexpr int PF_W_BYTES = 128 * 128;                    // a CTA's 128 weight rows x 64 bf16
constexpr int PF_CHUNK = 32;                             // positions per epilogue round
constexpr int PF_EPI_WARPS = 8;                          // two per TMEM lane quarter
constexpr int PF_THREADS = 64 + 32 * PF_EPI_WARPS;
constexpr int PF_XROW = PF_CHUNK / 2 + 1;                // exchange row: half a round's positions, padded
constexpr int PF_STAGING = 2 * 128 * PF_XROW;            // fp32 exchange of the two epilogue groups
#ifndef SDSAT_PF_GROUP
#define SDSAT_PF_GROUP 8
#endif
constexpr int PF_GROUP = SDSAT_PF_GROUP;
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
  static constexpr int ROUNDS = TOK / (2 * PF_CHUNK);    // epilogue rounds of each of the two warp groups
  static constexpr int NBAR = 2 * STAGES + 6;
  static constexpr size_t SMEM = 1024 + (size_t)RING + PF_STAGING * 4 + NBAR * 8 + 64;
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
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + PF_STAGING);
  uint64_t* full = bars;                  // rank 0: both CTAs' weights and positions landed (TMA)
  uint64_t* empty = bars + S;     // the stage was consumed by the tensor cores
  uint64_t* acc_full = bars + 2 * S;   // [2] accumulator ready
  uint64_t* acc_empty = acc_full + 2;          // [2] rank 0: accumulator drained in both CTAs
  uint64_t* drain = acc_empty + 2;
  uint64_t* red_bar = drain + 1;               // parts of the tile being reduced landed (bulk copies)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(red_bar + 1);
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
      const uint64_t pol_w = l2_policy_evict_normal();  // a weight tile is read by the pairs of every position block
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
    float* xch = staging + grp * 128 * PF_XROW;
    const uint32_t acc_empty0 = mapa_shared(smem_u32(acc_empty), 0);
    const int U = p.sk_tiles * p.kc;
    pdl_wait();   // residual rows and outputs belong to the previous kernels' results
    if (p.trace.rec) t_wait = globaltimer_ns();
    int seg = 0;
    PfWalk w(p, pair);
    for (; w.next(); ++seg) {
      int wp, tb;
      pf_tile(p, w.tile, wp, tb);
      const int wt = 2 * wp + rank;
      const int buf = seg & 1;
      const int mt = tb * TOK;   // the tile's first position
      const bool got = named_bar_and(1, NE, mbar_wait_bounded(&acc_full[buf], (seg >> 1) & 1, abort_flag, p.err));
      if (!got) break;
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
      const bool shared = w.k1 - w.k0 < p.kc;
      const int vr = min(TOK, p.M - mt);   // the tile's positions
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
      // Rounds of 2 x 32 positions.  This code runs a few times per launch and is fetched cold,
      // so it stays rolled: with the rounds unrolled the epilogue took twice as long.
      bool ok = true;
#pragma unroll 1
      for (int b0 = 0; b0 < vr; b0 += 2 * PF_CHUNK) {
        const int c0 = b0 + grp * PF_CHUNK, m0 = mt + c0;
        if (batch && b0 % batch == 0) {
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
          const uint32_t ph = (b0 / batch) & 1;
          ok = named_bar_and(1, NE, mbar_wait_bounded(red_bar, ph, abort_flag, p.err));
          if (!ok) {
            if (tid == 0) pf_drain(red_bar, ph);   // copies in flight land before the CTA exits
            break;
          }
        }
        if (c0 >= vr) break;   // the second group, in the tile's last round
        float y[PF_CHUNK];
        if (!shared) {
          load_acc(c0, y);
          if (b0 + 2 * PF_CHUNK >= TOK || c0 + 2 * PF_CHUNK >= vr) drained();
        } else {
#pragma unroll
          for (int j = 0; j < PF_CHUNK; ++j) y[j] = 0.f;
          if (batch) {
            const int rows = min(batch, vr - b0 / batch * batch);
            const float* src = reinterpret_cast<const float*>(stages) + (c0 - b0 / batch * batch) * 128 + r;
#pragma unroll 1
            for (int q = lo; q <= hi; ++q, src += rows * 128)
#pragma unroll
              for (int j = 0; j < PF_CHUNK; ++j) y[j] += src[j * 128];
          } else {
            // (positions past the tile's last read rows of the part that are not used)
#pragma unroll 1
            for (int q = lo; q <= hi; ++q) {
              const float* src = p.partials + ((size_t)(q * 2 + (q == lo)) * 2 + rank) * PF_TOK * 128 + c0 * 128 + r;
              float v[PF_CHUNK];
#pragma unroll
              for (int j = 0; j < PF_CHUNK; ++j) v[j] = __ldcg(src + j * 128);
#pragma unroll
              for (int j = 0; j < PF_CHUNK; ++j) y[j] += v[j];
            }
          }
        }
        if (p.epi == EPI_SWIGLU) {
          // tile rows 0-63: gate features 64*wt + r, rows 64-127: the matching up features; the
          // gate thread takes the round's first 16 positions, the up thread the other 16
          const int f = 64 * wt + (r & 63);
          const bool gate = r < 64;
#pragma unroll
          for (int j = 0; j < PF_CHUNK / 2; ++j) xch[r * PF_XROW + j] = gate ? y[16 + j] : y[j];
          named_bar_sync(2 + grp, 128);
          const float* other = xch + (r ^ 64) * PF_XROW;
          if (wt < p.n_wtiles && f < p.N) {
#pragma unroll
            for (int j = 0; j < PF_CHUNK / 2; ++j) {
              const int m = m0 + (gate ? j : 16 + j);
              if (m < p.M) {
                const float g = gate ? y[j] : other[j], up = gate ? other[j] : y[16 + j];
                const float a = g / (1.0f + expf(-g)) * up;
                const __nv_bfloat16 h = __float2bfloat16_rn(a);
                p.out_hi[(size_t)m * p.out_ld + f] = h;
                p.out_lo[(size_t)m * p.out_ld + f] = __float2bfloat16_rn(a - __bfloat162float(h));
              }
            }
          }
          named_bar_sync(2 + grp, 128);
        } else {
          const int n = 128 * wt + r;
          if (n < p.N) {
            if (p.epi == EPI_RESID) {
              float hv[PF_CHUNK];
#pragma unroll
              for (int j = 0; j < PF_CHUNK; ++j)
                hv[j] = (m0 + j < p.M) ? __ldcg(p.out + (size_t)(m0 + j) * p.out_ld + n) : 0.f;
#pragma unroll
              for (int j = 0; j < PF_CHUNK; ++j) y[j] += hv[j];
            }
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j)
              if (m0 + j < p.M) p.out[(size_t)(m0 + j) * p.out_ld + n] = y[j];
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

cudaError_t launch_prefill_gemm(PfGemmParams& p, int num_sms, cudaStream_t st, bool pdl) {
  const int tok = prefill_tok(p.M), P = std::max(1, std::min(num_sms / 2, g_pf_pairs));
  p.n_pairs_w = (p.n_wtiles + 1) / 2;
  p.n_tblocks = (p.M + tok - 1) / tok;
  p.group = std::min(p.n_tblocks, PF_GROUP * (128 / tok));
  const int T = p.n_pairs_w * p.n_tblocks, rem = T % P;
  p.sk_tiles = 0;
  p.sk_pairs = 0;
  if (rem && (P - rem) * p.kc >= 8 * P) {
    p.sk_tiles = rem;
    p.sk_pairs = std::max(rem, std::min(P, p.sk_tiles * p.kc / PF_SK_MIN));
    if (p.sk_pairs == rem) p.sk_tiles = p.sk_pairs = 0;   // nothing to split
  }
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg =
      pf_config(tok, std::min(P, std::max(p.sk_pairs, T - p.sk_tiles)), st, pdl, attr);
  return tok == 64 ? cudaLaunchKernelEx(&cfg, prefill_gemm_kernel<64>, p)
                   : cudaLaunchKernelEx(&cfg, prefill_gemm_kernel<128>, p);
}

// ---- RoPE + KV append of a prefill chunk ------------------------------------------------
// qkv [M][3R] (q | k | v, head-major columns) -> q rotated into qout [M][R]; k rotated and v
// into the cache slots len[seq] + m at position len[seq] + m (rotate-half pairing (i, i + hd/2)).
__global__ void __launch_bounds__(256) rope_kv_kernel(RopeKvParams p) {
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x;
  const int R = p.H * p.hd, half = p.hd >> 1;
  const int slot = __ldcg(p.len + p.seq) + m;
  int pos = slot;
  if (pos >= p.rope_len) {
    if (threadIdx.x == 0) set_error(p.err, ERR_POSITION);
    pos = p.rope_len - 1;
  }
  const bool fits = slot < p.cap;
  if (!fits && threadIdx.x == 0) set_error(p.err, ERR_CAPACITY);
  const float* row = p.qkv + (size_t)m * 3 * R;
  for (int idx = threadIdx.x; idx < R; idx += blockDim.x) {
    const int h = idx / p.hd, i = idx % p.hd;
    const int partner = i < half ? idx + half : idx - half;
    const float2 cs = p.rope[(size_t)pos * half + (i % half)];
    const float qa = row[idx], qp = row[partner];
    const float ka = row[R + idx], kp = row[R + partner];
    p.qout[(size_t)m * R + idx] = i < half ? qa * cs.x - qp * cs.y : qa * cs.x + qp * cs.y;
    if (fits) {
      const size_t o = (((size_t)p.seq * p.H + h) * p.cap + slot) * p.hd + i;
      p.k_layer[o] = __float2bfloat16_rn(i < half ? ka * cs.x - kp * cs.y : ka * cs.x + kp * cs.y);
      p.v_layer[o] = __float2bfloat16_rn(row[2 * R + idx]);
    }
  }
}

cudaError_t launch_rope_kv(const RopeKvParams& p, int M, cudaStream_t st, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(M);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, rope_kv_kernel, p);
}

}  // namespace sdsat
