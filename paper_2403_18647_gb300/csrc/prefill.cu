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
// does, so that the consuming GEMM only scales its result by each position's factor; SiLU(gate)
// * up as the down projection's bf16 hi + lo operand.  RMSNorm and RoPE as row kernels of their
// own cost two more passes over the chunk's rows each (2047 positions: 34 us per RMSNorm, 59
// us per RoPE + append).  Attention is prefill_attention.cu.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sdsat {

constexpr int PF_W_BYTES = 128 * 128;                    // a CTA's 128 weight rows x 64 bf16
constexpr int PF_CHUNK = 32;                             // positions per epilogue round
constexpr int PF_EPI_WARPS = 8;                          // two per TMEM lane quarter
constexpr int PF_THREADS = 64 + 32 * PF_EPI_WARPS;
constexpr int PF_STAGING = 2 * 128 * PF_CHUNK;           // fp32 exchange of the two epilogue groups
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
  static constexpr int ROUNDS = TOK / (2 * PF_CHUNK);    // epilogue rounds of each of the two warp groups
  static constexpr int NBAR = 2 * STAGES + 6;
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
    // exchange between the group's 128 rows: element (row, j) at row * 32 + (j ^ lane of the
    // row), so that a warp's rows fall on different banks
    float* xch = staging + grp * 128 * PF_CHUNK;
    int round = 0;
    const uint32_t acc_empty0 = mapa_shared(smem_u32(acc_empty), 0);
    const int U = p.sk_tiles * p.kc;
    pdl_wait();   // residual rows and outputs belong to the previous kernels' results
    if (p.trace.rec) t_wait = globaltimer_ns();
    const int len0 = p.epi == EPI_QKV ? __ldcg(p.len + p.seq) : 0;
    int seg = 0;
    PfWalk w(p, pair);
    for (; w.next(); ++seg) {
      int wp, tb;
      pf_tile(p, w.tile, wp, tb);
      const int wt = 2 * wp + rank;
      const int buf = seg & 1;
      const int mt = tb * TOK;   // the tile's first position
      const float* inv = s_inv + (seg & 1) * TOK;
      if (p.ssq_in) {
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
        if (p.ssq_in) {
#pragma unroll
          for (int j = 0; j < PF_CHUNK; ++j) y[j] *= inv[c0 + j];
        }
        if (p.epi == EPI_SWIGLU) {
          // tile rows 0-63: gate features 64*wt + r, rows 64-127: the matching up features; the
          // gate thread takes the round's first 16 positions, the up thread the other 16
          const int f = 64 * wt + (r & 63);
          const bool gate = r < 64;
#pragma unroll
          for (int j = 0; j < PF_CHUNK / 2; ++j) xch[r * PF_CHUNK + (j ^ lane)] = gate ? y[16 + j] : y[j];
          named_bar_sync(2 + grp, 128);
          const float* other = xch + (r ^ 64) * PF_CHUNK;
          if (wt < p.n_wtiles && f < p.N) {
#pragma unroll
            for (int j = 0; j < PF_CHUNK / 2; ++j) {
              const int m = m0 + (gate ? j : 16 + j);
              if (m < p.M) {
                const float x = other[j ^ lane];
                const float g = gate ? y[j] : x, up = gate ? x : y[16 + j];
                const float a = g / (1.0f + expf(-g)) * up;
                const __nv_bfloat16 h = __float2bfloat16_rn(a);
                p.out_hi[(size_t)m * p.out_ld + f] = h;
                p.out_lo[(size_t)m * p.out_ld + f] = __float2bfloat16_rn(a - __bfloat162float(h));
              }
            }
          }
          named_bar_sync(2 + grp, 128);
        } else if (p.epi == EPI_QKV) {
          // The tile lies in one of q, k, v and holds whole heads.  RoPE (rotate-half) pairs row
          // r with row r ^ hd/2; position m0 + j sits at slot (and position) len + m0 + j.
          const int R = p.rows_per_map, g = 128 * wt;
          const int which = (g >= R) + (g >= 2 * R);
          const int f = g - which * R + r, half = p.hd >> 1, i = f & (p.hd - 1);
          const int slot0 = len0 + m0;
          if (which < 2 && wt < p.n_wtiles) {
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j) xch[r * PF_CHUNK + (j ^ lane)] = y[j];
            named_bar_sync(2 + grp, 128);
            const float* other = xch + (r ^ half) * PF_CHUNK;
            const float sgn = i < half ? -1.f : 1.f;
            const float2* cs = p.rope + (i & (half - 1));
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j) {
              const float2 t = __ldg(cs + (size_t)min(slot0 + j, p.rope_len - 1) * half);
              y[j] = y[j] * t.x + sgn * (other[j ^ lane] * t.y);
            }
            named_bar_sync(2 + grp, 128);
          }
          if (wt < p.n_wtiles) {
            const int valid = min(PF_CHUNK, p.M - m0);
            if (which == 0) {
              const size_t o = (size_t)m0 * p.out_ld + f;
#pragma unroll
              for (int j = 0; j < PF_CHUNK; ++j)
                if (j < valid) {
                  const __nv_bfloat16 h = __float2bfloat16_rn(y[j]);
                  p.out_hi[o + (size_t)j * p.out_ld] = h;
                  p.out_lo[o + (size_t)j * p.out_ld] = __float2bfloat16_rn(y[j] - __bfloat162float(h));
                }
            } else {
              const int fits = min(valid, p.cap - slot0);
              __nv_bfloat16* dst = (which == 1 ? p.k_layer : p.v_layer) +
                                   ((size_t)(p.seq * p.H + f / p.hd) * p.cap + slot0) * p.hd + i;
#pragma unroll
              for (int j = 0; j < PF_CHUNK; ++j)
                if (j < fits) dst[j * p.hd] = __float2bfloat16_rn(y[j]);
              if (r == 0 && fits < valid) set_error(p.err, ERR_CAPACITY);
              if (r == 0 && slot0 + valid > p.rope_len) set_error(p.err, ERR_POSITION);
            }
          }
        } else {
          const int n = 128 * wt + r;
          const bool in = n < p.N;
          float* dst = p.out + (size_t)m0 * p.out_ld + n;
          const int valid = in ? min(PF_CHUNK, p.M - m0) : 0;
          if (p.epi == EPI_RESID) {
            float hv[PF_CHUNK];
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j) hv[j] = j < valid ? __ldcg(dst + (size_t)j * p.out_ld) : 0.f;
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j) y[j] += hv[j];
          }
#pragma unroll
          for (int j = 0; j < PF_CHUNK; ++j)
            if (j < valid) dst[(size_t)j * p.out_ld] = y[j];
          if (p.gain_next) {
            // the next RMSNorm's operand h * g, and this weight tile's sum of h^2 per position:
            // halving exchanges leave position j's sum over the warp's rows on lane j, the
            // group's four warps add up through shared memory (two buffers, one barrier)
            const float gn = in ? __bfloat162float(p.gain_next[n]) : 0.f;
            const size_t o = (size_t)m0 * p.out_ld + n;
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j) {
              const float x = y[j] * gn;
              const __nv_bfloat16 h = __float2bfloat16_rn(x);
              if (j < valid) {
                p.out_hi[o + (size_t)j * p.out_ld] = h;
                p.out_lo[o + (size_t)j * p.out_ld] = __float2bfloat16_rn(x - __bfloat162float(h));
              }
              y[j] = j < valid ? y[j] * y[j] : 0.f;
            }
#pragma unroll
            for (int o2 = 16; o2 > 0; o2 >>= 1) {
              const bool up = lane & o2;
#pragma unroll
              for (int j = 0; j < o2; ++j) {
                const float send = up ? y[j] : y[j + o2], keep = up ? y[j + o2] : y[j];
                y[j] = keep + __shfl_xor_sync(0xffffffffu, send, o2);
              }
            }
            float* part = xch + (round++ & 1) * 128;
            part[e * 32 + lane] = y[0];
            named_bar_sync(2 + grp, 128);
            if (e == 0 && m0 + lane < p.M && wt < p.n_wtiles)
              p.ssq_out[(size_t)(m0 + lane) * p.ssq_ld + wt] =
                  (part[lane] + part[32 + lane]) + (part[64 + lane] + part[96 + lane]);
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
  if (e == cudaSuccess) e = prefer_shared(prefill_gemm_kernel<128>);
  if (e == cudaSuccess) e = prefer_shared(prefill_gemm_kernel<64>);
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

}  // namespace sdsat
