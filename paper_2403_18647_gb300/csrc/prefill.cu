// Prefill: the prompt's positions through the model in chunks of up to PF_ROWS, before the
// decode loop.  Unlike the decode step (a handful of rows, bound by the weight stream), a
// chunk of hundreds of positions makes every projection a dense contraction, so it runs
// on a tiled tensor-core GEMM:
//
//   Y[m][n] = sum_k X[m][k] W[n][k], one CTA tile = 128 weight rows x 128 positions.
//
// The weight tile is the MMA's A operand (M = 128), the positions its B operand: the
// bf16 hi and lo parts of X stacked into one N = 256 operand, so one tcgen05.mma per
// 16-wide k-step computes W*Xhi and W*Xlo side by side in TMEM and the epilogue adds the
// two halves (fp32-like activations, exact bf16 weights, fp32 accumulation -- the decode
// path's precision).  One persistent CTA per SM (four 48 KB TMA stages, two 256-column
// TMEM accumulators so a tile's epilogue overlaps the next tile's MMAs); warp 0 streams
// TMA, warp 1 issues the MMAs, warps 2-5 drain TMEM.  Tiles are numbered weight-tile
// major, so the CTAs working at the same time share weight tiles through L2.
//
// Epilogues: store (q, k, v before RoPE), residual add (O and down projections), and
// SiLU(gate) * up written as the down projection's bf16 hi + lo operand.  RMSNorm and
// RoPE + the KV append are small row kernels here (the decode path folds them into the
// GEMMs); attention is the causal flash-attention kernel at the end of attention.cu.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sdsat {

constexpr int PF_STAGES = 6;
constexpr int PF_TOK = 128;                              // positions per tile
constexpr int PF_W_BYTES = 128 * 128;                    // a CTA's 128 weight rows x 64 bf16
constexpr int PF_X_BYTES = PF_TOK * 128;                 // 128 positions x 64 bf16: hi in rank 0, lo in rank 1
constexpr int PF_STAGE = PF_W_BYTES + PF_X_BYTES;        // 32 KB per CTA
constexpr int PF_ACC = 2 * PF_TOK;                       // TMEM columns of one accumulator (hi, lo)
constexpr int PF_CHUNK = 32;                             // positions per epilogue round
constexpr int PF_EPI_WARPS = 8;                          // two per TMEM lane quarter
constexpr int PF_THREADS = 64 + 32 * PF_EPI_WARPS;
constexpr int PF_XROW = PF_CHUNK / 2 + 1;                // exchange row: half a round's positions, padded
constexpr int PF_STAGING = 2 * 128 * PF_XROW;            // fp32 exchange of the two epilogue groups
constexpr int PF_NBAR = 2 * PF_STAGES + 5;
constexpr size_t PF_SMEM = 1024 + (size_t)PF_STAGES * PF_STAGE + PF_STAGING * 4 + PF_NBAR * 8 + 64;
#ifndef SDSAT_PF_GROUP
#define SDSAT_PF_GROUP 8
#endif
constexpr int PF_GROUP = SDSAT_PF_GROUP;
constexpr int PF_SK_MIN = 4;                             // chunks of a split-K share, at least

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
// whole tiles sk_tiles + pair, + P, ...  All roles of both CTAs walk the same list.
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

__global__ void __launch_bounds__(PF_THREADS, 1) prefill_gemm_kernel(const __grid_constant__ PfGemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stages = smem;
  float* staging = reinterpret_cast<float*>(smem + (size_t)PF_STAGES * PF_STAGE);
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + PF_STAGING);
  uint64_t* full = bars;                  // rank 0: both CTAs' weights and positions landed (TMA)
  uint64_t* empty = bars + PF_STAGES;     // the stage was consumed by the tensor cores
  uint64_t* acc_full = bars + 2 * PF_STAGES;   // [2] accumulator ready
  uint64_t* acc_empty = acc_full + 2;          // [2] rank 0: accumulator drained in both CTAs
  uint64_t* drain = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* s_last = reinterpret_cast<int*>(tmem_slot + 2);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank(), pair = (int)blockIdx.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < PF_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * PF_EPI_WARPS);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (threadIdx.x == 64) {
    const int nmaps = p.map_mode == MAP_QKV3 ? 3 : (p.map_mode == MAP_GATEUP ? 2 : 1);
    for (int i = 0; i < nmaps; ++i) tma_prefetch_desc(&p.tmap[i]);
    tma_prefetch_desc(&p.tmap_x[rank]);
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, 2 * PF_ACC);
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
        uint8_t* dst = stages + (size_t)s * PF_STAGE;
        tma_load_2d_pair(dst, &p.tmap[map0], bar, kc * 64, row0, pol_w);
        tma_load_2d_pair(dst + 8192, &p.tmap[map1], bar, kc * 64, row1, pol_w);
      };
      auto load_x = [&](int s, uint32_t bar, int k, int tb) {
        tma_load_2d_pair(stages + (size_t)s * PF_STAGE + PF_W_BYTES, &p.tmap_x[rank], bar, k * 64, tb * PF_TOK, pol_x);
      };
      // the weights of the first stages do not depend on the previous kernel
      int xk[PF_STAGES], xt[PF_STAGES], npre = 0;
      src();
#pragma unroll
      for (int s = 0; s < PF_STAGES; ++s) {
        xk[s] = kc;
        xt[s] = tb;
        if (!more) continue;
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * PF_STAGE);
        load_w(s, mapa_shared(smem_u32(&full[s]), 0));
        npre = s + 1;
        if (step() && more) src();
      }
      pdl_wait();   // the positions are the previous kernel's output
#pragma unroll
      for (int s = 0; s < PF_STAGES; ++s)
        if (s < npre) load_x(s, mapa_shared(smem_u32(&full[s]), 0), xk[s], xt[s]);
      int it = npre, s = it % PF_STAGES;
      uint32_t ph = 0;   // parity of the stage's previous use being consumed
      while (more) {
        if (!mbar_wait_bounded(&empty[s], ph, abort_flag, p.err)) break;
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * PF_STAGE);
        const uint32_t bar = mapa_shared(smem_u32(&full[s]), 0);
        load_w(s, bar);
        load_x(s, bar, kc, tb);
        ++it;
        if (++s == PF_STAGES) {
          s = 0;
          ph ^= 1u;
        }
        if (step() && more) src();
      }
      if (!*abort_flag) {
        // the CTA stays until the tensor cores have released its last stages (the commits of
        // rank 0 arrive on this CTA's barriers)
        for (int i = std::max(0, it - PF_STAGES); i < it; ++i)
          if (!mbar_wait_bounded(&empty[i % PF_STAGES], (i / PF_STAGES) & 1, abort_flag, p.err)) break;
      }
      if (*abort_flag) {   // let every copy in flight land before the CTA exits
        if (rank == 0) {
          for (int i = std::max(0, it - PF_STAGES); i < it; ++i) pf_drain(&full[i % PF_STAGES], (i / PF_STAGES) & 1);
        } else {           // counted on rank 0's barriers: 10 ms, far past any copy
          const uint64_t t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 < 10000000ull) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ tensor-core issue, for the pair
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(256, PF_ACC);
      int s = 0, seg = 0;
      uint32_t ph = 0;
      bool ok = true;
      PfWalk w(p, pair);
      while (ok && w.next()) {
        const int buf = seg & 1;
        if (!mbar_wait_bounded(&acc_empty[buf], ((seg >> 1) & 1) ^ 1, abort_flag, p.err)) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * PF_ACC;
        for (int kc = w.k0; kc < w.k1; ++kc) {
          if (!mbar_wait_bounded(&full[s], ph, abort_flag, p.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t wa = smem_u32(stages + (size_t)s * PF_STAGE);
          const uint32_t xb = wa + PF_W_BYTES;   // rows of Xhi here, of Xlo in rank 1
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma_bf16_pair(d, sdesc_sw128(wa + kk * 32), sdesc_sw128(xb + kk * 32), idesc,
                           (kc > w.k0 || kk > 0) ? 1u : 0u);
          umma_commit_pair(&empty[s]);
          if (++s == PF_STAGES) {
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
    int seg = 0;
    PfWalk w(p, pair);
    for (; w.next(); ++seg) {
      int wp, tb;
      pf_tile(p, w.tile, wp, tb);
      const int wt = 2 * wp + rank;
      const int buf = seg & 1;
      const int mt = tb * PF_TOK;   // the tile's first position
      const bool got = named_bar_and(1, NE, mbar_wait_bounded(&acc_full[buf], (seg >> 1) & 1, abort_flag, p.err));
      if (!got) break;
      tc_fence_after();
      const uint32_t lane_addr = tmem + ((uint32_t)(e * 32) << 16) + buf * PF_ACC;
      // hi + lo products of 32 positions; after the warp's last round the accumulator is drained
      auto load_acc = [&](int c0, float (&y)[PF_CHUNK]) {
        float ya[16], yb[16], la[16], lb[16];
        tmem_ld16(lane_addr + c0, ya);
        tmem_ld16(lane_addr + c0 + 16, yb);
        tmem_ld16(lane_addr + PF_TOK + c0, la);
        tmem_ld16(lane_addr + PF_TOK + c0 + 16, lb);
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
      int lo = 0, hi = 0;
      const bool shared = w.k1 - w.k0 < p.kc;
      if (shared) {
        // a split tile: publish this pair's part; the last contributor sums the parts in pair
        // order (deterministic) and runs the epilogue
        const int slot = w.k0 == 0;   // a share holds at most one part that starts its tile
        float* mine = p.partials + ((size_t)(pair * 2 + slot) * 2 + rank) * PF_TOK * 128;
        for (int c0 = grp * PF_CHUNK; c0 < PF_TOK && mt + c0 < p.M; c0 += 2 * PF_CHUNK) {
          float y[PF_CHUNK];
          load_acc(c0, y);
#pragma unroll
          for (int j = 0; j < PF_CHUNK; ++j)
            if (mt + c0 + j < p.M) __stcg(mine + (c0 + j) * 128 + r, y[j]);
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
      }
      for (int c0 = grp * PF_CHUNK; c0 < PF_TOK && mt + c0 < p.M; c0 += 2 * PF_CHUNK) {
        const int m0 = mt + c0;   // (uniform over the group's 128 threads)
        float y[PF_CHUNK];
        if (!shared) {
          load_acc(c0, y);
          if (c0 + 2 * PF_CHUNK >= PF_TOK || m0 + 2 * PF_CHUNK >= p.M) drained();
        } else {
#pragma unroll
          for (int j = 0; j < PF_CHUNK; ++j) y[j] = 0.f;
          for (int i = lo; i <= hi; ++i) {
            const float* src = p.partials + ((size_t)(i * 2 + (i == lo)) * 2 + rank) * PF_TOK * 128 + c0 * 128 + r;
#pragma unroll
            for (int j = 0; j < PF_CHUNK; ++j)
              if (m0 + j < p.M) y[j] += __ldcg(src + j * 128);
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
      if (!shared && mt + grp * PF_CHUNK >= p.M) drained();   // no round of its own in this tile
    }
  }

  tc_fence_before();
  cluster_sync_all();   // neither CTA leaves while the other may still signal its barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 2 * PF_ACC);
  }
}

namespace {
int g_pf_pairs = 0;   // CTA pairs resident at once
}

cudaError_t prefill_prepare() {
  cudaError_t e = cudaFuncSetAttribute(prefill_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PF_SMEM);
  if (e != cudaSuccess || g_pf_pairs > 0) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(PF_THREADS);
  cfg.dynamicSmemBytes = PF_SMEM;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, prefill_gemm_kernel, &cfg);
  if (e == cudaSuccess) g_pf_pairs = n;
  return e;
}

size_t prefill_partials(int num_sms) { return (size_t)(num_sms / 2) * 2 * 2 * PF_TOK * 128; }

cudaError_t launch_prefill_gemm(PfGemmParams& p, int num_sms, cudaStream_t st, bool pdl) {
  const int P = std::max(1, std::min(num_sms / 2, g_pf_pairs));
  p.n_pairs_w = (p.n_wtiles + 1) / 2;
  p.group = std::min(p.n_tblocks, PF_GROUP);
  const int T = p.n_pairs_w * p.n_tblocks, rem = T % P;
  p.sk_tiles = 0;
  p.sk_pairs = 0;
  if (rem && (P - rem) * p.kc >= 8 * P) {
    p.sk_tiles = rem;
    p.sk_pairs = std::max(rem, std::min(P, rem * p.kc / PF_SK_MIN));
    if (p.sk_pairs == rem) p.sk_tiles = p.sk_pairs = 0;   // nothing to split
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * std::min(P, std::max(p.sk_pairs, T - p.sk_tiles)));
  cfg.blockDim = dim3(PF_THREADS);
  cfg.dynamicSmemBytes = PF_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, prefill_gemm_kernel, p);
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
