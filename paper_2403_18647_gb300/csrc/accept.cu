// Target selection, verification and KV commit, plus the small kernels of the
// step (embedding gather, block-input building, explicit commit).
//
// Verification (Sec. 2.1.1, Eq. 3): with targets t_j (argmax or nucleus sample
// of block row j) and drafts d_i (the block's input token of row i), draft i is
// accepted while d_i == t_{i-1} for all i' <= i; the first mismatch stops the
// loop.  The emitted tokens are t_0 .. t_m and the committed KV length grows by
// 1 + m (the rejected rows, and in draft step 1 the adaptive-token rows, are
// rolled back by not being committed).
//
// One thread-block cluster per block row selects that row's target; the last row of a
// sequence (per-sequence counter, no waiting) runs the prefix scan and the commit.
//
// Tree blocks (Sec. 2.1.2): the rows are the nodes of a draft tree in
// topological order (parent[j] < j, row 0 the root).  Row j sits at position
// len + depth(j); a child is accepted when its parent is and its token equals
// the parent's target, and the deepest accepted node (lowest row among equally
// deep ones) ends the accepted path n_0 = 0, ..., n_m.  Its targets are
// emitted, and a compaction kernel moves the path's K and V rows to the slots
// len + 1 .. len + m before len advances by 1 + m.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sdsat {

// ---- the nucleus sampler's arithmetic -------------------------------------------
// exp(s) for s <= 0: Cody-Waite reduction with a two-part ln 2, degree-7 Taylor
// polynomial on |r| <= ln2/2 by Horner's rule, exact scaling by 2^n; every step
// is one correctly rounded fp32 operation (no contraction), so any IEEE
// implementation of the same steps gives the same bits.
__device__ __forceinline__ float exp_sd(float s) {
  if (!(s >= -87.0f)) return 0.0f;
  const float n = rintf(__fmul_rn(s, (float)1.4426950408889634));
  const float r = __fsub_rn(__fsub_rn(s, __fmul_rn(n, 0.693145751953125f)), __fmul_rn(n, (float)(0.6931471805599453 - 0.693145751953125)));
  float p = (float)(1.0 / 5040.0);        // 1/7!
  p = __fadd_rn(__fmul_rn(p, r), (float)(1.0 / 720.0));  // 1/6!
  p = __fadd_rn(__fmul_rn(p, r), (float)(1.0 / 120.0));  // 1/5!
  p = __fadd_rn(__fmul_rn(p, r), (float)(1.0 / 24.0));  // 1/4!
  p = __fadd_rn(__fmul_rn(p, r), (float)(1.0 / 6.0));  // 1/3!
  p = __fadd_rn(__fmul_rn(p, r), 0.5f);
  p = __fadd_rn(__fmul_rn(p, r), 1.0f);
  p = __fadd_rn(__fmul_rn(p, r), 1.0f);
  const float scale = __int_as_float(((int)n + 127) << 23);
  return __fmul_rn(p, scale);
}

// floor(w * 2^24) for 0 <= w <= 1, exactly, from the fp32 bits
__device__ __forceinline__ uint32_t fixed24(float w) {
  const uint32_t b = __float_as_uint(w);
  if (b == 0) return 0;
  const int sh = (int)((b >> 23) & 0xFF) - 127 + 1;   // W = mant * 2^(e - 23 + 24)
  const uint32_t mant = (b & 0x7FFFFFu) | 0x800000u;
  if (sh >= 0) return mant << sh;
  return sh <= -24 ? 0u : (mant >> (-sh));
}

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11)
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
    const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

// ---- the row's cluster -------------------------------------------------------------------
// One thread-block cluster per row: p.cs CTAs of ACC_THREADS threads; thread t of rank r owns
// the ids [ACC_SPAN r + ACC_EPT t, + ACC_EPT) (ascending id order is rank, thread, slot order).
// One CTA per row (1024 threads of 32 ids) left most SMs idle and ran its chain of dependent
// steps on four times the work per thread.  us per call, 32016 logits a row, one CTA per row (with
// a sorted list, or binary searches over the row) -> a cluster, and cuts by digits: 24 rows, top-p
// 0.95, T 0.2: 48.4 -> 14.4 (22.6 with the sort); with top-k 10: 34.5 -> 16.6; T 1 (row-wide):
// 101 -> 22.7 (46.8 with the searches); greedy 7.1 -> 5.0; 64 rows (512 CTAs, four on an SM):
// 48 -> 22.5, T 1: 101 -> 37.7, greedy 7.4 -> 6.3.  What is left is the chain of barriers and of
// instructions fetched cold, not bytes (3 MB).
// A sum over the row: the warps' totals meet in shared
// memory, warp 0 writes the CTA's total into every CTA of the cluster (distributed shared
// memory), and after one cluster barrier each warp reads the cluster's totals locally.  (Every
// warp reading every warp's total remotely was 15 us a sum with 24 rows.)  Two buffers
// alternate: one is written again only after the next barrier, which no CTA passes before
// every CTA has read it.
constexpr int ACC_THREADS = 512;
constexpr int ACC_EPT = 8;
constexpr int ACC_SPAN = ACC_THREADS * ACC_EPT;   // 4096 ids per CTA, vocab <= 32768
constexpr int ACC_WARPS = ACC_THREADS / 32;
constexpr int ACC_CS = 8;                         // most CTAs of a row
constexpr int ACC_WORDS = 4;                      // most 64-bit words summed together
static_assert(ACC_WARPS == 16 && ACC_CS == 8 && ACC_WORDS == 4, "eight lanes of a warp per word");

struct AccSlots {
  unsigned long long w[2][ACC_WARPS * ACC_WORDS];   // this CTA's warps
  unsigned long long c[2][ACC_CS * ACC_WORDS];      // the cluster's CTAs, written by each of them
};

__device__ __forceinline__ void st_dsmem_u64(uint32_t addr, uint64_t v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t ld_dsmem_u64(uint32_t addr) {
  uint64_t v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// a warp's total of per-thread sums below 2^29
__device__ __forceinline__ uint64_t warp_total(uint32_t v) {
  const uint64_t hi = __reduce_add_sync(0xffffffffu, v >> 12);
  return (hi << 12) + __reduce_add_sync(0xffffffffu, v & 4095u);
}

struct Row {   // the row's cluster, seen from one thread
  AccSlots* slots;
  int cs, rank, ph;
  // v[n]: this warp's values (every lane); afterwards combine() of them over the row, and with
  // `before` the sum of word 0 over the warps that come before this one in id order.  Eight lanes
  // per word, so all words go through the same three shuffles.
  template <int N, typename F>
  __device__ void reduce(uint64_t (&v)[N], uint64_t identity, F combine, uint64_t* before = nullptr) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, n = lane >> 3, i = lane & 7;
    unsigned long long* mine = slots->w[ph & 1];
    unsigned long long* all = slots->c[ph & 1];
    ++ph;
    auto over8 = [&](uint64_t t) {
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) t = combine(t, (uint64_t)__shfl_xor_sync(0xffffffffu, t, o));
      return t;
    };
    if (lane == 0)
#pragma unroll
      for (int k = 0; k < N; ++k) mine[k * ACC_WARPS + w] = v[k];
    __syncthreads();
    if (w == 0) {
      const uint64_t t = over8(n < N ? combine((uint64_t)mine[n * ACC_WARPS + i], (uint64_t)mine[n * ACC_WARPS + 8 + i]) : identity);
      if (n < N && i < cs) st_dsmem_u64(mapa_shared(smem_u32(&all[n * ACC_CS + rank]), i), t);
    }
    cluster_sync_all();
    const uint64_t t = n < N && i < cs ? all[n * ACC_CS + i] : identity;
    if (before)   // earlier CTAs, then earlier warps of this one
      *before = warp_sum_u64((lane < rank ? t : 0) + (lane < w ? mine[lane] : 0));
    const uint64_t r = over8(t);
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = __shfl_sync(0xffffffffu, r, 8 * k);
  }
  template <int N>
  __device__ void sum(uint64_t (&v)[N], uint64_t* before = nullptr) {
    reduce<N>(v, 0, [](uint64_t a, uint64_t b) { return a + b; }, before);
  }
  __device__ uint64_t largest(uint64_t warp_value) {
    uint64_t v[1] = {warp_value};
    reduce<1>(v, 0, [](uint64_t a, uint64_t b) { return a > b ? a : b; });
    return v[0];
  }
  __device__ uint64_t sum(uint64_t warp_value) {
    uint64_t v[1] = {warp_value};
    sum<1>(v);
    return v[0];
  }
  // exclusive prefix over the row's threads, in id order
  __device__ uint64_t exscan(uint64_t v) {
    const int lane = threadIdx.x & 31;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    uint64_t t[1] = {__shfl_sync(0xffffffffu, x, 31)}, before;
    sum<1>(t, &before);
    return before + x - v;
  }
};

// ---- block-wide sums (the list runs in one CTA) --------------------------------------------
__device__ __forceinline__ uint64_t block_sum_u64(uint64_t v, uint64_t* red) {
  v = warp_sum_u64(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  return warp_sum_u64(l < ACC_WARPS ? red[l] : 0);
}

// exclusive prefix sum over threads (in thread order) of v
__device__ __forceinline__ uint64_t block_exscan_u64(uint64_t v, uint64_t* red) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  uint64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (l >= o) x += y;
  }
  __syncthreads();
  if (l == 31) red[w] = x;
  __syncthreads();
  return warp_sum_u64(l < w ? red[l] : 0) + x - v;
}

// ---- greedy: argmax with the lowest id on ties, NaN as -inf ----------------------------
// (float value ordered as an unsigned word, inverted id): larger is heavier, then lower id
__device__ __forceinline__ uint64_t arg_key(float x, int id) {
  const uint32_t b = __float_as_uint(x);
  return ((uint64_t)((b & 0x80000000u) ? ~b : b | 0x80000000u) << 32) | (uint32_t)(0x7FFFFFFF - id);
}

__device__ int row_argmax(const float* row, int V, uint32_t* err, Row& rw) {
  float best = -INFINITY;
  int bi = 0;   // (a thread without ids, or with NaN alone, loses to any other: see the key)
  bool nan = false, any = false;
  auto take = [&](float x, int i) {
    if (x != x) {
      nan = true;
      x = -INFINITY;
    }
    x += 0.f;   // -0 counts as +0
    if (!any || x > best) {
      any = true;
      best = x;
      bi = i;
    }
  };
  // float4 loads, a round of RN per thread issued before any is compared; the row's CTAs take
  // its rounds in turn, a thread visits its ids in increasing order
  constexpr int RN = 2;
  const int nthr = rw.cs * ACC_THREADS, tid = rw.rank * ACC_THREADS + threadIdx.x;
  const bool vec = (reinterpret_cast<uintptr_t>(row) & 15u) == 0;
  const int V4 = vec ? V / 4 : 0;
  for (int i0 = 0; i0 < V4; i0 += RN * nthr) {
    float4 v[RN];
#pragma unroll
    for (int u = 0; u < RN; ++u) {
      const int i = i0 + u * nthr + tid;
      if (i < V4) v[u] = __ldcg(reinterpret_cast<const float4*>(row) + i);
    }
#pragma unroll
    for (int u = 0; u < RN; ++u) {
      const int i = i0 + u * nthr + tid;
      if (i < V4) {
        take(v[u].x, 4 * i);
        take(v[u].y, 4 * i + 1);
        take(v[u].z, 4 * i + 2);
        take(v[u].w, 4 * i + 3);
      }
    }
  }
  for (int i = 4 * V4 + tid; i < V; i += nthr) take(__ldcg(row + i), i);
  if (nan) set_error(err, ERR_NAN_LOGITS);
  uint64_t key = any ? arg_key(best, bi) : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) key = max(key, (uint64_t)__shfl_xor_sync(0xffffffffu, key, o));
  key = rw.largest(key);
  return 0x7FFFFFFF - (int)(uint32_t)key;
}

// ---- nucleus: the fixed-point top-k / top-p sampler ------------------------------------
// The kept set is a prefix of the order (W desc, id asc): every W above a cut x, and the first
// `ties` ids with W == x.  The cut (of a count for top-k, of a mass for top-p) is found digit by
// digit: three histograms of 256 bins over W - 1, highest digit first, each scanned from the
// heaviest bin to the one where the running sum reaches what is needed.
//
// The kept set lies among the heaviest weights.  With a floor such that the elements with W >=
// floor provably contain it (top-k: at least k of them, or all non-zero weights; top-p alone:
// their mass reaches the top-p threshold), those elements go in ascending id order into rank 0's
// shared memory, and that CTA finishes the row with block barriers only.  Otherwise (more than
// NUC_LIST_MAX of them) the same steps run over all ids, with histograms summed over the cluster.
constexpr int NUC_LIST_MAX = 4096;
constexpr int NUC_FLOORS = 7;

struct NucSmem {
  unsigned long long key[NUC_LIST_MAX];     // the list (rank 0): W << 32 | id, ascending id
  uint32_t own[ACC_EPT * ACC_THREADS];      // [slot][thread]: the threads' logits, then their W
  uint32_t lo[256], hi[256];                // histogram: sums of W & 4095 (or counts) and of W >> 12; 0 between uses
  unsigned long long bins[2][256];          // row-wide: this CTA's histogram, for the cluster
  unsigned long long above;
  int digit, pick;
};

// The largest x whose sum over the elements with W >= x is >= need (1 <= need <= their total), W
// itself summed or (COUNT) their number, and `above`, the sum over W > x.  each(f) calls f(W) for
// this thread's elements; a W of 0 is in no sum.  ROW: over the cluster, otherwise over the block.
template <bool COUNT, bool ROW, typename E>
__device__ __forceinline__ uint32_t weight_cut(NucSmem& L, E each, uint64_t need, uint64_t& above, uint64_t* red, Row& rw) {
  uint32_t prefix = 0;   // the digits of x - 1 found so far
  above = 0;
#pragma unroll 1
  for (int sh = 16; sh >= 0; sh -= 8) {
    each([&](uint32_t W) {
      const uint32_t u = W - 1;
      if (W == 0 || (u >> sh) >> 8 != prefix) return;
      const uint32_t b = (u >> sh) & 255u;
      atomicAdd(&L.lo[b], COUNT ? 1u : W & 4095u);     // <= 2^24 with 4096 elements a CTA
      if (!COUNT) atomicAdd(&L.hi[b], W >> 12);
    });
    __syncthreads();
    const int b = 255 - (int)threadIdx.x;   // one bin per thread, heaviest first
    uint64_t v = 0;
    if (b >= 0) {
      v = ((uint64_t)L.hi[b] << 12) + L.lo[b];
      L.lo[b] = L.hi[b] = 0;
    }
    if (ROW) {   // (a buffer is written again after another cluster barrier, when every CTA has read it:
                 // two steps later, or after the row sum between two cuts)
      unsigned long long* mine = L.bins[(sh >> 3) & 1];
      if (b >= 0) mine[b] = v;
      cluster_sync_all();
      v = 0;
      if (b >= 0)
        for (int c = 0; c < rw.cs; ++c) v += ld_dsmem_u64(mapa_shared(smem_u32(&mine[b]), c));
    }
    const uint64_t before = above + block_exscan_u64(v, red);
    if (before < need && before + v >= need) {   // one thread
      L.digit = b;
      L.above = before;
    }
    __syncthreads();
    prefix = prefix << 8 | (uint32_t)L.digit;
    above = L.above;
  }
  return prefix + 1;
}

// ceil(P S / 2^24), and 1 where that is 0 (the heaviest candidate is always kept)
__device__ __forceinline__ uint64_t top_p_need(const AcceptParams& p, uint64_t S) {
  const uint64_t prod = (uint64_t)p.p_fixed * S;   // P <= 2^24, S < 2^40
  return max((uint64_t)1, (prod >> 24) + ((prod & 0xFFFFFFull) ? 1 : 0));
}

// Steps 4-5: the kept set's cut.  each as above; total: sum of
// W over every id; k: candidates (0: all).  Kept are W > x and the first `ties` ids with W == x,
// together `mass`.
template <bool ROW, typename E, typename S>
__device__ __forceinline__ void kept_cut(const AcceptParams& p, NucSmem& L, E each, S total_of, uint64_t total,
                                         uint32_t k, uint64_t* red, Row& rw, uint32_t& x, uint64_t& ties, uint64_t& mass) {
  uint64_t need, above;
  x = 0;
  if (k) {   // 4. the k largest, then their mass
    const uint32_t xk = weight_cut<true, ROW>(L, each, k, above, red, rw);
    uint64_t gt = 0;
    each([&](uint32_t W) { gt += W > xk ? W : 0u; });
    gt = total_of(gt);
    need = top_p_need(p, gt + (k - above) * xk);
    if (gt < need) x = xk, above = gt;   // the top-k cut's own weight; heavier ones otherwise
  } else {
    need = top_p_need(p, total);
  }
  if (x == 0) x = weight_cut<false, ROW>(L, each, need, above, red, rw);   // 5.
  ties = need - above <= x ? 1 : (need - above + x - 1) / x;
  mass = above + ties * x;
}

// A prefix of elements in ascending id order as one word: the mass of those above the cut and
// the number at it (mass <= 2^39, number <= 2^15), and the kept mass that it stands for.
__device__ __forceinline__ uint64_t kept_word(uint32_t W, uint32_t x) { return W > x ? W : (W == x ? 1ull << 40 : 0ull); }
__device__ __forceinline__ uint64_t kept_mass(uint64_t word, uint32_t x, uint64_t ties) {
  return (word & ((1ull << 40) - 1)) + min(word >> 40, (uint64_t)ties) * x;
}

// The row's sampled id (valid in rank 0).  Every CTA of the cluster passes the same barriers:
// every branch is taken on values that the whole row shares.  These steps run once a call, so
// their instructions are fetched cold: loops over a thread's ids stay rolled, through shared memory.
__device__ __forceinline__ int row_nucleus(const AcceptParams& p, const float* row, int position, int seq,
                                           uint64_t* red, Row& rw, NucSmem& L) {
  const int V = p.V, tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int base = rw.rank * ACC_SPAN + tid * ACC_EPT;
  uint32_t* own = L.own + tid;   // slot e at own[e * ACC_THREADS]
  if (tid < 256) L.lo[tid] = L.hi[tid] = 0;
  float mx = -INFINITY;
  {
    // 1. logits (NaN -> -inf; ids >= V are -inf, hence W = 0) and the row maximum
    float l[ACC_EPT];
    if ((reinterpret_cast<uintptr_t>(row) & 15u) == 0 && base + ACC_EPT <= V) {
#pragma unroll
      for (int e = 0; e < ACC_EPT; e += 4) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(row + base + e));
        l[e] = v.x; l[e + 1] = v.y; l[e + 2] = v.z; l[e + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < ACC_EPT; ++e) l[e] = base + e < V ? __ldcg(row + base + e) : -INFINITY;
    }
    bool nan = false;
#pragma unroll
    for (int e = 0; e < ACC_EPT; ++e) {
      if (l[e] != l[e]) {
        nan = true;
        l[e] = -INFINITY;
      }
      mx = fmaxf(mx, l[e]);
      own[e * ACC_THREADS] = __float_as_uint(l[e]);
    }
    if (nan) set_error(p.err, ERR_NAN_LOGITS);
    // (ordered as in arg_key)
    const uint32_t ord = (uint32_t)rw.largest(__reduce_max_sync(0xffffffffu, (uint32_t)(arg_key(mx, 0) >> 32)));
    mx = __uint_as_float((ord & 0x80000000u) ? ord & 0x7FFFFFFFu : ~ord);
  }
  // 2-3. W_i = floor(exp((l_i - max) / T) * 2^24), which is 0 where (l_i - max) / T < -17 (e^-17 <
  // 2^-24 by a third, far more than any rounding here).  Floors 0-6: 2^24 (the largest weight),
  // 2^22, 2^20, 2^18, 2^16 (ratio 2^-8), 2^8 (2^-16), then 1 (every non-zero weight): the number
  // of weights above each, 10 bits a field, and the mass above the last three.
  const bool topk = p.top_k > 0 && p.top_k < V;
  const float cut = -17.0f * p.temperature;
  uint32_t c02 = 0, c35 = 0, c6 = 0, m4 = 0, m5 = 0, m6 = 0;   // (counts <= 8, masses <= 2^27)
#pragma unroll 1
  for (int e = 0; e < ACC_EPT; ++e) {
    const float d = __fsub_rn(__uint_as_float(own[e * ACC_THREADS]), mx);
    uint32_t W = 0;
    if (!(d < cut)) W = fixed24(exp_sd(__fdiv_rn(d, p.temperature)));
    own[e * ACC_THREADS] = W;
    if (W) {
      c02 += (W >> 24) + ((W >> 22 ? 1u : 0u) << 10) + ((W >> 20 ? 1u : 0u) << 20);
      c35 += (W >> 18 ? 1u : 0u) + ((W >> 16 ? 1u : 0u) << 10) + ((W >> 8 ? 1u : 0u) << 20);
      c6 += 1;
      m4 += W >> 16 ? W : 0u;
      m5 += W >> 8 ? W : 0u;
      m6 += W;
    }
  }
  // 6. the 64-bit draw keyed by (produced position, sequence)
  uint32_t ctr[4] = {(uint32_t)position, (uint32_t)seq, 0u, 0u};
  philox4x32_10(ctr, (uint32_t)(p.seed & 0xFFFFFFFFull), (uint32_t)(p.seed >> 32));
  const uint64_t rnd = ((uint64_t)ctr[0] << 32) | ctr[1];

  // Row totals.  Top-k: 16-bit counts (<= 32768) of floors 0-3 and 4-6; top-p alone: the counts
  // of floors 4-6 and the three masses.
  const uint32_t r35 = __reduce_add_sync(0xffffffffu, c35), r6 = __reduce_add_sync(0xffffffffu, c6);
  const uint64_t n46 = (uint64_t)((r35 >> 10) & 1023u) | (uint64_t)(r35 >> 20) << 16 | (uint64_t)r6 << 32;
  uint64_t t[ACC_WORDS] = {n46, warp_total(m6), 0, 0};
  if (topk) {
    const uint32_t r02 = __reduce_add_sync(0xffffffffu, c02);
    t[2] = (uint64_t)(r02 & 1023u) | (uint64_t)((r02 >> 10) & 1023u) << 16 | (uint64_t)(r02 >> 20) << 32 |
           (uint64_t)(r35 & 1023u) << 48;
  } else {
    t[2] = warp_total(m4);
    t[3] = warp_total(m5);
  }
  const int buf = rw.ph & 1;
  rw.sum<ACC_WORDS>(t);
  const uint64_t S_all = t[1];
  const int n_all = (int)((t[0] >> 32) & 0xFFFF);   // non-zero weights
  if (n_all == 0) return 0;   // every weight 0 (all-NaN row): the lowest candidate, id 0
  const uint32_t k = topk ? min((uint32_t)p.top_k, (uint32_t)n_all) : 0u;

  // the highest floor whose elements provably hold the candidates (top-k) or the kept prefix
  int f = -1, nf = 0;
  const uint64_t need_all = top_p_need(p, S_all);
#pragma unroll
  for (int i = 0; i < NUC_FLOORS; ++i) {
    if (i < 4 && !topk) continue;
    const int n = (int)((i < 4 ? t[2] >> (16 * i) : t[0] >> (16 * (i - 4))) & 0xFFFF);
    const bool holds = topk ? n >= (int)k : (i == 4 ? t[2] : i == 5 ? t[3] : S_all) >= need_all;
    if (f < 0 && n <= NUC_LIST_MAX && holds) f = i, nf = n;
  }
  if (f >= 0) {
    const uint32_t floor_w = f <= 4 ? 1u << (24 - 2 * f) : (f == 5 ? 256u : 1u);
    // this thread's place in the list: the CTAs and warps before (from the totals just
    // summed), then the lanes before
    uint32_t mine = 0;
#pragma unroll
    for (int e = 0; e < ACC_EPT; ++e) mine += own[e * ACC_THREADS] >= floor_w;
    if (__any_sync(0xffffffffu, mine != 0)) {
      const int word = f < 4 ? 2 : 0, sh = 16 * (f & 3);
      uint32_t at = 0, x = mine;
      if (lane < rw.rank) at += (uint32_t)(rw.slots->c[buf][word * ACC_CS + lane] >> sh) & 0xFFFFu;
      if (lane < w) at += (uint32_t)(rw.slots->w[buf][word * ACC_WARPS + lane] >> sh) & 0xFFFFu;
      at = __reduce_add_sync(0xffffffffu, at);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      uint32_t dst = mapa_shared(smem_u32(&L.key[0]), 0) + (at + x - mine) * 8;
#pragma unroll 1
      for (int e = 0; mine; ++e) {
        const uint32_t W = own[e * ACC_THREADS];
        if (W >= floor_w) {
          st_dsmem_u64(dst, (uint64_t)W << 32 | (uint32_t)(base + e));
          dst += 8;
          --mine;
        }
      }
    }
    cluster_sync_all();   // the list is complete
    if (rw.rank) return 0;
    uint32_t x;
    uint64_t ties, mass;
    kept_cut<false>(
        p, L, [&](auto f) { for (int i = tid; i < nf; i += ACC_THREADS) f((uint32_t)(L.key[i] >> 32)); },
        [&](uint64_t v) { return block_sum_u64(v, red); }, S_all, k, red, rw, x, ties, mass);
    // 7. the first kept id (ascending) whose inclusive cumulative weight exceeds tau
    const uint64_t tau = __umul64hi(rnd, mass);
    const int per = (nf + ACC_THREADS - 1) / ACC_THREADS, i0 = min(tid * per, nf), i1 = min(i0 + per, nf);
    uint64_t sum = 0;
    for (int i = i0; i < i1; ++i) sum += kept_word((uint32_t)(L.key[i] >> 32), x);
    uint64_t word = block_exscan_u64(sum, red);
    if (kept_mass(word, x, ties) <= tau && kept_mass(word + sum, x, ties) > tau) {
      int i = i0 - 1;
      do word += kept_word((uint32_t)(L.key[++i] >> 32), x);
      while (kept_mass(word, x, ties) <= tau);
      L.pick = (int)(uint32_t)L.key[i];
    }
    __syncthreads();
    return L.pick;
  }

  // ---- the same over all ids
  uint32_t x;
  uint64_t ties, mass;
  auto each = [&](auto f) { for (int e = 0; e < ACC_EPT; ++e) f(own[e * ACC_THREADS]); };
  kept_cut<true>(
      p, L, each, [&](uint64_t v) { return rw.sum(warp_sum_u64(v)); }, S_all, k, red, rw, x, ties, mass);
  const uint64_t tau = __umul64hi(rnd, mass);
  uint64_t sum = 0;
  each([&](uint32_t W) { sum += kept_word(W, x); });
  uint64_t word = rw.exscan(sum);
  uint32_t hit = 0;   // id + 1 in the one thread that holds it
  if (kept_mass(word, x, ties) <= tau && kept_mass(word + sum, x, ties) > tau) {
    int e = -1;
    do word += kept_word(own[++e * ACC_THREADS], x);
    while (kept_mass(word, x, ties) <= tau);
    hit = base + e + 1;
  }
  return (int)rw.sum(warp_total(hit)) - 1;
}

// parent of tree row i (0 < i < q): an earlier row; anything else is flagged and read as the root
__device__ __forceinline__ int tree_parent(const int* par, int i, uint32_t* err) {
  int pi = __ldcg(par + i);
  if (pi < 0 || pi >= i) {
    set_error(err, ERR_TREE);
    pi = 0;
  }
  return pi;
}

// depth of tree row j (the root has depth 0); at most j steps since parents are earlier rows
__device__ __forceinline__ int tree_depth(const int* par, int j, uint32_t* err) {
  int d = 0;
  for (int i = j; i > 0; i = tree_parent(par, i, err)) ++d;
  return d;
}

// (greedy apart: 4.97 us instead of 5.19 with 24 rows; four CTAs an SM instead of two: 64 rows 22.5
// instead of 24.2 us, greedy 6.3 instead of 7.3)
template <bool NUCLEUS>
__global__ void __launch_bounds__(ACC_THREADS, 4) accept_kernel(const AcceptParams p) {
  extern __shared__ __align__(16) uint8_t acc_smem[];   // NucSmem (nucleus only)
  __shared__ AccSlots slots;
  __shared__ uint64_t red[ACC_WARPS];
  cluster_arrive_thread();
  pdl_wait();
  pdl_trigger();
  cluster_wait_thread();   // every CTA of the row has started: its shared memory may be written
  Row rw{&slots, p.cs, (int)cluster_ctarank(), 0};
  const int j = blockIdx.x / p.cs, sl = blockIdx.y, s = p.seq0 + sl;
  const float* row = p.logits + (size_t)(sl * p.q + j) * p.V;
  int t;
  if constexpr (!NUCLEUS) {
    t = row_argmax(row, p.V, p.err, rw);
  } else {
    // the produced token's position: one past the row's own (len + j, or len + depth(j))
    const int position = __ldcg(p.len + s) + (p.parent ? tree_depth(p.parent + sl * p.q, j, nullptr) : j) + 1;
    t = row_nucleus(p, row, position, s, red, rw, *reinterpret_cast<NucSmem*>(acc_smem));
  }
  // the last row of a sequence (per-sequence counter) verifies and commits
  if (rw.rank || threadIdx.x) return;
  p.targets[sl * p.q + j] = t;
  if (atomic_add_acq_rel_gpu(p.counters + sl, 1) != p.q - 1) return;
  int tg[SDSAT_ATT_MAXQ];
  for (int i = 0; i < p.q; ++i) tg[i] = __ldcg(p.targets + sl * p.q + i);
  int m = 0;
  if (!p.parent) {
    const int nv = p.n_verify_dev ? min(max(__ldcg(p.n_verify_dev + sl), 0), p.q - 1) : p.n_verify;
    for (int i = 1; i <= nv; ++i) {                 // Eq. 3: prefix of matching drafts
      if (__ldcg(p.drafts + sl * p.q + i) != tg[i - 1]) break;
      m = i;
    }
    for (int i = 0; i < p.q; ++i) p.out_tokens[sl * p.q + i] = tg[i];
  } else {
    // Sec. 2.1.2: the longest branch accepted by the chain test applied along every branch
    const int* par = p.parent + sl * p.q;
    int dep[SDSAT_ATT_MAXQ], path[SDSAT_ATT_MAXQ];
    uint32_t accm = 1u;
    int best = 0;
    dep[0] = 0;
    for (int i = 1; i < p.q; ++i) {
      const int pi = tree_parent(par, i, p.err);
      dep[i] = dep[pi] + 1;
      if (((accm >> pi) & 1u) && __ldcg(p.drafts + sl * p.q + i) == tg[pi]) {
        accm |= 1u << i;
        if (dep[i] > dep[best]) best = i;
      }
    }
    m = dep[best];
    for (int d = m, i = best; d >= 0; --d) {
      path[d] = i;
      if (d > 0) i = tree_parent(par, i, nullptr);
    }
    for (int i = 0; i < p.q; ++i) {
      p.out_tokens[sl * p.q + i] = i <= m ? tg[path[i]] : -1;
      if (p.path) p.path[sl * p.q + i] = i <= m ? path[i] : -1;
    }
    // the compaction kernel's input: committed length before this step, m, the path rows
    int* w = p.tree_ws + sl * TREE_WS_STRIDE;
    w[0] = __ldcg(p.len + s);
    w[1] = m;
    for (int i = 0; i <= m; ++i) w[2 + i] = path[i];
  }
  p.accepted_len[sl] = 1 + m;
  if (p.commit) {
    const int nl = __ldcg(p.len + s) + 1 + m;
    if (nl <= p.cap) p.len[s] = nl;
    else set_error(p.err, ERR_CAPACITY);
    if (p.emitted) p.emitted[s] += 1 + m;
  }
  p.counters[sl] = 0;
}

static cudaLaunchConfig_t make_cfg(dim3 grid, dim3 block, cudaStream_t st, bool pdl, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cfg;
}

cudaError_t launch_accept(const AcceptParams& p0, cudaStream_t st, bool pdl) {
  AcceptParams p = p0;
  p.cs = std::min(ACC_CS, (p.V + ACC_SPAN - 1) / ACC_SPAN);   // (a larger vocabulary is greedy only)
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = make_cfg(dim3(p.q * p.cs, p.nb), dim3(ACC_THREADS), st, pdl, attr);
  cfg.dynamicSmemBytes = p.temperature > 0.f ? sizeof(NucSmem) : 0;
  attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
  attr[cfg.numAttrs].val.clusterDim.x = p.cs;
  attr[cfg.numAttrs].val.clusterDim.y = 1;
  attr[cfg.numAttrs].val.clusterDim.z = 1;
  ++cfg.numAttrs;
  return p.temperature > 0.f ? cudaLaunchKernelEx(&cfg, accept_kernel<true>, p) : cudaLaunchKernelEx(&cfg, accept_kernel<false>, p);
}

// ---- RMSNorm into the GEMM operand ------------------------------------------------------
// x = h * rsqrt(mean(h^2) + eps) * g (Llama's RMSNorm, fp32), stored as bf16 hi + lo with
// hi = bf16(x), lo = bf16(x - hi), so hi + lo carries ~16 significant bits of x.  With
// tokens != null the row is first gathered from the embedding table (h = E[token]).
__device__ __forceinline__ void split_store(float v, __nv_bfloat16* hi, __nv_bfloat16* lo) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  *hi = h;
  *lo = __float2bfloat16_rn(v - __bfloat162float(h));
}

__global__ void __launch_bounds__(256) rmsnorm_kernel(const int* tokens, const __nv_bfloat16* E, int V, float* h,
                                                      int d, const __nv_bfloat16* g, float eps, __nv_bfloat16* xhi,
                                                      __nv_bfloat16* xlo, uint32_t* err) {
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x;
  float* hr = h + (size_t)m * d;
  const __nv_bfloat16* er = nullptr;
  if (tokens) {
    int t = __ldcg(tokens + m);
    if (t < 0 || t >= V) {
      if (threadIdx.x == 0) set_error(err, ERR_TOKEN);
      t = 0;
    }
    er = E + (size_t)t * d;
  }
  float ss = 0.f;
  for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) {
    float4 v;
    if (er) {
      const __nv_bfloat162* e2 = reinterpret_cast<const __nv_bfloat162*>(er + i);
      const float2 a = __bfloat1622float2(e2[0]), b = __bfloat1622float2(e2[1]);
      v = make_float4(a.x, a.y, b.x, b.y);
      *reinterpret_cast<float4*>(hr + i) = v;
    } else {
      v = __ldcg(reinterpret_cast<const float4*>(hr + i));
    }
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x < 32) {
    float t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) red[0] = t;
  }
  __syncthreads();
  const float inv = 1.0f / sqrtf(red[0] / (float)d + eps);
  for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(hr + i));
    const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      split_store(vv[e] * inv * __bfloat162float(g[i + e]), xhi + (size_t)m * d + i + e, xlo + (size_t)m * d + i + e);
  }
}

cudaError_t launch_rmsnorm(const int* tokens, const __nv_bfloat16* E, int V, float* h, int d, int M,
                           const __nv_bfloat16* gain, float eps, __nv_bfloat16* xhi, __nv_bfloat16* xlo,
                           uint32_t* err, cudaStream_t st, bool pdl) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(M), dim3(256), st, pdl, attr);
  return cudaLaunchKernelEx(&cfg, rmsnorm_kernel, tokens, E, V, h, d, gain, eps, xhi, xlo, err);
}

__global__ void split_kernel(const float* x, int n, __nv_bfloat16* xhi, __nv_bfloat16* xlo) {
  pdl_wait();
  pdl_trigger();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) split_store(__ldcg(x + i), xhi + i, xlo + i);
}

cudaError_t launch_split(const float* x, int M, int K, __nv_bfloat16* xhi, __nv_bfloat16* xlo, cudaStream_t st,
                         bool pdl) {
  cudaLaunchAttribute attr[1];
  const int n = M * K;
  cudaLaunchConfig_t cfg = make_cfg(dim3((n + 255) / 256), dim3(256), st, pdl, attr);
  return cudaLaunchKernelEx(&cfg, split_kernel, x, n, xhi, xlo);
}

// ---- block input of draft step 1 (mode 1) and draft step 2 (mode 2) --------------------
// The previous block had prev_q rows per sequence.  Mode 2 builds `width` chains of k drafts
// below the root (width 1: the chain block; row 1 + w*k + i - 1 holds branch w's draft for
// position len + i, from table w).
__global__ void build_block_kernel(BuildParams b) {
  pdl_wait();
  pdl_trigger();
  const int sl = blockIdx.x, j = threadIdx.x;
  const int* prev = b.prev_out + sl * b.prev_q;
  if (b.mode == 3) {
    // pipelined blocks [x_0, r_1 .. r_k, a_1 .. a_k]: mode A (drafts known) after a mode-S
    // block or after a mode-A block that accepted all k drafts, else mode S (r_i = a_i);
    // x_0 = the newest emitted token, the drafts the k targets after it
    const int acc = __ldcg(b.prev_acc + sl);
    const bool a_mode = __ldcg(b.pipe_mode + sl) == 0 || acc == b.k + 1;
    __syncthreads();   // every thread has read the previous mode before thread 0 replaces it
    if (j == 0) {
      b.pipe_mode[sl] = a_mode ? 1 : 0;
      b.pipe_nverify[sl] = a_mode ? b.k : 0;
    }
    if (j >= b.q) return;
    int t;
    if (j == 0) {
      t = __ldcg(prev + acc - 1);
    } else if (j <= b.k && a_mode) {
      t = b.table ? __ldcg(b.table + (size_t)sl * b.table_stride + __ldcg(b.len + sl) + j) : __ldcg(prev + acc - 1 + j);
    } else {
      t = b.adaptive[(j - 1) % b.k];
    }
    b.tokens[sl * b.q + j] = t;
    return;
  }
  if (j >= b.q) return;
  int t;
  if (b.mode == 1) {
    t = (j == 0) ? __ldcg(prev + __ldcg(b.prev_acc + sl) - 1) : b.adaptive[j - 1];
  } else if (j == 0) {
    t = __ldcg(prev);
  } else {
    const int w = (j - 1) / b.k, i = (j - 1) % b.k + 1;
    if (b.table)
      t = __ldcg(b.table + ((size_t)w * b.table_batch + sl) * b.table_stride + __ldcg(b.len + sl) + i);
    else
      t = __ldcg(prev + i);
  }
  b.tokens[sl * b.q + j] = t;
}

cudaError_t launch_build_block(const BuildParams& b, cudaStream_t st, bool pdl) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(b.nb), dim3(32), st, pdl, attr);
  return cudaLaunchKernelEx(&cfg, build_block_kernel, b);
}

// ---- tree blocks: positions and attention masks, and the commit's KV compaction ----------
// Row j of a tree block: position len + depth(j) and the mask of the block rows it attends
// (its ancestors and itself).  One thread per row.
__global__ void tree_prep_kernel(const int* parent, const int* len, int nb, int q, int* pos, uint32_t* anc,
                                 uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  const int r = threadIdx.x;
  if (r >= nb * q) return;
  const int sl = r / q, j = r % q;
  const int* par = parent + sl * q;
  if (j == 0 && __ldcg(par) != -1) set_error(err, ERR_TREE);
  uint32_t m = 1u << j;
  int d = 0;
  for (int i = j; i > 0; ++d) {
    i = tree_parent(par, i, err);
    m |= 1u << i;
  }
  pos[r] = __ldcg(len + sl) + d;
  anc[r] = m;
}

cudaError_t launch_tree_prep(const int* parent, const int* len, int nb, int q, int* pos, uint32_t* anc,
                             uint32_t* err, cudaStream_t st, bool pdl) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(1), dim3(TREE_MAX_ROWS), st, pdl, attr);
  return cudaLaunchKernelEx(&cfg, tree_prep_kernel, parent, len, nb, q, pos, anc, err);
}

// Slot len0 + i receives the K and V rows of slot len0 + n_i (i = 1..m; n_i >= i, so no
// source is overwritten before it is read).  One CTA per (layer, head) and sequence, 16-byte
// chunks.
__global__ void tree_compact_kernel(const int* ws, int H, int hd, int cap, int batch, __nv_bfloat16* kc,
                                    __nv_bfloat16* vc) {
  pdl_wait();
  pdl_trigger();
  const int l = blockIdx.x / H, h = blockIdx.x % H, s = blockIdx.y;
  const int* w = ws + s * TREE_WS_STRIDE;
  const int len0 = __ldcg(w), m = __ldcg(w + 1);
  const int chunks = hd / 8;   // 16-byte chunks per row
  const size_t off = (((size_t)l * batch + s) * H + h) * cap * hd;
  for (int x = threadIdx.x; x < 2 * m * chunks; x += blockDim.x) {
    const int which = x / (m * chunks), rem = x % (m * chunks);
    const int i = 1 + rem / chunks, ch = rem % chunks;
    const int n = __ldcg(w + 2 + i);
    if (n == i || len0 + n >= cap) continue;
    __nv_bfloat16* base = (which ? vc : kc) + off;
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(base + (size_t)(len0 + n) * hd) + ch);
    __stcg(reinterpret_cast<uint4*>(base + (size_t)(len0 + i) * hd) + ch, v);
  }
}

cudaError_t launch_tree_compact(const int* ws, int nb, int L, int H, int hd, int cap, int batch,
                                __nv_bfloat16* k, __nv_bfloat16* v, cudaStream_t st, bool pdl) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(L * H, nb), dim3(64), st, pdl, attr);
  return cudaLaunchKernelEx(&cfg, tree_compact_kernel, ws, H, hd, cap, batch, k, v);
}

// ---- the bounded wait, run out on purpose (a test hook) ----------------------------------
// One CTA waits on an mbarrier that nothing arrives on, through the same bounded wait every
// kernel uses: after WAIT_LIMIT_NS it sets ERR_TIMEOUT and returns; nothing faults.
__global__ void wait_timeout_kernel(uint32_t* err) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  mbar_wait_bounded(&bar, 0, &abort_flag, err);
}

cudaError_t launch_wait_timeout(uint32_t* err, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(32);
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, wait_timeout_kernel, err);
}

// ---- explicit commit / rollback, and prefill commit --------------------------------------
__global__ void commit_kernel(int* len, const int* new_len, int nb, int cap, uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  const int s = threadIdx.x;
  if (s >= nb) return;
  int v = __ldcg(new_len + s);
  if (v < 0 || v > cap) {
    set_error(err, ERR_CAPACITY);
    v = v < 0 ? 0 : cap;
  }
  len[s] = v;
}

cudaError_t launch_commit(int* len, const int* new_len, int nb, int cap, uint32_t* err, cudaStream_t st,
                          bool pdl) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(1), dim3(64), st, pdl, attr);
  return cudaLaunchKernelEx(&cfg, commit_kernel, len, new_len, nb, cap, err);
}

__global__ void add_len_kernel(int* len, int seq, int n, int cap, uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  const int v = __ldcg(len + seq) + n;
  if (v > cap) set_error(err, ERR_CAPACITY);
  len[seq] = v > cap ? cap : v;
}

cudaError_t launch_add_len(int* len, int seq, int n, int cap, uint32_t* err, cudaStream_t st, bool pdl) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(1), dim3(1), st, pdl, attr);
  return cudaLaunchKernelEx(&cfg, add_len_kernel, len, seq, n, cap, err);
}

__global__ void exp_kernel(const float* in, float* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = exp_sd(in[i]);
}

cudaError_t accept_prepare() {
  cudaError_t e = cudaFuncSetAttribute(accept_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NucSmem));
  if (e == cudaSuccess) e = prefer_shared(accept_kernel<true>);
  if (e == cudaSuccess) e = prefer_shared(accept_kernel<false>);
  if (e == cudaSuccess) e = prefer_shared(rmsnorm_kernel);
  if (e == cudaSuccess) e = prefer_shared(split_kernel);
  if (e == cudaSuccess) e = prefer_shared(build_block_kernel);
  if (e == cudaSuccess) e = prefer_shared(tree_prep_kernel);
  if (e == cudaSuccess) e = prefer_shared(tree_compact_kernel);
  if (e == cudaSuccess) e = prefer_shared(commit_kernel);
  if (e == cudaSuccess) e = prefer_shared(add_len_kernel);
  return e;
}

cudaError_t launch_exp(const float* in, float* out, int n, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((n + 255) / 256);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, exp_kernel, in, out, n);
}

}  // namespace sdsat
