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
// steps on four times the work per thread.  us per call, 32016 logits a row, one CTA per row ->
// a cluster: 24 rows, top-p 0.95, T 0.2: 48.4 -> 22.5; with top-k 10: 34.5 -> 16.7; T 1 (row-wide
// searches): 101 -> 47; greedy 7.1 -> 5.0; 64 rows (512 CTAs, more than one wave): 48 -> 36, T 1:
// 101 -> 93, greedy 7.35 -> 7.4.  What is left is the chain of barriers, not bytes (3 MB).
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
constexpr int ACC_WORDS = 5;                      // 64-bit words of one warp's slot

struct AccSlots {
  unsigned long long w[2][ACC_WARPS * ACC_WORDS];   // this CTA's warps
  unsigned long long c[2][ACC_CS * ACC_WORDS];      // the cluster's CTAs, written by each of them
};

__device__ __forceinline__ void st_dsmem_u64(uint32_t addr, uint64_t v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
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
  // `before` the sum of word 0 over the warps that come before this one in id order
  template <int N, typename F>
  __device__ void reduce(uint64_t (&v)[N], uint64_t identity, F combine, uint64_t* before = nullptr) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long* mine = slots->w[ph & 1];
    unsigned long long* all = slots->c[ph & 1];
    ++ph;
    if (lane == 0)
#pragma unroll
      for (int n = 0; n < N; ++n) mine[w * N + n] = v[n];
    __syncthreads();
    if (w == 0) {
#pragma unroll
      for (int n = 0; n < N; ++n) {
        uint64_t t = lane < ACC_WARPS ? mine[lane * N + n] : identity;
#pragma unroll
        for (int o = ACC_WARPS / 2; o > 0; o >>= 1) t = combine(t, (uint64_t)__shfl_xor_sync(0xffffffffu, t, o));
        t = __shfl_sync(0xffffffffu, t, 0);
        if (lane < cs) st_dsmem_u64(mapa_shared(smem_u32(&all[rank * N + n]), lane), t);
      }
    }
    cluster_sync_all();
#pragma unroll
    for (int n = 0; n < N; ++n) {
      uint64_t t = lane < cs ? all[lane * N + n] : identity;
      if (n == 0 && before)   // earlier CTAs, then earlier warps of this one
        *before = warp_sum_u64((lane < rank ? t : 0) + (lane < w ? mine[lane * N] : 0));
#pragma unroll
      for (int o = ACC_CS / 2; o > 0; o >>= 1) t = combine(t, (uint64_t)__shfl_xor_sync(0xffffffffu, t, o));
      v[n] = __shfl_sync(0xffffffffu, t, 0);
    }
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
  // exclusive prefix over the row's threads, in id order, of v < 2^29
  __device__ uint64_t exscan(uint32_t v) {
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
// A thread keeps the weights W (uint32, <= 2^24) of its ids in registers.  Selections are
// predicates on (W, id); per-thread sums fit 32 bits, row sums 64.
struct Cut {
  uint32_t xk;  // top-k: candidates are W > xk, or W == xk and id <= idk
  int idk;
  uint32_t xp;  // top-p: kept candidates are W > xp, or W == xp and id <= idp
  int idp;
};
enum Pred : int {
  P_GE = 1,         // W >= x
  P_GT = 2,         // W > x
  P_EQ = 3,         // W == x
  P_CAND = 4,       // candidate
  P_CAND_GE = 5,    // candidate and W >= x
  P_CAND_GT = 6,    // candidate and W > x
  P_CAND_EQ = 7,    // candidate and W == x
  P_KEPT = 8,       // kept
};

template <int P>
__device__ __forceinline__ bool pred(uint32_t W, int id, const Cut& c, uint32_t x) {
  const bool cand = W > c.xk || (W == c.xk && id <= c.idk);
  switch (P) {
    case P_GE: return W >= x;
    case P_GT: return W > x;
    case P_EQ: return W == x;
    case P_CAND: return cand;
    case P_CAND_GE: return cand && W >= x;
    case P_CAND_GT: return cand && W > x;
    case P_CAND_EQ: return cand && W == x;
    default: return cand && (W > c.xp || (W == c.xp && id <= c.idp));
  }
}

// per-thread sum of W (COUNT: number of ids) over the owned ids selected by P (< 2^28)
template <int P, bool COUNT>
__device__ __forceinline__ uint32_t lsum(const uint32_t (&W)[ACC_EPT], int base, const Cut& c, uint32_t x) {
  uint32_t s = 0;
#pragma unroll
  for (int e = 0; e < ACC_EPT; ++e)
    if (pred<P>(W[e], base + e, c, x)) s += COUNT ? 1u : W[e];
  return s;
}
template <int P, bool COUNT>
__device__ __forceinline__ uint64_t row_sum(const uint32_t (&W)[ACC_EPT], int base, const Cut& c, uint32_t x, Row& rw) {
  return rw.sum(warp_total(lsum<P, COUNT>(W, base, c, x)));
}

// largest x in [0, 2^24] whose row total of lsum<P, COUNT>(x) is >= need (monotone in x); three
// thresholds a step: a step is one cluster barrier, whose latency outweighs the sums
template <int P, bool COUNT>
__device__ __forceinline__ uint32_t search_threshold(const uint32_t (&W)[ACC_EPT], int base, const Cut& c,
                                                     uint64_t need, Row& rw) {
  uint32_t lo = 0, hi = 1u << 24;
  while (lo < hi) {
    const uint32_t d = (hi - lo + 3) / 4;
    const uint32_t x[3] = {min(lo + d, hi), min(lo + 2 * d, hi), min(lo + 3 * d, hi)};
    uint64_t t[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) t[i] = warp_total(lsum<P, COUNT>(W, base, c, x[i]));
    rw.sum<3>(t);
    uint32_t nlo = lo, nhi = hi;
#pragma unroll
    for (int i = 2; i >= 0; --i) {
      if (t[i] >= need) nlo = max(nlo, x[i]);
      else nhi = x[i] - 1;   // (the last assignment is the lowest failing threshold's)
    }
    lo = nlo;
    hi = nhi;
  }
  return lo;
}

// the n-th (n >= 1) smallest id selected by P, or INT_MAX if there are fewer
template <int P>
__device__ __forceinline__ int nth_id(const uint32_t (&W)[ACC_EPT], int base, const Cut& c, uint32_t x,
                                      uint64_t n, Row& rw) {
  const uint32_t mine = lsum<P, true>(W, base, c, x);
  uint64_t k = rw.exscan(mine);
  uint32_t hit = 0;   // id + 1 in the one thread that holds it
  if (k < n && k + mine >= n) {
#pragma unroll
    for (int e = 0; e < ACC_EPT; ++e)
      if (pred<P>(W[e], base + e, c, x) && ++k == n) hit = base + e + 1;
  }
  const uint64_t id = rw.sum(warp_total(hit));
  return id ? (int)id - 1 : 0x7FFFFFFF;
}

// ---- the sampler on a compacted list ----------------------------------------------------
// The kept set is a prefix of the order (W desc, id asc), so it lies among the heaviest
// weights.  With a floor F such that the elements with W >= F provably contain it (top-k:
// at least k of them, or all non-zero weights; top-p alone: their mass reaches the top-p
// threshold), those elements go in ascending id order into rank 0's shared memory, and that
// CTA finishes the row.  Otherwise the row-wide searches over all ids run.
constexpr int NUC_LIST_MAX = 4096;
constexpr int NUC_FLOORS = 7;
// floor f: 2^24 (the largest weight), 2^22, 2^20, 2^18, 2^16 (ratio 2^-8), 2^8 (2^-16), then 1
// (every non-zero weight).  Weights of bucket b (nuc_bucket) are >= the floors f >= b.
__device__ __forceinline__ int nuc_bucket(uint32_t w) {
  if (w == 0) return NUC_FLOORS;
  const int e = 31 - __clz(w);
  return e >= 16 ? (25 - e) >> 1 : (e >= 8 ? 5 : 6);
}

struct NucList {
  unsigned long long key[NUC_LIST_MAX];      // nuc_key of the list's elements, ascending id
  unsigned long long sorted[NUC_LIST_MAX];   // the same in descending order
  unsigned long long kstar, sk;              // the kept prefix's last key and its mass
  int pick;
};

__device__ __forceinline__ uint64_t nuc_key(uint32_t w, int id) {   // larger: heavier, then lower id
  return ((uint64_t)w << 32) | (uint32_t)(0x7FFFFFFF - id);
}

// Steps 4-7 on the list (warp 0) when the candidates (top-k, k <= 32) or, without top-k, the
// kept prefix have at most 32 elements: up to 32 rounds of "largest key below the previous
// one" put them on the lanes in (W desc, id asc) order.  Returns -1 when this does not apply.
__device__ int list_small(const AcceptParams& p, const NucList& L, int n, uint64_t S_all, bool topk, uint64_t rnd) {
  const int lane = threadIdx.x & 31;
  if (topk && p.top_k > 32) return -1;
  uint64_t thr = 0;
  if (!topk) {
    const uint64_t prod = (uint64_t)p.p_fixed * S_all;
    thr = (prod >> 24) + ((prod & 0xFFFFFFull) ? 1 : 0);
  }
  const int rounds = topk ? min(p.top_k, n) : min(32, n);
  uint64_t prev = ~0ull, mine = 0, C = 0;
  int nc = 0;
  bool done = topk;
  for (int r = 0; r < rounds && !(nc > 0 && !topk && C >= thr); ++r) {
    uint64_t best = 0;
    for (int i = lane; i < n; i += 32) {
      const uint64_t k = L.key[i];
      if (k < prev && k > best) best = k;
    }
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(best >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(best >> 32) == hi ? (uint32_t)best : 0u);
    prev = ((uint64_t)hi << 32) | lo;
    if (lane == r) mine = prev;
    ++nc;
    C += hi;   // the round's weight
  }
  if (!topk) done = C >= thr;   // the kept prefix: the first nc elements reach the threshold
  if (!done) return -1;
  const uint32_t w = lane < nc ? (uint32_t)(mine >> 32) : 0u;
  const int id = 0x7FFFFFFF - (int)(uint32_t)mine;
  bool kept = lane < nc;
  if (topk) {
    // candidates = the nc lanes; kept = the shortest prefix whose mass reaches thr
    const uint64_t S = __reduce_add_sync(0xffffffffu, w);
    const uint64_t prod = (uint64_t)p.p_fixed * S;
    const uint64_t t = (prod >> 24) + ((prod & 0xFFFFFFull) ? 1 : 0);
    uint32_t incl = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    kept = kept && (lane == 0 || (uint64_t)(incl - w) < t);
  }
  const uint32_t kw = kept ? w : 0u;
  const uint64_t Sk = __reduce_add_sync(0xffffffffu, kw);
  const uint64_t tau = __umul64hi(rnd, Sk);
  // ascending-id cumulative weight of the kept elements up to and including this lane's
  uint64_t cum = 0;
  for (int j = 0; j < nc; ++j) {
    const uint32_t wj = __shfl_sync(0xffffffffu, kw, j);
    const int idj = __shfl_sync(0xffffffffu, id, j);
    if (idj <= id) cum += wj;
  }
  const uint32_t m = __ballot_sync(0xffffffffu, kept && cum > tau && cum - kw <= tau);
  return __shfl_sync(0xffffffffu, id, __ffs(m) - 1);
}

// L.sorted = the n2 (a power of two >= 32, the list's n keys and zeros) keys in descending
// order: bitonic; distances below 32 stay in the warp (element i is on lane i & 31), so 1024
// keys take 15 block barriers and not 55.
__device__ void list_sort(NucList& L, int n, int n2) {
  constexpr int PER = NUC_LIST_MAX / ACC_THREADS;
  auto in_warp = [&](uint64_t x, int i, int k, int j) {   // distances j .. 1 of the merge of size k
    for (; j > 0; j >>= 1) {
      const uint64_t y = __shfl_xor_sync(0xffffffffu, x, j);
      // descending blocks where bit k of i is clear: the lower element keeps the larger key
      const bool keep_max = ((i & k) == 0) == ((i & j) == 0);
      x = keep_max ? max(x, y) : min(x, y);
    }
    return x;
  };
#pragma unroll 1
  for (int r = 0; r < PER; ++r) {
    const int i = threadIdx.x + r * ACC_THREADS;
    if (i >= n2) break;   // (whole warps)
    uint64_t x = i < n ? L.key[i] : 0ull;   // padding sorts last (every list W >= 1)
    for (int k = 2; k <= 32; k <<= 1) x = in_warp(x, i, k, k >> 1);
    L.sorted[i] = x;
  }
  for (int k = 64; k <= n2; k <<= 1) {
    for (int j = k >> 1; j >= 32; j >>= 1) {
      __syncthreads();
      for (int i = threadIdx.x; i < n2; i += ACC_THREADS) {
        const int l = i ^ j;
        if (l > i) {
          const uint64_t a = L.sorted[i], b = L.sorted[l];
          if (((i & k) == 0) == (a < b)) {
            L.sorted[i] = b;
            L.sorted[l] = a;
          }
        }
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int r = 0; r < PER; ++r) {
      const int i = threadIdx.x + r * ACC_THREADS;
      if (i >= n2) break;
      L.sorted[i] = in_warp(L.sorted[i], i, k, 16);
    }
  }
  __syncthreads();
}

// Steps 4-7 on the list with the whole CTA.  The list holds the first n elements of the order
// (W desc, id asc), in ascending id.  Its keys are sorted once, so the candidates (the first
// min(k, n)), their mass, the kept prefix (the shortest one whose mass reaches
// ceil(P S / 2^24)) and its mass are prefix sums of the sorted weights.  The pick then scans
// the list itself in ascending id with "kept" = key >= the kept prefix's last key.
__device__ int list_sorted_select(const AcceptParams& p, NucList& L, int n, uint64_t S_all, uint64_t rnd,
                                  uint64_t* red) {
  int n2 = 32;
  while (n2 < n) n2 <<= 1;
  list_sort(L, n, n2);
  // candidates and the kept prefix: thread t holds `per` consecutive sorted elements
  const int per = (n + ACC_THREADS - 1) / ACC_THREADS, i0 = threadIdx.x * per, i1 = min(i0 + per, n);
  const bool topk = p.top_k > 0 && p.top_k < p.V;
  const int nc = topk ? min(p.top_k, n) : n;
  uint64_t wsum = 0;
  for (int i = i0; i < min(i1, nc); ++i) wsum += L.sorted[i] >> 32;
  const uint64_t S = topk ? block_sum_u64(wsum, red) : S_all;
  const uint64_t prod = (uint64_t)p.p_fixed * S;
  const uint64_t thr = (prod >> 24) + ((prod & 0xFFFFFFull) ? 1 : 0);
  const uint64_t before = block_exscan_u64(wsum, red);
  // the first sorted index whose inclusive mass reaches thr (index 0 when thr = 0); the list
  // provably holds it
  if (thr == 0 ? threadIdx.x == 0 : (before < thr && before + wsum >= thr)) {
    uint64_t cum = before;
    for (int i = i0; i < i1; ++i) {
      cum += L.sorted[i] >> 32;
      if (cum >= thr) {
        L.kstar = L.sorted[i];
        L.sk = cum;
        break;
      }
    }
  }
  __syncthreads();
  const uint64_t kstar = L.kstar, Sk = L.sk;
  const uint64_t tau = __umul64hi(rnd, Sk);
  // 7. the first kept id (ascending) whose inclusive cumulative weight exceeds tau
  uint64_t mine = 0;
  for (int i = i0; i < i1; ++i)
    if (L.key[i] >= kstar) mine += L.key[i] >> 32;
  const uint64_t below = block_exscan_u64(mine, red);
  if (below <= tau && below + mine > tau) {
    uint64_t cum = below;
    for (int i = i0; i < i1; ++i)
      if (L.key[i] >= kstar) {
        cum += L.key[i] >> 32;
        if (cum > tau) {
          L.pick = 0x7FFFFFFF - (int)(uint32_t)L.key[i];
          break;
        }
      }
  }
  __syncthreads();
  return L.pick;
}

// The row's sampled id (valid in rank 0).  Every CTA of the cluster passes the same barriers:
// every branch is taken on values that the whole row shares.
__device__ __forceinline__ int row_nucleus(const AcceptParams& p, const float* row, int position, int seq,
                                           uint64_t* red, Row& rw, NucList& L) {
  const int V = p.V;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int base = rw.rank * ACC_SPAN + threadIdx.x * ACC_EPT;
  uint32_t W[ACC_EPT];
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
    float mx = -INFINITY;
#pragma unroll
    for (int e = 0; e < ACC_EPT; ++e) {
      if (l[e] != l[e]) {
        nan = true;
        l[e] = -INFINITY;
      }
      mx = fmaxf(mx, l[e]);
    }
    if (nan) set_error(p.err, ERR_NAN_LOGITS);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    // (ordered as in arg_key, with id bits that do not matter)
    const uint32_t ord = (uint32_t)(rw.largest(arg_key(mx, 0)) >> 32);
    mx = __uint_as_float((ord & 0x80000000u) ? ord & 0x7FFFFFFFu : ~ord);
    // 2-3. W_i = floor(exp((l_i - max) / T) * 2^24)
#pragma unroll
    for (int e = 0; e < ACC_EPT; ++e) W[e] = fixed24(exp_sd(__fdiv_rn(__fsub_rn(l[e], mx), p.temperature)));
  }
  // 6. the 64-bit draw keyed by (produced position, sequence)
  uint32_t ctr[4] = {(uint32_t)position, (uint32_t)seq, 0u, 0u};
  philox4x32_10(ctr, (uint32_t)(p.seed & 0xFFFFFFFFull), (uint32_t)(p.seed >> 32));
  const uint64_t rnd = ((uint64_t)ctr[0] << 32) | ctr[1];

  // ---- the list path: counts (and, without top-k, masses) of the weights above each floor
  const bool topk = p.top_k > 0 && p.top_k < V;
  {
    // per-thread counts (<= 8) of the floors in 16-bit fields: floors 0-3 and 4-6
    uint64_t c03 = 0, c46 = 0;
    uint32_t m4 = 0, m5 = 0, m6 = 0;   // masses >= floors 4, 5, 6 (< 2^28)
#pragma unroll
    for (int e = 0; e < ACC_EPT; ++e) {
      const int b = nuc_bucket(W[e]);
#pragma unroll
      for (int f = 0; f < 4; ++f) c03 += b <= f ? 1ull << (16 * f) : 0ull;
#pragma unroll
      for (int f = 4; f < NUC_FLOORS; ++f) c46 += b <= f ? 1ull << (16 * (f - 4)) : 0ull;
      m4 += b <= 4 ? W[e] : 0u;
      m5 += b <= 5 ? W[e] : 0u;
      m6 += W[e];
    }
    // (warp totals of a field <= 256, row totals <= 32768)
    auto add16 = [&](uint64_t v) {
      return ((uint64_t)__reduce_add_sync(0xffffffffu, (uint32_t)(v >> 32)) << 32) |
             __reduce_add_sync(0xffffffffu, (uint32_t)v);
    };
    uint64_t t[ACC_WORDS] = {add16(c03), add16(c46), warp_total(m4), warp_total(m5), warp_total(m6)};
    const int buf = rw.ph & 1;
    rw.sum<ACC_WORDS>(t);
    const unsigned long long *warps = rw.slots->w[buf], *ctas = rw.slots->c[buf];
    int N[NUC_FLOORS];
#pragma unroll
    for (int f = 0; f < NUC_FLOORS; ++f) N[f] = (int)(((f < 4 ? t[0] : t[1]) >> (16 * (f & 3))) & 0xFFFF);
    const uint64_t Sf[3] = {t[2], t[3], t[4]};
    const uint64_t S_all = Sf[2];
    uint64_t thr_all = 0;
    if (!topk) {
      const uint64_t prod = (uint64_t)p.p_fixed * S_all;
      thr_all = (prod >> 24) + ((prod & 0xFFFFFFull) ? 1 : 0);
    }
    // the highest floor whose elements provably hold the candidates (top-k) or the kept prefix
    int f = -1;
#pragma unroll
    for (int i = 0; i < NUC_FLOORS; ++i) {
      const bool holds = topk ? (N[i] >= p.top_k || N[i] == N[6]) : (i >= 4 && Sf[i - 4] >= thr_all);
      if (f < 0 && N[i] <= NUC_LIST_MAX && holds) f = i;
    }
    if (N[6] == 0) return 0;   // every weight 0 (all-NaN row): the lowest candidate, id 0
    if (f >= 0) {
      int nf = 0;
#pragma unroll
      for (int i = 0; i < NUC_FLOORS; ++i) nf = i == f ? N[i] : nf;
      // this thread's place in the list: the CTAs and warps before (from the totals just
      // summed), then the lanes before
      const int word = f >> 2, sh = 16 * (f & 3);
      uint64_t at = 0;
      if (lane < rw.rank) at += (ctas[lane * ACC_WORDS + word] >> sh) & 0xFFFF;
      if (lane < w) at += (warps[lane * ACC_WORDS + word] >> sh) & 0xFFFF;
      at = warp_sum_u64(at);
      uint32_t mine = 0;
#pragma unroll
      for (int e = 0; e < ACC_EPT; ++e) mine += nuc_bucket(W[e]) <= f;
      uint32_t x = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      uint32_t dst = mapa_shared(smem_u32(&L.key[0]), 0) + ((uint32_t)at + x - mine) * 8;
#pragma unroll
      for (int e = 0; e < ACC_EPT; ++e)
        if (nuc_bucket(W[e]) <= f) {
          st_dsmem_u64(dst, nuc_key(W[e], base + e));
          dst += 8;
        }
      cluster_sync_all();   // the list is complete
      if (rw.rank) return 0;
      // a kept set (or top-k) of at most 32 on the lanes of one warp when that is cheap: a
      // small top-k, or a short list; otherwise, or when it does not apply, the sorted list
      if ((topk && p.top_k <= 32) || nf <= 64) {
        if (w == 0) {
          const int pick = list_small(p, L, nf, S_all, topk, rnd);
          if (lane == 0) L.pick = pick;
        }
        __syncthreads();
        const int pick = L.pick;
        if (pick >= 0) return pick;
        __syncthreads();   // L.pick is written again
      }
      return list_sorted_select(p, L, nf, S_all, rnd, red);
    }
  }

  // ---- the row-wide path over all ids
  Cut c;
  c.xk = 0;
  c.idk = 0x7FFFFFFF;
  c.xp = 0;
  c.idp = 0x7FFFFFFF;
  // 4. top-k candidates
  if (topk) {
    c.xk = search_threshold<P_GE, true>(W, base, c, (uint64_t)p.top_k, rw);
    const uint64_t above = row_sum<P_GT, true>(W, base, c, c.xk, rw);
    c.idk = nth_id<P_EQ>(W, base, c, c.xk, (uint64_t)p.top_k - above, rw);
  }
  // 5. top-p over the candidates: thr = ceil(P * S / 2^24), P <= 2^24, S < 2^40
  const uint64_t S = row_sum<P_CAND, false>(W, base, c, 0, rw);
  const uint64_t prod = (uint64_t)p.p_fixed * S;
  const uint64_t thr = (prod >> 24) + ((prod & 0xFFFFFFull) ? 1 : 0);
  c.xp = search_threshold<P_CAND_GE, false>(W, base, c, thr, rw);
  uint64_t ab[2] = {warp_total(lsum<P_CAND_GT, false>(W, base, c, c.xp)),
                    warp_total(lsum<P_CAND_GT, true>(W, base, c, c.xp))};
  rw.sum<2>(ab);
  uint64_t ties = thr > ab[0] ? (thr - ab[0] + c.xp - 1) / c.xp : 0;
  if (ab[1] == 0 && ties == 0) ties = 1;
  c.idp = ties == 0 ? -1 : nth_id<P_CAND_EQ>(W, base, c, c.xp, ties, rw);
  // 7. the first kept id (ascending) whose inclusive cumulative weight exceeds tau
  const uint32_t mine = lsum<P_KEPT, false>(W, base, c, 0);
  const uint64_t Sk = rw.sum(warp_total(mine));
  const uint64_t tau = __umul64hi(rnd, Sk);
  const uint64_t before = rw.exscan(mine);
  uint32_t hit = 0;   // id + 1 in the one thread that holds it
  if (before <= tau && before + mine > tau) {
    uint64_t cum = before;
#pragma unroll
    for (int e = 0; e < ACC_EPT; ++e) {
      if (pred<P_KEPT>(W[e], base + e, c, 0)) {
        cum += W[e];
        if (cum > tau && !hit) hit = base + e + 1;
      }
    }
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

__global__ void __launch_bounds__(ACC_THREADS) accept_kernel(const AcceptParams p) {
  extern __shared__ __align__(16) uint8_t acc_smem[];   // NucList (nucleus only)
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
  if (p.temperature <= 0.f) {
    t = row_argmax(row, p.V, p.err, rw);
  } else {
    // the produced token's position: one past the row's own (len + j, or len + depth(j))
    const int position = __ldcg(p.len + s) + (p.parent ? tree_depth(p.parent + sl * p.q, j, nullptr) : j) + 1;
    t = row_nucleus(p, row, position, s, red, rw, *reinterpret_cast<NucList*>(acc_smem));
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
  cfg.dynamicSmemBytes = p.temperature > 0.f ? sizeof(NucList) : 0;
  attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
  attr[cfg.numAttrs].val.clusterDim.x = p.cs;
  attr[cfg.numAttrs].val.clusterDim.y = 1;
  attr[cfg.numAttrs].val.clusterDim.z = 1;
  ++cfg.numAttrs;
  return cudaLaunchKernelEx(&cfg, accept_kernel, p);
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
  cudaError_t e = cudaFuncSetAttribute(accept_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NucList));
  if (e == cudaSuccess) e = prefer_shared(accept_kernel);
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
