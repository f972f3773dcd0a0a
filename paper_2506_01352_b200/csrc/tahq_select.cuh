// Sec. 3.2 and 3.4 between scoring and quantise + pack (sm_100a): the exact top-k_hi selection of every ranking group,
// the bit map and the running count of higher-width tiles; the scores of allocation tiles wider than the quantisation
// tile.
#pragma once

#include <cooperative_groups.h>

#include "tahq_lanes.cuh"

namespace tahq {

namespace cg = cooperative_groups;

constexpr int kSelThreads = 512;       // threads per CTA of select_kernel: two CTAs fit on an SM
constexpr int kClKeys = 4096;          // candidate keys that are ranked in shared memory
constexpr int kClMaxCtas = 16;
constexpr int kHeld = 8;               // scores a thread keeps in registers
constexpr int kCoarse = 64, kFine = kBins / kCoarse;

// ------------------------------------------------------------------------------------------
// Eq. 1-2 over allocation tiles wider than the quantisation tile (Sec. 3.2, A = m * G, up to 8192
// channels): one warp per allocation tile, exact arithmetic in the summation order of the pairwise tree
// -- eight consecutive elements inside a lane, then neighbouring lanes (a lane without a neighbour
// waits for the next level), then the sums of successive rounds of 256 elements in the same way.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_tree(float x, uint32_t n, int lane) {   // n <= 32 values, one per lane
#pragma unroll
  for (int h = 1; h < 32; h *= 2) {
    const float y = __shfl_down_sync(kFull, x, h);
    if ((lane & (2 * h - 1)) == 0 && (uint32_t)(lane + h) < n) x = x + y;
  }
  return __shfl_sync(kFull, x, 0);
}
// U rounds of 256 elements go at a time: their loads and the steps of their trees are in flight together (one after the
// other, the 16 rounds of a 2048-channel tile were a chain of load and shuffle latencies: 4096 x 2048 bf16 13.7 -> 10.8 us with two logarithms to an instruction).
template <bool BF16, int U, class F>
__device__ __forceinline__ float alloc_tree(const uint8_t *base, uint32_t n_oct, int lane, F &&f) {
  const uint32_t rounds = (n_oct + 31) / 32;
  float rs = 0.0f;   // lane r keeps the sum of round r
  for (uint32_t r = 0; r < rounds; r += U) {
    float v[U][8], x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t o = (r + u) * 32 + lane;
      if (o < n_oct) {
        if constexpr (BF16) {
          const uint4 w = __ldg(reinterpret_cast<const uint4 *>(base) + o);
          const uint32_t t[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            v[u][2 * j] = fabsf(__uint_as_float(t[j] << 16));
            v[u][2 * j + 1] = fabsf(__uint_as_float(t[j] & 0xffff0000u));
          }
        } else {
          const float4 p = __ldg(reinterpret_cast<const float4 *>(base) + 2 * o);
          const float4 q = __ldg(reinterpret_cast<const float4 *>(base) + 2 * o + 1);
          v[u][0] = fabsf(p.x); v[u][1] = fabsf(p.y); v[u][2] = fabsf(p.z); v[u][3] = fabsf(p.w);
          v[u][4] = fabsf(q.x); v[u][5] = fabsf(q.y); v[u][6] = fabsf(q.z); v[u][7] = fabsf(q.w);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) v[u][k] = 0.0f;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if ((r + u) * 32 + lane < n_oct) {
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
          const float2 t = f(f2(v[u][k], v[u][k + 1]));
          v[u][k] = t.x;
          v[u][k + 1] = t.y;
        }
      }
      x[u] = tree8(v[u]);
    }
    if ((r + U) * 32 <= n_oct) {   // whole rounds: the tree as xor shuffles (addition commutes: every lane ends with its sum)
#pragma unroll
      for (int h = 1; h < 32; h *= 2)
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = x[u] + __shfl_xor_sync(kFull, x[u], h);
#pragma unroll
      for (int u = 0; u < U; ++u) rs = (uint32_t)lane == r + u ? x[u] : rs;
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t o = (r + u) * 32, n = o < n_oct ? (n_oct - o < 32u ? n_oct - o : 32u) : 0u;
        const float t = warp_tree(x[u], n, lane);
        rs = (uint32_t)lane == r + u ? t : rs;
      }
    }
  }
  return warp_tree(rs, rounds, lane);
}
template <bool BF16, int U>
__global__ void __launch_bounds__(kThreads) alloc_score_kernel(const Args a) {
  const int lane = threadIdx.x & 31;
  const uint64_t warp = ((uint64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * kThreads) >> 5;
  const uint32_t A = a.alloc_m * a.tile, n_oct = A / 8;
  const uint64_t n_alloc = a.n_tiles / a.alloc_m;
  TraceScope trace(a.trace, 1);
  grid_dependency_wait();
  trace.started();
  clear_bitmap(a);
  for (uint64_t t = warp; t < n_alloc; t += n_warps) {
    const uint8_t *base = a.in + t * (uint64_t)A * (BF16 ? 2 : 4);
    const float L1 = alloc_tree<BF16, U>(base, n_oct, lane, [](float2 m) { return m; });
    const float inv = __fdiv_rn(1.0f, L1 + a.eps_l1);
    const float S = alloc_tree<BF16, U>(base, n_oct, lane, [&](float2 m) {   // (scalar products: they are added to)
      const float2 p = f2(m.x * inv, m.y * inv), l = lg2_fma2(add2(p, f2(a.eps_log)));
      return f2(p.x * l.x, p.y * l.y);
    });
    if (lane == 0) a.scores[t] = ranked_score(0.0f - S);
  }
}

// ------------------------------------------------------------------------------------------
// Sec. 3.2: exact top-k_hi per ranking group.  One thread-block cluster of up to 16 CTAs per group, a slice of the
// group's scores to each CTA; what the CTAs have to tell each other -- histogram columns, candidate keys, counts --
// travels through distributed shared memory between two cluster barriers.
//
//   1  every CTA bins its scores, fine (4096 bins) and coarse (64)
//   2  after the first barrier every CTA reads the cluster's coarse counts, finds the coarse bin of the k_hi-th ranked
//      tile, reads the 64 fine counts inside it and has the threshold bin B
//   3  tiles well above / below bin B are decided: the bits of those above are the first version of the slice's
//      words.  The few inside the band are listed and get their exact score (8 lanes per tile of 64, straight from the
//      tensor, all in flight together); their ranking keys are stored into every CTA's copy of the key list (slots
//      handed out by the first CTA's counter)
//   4  after the second barrier every CTA ranks its copy of the list for itself, counts the band tiles of earlier
//      slices that made it and sets the bits of its own
//   5  the words of the slice leave as words of the bit map with their running counts.  A ranking group may start
//      anywhere in a word and a ranked tile may stand for several quantisation tiles (A > G): words that two slices
//      share are put together by atomicOr on zeroed memory.
//
// If there are more candidates than the list holds (thousands of near-equal scores) the cluster runs a radix selection
// over the slices instead (selection_by_radix).
// ------------------------------------------------------------------------------------------

// r-th largest (1-based) key of a sequence, radix select with 8 bits a pass.  get(i, key) returns
// false for entries that do not take part.
template <class Get>
__device__ __forceinline__ unsigned long long radix_select(uint64_t count, uint32_t r, Get &&get) {
  __shared__ uint32_t h[256];
  __shared__ uint32_t pick[2];
  // bits on which the keys differ: a pass over a digit that is the same in every key is skipped
  __shared__ unsigned long long s_or[kSelThreads / 32], s_and[kSelThreads / 32];
  unsigned long long orv = 0, andv = ~0ull;
  for (uint64_t i = threadIdx.x; i < count; i += blockDim.x) {
    unsigned long long key;
    if (get(i, key)) { orv |= key; andv &= key; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    orv |= __shfl_xor_sync(kFull, orv, o);
    andv &= __shfl_xor_sync(kFull, andv, o);
  }
  if ((threadIdx.x & 31) == 0) { s_or[threadIdx.x >> 5] = orv; s_and[threadIdx.x >> 5] = andv; }
  __syncthreads();
  for (int w = 0; w < (int)(blockDim.x / 32); ++w) { orv |= s_or[w]; andv &= s_and[w]; }
  const unsigned long long varying = orv ^ andv;
  unsigned long long prefix = 0, mask = 0;
  for (int shift = 56; shift >= 0; shift -= 8) {
    if (((varying >> shift) & 0xffull) == 0) {   // every key has the same digit here
      prefix |= orv & (0xffull << shift);
      mask |= 0xffull << shift;
      continue;
    }
    if (threadIdx.x < 256) h[threadIdx.x] = 0;
    __syncthreads();   // the digit counts are clear before anyone adds to them
    for (uint64_t i = threadIdx.x; i < count; i += blockDim.x) {
      unsigned long long key;
      if (get(i, key) && (key & mask) == prefix) atomicAdd(&h[(unsigned)(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      // lane L owns digits 255-8L .. 248-8L (descending); find where the running count reaches r
      const int top = 255 - 8 * (int)threadIdx.x;
      uint32_t mine = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) mine += h[top - j];
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o *= 2) {
        const uint32_t v = __shfl_up_sync(kFull, incl, o);
        if ((int)threadIdx.x >= o) incl += v;
      }
      uint32_t above = incl - mine;
      if (above < r && incl >= r) {
        for (int j = 0; j < 8; ++j) {
          const uint32_t c = h[top - j];
          if (above + c >= r) { pick[0] = (uint32_t)(top - j); pick[1] = r - above; break; }
          above += c;
        }
      }
    }
    __syncthreads();
    prefix |= (unsigned long long)pick[0] << shift;
    mask |= 0xffull << shift;
    r = pick[1];
    __syncthreads();
  }
  return prefix;
}

// exact score of tile `tp` by the NOCT lanes that share it (all 32 lanes of the warp call this)
__device__ __forceinline__ float exact_score_any(const uint8_t *tp, uint32_t noct, bool bf16, uint32_t sub, float eps_l1,
                                                 float eps_log) {
  if (bf16)
    return noct == 1   ? exact_score_coop<1, true>(tp, sub, eps_l1, eps_log)
           : noct == 2 ? exact_score_coop<2, true>(tp, sub, eps_l1, eps_log)
           : noct == 4 ? exact_score_coop<4, true>(tp, sub, eps_l1, eps_log)
           : noct == 8 ? exact_score_coop<8, true>(tp, sub, eps_l1, eps_log)
                       : exact_score_coop<16, true>(tp, sub, eps_l1, eps_log);
  return noct == 1   ? exact_score_coop<1, false>(tp, sub, eps_l1, eps_log)
         : noct == 2 ? exact_score_coop<2, false>(tp, sub, eps_l1, eps_log)
         : noct == 4 ? exact_score_coop<4, false>(tp, sub, eps_l1, eps_log)
         : noct == 8 ? exact_score_coop<8, false>(tp, sub, eps_l1, eps_log)
                     : exact_score_coop<16, false>(tp, sub, eps_l1, eps_log);
}

// r-th largest of n distinct keys in shared memory (n <= kClKeys), the same value returned to every thread: they go
// into kSelThreads buckets by score first and only the bucket that holds rank r is counted; thousands of equal scores
// fall through to the radix selection.
static __device__ __noinline__ unsigned long long rank_keys_shared(unsigned long long *s_keys, uint32_t n, uint32_t r,
                                                                      unsigned long long *s_few /* kSelThreads */) {
  __shared__ unsigned long long s_ans;
  __shared__ uint32_t s_cnt[kSelThreads];
  __shared__ uint32_t s_sub[kSelThreads];
  __shared__ uint32_t s_wsum[kSelThreads / 32];
  __shared__ uint32_t s_lo, s_hi, s_nsub, s_pick[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) { s_ans = ~0ull; s_lo = 0xffffffffu; s_hi = 0; s_nsub = 0; s_pick[0] = 0; s_pick[1] = 0; }
  s_cnt[threadIdx.x] = 0;
  __syncthreads();
  {   // the scores, mapped to unsigned integers of the same order: smallest and largest
    uint32_t mn = 0xffffffffu, mx = 0;
    for (uint32_t i = threadIdx.x; i < n; i += kSelThreads) {
      const uint32_t m = (uint32_t)(s_keys[i] >> 32);
      mn = m < mn ? m : mn;
      mx = m > mx ? m : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint32_t v = __shfl_xor_sync(kFull, mn, o), w = __shfl_xor_sync(kFull, mx, o);
      mn = v < mn ? v : mn;
      mx = w > mx ? w : mx;
    }
    if (lane == 0) { atomicMin(&s_lo, mn); atomicMax(&s_hi, mx); }
  }
  __syncthreads();
  const uint32_t lo_m = s_lo, span = s_hi - s_lo;
  // (a multiplication in binary32 instead of a 64-bit division per key: rounding keeps the map non-decreasing,
  // which is all the buckets need)
  const float per_bucket = span ? (float)(kSelThreads - 1) / (float)span : 0.0f;
  auto bucket_of = [&](unsigned long long key) {
    const uint32_t b = (uint32_t)((float)((uint32_t)(key >> 32) - lo_m) * per_bucket);
    return b < (uint32_t)kSelThreads - 1u ? b : (uint32_t)kSelThreads - 1u;
  };
  for (uint32_t i = threadIdx.x; i < n; i += kSelThreads) atomicAdd(&s_cnt[bucket_of(s_keys[i])], 1u);
  __syncthreads();
  {   // keys in the buckets above this thread's bucket (one bucket per thread)
    const uint32_t c = s_cnt[threadIdx.x];
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const uint32_t v = __shfl_down_sync(kFull, incl, o);
      if (lane + o < 32) incl += v;
    }
    if (lane == 0) s_wsum[warp] = incl;
    __syncthreads();
    uint32_t above = incl - c;
    for (int w = warp + 1; w < kSelThreads / 32; ++w) above += s_wsum[w];
    if (above < r && above + c >= r) { s_pick[0] = threadIdx.x; s_pick[1] = r - above; }
  }
  __syncthreads();
  const uint32_t bsel = s_pick[0], rsel = s_pick[1];
  if (rsel != 0 && s_cnt[bsel] <= (uint32_t)kSelThreads) {
    for (uint32_t i = threadIdx.x; i < n; i += kSelThreads)
      if (bucket_of(s_keys[i]) == bsel) s_sub[atomicAdd(&s_nsub, 1u)] = i;
    __syncthreads();
    const uint32_t ns = s_nsub;
    const unsigned long long mine = threadIdx.x < ns ? s_keys[s_sub[threadIdx.x]] : 0ull;
    if (threadIdx.x < ns) s_few[threadIdx.x] = mine;
    __syncthreads();
    if (threadIdx.x < ns) {
      uint32_t larger = 0;
      for (uint32_t i = 0; i < ns; ++i) larger += s_few[i] > mine ? 1u : 0u;
      if (larger == rsel - 1) s_ans = mine;
    }
    __syncthreads();
    return s_ans;
  }
  // thousands of equal scores: digit by digit
  return radix_select(n, r, [&](uint64_t i, unsigned long long &key) { key = s_keys[i]; return true; });
}

struct SelShared {
  uint32_t part[kClMaxCtas];     // tiles above the band in each CTA's slice
  uint32_t tot[kClMaxCtas];      // (radix) set bits in each CTA's words
  uint32_t n_keys;               // (first CTA) list slots handed out so far
  uint32_t n_total;              // candidates of the whole cluster (every CTA is told)
  uint32_t overflow;             // a slice has so many that the list is not made
  uint32_t digit_pick[3];        // radix selection: chosen digit, remaining rank, keys with that digit
  uint32_t key_bits[4];          // (radix) bits that some key of this CTA has, bits that all have; low and high words
  uint32_t red[32];              // sums of the warps
  uint32_t n_cand, n_above;      // the slice's candidates, its tiles above the band
};

// The CTA's dynamic shared memory.
struct SelMem {
  unsigned long long *keys;      // [kClKeys + kSelThreads] the cluster's candidate keys
  uint32_t *hist;                // [kBins]; later the words' running counts
  uint32_t *cand;                // [kClKeys] band tiles of the slice
  uint32_t *words;               // [kWordsShared]
  __device__ __forceinline__ SelMem() {
    extern __shared__ __align__(16) uint8_t smem_sel[];
    keys = reinterpret_cast<unsigned long long *>(smem_sel);
    hist = reinterpret_cast<uint32_t *>(keys + kClKeys + kSelThreads);
    cand = hist + kBins;
    words = cand + kClKeys;
  }
};

// A score on the axis of the bins, in steps, 16 to a bin (non-decreasing in the score; not yet cut to whole steps).  Scores
// lie in [0, log2 A]; three quarters of the bins are given to the top two units, where most tiles and the threshold are:
// with bins of one width a threshold in the dense part had 2.6 times as many candidates.
struct StepMap { float lo, hi, off; };   // max(s * lo, s * hi - off)
// Scores below zero (p + varsigma above one: tiles with a single large element) are in the first bin.
__device__ __forceinline__ float score_pos(float s, const StepMap &m) { return fmaxf(s * m.lo, __fmaf_rn(s, m.hi, -m.off)); }
__device__ __forceinline__ int score_step(float s, const StepMap &m) {
  return (int)fminf(fmaxf(score_pos(s, m), 0.0f), (float)(16 * kBins - 1));
}
// Screening scores differ from exact ones by less than 1e-4 (see tile_score_screen), 2.5 steps at most.  With k_hi-th largest
// screening score in bin B, a tile whose screening score lies more than twice that outside bin B is certainly inside or
// outside the top k_hi; six steps also cover the cut to whole steps.
constexpr int kScreenBand = 6;

// Exact scores of n listed tiles, `NOCT` lanes to a tile, by the warps of `threads` threads that call this together, as keys
// (at the tile's place in the list; i0: the slice's first tile) or as scores (at the tile's place in the slice).  Two tiles of a
// lane are on their way at a time, in a function of its own: one at a time, 131072 equal tiles took 152 us to select from
// instead of 138; with four, or without the call, select_kernel no longer fits its registers, which every encode pays for.
template <int NOCT, bool BF16>
__device__ __forceinline__ void exact_listed(const uint8_t *tiles, const uint32_t *list, uint32_t n, uint32_t thread, uint32_t threads,
                                             float eps_l1, float eps_log, uint32_t i0, unsigned long long *keys, float *scores) {
  constexpr uint32_t TB = NOCT * 8 * (BF16 ? 2 : 4);
  constexpr int U = 2;
  const uint32_t sub = thread % NOCT, per = threads / NOCT;
  for (uint32_t j0 = thread / NOCT; j0 - thread / NOCT < n; j0 += U * per) {
    float v[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u) load_abs_oct_global<BF16>(tiles + (uint64_t)list[j0 + u * per < n ? j0 + u * per : 0u] * TB, sub, v[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float ex = ranked_score(exact_score_of_octs<NOCT, true>(v[u], eps_l1, eps_log));
      const uint32_t j = j0 + u * per;
      if (j < n && sub == 0) {
        if (keys) keys[j] = rank_key(ex, i0 + list[j]);
        else scores[list[j]] = ex;
      }
    }
  }
}
static __device__ __noinline__ void exact_listed_any(const Args &a, const uint8_t *tiles, const uint32_t *list, uint32_t n, uint32_t thread,
                                                     uint32_t threads, uint32_t i0, unsigned long long *keys, float *scores) {
  auto run = [&](auto noct) {
    constexpr int N = decltype(noct)::value;
    if (a.bf16) exact_listed<N, true>(tiles, list, n, thread, threads, a.eps_l1, a.eps_log, i0, keys, scores);
    else exact_listed<N, false>(tiles, list, n, thread, threads, a.eps_l1, a.eps_log, i0, keys, scores);
  };
  switch (a.tile) {
    case 8: run(std::integral_constant<int, 1>{}); break;
    case 16: run(std::integral_constant<int, 2>{}); break;
    case 32: run(std::integral_constant<int, 4>{}); break;
    case 64: run(std::integral_constant<int, 8>{}); break;
    default: run(std::integral_constant<int, 16>{}); break;
  }
}

// More candidates than the key list holds, for thousands of equal scores or a very long group: a radix selection over the
// candidates of all slices, 8 bits a pass, gives the threshold key; every CTA sums the cluster's digit counts for itself.  A
// slice whose own candidates are all listed has their keys in shared memory; else every pass reads the slice, whose candidates
// have their exact score and whose other tiles +-infinity, from there if it fits and in place if not.  A digit that all keys
// share is skipped, and so is what lies behind a digit all of whose keys make it.  Sets the slice's words and returns the higher-width tiles of the slices before it.
// (Out of line: the usual path runs once per launch from a cold instruction cache and stays compact.)
static __device__ __noinline__ uint32_t selection_by_radix(const Args &a, uint32_t per_cta, int B, uint32_t rr, uint32_t *words, SelShared &sh) {
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t CS = cl.num_blocks(), rank = cl.block_rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const SelMem mem;
  unsigned long long *const s_keys = mem.keys;
  uint32_t *const s_cand = mem.cand, *const s_count = mem.hist /* [2][256] */, *const s_red = sh.red;
  const uint32_t ng = (uint32_t)a.rank_per_group, i0 = rank * per_cta, n_loc = i0 < ng ? (ng - i0 < per_cta ? ng - i0 : per_cta) : 0u;
  const uint64_t first = (uint64_t)(blockIdx.x / CS) * ng + i0;
  float *const sc = a.scores + first;
  const uint8_t *const tiles = a.in + first * (a.tile * (a.bf16 ? 2u : 4u));
  const int band = a.exact_scores ? 0 : kScreenBand, lo_v = B * 16 - band, hi_v = (B + 1) * 16 + band;
  const uint32_t nc = sh.n_cand;
  const bool listed = nc <= (uint32_t)kClKeys;
  float *const own = n_loc <= 2u * (kClKeys + kSelThreads) ? reinterpret_cast<float *>(s_keys) : sc;   // (not listed) the slice's scores
  if (listed) {
    if (a.exact_scores)
      for (uint32_t j = threadIdx.x; j < nc; j += kSelThreads) s_keys[j] = rank_key(sc[s_cand[j]], i0 + s_cand[j]);
    else
      exact_listed_any(a, tiles, s_cand, nc, threadIdx.x, kSelThreads, i0, s_keys, nullptr);
  } else {
    __syncthreads();   // the list, which holds a part of the candidates only, makes room for one of 128 per warp
    uint32_t *const mine = s_cand + warp * 128;
    for (uint32_t c0 = (uint32_t)warp * 128u; c0 < n_loc; c0 += 4u * kSelThreads) {
      uint32_t n = 0;
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) {
        const uint32_t i = c0 + 32u * k + lane;
        const float s = i < n_loc ? sc[i] : 0.0f;
        const int v = score_step(s, {a.step_lo, a.step_hi, a.step_off});
        const bool cand = i < n_loc && v >= lo_v && v < hi_v;
        if (i < n_loc) own[i] = cand ? s : __int_as_float(v >= hi_v ? 0x7f800000 : (int)0xff800000);
        const unsigned m = __ballot_sync(kFull, cand);
        if (cand) mine[n + (uint32_t)__popc(m & ((1u << lane) - 1u))] = i;
        n += (uint32_t)__popc(m);
      }
      if (a.exact_scores) continue;
      __syncwarp();
      exact_listed_any(a, tiles, mine, n, lane, 32u, i0, nullptr, own);
      __syncwarp();
    }
  }
  __syncthreads();
  // f(takes part, key) for every candidate of the slice; whole warps at a time
  auto each = [&](auto &&f) {
    if (listed) {
      for (uint32_t i = threadIdx.x; i - (uint32_t)lane < nc; i += kSelThreads) f(i < nc, i < nc ? s_keys[i] : 0ull);
    } else {
      for (uint32_t b = threadIdx.x; b - (uint32_t)lane < n_loc; b += 4 * kSelThreads) {
        float s[4];   // (the loads together: they may come from memory)
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) s[u] = b + u * kSelThreads < n_loc ? own[b + u * kSelThreads] : __int_as_float(0x7f800000);
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
          f((__float_as_uint(s[u]) & 0x7f800000u) != 0x7f800000u, rank_key(s[u], i0 + b + u * kSelThreads));
      }
    }
  };
  // bits on which the cluster's keys differ
  unsigned long long some = 0, all = ~0ull;
  each([&](bool in, unsigned long long key) {
    if (in) { some |= key; all &= key; }
  });
  auto reduce = [&]() {
    some = (unsigned long long)__reduce_or_sync(kFull, (uint32_t)(some >> 32)) << 32 | __reduce_or_sync(kFull, (uint32_t)some);
    all = (unsigned long long)__reduce_and_sync(kFull, (uint32_t)(all >> 32)) << 32 | __reduce_and_sync(kFull, (uint32_t)all);
  };
  if (threadIdx.x < 4) sh.key_bits[threadIdx.x] = threadIdx.x < 2 ? 0u : 0xffffffffu;
  s_count[threadIdx.x] = 0;
  static_assert(kSelThreads == 512, "a thread to each of the two times 256 counts");
  reduce();
  __syncthreads();
  if (lane == 0) {
    atomicOr(&sh.key_bits[0], (uint32_t)some);
    atomicOr(&sh.key_bits[1], (uint32_t)(some >> 32));
    atomicAnd(&sh.key_bits[2], (uint32_t)all);
    atomicAnd(&sh.key_bits[3], (uint32_t)(all >> 32));
  }
  cl.sync();
  some = 0;
  all = ~0ull;
  if (lane < (int)CS) {
    const uint32_t *k = cl.map_shared_rank(&sh, lane)->key_bits;
    some = (unsigned long long)k[1] << 32 | k[0];
    all = (unsigned long long)k[3] << 32 | k[2];
  }
  reduce();
  const unsigned long long varying = some ^ all;
  unsigned long long prefix = 0, mask = 0;
  uint32_t r = rr, buf = 0;
  for (int shift = 56; shift >= 0; shift -= 8) {
    if (((varying >> shift) & 0xffull) == 0) {
      prefix |= some & (0xffull << shift);
      mask |= 0xffull << shift;
      continue;
    }
    uint32_t *const s_digit = s_count + 256 * buf;
    each([&](bool in, unsigned long long key) {
      in = in && (key & mask) == prefix;
      const uint32_t d = (uint32_t)(key >> shift) & 255u;
      const unsigned m = __ballot_sync(kFull, in);
      if (m == 0u) return;
      // the warp's keys often share the digit: one addition then
      const uint32_t d0 = __shfl_sync(kFull, d, __ffs(m) - 1);
      if (__ballot_sync(kFull, in && d == d0) == m) {
        if (lane == 0) atomicAdd(&s_digit[d0], (uint32_t)__popc(m));
      } else if (in) {
        atomicAdd(&s_digit[d], 1u);
      }
    });
    cl.sync();
    // (the other half of the counts was read by everybody before this barrier)
    if (threadIdx.x < 256) s_count[256 * (buf ^ 1u) + threadIdx.x] = 0;
    uint32_t cnt = 0;   // thread d < 256: keys of the cluster with digit d
    if (threadIdx.x < 256)
      for (uint32_t q = 0; q < CS; ++q) cnt += cl.map_shared_rank(s_digit, q)[threadIdx.x];
    uint32_t incl = cnt;   // keys with a larger digit: suffix scan over the 256 counts (warps 0..7)
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const uint32_t v = __shfl_down_sync(kFull, incl, o);
      if (lane + o < 32) incl += v;
    }
    if (lane == 0 && warp < 8) s_red[warp] = incl;
    __syncthreads();
    if (threadIdx.x < 256) {
      uint32_t above = incl - cnt;
      for (int w = warp + 1; w < 8; ++w) above += s_red[w];
      if (above < r && above + cnt >= r) { sh.digit_pick[0] = threadIdx.x; sh.digit_pick[1] = r - above; sh.digit_pick[2] = cnt; }
    }
    __syncthreads();
    prefix |= (unsigned long long)sh.digit_pick[0] << shift;
    mask |= 0xffull << shift;
    r = sh.digit_pick[1];
    buf ^= 1u;
    if (sh.digit_pick[2] == r) break;   // all keys that begin like this make it
    __syncthreads();   // the pick is read, s_red is free
  }
  // the candidates against the threshold; the slices' counts have to be exchanged
  uint32_t bits_here = 0;
  if (listed) {
    for (uint32_t j = threadIdx.x; j < nc; j += kSelThreads)
      if (s_keys[j] >= prefix) {
        const uint32_t i = s_cand[j];
        atomicOr(&words[i >> 5], 1u << (i & 31u));
        ++bits_here;
      }
    if (threadIdx.x == 0) bits_here += sh.n_above;
  } else {
    for (uint32_t c0 = (uint32_t)warp * 32u; c0 < n_loc; c0 += kSelThreads) {
      const uint32_t i = c0 + lane;
      const unsigned m = __ballot_sync(kFull, i < n_loc && rank_key(own[i], i0 + i) >= prefix);   // +inf is above every threshold
      if (lane == 0) { words[c0 >> 5] = m; bits_here += (uint32_t)__popc(m); }
    }
  }
  bits_here = __reduce_add_sync(kFull, bits_here);
  __syncthreads();
  if (lane == 0) s_red[warp] = bits_here;
  __syncthreads();
  if (threadIdx.x < CS) {
    uint32_t T = 0;
    for (int w = 0; w < kSelThreads / 32; ++w) T += s_red[w];
    cl.map_shared_rank(&sh, threadIdx.x)->tot[rank] = T;
  }
  cl.sync();   // (the last time that a CTA touches another one's shared memory is before this)
  uint32_t before = 0;
  for (uint32_t q = 0; q < rank; ++q) before += sh.tot[q];
  return before;
}

// The bin among n ascending counts, held `per` to a lane by one warp, that holds the k-th largest, and the rank inside it.
template <int PER>
__device__ __forceinline__ void find_bin(const uint32_t (&c)[PER], uint32_t k, uint32_t &bin, uint32_t &rank_in) {
  const int lane = threadIdx.x & 31;
  uint32_t mine = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) mine += c[j];
  uint32_t incl = mine;   // counts in this lane's bins and higher
#pragma unroll
  for (int o = 1; o < 32; o *= 2) {
    const uint32_t v = __shfl_down_sync(kFull, incl, o);
    if (lane + o < 32) incl += v;
  }
  uint32_t above = incl - mine, b = 0, r = 0;
  const bool here = above < k && incl >= k;
#pragma unroll
  for (int j = PER - 1; j >= 0; --j) {
    if (above < k && above + c[j] >= k) { b = (uint32_t)(lane * PER + j); r = k - above; }
    above += c[j];
  }
  const unsigned m = __ballot_sync(kFull, here);
  const int src = m ? __ffs(m) - 1 : 0;   // (always found: k_hi is at most the number of tiles)
  bin = __shfl_sync(kFull, b, src);
  rank_in = __shfl_sync(kFull, r, src);
}

// Screening scores of n tiles from `first` on, by a CTA of the selection kernel, to shared and to global memory.
template <class C>
__device__ __forceinline__ void slice_scores(const Args &a, uint64_t first, uint32_t n, float *s_out, float *out) {
  using D = LaneCfg<C>;
  constexpr int P = D::P, TPR = D::TPR, NP = D::E / 2;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, sub = lane % P;
  const uint8_t *in = a.in + first * D::TB + sub * 64u;
  const uint32_t n_rounds = (n + TPR - 1) / TPR;
  uint32_t raw[16];
  auto load = [&](uint32_t r) {
    const uint32_t t = r * TPR + lane / P;
    load_64_bytes<false>(in + (uint64_t)(t < n ? t : 0u) * D::TB, raw);
  };
  uint32_t range = 0;   // see screen_range
  if (warp < n_rounds) load(warp);
  for (uint32_t r = warp; r < n_rounds; r += kSelThreads / 32) {
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] = raw[i];
    if (r + kSelThreads / 32 < n_rounds) load(r + kSelThreads / 32);
    float2 L[2], T[2];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      float2 v;
      if constexpr (C::BF16) bf2_add_f32(w[i] & 0x7fff7fffu, 1e-30f, v.x, v.y);
      else v = f2(fabsf(__uint_as_float(w[2 * i])) + 1e-30f, fabsf(__uint_as_float(w[2 * i + 1])) + 1e-30f);
      const float2 l = f2(lg2_approx(v.x), lg2_approx(v.y));
      if (i < 2) {
        L[i] = v;
        T[i] = f2(v.x * l.x, v.y * l.y);   // (scalar products: they feed the fused chain's addend)
      } else {
        L[i & 1] = add2(L[i & 1], v);
        T[i & 1] = fma2(v, l, T[i & 1]);
      }
    }
    const float2 L2 = add2(L[0], L[1]), T2 = add2(T[0], T[1]);
    float Ls = L2.x + L2.y, Ts = T2.x + T2.y;
#pragma unroll
    for (int h = 1; h < P; h *= 2) {
      Ls += __shfl_xor_sync(kFull, Ls, h);
      Ts += __shfl_xor_sync(kFull, Ts, h);
    }
    const float Lp = Ls + a.eps_l1;
    float rc;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(Lp));
    range = max(range, screen_range(Lp));
    const uint32_t t = r * TPR + lane / P;
    if (sub == 0 && t < n) {
      const float s = __fmaf_rn(lg2_approx(Lp), Ls, -Ts) * rc;
      s_out[t] = s;
      out[t] = s;
    }
  }
  if (__any_sync(kFull, range > kScreenRange))
    for (uint32_t r = warp; r < n_rounds; r += kSelThreads / 32)
      exact_scores_of<C::G / 8, C::BF16>(a.in + (first + r * TPR) * D::TB, n - r * TPR < TPR ? n - r * TPR : TPR, a.eps_l1, a.eps_log,
                                                s_out + r * TPR, out + r * TPR);
}

// HELD: a thread's scores stay in registers between binning and deciding (slices of up to kHeld * kSelThreads);
// longer slices are read again, from L2.
// C: void, or the tile configuration of a call whose (screening) scores are formed here instead of in a kernel in front
// (small tensors; groups of whole words): see fuse_scores.
template <bool HELD, class C>
__global__ void __launch_bounds__(kSelThreads, 2) select_kernel(const __grid_constant__ Args a, const uint32_t per_cta) {
  constexpr int NW = kSelThreads / 32;
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t CS = cl.num_blocks(), rank = cl.block_rank();
  const uint64_t g = blockIdx.x / CS;
  const uint32_t ng = (uint32_t)a.rank_per_group, k = (uint32_t)a.rank_k;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const StepMap map = {a.step_lo, a.step_hi, a.step_off};
  const SelMem mem;
  unsigned long long *const s_keys = mem.keys;
  uint32_t *const s_hist = mem.hist, *const s_cand = mem.cand, *const s_words = mem.words;
  __shared__ SelShared sh;
  __shared__ uint32_t s_coarse[kCoarse];      // the CTA's coarse counts
  __shared__ __align__(8) uint32_t s_sum[2][kCoarse];   // the cluster's coarse counts; its fine counts in the chosen coarse bin
  uint32_t *const s_red = sh.red;
  __shared__ uint32_t s_base, s_made;
  TraceScope trace(a.trace, 2);

  const uint32_t i0 = rank * per_cta;                                   // first tile of the slice, inside the group
  const uint32_t n_loc = i0 < ng ? (ng - i0 < per_cta ? ng - i0 : per_cta) : 0u;
  const uint32_t n_words = (n_loc + 31u) / 32u, n_it = (n_loc + 4 * kSelThreads - 1) / (4 * kSelThreads);
  // the slice's words (and running counts): in shared memory, or in the payload section, where the codes come later, when the
  // slice is very long
  const bool in_smem = per_cta <= 32u * kWordsShared;
  uint32_t *words = s_words, *wpre = s_hist;
  if (!in_smem) {
    words = a.words + g * 2ull * ((ng + 31u) / 32u + kClMaxCtas) + 2ull * (i0 / 32u);
    wpre = words + n_words;
  }
  for (uint32_t b = threadIdx.x; b < (uint32_t)kBins; b += kSelThreads) s_hist[b] = 0;
  if (threadIdx.x < 2 * kCoarse) s_sum[0][threadIdx.x] = 0;
  if (threadIdx.x == 0) { sh.n_keys = 0; sh.n_total = 0; sh.overflow = 0; sh.n_cand = 0; sh.n_above = 0; s_made = 0; }
  grid_dependency_wait();   // the scores are the score kernel's (or the tensor a kernel's in front)
  trace.started();
  float *sc = a.scores + g * (uint64_t)ng + i0;
  if constexpr (!std::is_void<C>::value) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.status = 0;   // nothing else of the workspace has to start at zero
    // into this CTA's key list, which nobody writes before the first cluster barrier; and to memory, for the radix
    slice_scores<C>(a, g * (uint64_t)ng + i0, n_loc, reinterpret_cast<float *>(s_keys), sc);
    __syncthreads();
  }
  // ---- 1: the slice's histogram.  In turn `it` warp w takes 128 tiles from 128 * (it * NW + w) on, a lane four of them.
  const bool vec = ((reinterpret_cast<uintptr_t>(sc)) & 15u) == 0;
  const float *const s_own = reinterpret_cast<const float *>(s_keys);
  auto first_of = [&](uint32_t it) { return (it * NW + (uint32_t)warp) * 128u + (uint32_t)lane * 4u; };
  auto left_of = [&](uint32_t it) { return (int)n_loc - (int)first_of(it); };   // tiles of the slice from the lane's first on
  auto load4 = [&](uint32_t it) -> float4 {   // zeroes behind the slice's end (told by their place, not by their value)
    const uint32_t i = first_of(it);
    if constexpr (!std::is_void<C>::value)   // (slices of whole words)
      return i < n_loc ? *reinterpret_cast<const float4 *>(s_own + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (vec && i + 4u <= n_loc) return __ldg(reinterpret_cast<const float4 *>(sc + i));
    return make_float4(i < n_loc ? __ldg(sc + i) : 0.0f, i + 1u < n_loc ? __ldg(sc + i + 1) : 0.0f,
                       i + 2u < n_loc ? __ldg(sc + i + 2) : 0.0f, i + 3u < n_loc ? __ldg(sc + i + 3) : 0.0f);
  };
  auto bin4 = [&](uint32_t it, const float4 &v) {
    const int left = left_of(it);
    if (left > 0) atomicAdd(&s_hist[score_step(v.x, map) >> 4], 1u);
    if (left > 1) atomicAdd(&s_hist[score_step(v.y, map) >> 4], 1u);
    if (left > 2) atomicAdd(&s_hist[score_step(v.z, map) >> 4], 1u);
    if (left > 3) atomicAdd(&s_hist[score_step(v.w, map) >> 4], 1u);
  };
  float4 held[kHeld / 4];   // the scores, or (long slices) the first ones
#pragma unroll
  for (int it = 0; it < kHeld / 4; ++it) held[it] = load4(it);
  __syncthreads();
  if constexpr (HELD) {
#pragma unroll
    for (int it = 0; it < kHeld / 4; ++it) bin4(it, held[it]);
  } else {
    for (uint32_t it0 = 0; it0 < n_it; it0 += kHeld / 4) {
      float4 cur[kHeld / 4];
#pragma unroll
      for (int j = 0; j < kHeld / 4; ++j) { cur[j] = held[j]; held[j] = load4(it0 + kHeld / 4 + j); }
#pragma unroll
      for (int j = 0; j < kHeld / 4; ++j) bin4(it0 + j, cur[j]);
    }
  }
  __syncthreads();
  {   // eight threads to a coarse bin (turned, so that few lanes meet in a bank)
    const uint32_t c = threadIdx.x >> 3, j = threadIdx.x & 7u;
    uint32_t sum = 0;
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i) sum += s_hist[c * kFine + j * 8u + ((i + j + 2u * c) & 7u)];
#pragma unroll
    for (int o = 1; o < 8; o *= 2) sum += __shfl_xor_sync(kFull, sum, o);
    if (j == 0) s_coarse[c] = sum;
  }
  cl.sync();
  // ---- 2: the bin of the k_hi-th ranked tile.  Reads of another CTA's shared memory take a few hundred cycles each and
  // share a narrow path: two per thread here and two below.  What follows them is done by every warp for itself.
  uint32_t Bc, kin, Bf, unused;
  auto cluster_sum = [&](const uint32_t *counts, uint32_t *sum) {   // kCoarse counts of every CTA
    static_assert(kCoarse == 64 && kFine == 64 && kSelThreads == 512 && kClMaxCtas <= 16, "two CTAs to a thread");
    const uint32_t c = threadIdx.x & 63u, r = threadIdx.x >> 6;
    uint32_t p = r < CS ? cl.map_shared_rank(counts, r)[c] : 0u;
    if (r + 8u < CS) p += cl.map_shared_rank(counts, r + 8u)[c];
    if (p) atomicAdd(&sum[c], p);
    __syncthreads();
  };
  cluster_sum(s_coarse, s_sum[0]);
  {
    const uint32_t c[2] = {s_sum[0][lane * 2], s_sum[0][lane * 2 + 1]};
    find_bin<2>(c, k, Bc, kin);
  }
  cluster_sum(s_hist + Bc * kFine, s_sum[1]);
  {
    const uint32_t c[2] = {s_sum[1][lane * 2], s_sum[1][lane * 2 + 1]};
    find_bin<2>(c, kin, Bf, unused);
  }
  // ---- 3: decide what is certain; list the band's tiles
  const int B = (int)(Bc * kFine + Bf), band = a.exact_scores ? 0 : kScreenBand;
  const int lo_v = B * 16 - band, hi_v = (B + 1) * 16 + band;
  {
    // step(s) >= v for a whole v > 0 is score_pos(s) >= v; the first bin has nothing below it, the last one nothing above
    const float lo_f = B > 0 ? (float)lo_v : __int_as_float(0xff800000), hi_f = hi_v > 16 * kBins - 1 ? __int_as_float(0x7f800000) : (float)hi_v;
    uint32_t n_above = 0;
    auto decide = [&](uint32_t it, const float4 &v) {
      const float t[4] = {score_pos(v.x, map), score_pos(v.y, map), score_pos(v.z, map), score_pos(v.w, map)};
      const int left = left_of(it);
      uint32_t above = 0, cand = 0;   // of the lane's four tiles
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        above |= t[j] >= hi_f ? 1u << j : 0u;   // (a zero behind the slice's end is above nothing)
        cand |= (j < left && !(t[j] >= hi_f) && !(t[j] < lo_f)) ? 1u << j : 0u;
      }
      // eight lanes hold a word
      uint32_t word = above << (4 * (lane & 7));
#pragma unroll
      for (int o = 1; o < 8; o *= 2) word |= __shfl_xor_sync(kFull, word, o);
      const uint32_t w = (it * NW + (uint32_t)warp) * 4u + (uint32_t)(lane >> 3);
      if ((lane & 7) == 0 && w < n_words) words[w] = word;   // the bits that are certain; the band's winners are added in step 4
      n_above += (uint32_t)__popc(above);
      if (__any_sync(kFull, cand != 0u)) {
        const uint32_t mine = (uint32_t)__popc(cand);
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o *= 2) {
          const uint32_t x = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += x;
        }
        uint32_t base = 0;
        if (lane == 31) base = atomicAdd(&sh.n_cand, incl);
        uint32_t slot = __shfl_sync(kFull, base, 31) + incl - mine;
        const uint32_t i = first_of(it);
        for (uint32_t m = cand; m; m &= m - 1u, ++slot)
          if (slot < (uint32_t)kClKeys) s_cand[slot] = i + (uint32_t)__ffs(m) - 1u;
      }
    };
    if constexpr (HELD) {
#pragma unroll
      for (int it = 0; it < kHeld / 4; ++it)
        if ((uint32_t)it < n_it) decide(it, held[it]);
    } else {
#pragma unroll
      for (int it = 0; it < kHeld / 4; ++it) held[it] = load4(it);
      for (uint32_t it0 = 0; it0 < n_it; it0 += kHeld / 4) {
        float4 cur[kHeld / 4];
#pragma unroll
        for (int j = 0; j < kHeld / 4; ++j) { cur[j] = held[j]; held[j] = load4(it0 + kHeld / 4 + j); }
#pragma unroll
        for (int j = 0; j < kHeld / 4; ++j)
          if (it0 + j < n_it) decide(it0 + j, cur[j]);
      }
    }
    n_above = __reduce_add_sync(kFull, n_above);
    if (lane == 0 && n_above) atomicAdd(&sh.n_above, n_above);
  }
  __syncthreads();
  // A slice with more than its part of what the list holds, or a quarter of that, is nearly always one of many like it (equal
  // scores): its keys are not made here, which would be for nothing, but in selection_by_radix.
  const uint32_t nc = sh.n_cand, n_listed = nc <= ((uint32_t)kClKeys >> (CS < 4u ? CS >> 1 : 2u)) ? nc : 0u;   // (CS: a power of two)
  if (threadIdx.x == 0) s_base = nc ? atomicAdd(&cl.map_shared_rank(&sh, 0)->n_keys, nc) : 0u;
  if (threadIdx.x < CS) {
    SelShared *o = cl.map_shared_rank(&sh, threadIdx.x);
    o->part[rank] = sh.n_above;
    if (nc) atomicAdd(&o->n_total, nc);
    if (nc != n_listed) o->overflow = 1;
  }
  const uint32_t tile_bytes = a.tile * (a.bf16 ? 2u : 4u);
  const uint8_t *tiles = a.in + (g * (uint64_t)ng + i0) * tile_bytes;   // (not used with wider allocation tiles: their scores are exact)
  {
    const uint32_t noct = a.exact_scores ? 1u : a.tile / 8, sub = (uint32_t)threadIdx.x % noct, per_round = (uint32_t)kSelThreads / noct;
    for (uint32_t j0 = 0; j0 < n_listed; j0 += per_round) {   // uniform trip count: whole warps take part
      const uint32_t j = j0 + threadIdx.x / noct;
      const bool live = j < n_listed;
      const uint32_t i = s_cand[live ? j : 0];
      const float ex = a.exact_scores ? sc[i] : ranked_score(exact_score_any(tiles + (uint64_t)i * tile_bytes, noct, a.bf16 != 0, sub,
                                                                             a.eps_l1, a.eps_log));
      if (j0 == 0) __syncthreads();   // s_base
      // the keys go into every CTA's copy of the list: nobody has to fetch them from one CTA afterwards
      const uint32_t at = s_base + j;
      if (live && at < (uint32_t)kClKeys) {
        const unsigned long long key = rank_key(ex, i0 + i);
        for (uint32_t r = sub; r < CS; r += noct) cl.map_shared_rank(s_keys, r)[at] = key;
      }
    }
  }
  cl.sync();
  // ---- 4: who of the band made it, found by every CTA for itself from its copy of the list (from here on nobody touches
  // another CTA's shared memory, unless the list overflowed)
  const uint32_t n = sh.n_total, p_lane = lane < (int)CS ? sh.part[lane] : 0u;
  const uint32_t nab = __reduce_add_sync(kFull, p_lane);   // tiles above the band
  uint32_t before = __reduce_add_sync(kFull, lane < (int)rank ? p_lane : 0u);   // ... in the slices before this one
  uint32_t rr = k - nab;   // candidates that get the higher width
  if (nab >= k || rr > n) {   // only possible if the screening error exceeded its bound
    if (rank == 0 && threadIdx.x == 0) atomicOr(a.status, 8u /* TAHQ_DEV_INTERNAL */);
    rr = rr > n ? n : 1u;
  }
  if (n > (uint32_t)kClKeys || sh.overflow) {
    before = selection_by_radix(a, per_cta, B, rr, words, sh);
  } else {
    // band tiles that made it: those of the slices before this one are counted, those of this slice get their bit
    auto won = [&](unsigned long long key) {
      const uint32_t idx = 0xffffffffu - (uint32_t)key;   // tile inside the group
      if (idx < i0) atomicAdd(&s_made, 1u);
      else if (idx - i0 < n_loc) atomicOr(&words[(idx - i0) >> 5], 1u << ((idx - i0) & 31u));
    };
    if (n <= 128u) {   // a warp to a key: it counts the larger ones (keys are distinct)
      for (uint32_t q = (uint32_t)warp; q < n; q += NW) {
        const unsigned long long mine = s_keys[q];
        uint32_t larger = 0;
        for (uint32_t i = 0; i < n; i += 32) larger += (uint32_t)__popc(__ballot_sync(kFull, i + lane < n && s_keys[i + lane] > mine));
        if (lane == 0 && larger < rr) won(mine);
      }
    } else {
      const unsigned long long theta = rank_keys_shared(s_keys, n, rr, s_keys + kClKeys);
      for (uint32_t i = threadIdx.x; i < n; i += kSelThreads)
        if (s_keys[i] >= theta) won(s_keys[i]);
    }
    __syncthreads();
    before += s_made;
  }
  before += (uint32_t)(g * a.rank_k);   // ranked tiles of the higher width in front of the slice, over the whole tensor

  // ---- 5: running counts, words, and out.  512 words at a time.
  uint32_t *const bitmap = reinterpret_cast<uint32_t *>(a.packed + a.off_bitmap);
  const uint64_t t0 = (g * (uint64_t)ng + i0) * a.alloc_m;   // first quantisation tile of the slice
  auto word_at = [&](uint32_t w) { return *(volatile const uint32_t *)(words + w); };   // (in global memory: changed by atomics)
  uint32_t carry = before, next = threadIdx.x < n_words ? word_at(threadIdx.x) : 0u;
  for (uint32_t w0 = 0; w0 < n_words; w0 += kSelThreads) {
    const uint32_t w = w0 + threadIdx.x, wv = next, c = (uint32_t)__popc(wv);
    next = w + kSelThreads < n_words ? word_at(w + kSelThreads) : 0u;   // (a round trip to L2 for a very long slice)
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const uint32_t v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    if (w0) __syncthreads();
    if (lane == 31) s_red[warp] = incl;
    __syncthreads();
    const uint32_t sum = lane < NW ? s_red[lane] : 0u;
    const uint32_t ex = carry + incl - c + __reduce_add_sync(kFull, lane < warp ? sum : 0u);
    carry += __reduce_add_sync(kFull, sum);
    if (w < n_words) {
      if (a.whole_words) {   // groups of whole words, A = G: the words are the bit map's
        bitmap[t0 / 32 + w] = wv;
        a.pre[t0 / 32 + w] = ex;
      } else {
        wpre[w] = ex;
      }
    }
  }
  if (a.whole_words) return;
  __syncthreads();
  const uint32_t m = a.alloc_m, off = (uint32_t)(t0 & 31u);   // the slice starts at bit `off` of its first word
  const uint64_t n_out = (uint64_t)n_loc * m + off;           // bits from the start of that word
  if (n_loc == 0) return;
  for (uint32_t j = threadIdx.x; (uint64_t)j * 32u < n_out; j += kSelThreads) {
    const uint64_t word = t0 / 32 + j;
    const int64_t q0 = (int64_t)j * 32 - off;                 // the word's first tile, from the slice's first (negative: not ours)
    uint32_t bits = 0;
    if (m == 1u) {
      if (q0 < 0) {
        bits = word_at(0) << off;
      } else {
        const uint32_t w = (uint32_t)q0 >> 5;
        bits = __funnelshift_r(word_at(w), w + 1u < n_words ? word_at(w + 1u) : 0u, (uint32_t)q0 & 31u);
      }
    } else {
      const uint32_t q_end = n_out < (uint64_t)(j + 1) * 32u ? (uint32_t)(n_out - off) : (uint32_t)(q0 + 32);
      for (uint32_t q = q0 < 0 ? 0u : (uint32_t)q0; q < q_end;) {   // a ranked tile's run of quantisation tiles at a time
        const uint32_t r = q / m, e = (r + 1u) * m < q_end ? (r + 1u) * m : q_end, len = e - q;
        if ((word_at(r >> 5) >> (r & 31u)) & 1u) bits |= (len >= 32u ? 0xffffffffu : (1u << len) - 1u) << (uint32_t)((int64_t)q - q0);
        q = e;
      }
    }
    if (q0 >= 0 && (uint64_t)(j + 1) * 32u <= n_out) bitmap[word] = bits;
    else atomicOr(bitmap + word, bits);   // shared with a neighbouring slice or group
    if (q0 >= 0) {
      const uint32_t r = (uint32_t)q0 / m, in = (uint32_t)q0 - r * m;
      a.pre[word] = m * (wpre[r >> 5] + (uint32_t)__popc(word_at(r >> 5) & ((1u << (r & 31u)) - 1u))) + (((word_at(r >> 5) >> (r & 31u)) & 1u) ? in : 0u);
    }
  }
}

}  // namespace tahq
