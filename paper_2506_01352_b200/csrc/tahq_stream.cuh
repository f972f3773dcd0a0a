// Warp-streaming kernels of the TAH-Quant boundary codec (sm_100a): scores (Eq. 1-2), quantise + pack
// (Eq. 3-4, Sec. 3.2-3.4), decode (Sec. 3.3).
//
// A lane owns a "row": a whole tile (G = 8 ... 64), or half of a 128-wide tile, whose two halves sit in
// neighbouring lanes and meet in a few shuffles (the score's two sums, the range, the two largest
// magnitudes, the butterfly's last stage).  Every warp is an independent worker: it streams units of 32
// consecutive rows through a private ring of slots in shared memory and never meets a CTA-wide barrier
// in its loop.  Rows of 128 bytes arrive by one tiled TMA copy per unit on the warp's own mbarriers,
// other row sizes by 16-byte cp.async.  Two things make the independence possible.
//   * Sec. 3.2 / 3.4: the widths are known before quantise + pack starts: the selection has written the
//     bit map and, per bit-map word, the number of higher-width tiles in front of it.
//   * Eq. 3-4: tiles that pass the pivot test cost about three times as much as the others.  A lane
//     handles an unflagged tile on the spot; tiles that may be flagged are only noted in a queue of
//     row indices private to the warp.  When 32 are queued, their rows are fetched again (from L2,
//     where they were a moment ago) into a 32-row stage of the warp, and one iteration later the whole
//     warp runs the flagged path on them, one lane per row, in a routine that is not inlined (the
//     hot loop stays small enough for the instruction cache).  All warps therefore do the same
//     amount of work and no lane idles through the long path.  Decode holds transformed tiles back
//     in the same way.
#pragma once

#include <cuda.h>   // CUtensorMap (type only; the driver entry point is looked up at run time)

#include <type_traits>

#include "tahq_kernels.cuh"

namespace tahq {

constexpr int kWarps = kThreads / 32;
constexpr int kSegWords = 512;    // bit-map words (units) a CTA keeps in shared memory at a time

template <class C>
struct StreamCfg {
  static constexpr int UNIT_BYTES = 32 * C::ROWB;   // 32 rows (a row = what one lane owns: a tile, or half of a 128-wide one)
  static constexpr int WORDS = C::ROWB / 4;         // 32-bit words of one row
  // ring slots plus the stage of re-fetched rows, then the warps' mbarriers
  static constexpr int smem_bytes(int nst) { return kWarps * (nst + 1) * UNIT_BYTES + 256; }
};

// cp.async of unit u (tiles 32u .. 32u+31) into a warp-private slot, rows swizzled as everywhere
template <class C>
__device__ __forceinline__ void warp_issue_unit(const uint8_t *in, uint64_t n_tiles, uint64_t u, uint8_t *slot,
                                                int lane) {
  const uint64_t tile0 = u * 32;
  const uint8_t *src = in + tile0 * (uint64_t)C::ROWB + (size_t)lane * 16;
  if (tile0 + 32 <= n_tiles) {
#pragma unroll
    for (int i = 0; i < C::CPR; ++i) {
      const int piece = i * 32 + lane;
      cp_async16(slot + (size_t)phys_chunk<C>(piece / C::CPR, piece % C::CPR) * 16, src + (size_t)i * 512, 16);
    }
  } else {
    const uint32_t valid_bytes = tile0 < n_tiles ? (uint32_t)(n_tiles - tile0) * C::ROWB : 0u;
#pragma unroll
    for (int i = 0; i < C::CPR; ++i) {
      const int piece = i * 32 + lane;
      const bool ok = (uint32_t)piece * 16u < valid_bytes;
      cp_async16(slot + (size_t)phys_chunk<C>(piece / C::CPR, piece % C::CPR) * 16, ok ? src + (size_t)i * 512 : in,
                 ok ? 16 : 0);
    }
  }
}

// A warp's ring of unit slots.  Rows of 128 bytes arrive by one tiled TMA copy per unit, issued by
// lane 0 and completing on the slot's mbarrier: the hardware's 128-byte swizzle is exactly the XOR
// pattern of phys_chunk (slots are 1024-byte aligned), and rows past the end of the tensor come as
// zeros.  Other row sizes use 16-byte cp.async per lane and commit groups.
template <class C, int NST>
struct UnitRing {
  static_assert(kWarps * NST * 8 <= 256, "the warps' mbarriers live in the 256 bytes behind the ring slots");
  uint8_t *base;
  unsigned long long *bar;   // [NST], this warp's
  const void *tmap;          // nullptr: cp.async
  uint32_t phases;           // bit s = parity slot s waits for next
  int lane;
  __device__ __forceinline__ void init(uint8_t *b, unsigned long long *br, const void *tm, int ln) {
    base = b; bar = br; tmap = tm; phases = 0; lane = ln;
    if (tmap) {
      if (lane == 0) {
#pragma unroll
        for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
        mbar_init_fence();
      }
      __syncwarp();
    }
  }
  __device__ __forceinline__ uint8_t *slot(int s) const { return base + (size_t)s * StreamCfg<C>::UNIT_BYTES; }
  // fill slot s with unit u; every lane is done reading the slot (the caller has synchronised the warp)
  __device__ __forceinline__ void issue(const Args &a, uint64_t u, int s) {
    if (tmap) {
      if (lane == 0) {
        fence_async_proxy();   // the lanes' reads of the slot are ordered before the asynchronous write
        mbar_expect_tx(&bar[s], StreamCfg<C>::UNIT_BYTES);
        tma_load_rows(slot(s), tmap, (int)(u * 32), &bar[s]);
      }
    } else {
      warp_issue_unit<C>(a.in, a.n_tiles * C::LPT, u, slot(s), lane);
    }
  }
  __device__ __forceinline__ void commit() const {   // one group per round, issued or not
    if (!tmap) cp_async_commit();
  }
  // the unit issued into slot s has landed (call once per issue, in issue order)
  __device__ __forceinline__ void wait(const Args &a, int s) {
    if (tmap) {
      if (!mbar_wait(&bar[s], (phases >> s) & 1u)) atomicOr(a.status, 4u /* TAHQ_DEV_TIMEOUT */);
      phases ^= 1u << s;
    } else {
      cp_async_wait<NST - 1>();
    }
    __syncwarp();
  }
};

// a row: shared memory -> registers (raw words)
template <class C>
__device__ __forceinline__ void row_load_words(const uint8_t *stage, int row, uint32_t (&w)[C::ROWB / 4]) {
#pragma unroll
  for (int q = 0; q < C::CPR; ++q) {
    const uint4 v = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, q) * 16);
    w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
  }
}
// smallest and largest element of a row held as raw words
template <class C>
__device__ __forceinline__ void words_minmax(const uint32_t (&w)[C::ROWB / 4], float &mn, float &mx) {
  constexpr int NW = C::ROWB / 4;
  if constexpr (C::BF16) {
    uint32_t lo0 = bf2_min(w[0], w[2]), hi0 = bf2_max(w[0], w[2]);
    uint32_t lo1 = bf2_min(w[1], w[3]), hi1 = bf2_max(w[1], w[3]);
#pragma unroll
    for (int j = 4; j < NW; j += 4) {
      lo0 = bf2_min(lo0, bf2_min(w[j], w[j + 2])); hi0 = bf2_max(hi0, bf2_max(w[j], w[j + 2]));
      lo1 = bf2_min(lo1, bf2_min(w[j + 1], w[j + 3])); hi1 = bf2_max(hi1, bf2_max(w[j + 1], w[j + 3]));
    }
    lo0 = bf2_min(lo0, lo1); hi0 = bf2_max(hi0, hi1);
    mn = fminf(__uint_as_float(lo0 << 16), __uint_as_float(lo0 & 0xffff0000u));
    mx = fmaxf(__uint_as_float(hi0 << 16), __uint_as_float(hi0 & 0xffff0000u));
  } else {
    float l0 = fminf(__uint_as_float(w[0]), __uint_as_float(w[2])), h0 = fmaxf(__uint_as_float(w[0]), __uint_as_float(w[2]));
    float l1 = fminf(__uint_as_float(w[1]), __uint_as_float(w[3])), h1 = fmaxf(__uint_as_float(w[1]), __uint_as_float(w[3]));
#pragma unroll
    for (int j = 4; j < NW; j += 4) {
      l0 = fminf(l0, fminf(__uint_as_float(w[j]), __uint_as_float(w[j + 2])));
      h0 = fmaxf(h0, fmaxf(__uint_as_float(w[j]), __uint_as_float(w[j + 2])));
      l1 = fminf(l1, fminf(__uint_as_float(w[j + 1]), __uint_as_float(w[j + 3])));
      h1 = fmaxf(h1, fmaxf(__uint_as_float(w[j + 1]), __uint_as_float(w[j + 3])));
    }
    mn = fminf(l0, l1);
    mx = fmaxf(h0, h1);
  }
}

// ------------------------------------------------------------------------------------------
// Eq. 1-2: scores only, no group boundaries -- a warp streams units of 32 rows and stores their scores.  (Screening
// scores of bfloat16 tiles of 32 and more: score_lanes_kernel.)
// ------------------------------------------------------------------------------------------

template <class C, int NST, bool EXACT>
__global__ void __launch_bounds__(kThreads, 2) score_kernel(const Args a, const __grid_constant__ CUtensorMap tmap) {
  using S = StreamCfg<C>;
  extern __shared__ __align__(1024) uint8_t smem_sc[];
  uint8_t *const smem = smem_sc;
  unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem + (size_t)kWarps * NST * S::UNIT_BYTES);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  TraceScope trace(a.trace, 1);
  UnitRing<C, NST> ring;
  ring.init(smem + (size_t)warp * NST * S::UNIT_BYTES, bars + warp * NST,
            (a.use_tma && (smem_u32(smem) & 1023u) == 0) ? &tmap : nullptr, lane);
  const uint64_t n_units = (a.n_tiles * C::LPT + 31) / 32;   // units of 32 rows
  const uint64_t u0 = n_units * blockIdx.x / gridDim.x, u1 = n_units * (blockIdx.x + 1ull) / gridDim.x;
  const uint32_t stride = kWarps, first = warp;
  const uint32_t nu = (uint32_t)(u1 - u0);
  auto unit_of = [&](uint32_t k) -> uint64_t { return u1 - 1 - k; };
  grid_dependency_wait();   // the tensor may be the work of the kernel in front
  trace.started();
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.status = 0;   // nothing else of the workspace has to start at zero
  // The CTA's stretch is read back to front: the units read last are the ones the encoder, which walks the same
  // stretch front to back right afterwards, asks for first, while they are still in L2.
#pragma unroll
  for (int s = 0; s < NST; ++s) {
    const uint32_t k = first + (uint32_t)s * stride;
    if (k < nu) ring.issue(a, unit_of(k), s);
    ring.commit();
  }
  int slot = 0;
  uint32_t range = 0;   // (screening) see screen_range
  for (uint32_t k = first; k < nu; k += stride) {
    const uint64_t u = unit_of(k);
    ring.wait(a, slot);
    const uint8_t *stage = ring.slot(slot);
    const float s = EXACT ? ranked_score(tile_score<C>(stage, lane, a.eps_l1, a.eps_log)) : tile_score_screen<C>(stage, lane, a.eps_l1, range);
    __syncwarp();
    {
      const uint32_t kn = k + (uint32_t)NST * stride;
      if (kn < nu) ring.issue(a, unit_of(kn), slot);
      ring.commit();
    }
    slot = (slot + 1 == NST) ? 0 : slot + 1;
    const uint64_t tile = (u * 32 + lane) / C::LPT;
    if (tile < a.n_tiles && (C::LPT == 1 || !(lane & 1))) a.scores[tile] = s;
  }
  cp_async_wait<0>();
  if constexpr (!EXACT) {
    constexpr uint32_t TPU = 32 / C::LPT;   // tiles of a unit
    if (__any_sync(kFull, range > kScreenRange))   // (rows behind the last tile are zeroes and may say so too)
      for (uint32_t k = first; k < nu; k += stride) {
        const uint64_t tile = unit_of(k) * TPU, left = a.n_tiles - tile;
        exact_scores_of<C::G / 8, C::BF16>(a.in + tile * (uint64_t)(C::G * C::ESZ), left < TPU ? (uint32_t)left : TPU, a.eps_l1,
                                                  a.eps_log, a.scores + tile, nullptr);
      }
  }
}

template <class C> using WidthOf = typename std::conditional<(C::G <= 32), WidthConst, WidthNone>::type;

// Sec. 3.3-3.4 for a row that is not transformed, straight from its raw words: zero-point and scale
// from the known range, codes (computed once), then the bit stream at the lane's own width.
// Returns the stored {scale, zero}.
template <class C, bool SR>
__device__ __forceinline__ uint32_t encode_plain_words(const uint32_t (&w)[C::ROWB / 4], float mn, float mx,
                                                       uint32_t bits, bool hi, const WidthOf<C> &wc, bool narrow, uint32_t *dst,
                                                       unsigned long long seed, unsigned long long first) {
  const Quantiser q = make_quantiser(mn, mx, bits, hi, wc);
  if constexpr (SR) {
    float d[C::EPT];
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i) {
      if constexpr (C::BF16) bf2_add_f32(w[i], -q.z, d[2 * i], d[2 * i + 1]);
      else { d[2 * i] = __uint_as_float(w[2 * i]) - q.z; d[2 * i + 1] = __uint_as_float(w[2 * i + 1]) - q.z; }
    }
    stochastic_codes<C::EPT>(d, q.inv_s, q.qmax, seed, first);
    auto tk = [&](int k) { return d[k]; };
    if constexpr (C::EPT < 32) pack_store_small<C::EPT>(tk, bits, reinterpret_cast<uint8_t *>(dst));
    else if (narrow) pack_store_narrow<C::EPT>(tk, bits, dst);
    else pack_row<C::EPT>(tk, bits, dst);
    return q.sz;
  }
  const float ymin = (mn - q.z) * q.inv_s, ymax = (mx - q.z) * q.inv_s;
  const bool safe = ymin >= -0.4999f && ymax < q.qmax + 0.4999f;
  const float nz = -q.z;   // x + (-z) is x - z
  const float2 is = f2(q.inv_s), mg = f2(kMagic);
  // the codes are formed where the packing asks for them, pair by pair: no array of 64 values stays live
  auto pair = [&](int i) {
    float2 d;
    if constexpr (C::BF16) bf2_add_f32(w[i], nz, d.x, d.y);
    else d = add2(f2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1])), f2(nz));
    return fma2(d, is, mg);
  };
  if (__all_sync(__activemask(), safe)) {
    auto tk = [&](int k) { const float2 t = pair(k >> 1); return (k & 1) ? t.y : t.x; };
    if constexpr (C::EPT < 32) pack_store_small<C::EPT>(tk, bits, reinterpret_cast<uint8_t *>(dst));
    else if (narrow) pack_store_narrow<C::EPT>(tk, bits, dst);   // every width of this call is at most 4 bits
    else pack_row<C::EPT>(tk, bits, dst);
  } else {
    const float top = kMagic + q.qmax;
    auto tk = [&](int k) {
      const float2 t = pair(k >> 1);
      return fminf(fmaxf((k & 1) ? t.y : t.x, kMagic), top);
    };
    if constexpr (C::EPT < 32) pack_store_small<C::EPT>(tk, bits, reinterpret_cast<uint8_t *>(dst));
    else if (narrow) pack_store_narrow<C::EPT>(tk, bits, dst);
    else pack_row<C::EPT>(tk, bits, dst);
  }
  return q.sz;
}

// Eq. 3-4 + Sec. 3.3-3.4 for a queued row (shared memory): exact pivot test, pivot swap, Hadamard,
// range, codes, bit stream, stores.
template <class C, bool SR>
__device__ __noinline__ void encode_queued_row(float tau, float eps_ratio, uint8_t *queue, int row, uint32_t bits,
                                               bool hi, const WidthOf<C> wc, bool narrow, uint32_t *dst, uint32_t *sz, uint8_t *pv,
                                               unsigned long long seed, unsigned long long first) {
  float a1, a2;
  row_top2<C>(queue, row, a1, a2);
  const float t1 = a2 + eps_ratio;
  const float t2 = tau * t1;
  const bool flag = a1 > t2;   // Eq. 3
  int d = 0;
  if (flag) {   // Eq. 4: the pivot swap P_d, done in shared memory before the row is loaded
    d = row_first_index_of<C>(queue, row, a1);
    row_swap_0_d<C, !C::BF16>(queue, row, d);
    asm volatile("" ::: "memory");
  }
  float2 p[C::EPT / 2];
  load_row_pairs<C>(queue, row, p);
  // Eq. 4: (1/sqrt G) H_G.  For G = 64 the factor is a power of two: the products are exact, so the
  // factor is applied to the range and inside the quantiser's subtraction instead of element by element.
  constexpr bool kFold = C::G == 64 || C::G == 16;
  if (flag) {
    butterfly2<C::EPT / 2>(p);
    if (!kFold) {
#pragma unroll
      for (int i = 0; i < C::EPT / 2; ++i)   // scalar products: they are added to right after
        p[i] = f2(p[i].x * hadamard_scale<C>(), p[i].y * hadamard_scale<C>());
    }
  }
  float mn = fminf(p[0].x, p[0].y), mx = fmaxf(p[0].x, p[0].y);
#pragma unroll
  for (int i = 1; i < C::EPT / 2; ++i) {
    mn = fminf(mn, fminf(p[i].x, p[i].y));
    mx = fmaxf(mx, fmaxf(p[i].x, p[i].y));
  }
  const float pre = (kFold && flag) ? hadamard_scale<C>() : 1.0f;
  mn *= pre;
  mx *= pre;
  const Quantiser q = make_quantiser(mn, mx, bits, hi, wc);
  if constexpr (SR) {
    float d[C::EPT];
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i) {
      d[2 * i] = __fmaf_rn(p[i].x, pre, -q.z);
      d[2 * i + 1] = __fmaf_rn(p[i].y, pre, -q.z);
    }
    stochastic_codes<C::EPT>(d, q.inv_s, q.qmax, seed, first);
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i) p[i] = f2(d[2 * i], d[2 * i + 1]);
  } else {
    quantise_pairs<C::EPT / 2>(p, pre, mn, mx, q);
  }
  *sz = q.sz;
  *pv = flag ? (uint8_t)(0x80 | d) : (uint8_t)0;
  auto tk = [&](int k) { return (k & 1) ? p[k >> 1].y : p[k >> 1].x; };
  if constexpr (C::EPT < 32) pack_store_small<C::EPT>(tk, bits, reinterpret_cast<uint8_t *>(dst));
  else if (narrow) pack_store_narrow<C::EPT>(tk, bits, dst);
  else pack_row<C::EPT>(tk, bits, dst);
}

// The same for a 128-wide tile, whose halves are two neighbouring rows of the stage owned by lanes 2j and
// 2j+1.  All 32 lanes call it (`live`: the row is a queued one); what crosses the two lanes: the merge of the
// halves' two largest magnitudes (the lower half wins a tie: it holds the lower indices), the pivot swap
// (element 0 of the lower half with element d of either), the butterfly's last stage (stride 64), the range.
template <class C, bool SR>
__device__ __noinline__ void encode_queued_pair(float tau, float eps_ratio, uint8_t *queue, int row, bool live,
                                                uint32_t bits, bool hi, const WidthOf<C> wc, bool narrow, uint32_t *dst, uint32_t *sz, uint8_t *pv,
                                                unsigned long long seed, unsigned long long first) {
  const int half = row & 1;
  float a1, a2;
  row_top2<C>(queue, row, a1, a2);
  bool lower_wins;
  {
    const float o1 = __shfl_xor_sync(kFull, a1, 1), o2 = __shfl_xor_sync(kFull, a2, 1);
    const float l1 = half ? o1 : a1, l2 = half ? o2 : a2, u1 = half ? a1 : o1, u2 = half ? a2 : o2;
    lower_wins = l1 >= u1;
    a1 = lower_wins ? l1 : u1;
    a2 = lower_wins ? fmaxf(l2, u1) : fmaxf(u2, l1);
  }
  const float t1 = a2 + eps_ratio;
  const float t2 = tau * t1;
  const bool flag = a1 > t2;   // Eq. 3
  const int owner = lower_wins ? 0 : 1;
  int dl = 0;
  if (flag && half == owner) dl = row_first_index_of<C>(queue, row, a1);
  dl = __shfl_sync(kFull, dl, (row & ~1) + owner);
  const int d = owner * C::EPT + dl;
  if (flag && half == 0) {   // Eq. 4: the pivot swap P_d, in shared memory
    constexpr int EPC = 16 / C::ESZ;
    uint8_t *p0 = queue + (size_t)phys_chunk<C>(row, 0) * 16;
    uint8_t *pd = queue + (size_t)phys_chunk<C>(row + owner, dl / EPC) * 16 + (size_t)(dl % EPC) * C::ESZ;
    if constexpr (C::BF16) {
      const uint16_t x0 = *reinterpret_cast<uint16_t *>(p0), xd = *reinterpret_cast<uint16_t *>(pd);
      *reinterpret_cast<uint16_t *>(p0) = xd;
      *reinterpret_cast<uint16_t *>(pd) = x0;
    } else {
      const uint32_t x0 = *reinterpret_cast<uint32_t *>(p0), xd = *reinterpret_cast<uint32_t *>(pd);
      *reinterpret_cast<uint32_t *>(p0) = xd;
      *reinterpret_cast<uint32_t *>(pd) = x0;
    }
  }
  __syncwarp();
  float2 p[C::EPT / 2];
  load_row_pairs<C>(queue, row, p);
  const unsigned fm = __ballot_sync(kFull, flag);
  if (flag) {   // Eq. 4: (1/sqrt G) H_G -- strides 1 .. 32 inside the lane, stride 64 across the two lanes
    butterfly2<C::EPT / 2>(p);
    const float2 sg = f2(half ? -1.0f : 1.0f);
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i) {   // lower half: own + other; upper half: other - own (products by +-1 are exact)
      const float2 o = f2(__shfl_xor_sync(fm, p[i].x, 1), __shfl_xor_sync(fm, p[i].y, 1));
      p[i] = fma2(p[i], sg, o);
    }
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i)   // scalar products: they are added to right after
      p[i] = f2(p[i].x * hadamard_scale<C>(), p[i].y * hadamard_scale<C>());
  }
  float mn = fminf(p[0].x, p[0].y), mx = fmaxf(p[0].x, p[0].y);
#pragma unroll
  for (int i = 1; i < C::EPT / 2; ++i) {
    mn = fminf(mn, fminf(p[i].x, p[i].y));
    mx = fmaxf(mx, fmaxf(p[i].x, p[i].y));
  }
  mn = fminf(mn, __shfl_xor_sync(kFull, mn, 1));
  mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 1));
  const Quantiser q = make_quantiser(mn, mx, bits, hi, wc);
  if constexpr (SR) {
    float dd[C::EPT];
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i) {
      dd[2 * i] = p[i].x - q.z;
      dd[2 * i + 1] = p[i].y - q.z;
    }
    stochastic_codes<C::EPT>(dd, q.inv_s, q.qmax, seed, first);
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i) p[i] = f2(dd[2 * i], dd[2 * i + 1]);
  } else {
    quantise_pairs<C::EPT / 2>(p, 1.0f, mn, mx, q);
  }
  if (!live) return;
  if (half == 0) {
    *sz = q.sz;
    *pv = flag ? (uint8_t)(0x80 | d) : (uint8_t)0;
  }
  auto tk = [&](int k) { return (k & 1) ? p[k >> 1].y : p[k >> 1].x; };
  if (narrow) pack_store_narrow<C::EPT>(tk, bits, dst);
  else pack_row<C::EPT>(tk, bits, dst);
}

// Exclusive running count of set bits over the nw bit-map words of a segment (barriers inside):
// s_pre[i] = first + bits of words before i; returns the segment's total.
__device__ __forceinline__ uint32_t scan_segment(const uint32_t *s_bm, uint32_t nw, uint32_t first, uint32_t *s_pre,
                                                 uint32_t *s_wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int PER = kSegWords / kThreads;
  uint32_t c[PER], mine = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const uint32_t i = threadIdx.x * PER + j;
    c[j] = i < nw ? (uint32_t)__popc(s_bm[i]) : 0u;
    mine += c[j];
  }
  uint32_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o *= 2) {
    const uint32_t v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_wsum[warp] = incl;
  __syncthreads();
  uint32_t before = incl - mine + first, total = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t v = s_wsum[w];
    before += w < warp ? v : 0u;
    total += v;
  }
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const uint32_t i = threadIdx.x * PER + j;
    if (i < nw) s_pre[i] = before;
    before += c[j];
  }
  __syncthreads();
  return total;
}

constexpr int kQueueCap = 64;   // tile indices a warp can hold back (32 left over + 32 of one unit)

// ------------------------------------------------------------------------------------------
// Quantise + pack.  The bit-map word of a unit of 32 tiles is in the packed buffer already and a.pre[unit] is the
// number of higher-width tiles before it, so a warp needs nothing from the rest of its CTA -- no pass over the
// scores, no scan, no look-back over the CTAs -- and starts on its first unit at once.  NARROW: no width above 4 bits
// in this call (compiling the unit loop for the one case it meets makes it 1.5 us faster on the LLaMA-7B shape than
// finding out at run time).
// ------------------------------------------------------------------------------------------
template <class C, int NST, bool SR, bool NARROW>
__global__ void __launch_bounds__(kThreads, 2) quant2_kernel(const Args a, const __grid_constant__ CUtensorMap tmap) {
  using S = StreamCfg<C>;
  extern __shared__ __align__(1024) uint8_t smem_q2[];
  uint8_t *const smem = smem_q2;
  unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem + (size_t)kWarps * (NST + 1) * S::UNIT_BYTES);
  __shared__ uint32_t s_qtile[kWarps][kQueueCap];   // held-back tile: (tile - first tile of the CTA) * 2 + higher width
  __shared__ uint32_t s_qhib[kWarps][kQueueCap];    // held-back tile: higher-width tiles before it, from the CTA's first
  __shared__ uint32_t s_pool[2][kWarps * 32];        // the warps' last, partly filled batches, pooled at the end
  __shared__ uint32_t s_pool_n;
  if (threadIdx.x == 0) s_pool_n = 0;   // (read only after the barrier further down)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int R = C::LPT;        // lanes (rows) per tile
  constexpr int TPU = 32 / R;      // tiles per unit of 32 rows
  const int half = lane & (R - 1);
  TraceScope trace(a.trace, 3);
  UnitRing<C, NST> ring;
  ring.init(smem + (size_t)warp * (NST + 1) * S::UNIT_BYTES, bars + warp * NST,
            (a.use_tma && (smem_u32(smem) & 1023u) == 0) ? &tmap : nullptr, lane);
  uint8_t *fstage = ring.slot(NST);   // rows fetched again for the flagged path (always by cp.async)
  uint32_t *sz32 = reinterpret_cast<uint32_t *>(a.packed + a.off_sz);
  uint8_t *pivot = a.packed + a.off_pivot;
  uint32_t *bitmap = reinterpret_cast<uint32_t *>(a.packed + a.off_bitmap);
  uint8_t *payload = a.packed + a.off_payload;
  constexpr uint32_t kTB = C::G / 8;   // bytes of a tile's codes per bit of width

  const uint64_t n_rows = a.n_tiles * R, n_units = (n_rows + 31) / 32, n_words = (a.n_tiles + 31) / 32;
  const uint64_t u0 = n_units * blockIdx.x / gridDim.x, u1 = n_units * (blockIdx.x + 1ull) / gridDim.x;
  const uint64_t row_cta = u0 * 32, tile_cta = u0 * TPU;
  const uint32_t nu = (uint32_t)(u1 - u0);
  grid_dependency_wait();   // bit map and running counts are the selection kernel's; the tensor may be a kernel's too
  trace.started();
#pragma unroll
  for (int s = 0; s < NST; ++s) {
    const uint32_t k = warp + (uint32_t)s * kWarps;
    if (k < nu) ring.issue(a, u0 + k, s);
    ring.commit();
  }
  if (blockIdx.x == 0) {   // header and the zero padding behind every section
    if (threadIdx.x == 0 && !a.mixed) *a.status = 0;   // (with two widths in use the score kernel has done it)
    if (threadIdx.x < 32) reinterpret_cast<uint32_t *>(a.packed)[threadIdx.x] = a.header[threadIdx.x];
    for (int s = 0; s < 4; ++s) {
      const uint64_t from = s == 0 ? a.off_bitmap + 4 * n_words : s == 1 ? a.off_sz + 4 * a.n_tiles
                          : s == 2 ? a.off_pivot + a.n_tiles : a.off_payload + a.payload_bytes;
      const uint64_t to = s == 0 ? a.off_sz : s == 1 ? a.off_pivot : s == 2 ? a.off_payload : a.total_bytes;
      for (uint64_t o = from + threadIdx.x; o < to; o += kThreads) a.packed[o] = 0;
    }
  }

  uint32_t qhead = 0, qn = 0;   // this warp's queue of held-back tiles (circular)
  uint32_t f_n = 0;             // rows on their way into (or waiting in) fstage
  uint32_t f_tile = 0, f_hib = 0;   // lane j's row of fstage: (row - first row of the CTA) * 2 + higher width; count
  const uint64_t row_bytes = (uint64_t)C::ROWB;
  const bool narrow = NARROW;
  const uint32_t lo = a.lo;
  const WidthOf<C> wc(lo);

  // fetch the rows of the first n (<= 32) queued tiles again; lane j keeps the j-th tile's particulars
  auto gather = [&](uint32_t n) {
    f_tile = s_qtile[warp][(qhead + lane) & (kQueueCap - 1)];
    f_hib = s_qhib[warp][(qhead + lane) & (kQueueCap - 1)];
#pragma unroll
    for (int i = 0; i < C::CPR; ++i) {
      const int piece = i * 32 + lane, r = piece / C::CPR, q = piece % C::CPR;
      const uint32_t tr = __shfl_sync(kFull, f_tile, r) >> 1;
      const bool ok = (uint32_t)r < n;
      cp_async16(fstage + (size_t)phys_chunk<C>(r, q) * 16,
                 ok ? a.in + (row_cta + tr) * row_bytes + (size_t)q * 16 : a.in, ok ? 16 : 0);
    }
    cp_async_commit();
    f_n = n;
    qhead = (qhead + n) & (kQueueCap - 1);
    qn -= n;
  };
  // Eq. 3-4 on the rows of fstage, lane j on row j
  auto run_flagged = [&]() {
    if constexpr (R == 1) {
      if ((uint32_t)lane < f_n) {
        const uint64_t tile = tile_cta + (f_tile >> 1);
        const uint64_t off = (uint64_t)kTB * ((uint64_t)lo * tile + f_hib);
        encode_queued_row<C, SR>(a.tau, a.eps_ratio, fstage, lane, lo + (f_tile & 1u), (f_tile & 1u) != 0u, wc, narrow,
                                 reinterpret_cast<uint32_t *>(payload + off), sz32 + tile, pivot + tile, a.seed,
                                 tile * (unsigned long long)C::G);
      }
    } else {   // the two rows of a tile are queued together and sit in neighbouring lanes
      const bool live = (uint32_t)lane < f_n;
      const uint64_t tile = live ? tile_cta + (f_tile >> 2) : 0;
      const uint32_t bits = lo + (f_tile & 1u);
      const uint64_t off = live ? (uint64_t)kTB * ((uint64_t)lo * tile + f_hib) + (uint64_t)half * (C::EPT / 8) * bits : 0;
      encode_queued_pair<C, SR>(a.tau, a.eps_ratio, fstage, lane, live, bits, (f_tile & 1u) != 0u, wc, narrow,
                                reinterpret_cast<uint32_t *>(payload + off), sz32 + tile, pivot + tile, a.seed,
                                tile * (unsigned long long)C::G + (unsigned)(half * C::EPT));
    }
    f_n = 0;
    __syncwarp();
  };

  int slot = 0;
  const uint32_t n_rel = n_rows - row_cta < 0xffffffffull ? (uint32_t)(n_rows - row_cta) : 0xffffffffu;   // rows from the CTA's first
  // the unit's bit-map word and running count, asked for one round ahead
  uint32_t word_n = 0, pre_n = 0;
  if (a.mixed && (uint32_t)warp < nu) { word_n = __ldg(bitmap + (u0 + warp) / R); pre_n = __ldg(a.pre + (u0 + warp) / R); }
  for (uint32_t su = warp; su < nu; su += kWarps) {   // su = unit index inside the CTA's range
    const uint32_t word = word_n, pre = pre_n;
    if (a.mixed && su + kWarps < nu) { word_n = __ldg(bitmap + (u0 + su + kWarps) / R); pre_n = __ldg(a.pre + (u0 + su + kWarps) / R); }
    if (f_n && ring.tmap) cp_async_wait<0>();   // the rows fetched again one round ago (their own group here)
    ring.wait(a, slot);                         // this unit has landed (cp.async: and so have those rows)
    if (f_n) run_flagged();
    if (qn >= 32u) gather(32u);

    uint8_t *stage = ring.slot(slot);
    uint32_t w[S::WORDS];
    row_load_words<C>(stage, lane, w);
    __syncwarp();
    {   // the slot is free again: fetch the unit that comes NST rounds later
      const uint32_t sn = su + (uint32_t)NST * kWarps;
      if (sn < nu) ring.issue(a, u0 + sn, slot);
      ring.commit();
    }
    slot = (slot + 1 == NST) ? 0 : slot + 1;

    if (!a.mixed && lane == 0 && (R == 1 || !((u0 + su) & 1))) bitmap[(u0 + su) / R] = 0;
    const uint32_t bp = R == 1 ? (uint32_t)lane : (uint32_t)(((u0 + su) & 1) * 16 + (lane >> 1));   // the tile's bit in the word
    const uint32_t hi = (word >> bp) & 1u;
    const uint32_t trel = su * 32u + lane;   // row - first row of the CTA
    const bool live = trel < n_rel;
    const uint32_t hib = pre + (uint32_t)__popc(word & ((1u << bp) - 1u));   // higher-width tiles before this one, whole tensor

    // Eq. 3, first look: the second-largest magnitude is at least the smaller of |min| and |max| (they
    // sit at different positions, or every element is equal), so a tile whose largest magnitude does
    // not exceed tau * (that + varrho) cannot be flagged.  The others are held back for the exact test.
    float mn, mx;
    words_minmax<C>(w, mn, mx);
    if constexpr (R == 2) {
      mn = fminf(mn, __shfl_xor_sync(kFull, mn, 1));
      mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 1));
    }
    const float m_big = fmaxf(fabsf(mn), fabsf(mx)), m_small = fminf(fabsf(mn), fabsf(mx));
    const bool maybe = live && m_big > a.tau * (m_small + a.eps_ratio);
    const unsigned held = __ballot_sync(kFull, maybe);
    if (maybe) {
      const uint32_t e = (qhead + qn + (uint32_t)__popc(held & ((1u << lane) - 1u))) & (kQueueCap - 1);
      s_qtile[warp][e] = (trel << 1) | hi;
      s_qhib[warp][e] = hib;
    }
    qn += (uint32_t)__popc(held);
    if (live && !maybe) {
      const uint64_t tile = tile_cta + trel / R;
      const uint64_t off = (uint64_t)kTB * ((uint64_t)lo * tile + hib) + (uint64_t)half * (C::EPT / 8) * (lo + hi);
      const uint32_t szw = encode_plain_words<C, SR>(w, mn, mx, lo + hi, hi != 0u, wc, narrow, reinterpret_cast<uint32_t *>(payload + off),
                                                     a.seed, tile * (unsigned long long)C::G + (unsigned)(half * C::EPT));
      if (R == 1 || half == 0) {
        sz32[tile] = szw;
        pivot[tile] = 0;
      }
    }
    __syncwarp();
  }
  cp_async_wait<0>();
  __syncwarp();
  // ---- what is still held back: full batches first, then the warps pool their remainders so that the
  // CTA runs as few partly filled batches as possible (on a small tensor these are half of all batches)
  if (f_n) run_flagged();
  while (qn >= 32u) {
    gather(32u);
    cp_async_wait<0>();
    __syncwarp();
    run_flagged();
  }
  {
    uint32_t base = 0;
    if (lane == 0 && qn) base = atomicAdd(&s_pool_n, qn);
    base = __shfl_sync(kFull, base, 0);
    if ((uint32_t)lane < qn) {
      s_pool[0][base + lane] = s_qtile[warp][(qhead + lane) & (kQueueCap - 1)];
      s_pool[1][base + lane] = s_qhib[warp][(qhead + lane) & (kQueueCap - 1)];
    }
    __syncthreads();
    const uint32_t n = s_pool_n;
    for (uint32_t t0 = (uint32_t)warp * 32u; t0 < n; t0 += kWarps * 32u) {
      const uint32_t cnt = n - t0 < 32u ? n - t0 : 32u;
      s_qtile[warp][lane] = (uint32_t)lane < cnt ? s_pool[0][t0 + lane] : 0u;   // through the warp's own queue
      s_qhib[warp][lane] = (uint32_t)lane < cnt ? s_pool[1][t0 + lane] : 0u;
      __syncwarp();
      qhead = 0;
      qn = cnt;
      gather(cnt);
      cp_async_wait<0>();
      __syncwarp();
      run_flagged();
    }
  }
}

// ------------------------------------------------------------------------------------------
// Decode of tiles of 8 and 16 elements, warp-streaming (Sec. 3.3, Algorithm 1 line 5); wider tiles: tahq_lanes.cuh
// ------------------------------------------------------------------------------------------

// Transformed tiles (Eq. 4 inverted): codes from the packed buffer, z + q*s, the butterfly, the
// scale, the row into the warp's output stage, coordinates 0 and d swapped back there.
template <class C>
__device__ __noinline__ void decode_flagged_row(const uint8_t *codes, uint32_t bits, uint32_t szw, uint32_t pvb,
                                                uint8_t *ostage, int row) {
  float s = __half2float(__ushort_as_half((unsigned short)(szw & 0xffffu)));
  float z = __half2float(__ushort_as_half((unsigned short)(szw >> 16)));
  // 1/sqrt(G) is a power of two for G = 16: scaling s and z by it beforehand scales every later value
  // by it exactly, so the result has the same bits as multiplying at the end
  constexpr bool kFold = C::G == 16;
  if (kFold) { s *= hadamard_scale<C>(); z *= hadamard_scale<C>(); }
  float x[C::EPT];
  dequant_small<C::EPT>(codes, bits, s, z, x);
  float2 p[C::EPT / 2];
#pragma unroll
  for (int i = 0; i < C::EPT / 2; ++i) p[i] = f2(x[2 * i], x[2 * i + 1]);
  butterfly2<C::EPT / 2>(p);
  if (!kFold) {
#pragma unroll
    for (int i = 0; i < C::EPT / 2; ++i) p[i] = mul2(p[i], f2(hadamard_scale<C>()));   // feeds no addition
  }
#pragma unroll
  for (int i = 0; i < C::EPT / 2; ++i) { x[2 * i] = p[i].x; x[2 * i + 1] = p[i].y; }
#pragma unroll
  for (int q = 0; q < C::CPR; ++q)
    *reinterpret_cast<uint4 *>(ostage + (size_t)phys_chunk<C>(row, q) * 16) = row_piece<C>(x, q);
  asm volatile("" ::: "memory");
  row_swap_0_d<C, !C::BF16>(ostage, row, pvb & (C::G - 1));   // masked: a foreign buffer cannot reach outside the row
}

template <class C>
struct DecStreamCfg {
  static_assert(C::G <= 16, "wider tiles: decode_lanes_kernel");
  static constexpr int NST = C::BF16 ? 3 : 2;
  static constexpr int PAY = 32 * C::EPT + 16;          // a unit's codes at 8 bits, from the 16-byte boundary below
  static constexpr int SLOT = PAY + 32 * 4 + 32;        // + scale/zero words + pivot bytes
  static constexpr int OUT = 32 * C::ROWB;              // the unit's rows on their way out
  static constexpr int WARP = NST * SLOT + OUT;
  static constexpr int TOTAL = kWarps * WARP;
};

template <class C>
__global__ void __launch_bounds__(kThreads, 2) decode_stream_kernel(const Args a) {
  using S = DecStreamCfg<C>;
  constexpr int NST = S::NST;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint32_t s_bm[kSegWords];
  __shared__ uint32_t s_pre[kSegWords];
  __shared__ uint32_t s_wsum[kWarps];
  __shared__ uint32_t s_q[kWarps][4][kQueueCap];   // held-back tiles: tile - first tile of the CTA, higher-width tiles
                                                   // before it (and the width bit), scale/zero word, pivot byte
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int TPU = 32;          // tiles per unit
  const unsigned lt = (1u << lane) - 1u;
  TraceScope trace(a.trace, 5);
  grid_dependency_wait();   // the look-back flags are cleared by the kernel in front
  trace.started();
  uint8_t *ring = smem + (size_t)warp * S::WARP;
  uint8_t *ostage = ring + (size_t)NST * S::SLOT;
  const uint32_t *bitmap = reinterpret_cast<const uint32_t *>(a.packed + a.off_bitmap);
  const uint8_t *payload = a.packed + a.off_payload;

  const uint64_t n_units = (a.n_tiles + TPU - 1) / TPU;
  const uint64_t u0 = n_units * blockIdx.x / gridDim.x, u1 = n_units * (blockIdx.x + 1ull) / gridDim.x;
  const uint64_t tile_cta = u0 * TPU;

  // The prologue's loads from global memory -- the header, the bit-map bits of the CTA's first units, the words in
  // front of its slice -- are all requested before the first barrier: one round trip to L2 instead of three.
  const bool checks = blockIdx.x == 0 || a.own_prefix;
  const uint32_t hdr_w = (checks && threadIdx.x < 32) ? __ldg(reinterpret_cast<const uint32_t *>(a.packed) + threadIdx.x) : 0u;
  // the bit-map word of unit i of the tensor, bits beyond the last tile cleared
  auto bm_raw = [&](uint64_t i) -> uint32_t {
    if (!a.mixed) return 0u;
    const uint64_t left = a.n_tiles - i * TPU;
    return __ldg(bitmap + i) & (left >= (uint64_t)TPU ? 0xffffffffu : ((1u << (uint32_t)left) - 1u));
  };
  static_assert(kSegWords == 2 * kThreads, "two units of the first segment per thread");
  uint32_t first_bits[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const uint64_t i = u0 + threadIdx.x + (uint32_t)k * kThreads;
    first_bits[k] = (i < u1) ? bm_raw(i) : 0u;
  }
  uint32_t own_before = 0;   // a.own_prefix: this thread's share of the higher-width tiles before the CTA's slice
  if (a.own_prefix && a.mixed) {   // words before u0 are whole: 128-bit loads, then the last few one by one
    const uint4 *b4 = reinterpret_cast<const uint4 *>(bitmap);
    const uint64_t nwb = u0;                     // words before the slice (at most 65536 here)
    const uint32_t n4 = (uint32_t)(nwb / 4);
    // eight loads in flight per thread: the words sit in L2, and the CTAs at the end of the tensor, which count
    // the most, set the kernel's end (one load at a time cost the last CTA 3.5 us on the LLaMA-7B shape)
    for (uint32_t i = threadIdx.x; i < n4; i += 8u * kThreads) {
      uint4 v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t k = i + (uint32_t)j * kThreads;
        v[j] = k < n4 ? __ldg(b4 + k) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) own_before += __popc(v[j].x) + __popc(v[j].y) + __popc(v[j].z) + __popc(v[j].w);
    }
    if (threadIdx.x < (uint32_t)(nwb - (uint64_t)n4 * 4)) own_before += __popc(__ldg(bitmap + (uint64_t)n4 * 4 + threadIdx.x));
  }
  // CTA 0 compares the received header with the one these parameters produce; what it finds travels
  // with the offset prefix, so a refused buffer leaves the output untouched.
  // (On a small tensor, a.own_prefix, every CTA does this itself and counts the bit map in front of its slice
  // itself: no look-back, nothing that has to be cleared beforehand, one launch; the last CTA writes the status.)
  bool refuse = false;
  if (checks) {
    refuse = __syncthreads_or(threadIdx.x < 32 && hdr_w != a.header[threadIdx.x]) != 0;
    if (refuse && threadIdx.x == 0 && !a.own_prefix) atomicOr(a.status, 1u /* TAHQ_DEV_BAD_HEADER */);
  }
  auto bm_word = [&](uint64_t i) -> uint32_t { return refuse ? 0u : bm_raw(i); };
  if (u0 == u1) {   // (never the last CTA)
    bool stop;
    if (!a.own_prefix) cta_exclusive_prefix(a, 0, refuse, stop);
    return;
  }
  const bool single = u1 - u0 <= (uint64_t)kSegWords;
  uint64_t counted = 0;
  if (!single) {
    uint32_t n = 0;
    for (uint64_t i = u0 + threadIdx.x; i < u1; i += kThreads) n += __popc(bm_word(i));
    counted = block_sum(n);
  }

  uint64_t base_hi = 0;
  uint32_t seg_hi = 0;
  uint32_t qhead = 0, qn = 0;

  // cp.async of unit u's codes, scale/zero words and pivot bytes into a slot; `hib` = higher-width tiles
  // of the CTA before the unit.  A unit whose codes would reach past the payload (corrupt bit map) is
  // not fetched.
  // Inside the loops everything is relative to the CTA's first tile and first payload byte (32-bit).
  // pay_off0 = byte offset of the CTA's first code in the payload, known after the look-back.
  uint64_t pay_off0 = 0;
  const uint32_t n_rel = a.n_tiles - tile_cta < 0xffffffffull ? (uint32_t)(a.n_tiles - tile_cta) : 0xffffffffu;
  // bytes [off, off + len) of the CTA's codes belong to the unit whose first tile is trel0 (relative)
  auto unit_range = [&](uint32_t trel0, uint32_t hib, uint32_t word, uint32_t &off, uint32_t &len) {
    const uint32_t left = n_rel - trel0;
    const uint32_t nv = left < (uint32_t)TPU ? left : (uint32_t)TPU;
    off = (uint32_t)(C::G / 8) * (a.lo * trel0 + hib);
    len = (uint32_t)(C::G / 8) * (a.lo * nv + (uint32_t)__popc(word));
    return pay_off0 + off + len <= a.payload_bytes;   // a corrupt bit map must not lead outside the buffer
  };
  // cp.async of a unit's codes (from the 16-byte boundary below them), scale/zero words and pivot bytes
  auto issue = [&](uint32_t trel0, uint32_t su, uint8_t *slot) {   // su = unit index inside the segment
    uint32_t off, len;
    if (unit_range(trel0, s_pre[su], s_bm[su], off, len)) {
      const uint64_t g = pay_off0 + off;
      const uint8_t *src = payload + (g & ~15ull);
      const uint32_t npieces = ((uint32_t)(g & 15ull) + len + 15u) >> 4;
#pragma unroll
      for (int i = 0; i < (S::PAY + 511) / 512; ++i)
        if ((uint32_t)(i * 32 + lane) < npieces)
          cp_async16(slot + (size_t)(i * 32 + lane) * 16, src + (size_t)(i * 32 + lane) * 16, 16);
      const uint64_t t0 = tile_cta + trel0;
      if (lane < TPU / 4) cp_async16(slot + S::PAY + lane * 16, a.packed + a.off_sz + t0 * 4 + lane * 16, 16);
      else if (lane >= 8 && lane < 8 + TPU / 16)
        cp_async16(slot + S::PAY + 128 + (lane - 8) * 16, a.packed + a.off_pivot + t0 + (lane - 8) * 16, 16);
    }
  };
  auto prime = [&](uint64_t s0, uint64_t s1) {
#pragma unroll
    for (int st = 0; st < NST; ++st) {
      const uint64_t u = s0 + warp + (uint64_t)st * kWarps;
      if (u < s1) issue((uint32_t)(u - u0) * TPU, (uint32_t)(u - s0), ring + (size_t)st * S::SLOT);
      cp_async_commit();
    }
  };
  // the warp's output stage leaves: row r goes to row `tile_of(r)` of the tensor if bit r of `rows` is set
  auto copy_out = [&](unsigned rows, auto &&tile_of) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < C::CPR; ++i) {
      const int piece = i * 32 + lane, r = piece / C::CPR, q = piece % C::CPR;
      const uint64_t t = tile_of(r);
      if ((rows >> r) & 1u)   // streaming store: the tensor is not read again by this library
        __stcs(reinterpret_cast<uint4 *>(a.out + t * (uint64_t)C::ROWB + (size_t)q * 16),
               *reinterpret_cast<const uint4 *>(ostage + (size_t)phys_chunk<C>(r, q) * 16));
    }
    __syncwarp();
  };
  // the same for the 32 consecutive tiles of a unit: one base address, constant strides
  auto copy_out_unit = [&](unsigned rows, uint8_t *dst0) {   // dst0 = first byte of the unit's rows + lane * 16
    __syncwarp();
#pragma unroll
    for (int i = 0; i < C::CPR; ++i) {
      const int piece = i * 32 + lane, r = piece / C::CPR, q = piece % C::CPR;
      const uint4 v = *reinterpret_cast<const uint4 *>(ostage + (size_t)phys_chunk<C>(r, q) * 16);
      if (rows == 0xffffffffu || ((rows >> r) & 1u)) __stcs(reinterpret_cast<uint4 *>(dst0 + (size_t)i * 512), v);
    }
    __syncwarp();
  };
  // the first n (<= 32) held-back tiles, lane j on the j-th
  auto run_flagged = [&](uint32_t n) {
    const uint32_t e = (qhead + lane) & (kQueueCap - 1);
    const uint32_t ft = s_q[warp][0][e], fh = s_q[warp][1][e];   // tile - first tile of the CTA; count * 2 + width bit
    if ((uint32_t)lane < n) {
      const uint32_t off = (uint32_t)(C::G / 8) * (a.lo * ft + (fh >> 1));
      decode_flagged_row<C>(payload + pay_off0 + off, a.lo + (fh & 1u), s_q[warp][2][e], s_q[warp][3][e], ostage, lane);
    }
    copy_out(n >= 32u ? 0xffffffffu : ((1u << n) - 1u), [&](int r) { return tile_cta + __shfl_sync(kFull, ft, r); });
    qhead = (qhead + n) & (kQueueCap - 1);
    qn -= n;
  };

  for (uint64_t s0 = u0; s0 < u1; s0 += kSegWords) {
    const uint64_t s1 = s0 + kSegWords < u1 ? s0 + kSegWords : u1;
    const uint32_t nw = (uint32_t)(s1 - s0);
    if (s0 != u0) __syncthreads();   // every warp is done with the previous segment's words
    if (s0 == u0) {
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (threadIdx.x + (uint32_t)k * kThreads < nw) s_bm[threadIdx.x + (uint32_t)k * kThreads] = refuse ? 0u : first_bits[k];
    } else {
      for (uint32_t i = threadIdx.x; i < nw; i += kThreads) s_bm[i] = bm_word(s0 + i);
    }
    __syncthreads();
    const uint32_t seg_total = scan_segment(s_bm, nw, seg_hi, s_pre, s_wsum);
    if (s0 == u0) {   // Sec. 3.4: higher-width tiles of all CTAs before this one; what CTA 0 found in the header
      bool stop;
      const uint64_t mine = single ? (uint64_t)seg_total : counted;
      if (a.own_prefix) {
        base_hi = block_sum(refuse ? 0u : own_before);
        stop = refuse;
        if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0)
          *a.status = (refuse ? 1u /* TAHQ_DEV_BAD_HEADER */ : 0u) |
                      ((a.mixed && !refuse && base_hi + mine != a.n_groups * a.k_hi) ? 2u /* TAHQ_DEV_BAD_BITMAP */ : 0u);
      } else {
        base_hi = cta_exclusive_prefix(a, mine, refuse, stop);
        if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0 && a.mixed && !stop && base_hi + mine != a.n_groups * a.k_hi)
          atomicOr(a.status, 2u /* TAHQ_DEV_BAD_BITMAP */);
      }
      if (stop) return;
      pay_off0 = (uint64_t)(C::G / 8) * ((uint64_t)a.lo * tile_cta + base_hi);
    }
    prime(s0, s1);

    int slot_i = 0;
    const uint32_t su1 = (uint32_t)(s1 - s0), seg_rel = (uint32_t)(s0 - u0) * TPU;   // (tiles)
    for (uint32_t su = warp; su < su1; su += kWarps) {   // su = unit index inside the segment
      cp_async_wait<NST - 1>();
      __syncwarp();
      if (qn >= 32u) run_flagged(32u);

      uint8_t *slot = ring + (size_t)slot_i * S::SLOT;
      const uint32_t word = s_bm[su], pre = s_pre[su];
      const uint32_t hi = (word >> lane) & 1u;
      const uint32_t hib = pre + (uint32_t)__popc(word & lt);
      const uint32_t trel0 = seg_rel + su * TPU, trel = trel0 + lane;   // relative to the CTA's first tile
      uint32_t off, len;
      const bool fits = unit_range(trel0, pre, word, off, len);
      const bool live = trel < n_rel && fits;
      const uint32_t szw = reinterpret_cast<const uint32_t *>(slot + S::PAY)[lane];
      const uint32_t pvb = live ? slot[S::PAY + 128 + lane] : 0u;
      const bool flagged = (pvb & 0x80u) != 0;
      const unsigned held = __ballot_sync(kFull, flagged);
      if (flagged) {   // Eq. 4 inverted costs three times the plain path: held back until 32 have gathered
        const uint32_t e = (qhead + qn + (uint32_t)__popc(held & lt)) & (kQueueCap - 1);
        s_q[warp][0][e] = trel;
        s_q[warp][1][e] = (hib << 1) | hi;
        s_q[warp][2][e] = szw;
        s_q[warp][3][e] = pvb;
      }
      qn += (uint32_t)__popc(held);
      if (live && !flagged) {
        const float s = __half2float(__ushort_as_half((unsigned short)(szw & 0xffffu)));
        const float z = __half2float(__ushort_as_half((unsigned short)(szw >> 16)));
        const uint8_t *codes = slot + (uint32_t)((pay_off0 + off) & 15ull) + (uint32_t)(C::G / 8) * (a.lo * lane + (hib - pre));
        float x[C::EPT];
        dequant_small<C::EPT>(codes, a.lo + hi, s, z, x);
#pragma unroll
        for (int q = 0; q < C::CPR; ++q)
          *reinterpret_cast<uint4 *>(ostage + (size_t)phys_chunk<C>(lane, q) * 16) = row_piece<C>(x, q);
      }
      __syncwarp();
      {   // the slot is free again
        const uint32_t sn = su + (uint32_t)NST * kWarps;
        if (sn < su1) issue(seg_rel + sn * TPU, sn, slot);
        cp_async_commit();
      }
      slot_i = (slot_i + 1 == NST) ? 0 : slot_i + 1;
      copy_out_unit(__ballot_sync(kFull, live && !flagged),
                    a.out + (tile_cta + trel0) * (uint64_t)C::ROWB + (size_t)lane * 16);
    }
    cp_async_wait<0>();
    __syncwarp();
    seg_hi += seg_total;
  }
  while (qn) run_flagged(qn < 32u ? qn : 32u);
}

}  // namespace tahq
