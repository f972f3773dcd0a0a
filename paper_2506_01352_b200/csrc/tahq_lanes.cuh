// Tile kernels in which a lane holds 64 bytes of the tensor (sm_100a): 32 elements of bfloat16 or 16 of binary32, so
// that a tile of 32, 64 or 128 elements belongs to 1 ... 8 neighbouring lanes.  Few values to a lane mean 80 registers
// and 24 warps on an SM (a lane that holds a whole tile needs 128 and gets 16), and the tensor moves between
// registers and memory in whole 32-byte sectors without a stage in shared memory.
//
// A warp works on "rounds" of 32 / P tiles (P lanes to a tile), the CTA's rounds dealt out over its warps one by one,
// and asks for the next round's bytes before it works on the current one.  Tiles that are transformed (Eq. 4) cost
// twice as much as the others: they are put aside, lane by lane with what the lane has loaded of them, in a queue
// of the warp in shared memory, and when a whole warp's worth has gathered they make up a round of their own.
#pragma once

#include "tahq_stream.cuh"

namespace tahq {

// one CTA per SM: the bit map in front of a CTA's tiles is counted once per SM, not once per few warps
constexpr int kLaneThreads = 768;
constexpr int kLaneWarps = kLaneThreads / 32;   // (a multiple of every P: a lane's bit in the bit-map words is fixed)

template <class C>
struct LaneCfg {
  static constexpr int E = 64 / C::ESZ;        // elements of a lane
  static constexpr int P = C::G / E;           // lanes of a tile
  static constexpr int TPR = 32 / P;           // tiles of a round
  static constexpr int TB = C::G * C::ESZ;     // bytes of a tile
  static_assert(kLaneWarps % P == 0, "a warp's rounds take the same part of their bit-map word");
};

template <bool WIDE>
__device__ __forceinline__ void store_64_bytes(uint8_t *dst, const uint32_t (&o)[16]) {
#pragma unroll
  for (int i = 0; i < 16; i += 8) {
    if constexpr (WIDE) {   // (streaming: the tensor is not read again by this library)
      asm volatile("st.global.cs.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 4 * i), "r"(o[i]),
                   "r"(o[i + 1]), "r"(o[i + 2]), "r"(o[i + 3]), "r"(o[i + 4]), "r"(o[i + 5]), "r"(o[i + 6]), "r"(o[i + 7])
                   : "memory");
    } else {                // the tensor's base is only 16-byte aligned
      __stcs(reinterpret_cast<uint4 *>(dst + 4 * i), make_uint4(o[i], o[i + 1], o[i + 2], o[i + 3]));
      __stcs(reinterpret_cast<uint4 *>(dst + 4 * i) + 1, make_uint4(o[i + 4], o[i + 5], o[i + 6], o[i + 7]));
    }
  }
}

// Words of a lane's codes.  32 codes of W bits are W whole words; 16 codes start on a half word if W is odd and the
// lane is, and lie in W / 2 words rounded up (`half`: 16 if they do, else 0).
template <int E, int NWORD>
__device__ __forceinline__ void load_codes(const uint32_t *tile, uint32_t sub, uint32_t W, uint32_t (&w)[NWORD]) {
  const uint32_t first = E == 32 ? sub * W : (sub * W) >> 1;
  const uint32_t n = E == 32 ? W : (W + 1) >> 1;
#pragma unroll
  for (int j = 0; j < NWORD; ++j) w[j] = (j < E / 16 || (uint32_t)j < n) ? __ldg(tile + first + j) : 0u;
}

// z + q*s for a lane's codes of W = 2, 3 or 4 bits (W is a lane's own value): eight codes -- W whole bytes -- are
// brought to the bottom of a word, masked where they sit and OR-ed into the mantissa of 2^23 (giving 2^23 + q*2^p
// exactly); one subtraction and one fused multiply-add with s*2^-p give the same bits as fma((float)q, s, z).
template <int E, int NWORD>
__device__ __forceinline__ void dequant_narrow_lane(const uint32_t (&w)[NWORD], uint32_t sub, uint32_t W, float s, float z,
                                                    float2 (&p)[E / 2]) {
  uint32_t g[E / 8];
  if constexpr (E == 32) {
    g[0] = w[0];
    g[1] = __funnelshift_rc(w[0], w[1], 8u * W);          // (16, 24 or 32: the clamped form shifts by a whole word)
    g[2] = __funnelshift_rc(w[1], w[2], 16u * W - 32u);   // (0, 16 or 32)
    const bool two = W == 2u;
    g[3] = __funnelshift_rc(two ? w[1] : w[2], two ? 0u : w[3], two ? 16u : 24u * W - 64u);   // (16; 8 or 32)
  } else {
    const uint32_t sh = (sub & W & 1u) * 16u;
    const uint32_t v0 = __funnelshift_r(w[0], w[1], sh), v1 = w[1] >> sh;
    g[0] = v0;
    g[1] = __funnelshift_rc(v0, v1, 8u * W);
  }
  uint32_t two23;
  asm volatile("mov.u32 %0, 0x4B000000;" : "=r"(two23));
  const float step = __uint_as_float((127u - W) << 23);   // 2^-W
  uint32_t mk[4];
  float sc[4];
  mk[0] = (1u << W) - 1u;
  sc[0] = s;
#pragma unroll
  for (int i = 1; i < 4; ++i) { mk[i] = mk[i - 1] << W; sc[i] = sc[i - 1] * step; }   // s * 2^-(W i), exact
#pragma unroll
  for (int j = 0; j < E / 8; ++j) {
    const uint32_t hi = g[j] >> (4u * W);
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      uint32_t m0, m1;
      asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(m0) : "r"(i < 4 ? g[j] : hi), "r"(mk[i & 3]), "r"(two23));
      asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(m1) : "r"(i < 4 ? g[j] : hi), "r"(mk[(i + 1) & 3]), "r"(two23));
      const float2 f = add2(f2(__uint_as_float(m0), __uint_as_float(m1)), f2(-8388608.0f));   // q * 2^p, exact
      p[4 * j + i / 2] = fma2(f, f2(sc[i & 3], sc[(i + 1) & 3]), f2(z));
    }
  }
}
template <int W, int E, int NWORD>
__device__ __forceinline__ void dequant_lane_w(const uint32_t (&w)[NWORD], uint32_t sub, float s, float z, float2 (&p)[E / 2]) {
  float x[E];
  if constexpr (E == 16 && W % 2) {
    const uint32_t sh = (sub & 1u) * 16u;
    uint32_t v[NWORD];
#pragma unroll
    for (int j = 0; j < NWORD; ++j) v[j] = __funnelshift_r(w[j], j + 1 < NWORD ? w[j + 1 < NWORD ? j + 1 : j] : 0u, sh);
    unpack_dequant<W, E>(v, s, z, x);
  } else {
    unpack_dequant<W, E>(w, s, z, x);
  }
#pragma unroll
  for (int i = 0; i < E / 2; ++i) p[i] = f2(x[2 * i], x[2 * i + 1]);
}
template <bool NARROW, int E, int NWORD>
__device__ __forceinline__ void dequant_lane(const uint32_t (&w)[NWORD], uint32_t sub, uint32_t W, float s, float z,
                                             float2 (&p)[E / 2]) {
  if constexpr (NARROW) {
    dequant_narrow_lane<E, NWORD>(w, sub, W, s, z, p);
  } else {   // wider codes: the two widths of a call are neighbours, and most calls have one
    switch (W) {
      case 4: dequant_lane_w<4, E>(w, sub, s, z, p); break;
      case 5: dequant_lane_w<5, E>(w, sub, s, z, p); break;
      case 6: dequant_lane_w<6, E>(w, sub, s, z, p); break;
      case 7: dequant_lane_w<7, E>(w, sub, s, z, p); break;
      default: dequant_lane_w<8, E>(w, sub, s, z, p); break;
    }
    __syncwarp();
  }
}

// Butterfly of Eq. 4 on a tile spread over P lanes, E elements each: strides below E inside the lane, the others
// between lanes (lower half: own + other; upper half: other - own; the products by +-1 are exact).
template <int E, int P>
__device__ __forceinline__ void butterfly_lanes(float2 (&p)[E / 2], uint32_t sub) {
  butterfly2<E / 2>(p);
#pragma unroll
  for (int h = 1; h < P; h *= 2) {
    const float2 sg = f2((sub & h) ? -1.0f : 1.0f);
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      const float2 o = f2(__shfl_xor_sync(kFull, p[i].x, h), __shfl_xor_sync(kFull, p[i].y, h));
      p[i] = fma2(p[i], sg, o);
    }
  }
}

// ------------------------------------------------------------------------------------------
// Decode (Sec. 3.3, Algorithm 1 line 5)
//
// Bound by instruction issue (0.6 per scheduler and cycle at 770 instructions per 32 tiles of 64) and, from a gibibyte
// on, half by the tensor's way to DRAM.  Against a lane per tile with the codes and rows staged in shared memory, 16
// warps per SM: 22.3 -> 18.6 us for 8192 x 4096 bf16 at 3.8 bits, 78.5 -> 74.3 us for 16384 x 5120 fp32, 323 -> 293 us
// for 65536 x 8192 bf16 with 1 % outlier channels, 12.5 -> 9.6 us for 8192 x 768 fp32, where a warp of the older
// kernel had three units of 32 tiles one after the other.  With 16 elements to a bf16 lane 22.6 us, with three
// CTAs of 8 warps per SM instead of one of 24 (each counting the bit map in front of it) 21.1 us.
// ------------------------------------------------------------------------------------------
template <class C, bool NARROW>
struct DecodeLanes {
  static constexpr int NWORD = C::BF16 ? (NARROW ? 4 : 8) : (NARROW ? 2 : 4);   // words of a lane's codes at the largest width
  // per warp: the queue of lanes put aside (two times 32: codes; scale/zero, tile, width and pivot) and the rows of a
  // round of them, where the pivot's coordinates change places
  static constexpr int WARP = 64 * (NWORD * 4 + 16) + 32 * 64;
  static constexpr int SMEM = kLaneWarps * WARP;
};

// The elements of a lane -> the tensor's type.
template <class C>
__device__ __forceinline__ void lane_words(const float2 (&p)[LaneCfg<C>::E / 2], uint32_t (&o)[16]) {
#pragma unroll
  for (int i = 0; i < LaneCfg<C>::E / 2; ++i) {
    if constexpr (C::BF16) {
      const __nv_bfloat162 h2 = __floats2bfloat162_rn(p[i].x, p[i].y);
      o[i] = *reinterpret_cast<const uint32_t *>(&h2);
    } else {
      o[2 * i] = __float_as_uint(p[i].x);
      o[2 * i + 1] = __float_as_uint(p[i].y);
    }
  }
}

// 32 lanes of the queue (the first n of them count), whole tiles with their lanes side by side: codes, the butterfly,
// coordinates 0 and d change places again, the rows leave.
template <class C, bool NARROW, bool WIDE_ST>
__device__ __forceinline__ void decode_flagged_round(const uint32_t *q_codes, const uint4 *q_info, uint4 *rows, uint32_t head,
                                                     uint32_t n, uint8_t *out_cta) {
  using D = LaneCfg<C>;
  constexpr int E = D::E, P = D::P, NWORD = DecodeLanes<C, NARROW>::NWORD;
  const uint32_t lane = threadIdx.x & 31u, sub = lane % P;
  const uint32_t at = (head + (lane < n ? lane : sub)) & 63u;
  const uint4 info = q_info[at];
  uint32_t w[NWORD];
#pragma unroll
  for (int j = 0; j < NWORD / 2; ++j) {
    const uint2 v = reinterpret_cast<const uint2 *>(q_codes)[64 * j + at];
    w[2 * j] = v.x; w[2 * j + 1] = v.y;
  }
  float s = __half2float(__ushort_as_half((unsigned short)(info.x & 0xffffu)));
  float z = __half2float(__ushort_as_half((unsigned short)(info.x >> 16)));
  // 1/sqrt(G) a power of two: scaling s and z beforehand scales every later value exactly, so the result has the
  // same bits as multiplying at the end
  constexpr bool kFold = C::G == 64 || C::G == 16;
  if (kFold) { s *= hadamard_scale<C>(); z *= hadamard_scale<C>(); }
  float2 p[E / 2];
  dequant_lane<NARROW, E>(w, sub, info.z & 15u, s, z, p);
  butterfly_lanes<E, P>(p, sub);
  if (!kFold) {
#pragma unroll
    for (int i = 0; i < E / 2; ++i) p[i] = mul2(p[i], f2(hadamard_scale<C>()));   // feeds no addition
  }
  uint32_t o[16];
  lane_words<C>(p, o);
  auto piece = [&](uint32_t l, uint32_t q) -> uint4 * { return rows + l * 4u + (q ^ ((l >> 1) & 3u)); };   // XOR-swizzled
#pragma unroll
  for (int q = 0; q < 4; ++q) *piece(lane, q) = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
  __syncwarp();
  if (sub == 0) {
    using T = typename std::conditional<C::BF16, uint16_t, uint32_t>::type;
    constexpr uint32_t EPP = 16 / C::ESZ;   // elements of a piece
    const uint32_t d = (info.z >> 4) & (C::G - 1);   // masked: a foreign buffer cannot reach outside the tile
    T *const p0 = reinterpret_cast<T *>(piece(lane, 0));
    T *const pd = reinterpret_cast<T *>(piece(lane + d / E, d % E / EPP)) + d % EPP;
    const T x0 = *p0, xd = *pd;
    *p0 = xd;
    *pd = x0;
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint4 v = *piece(lane, q);
    o[4 * q] = v.x; o[4 * q + 1] = v.y; o[4 * q + 2] = v.z; o[4 * q + 3] = v.w;
  }
  if (lane < n) store_64_bytes<WIDE_ST>(out_cta + (uint64_t)info.y * D::TB, o);
}

// MIXED: two widths in use.  With one, no offset depends on the bit map, and the codes are asked for along with the header
// (256 x 1344 fp32 at 3 bits 4.2 -> 2.0 us, 8192 x 2048 bf16 at 4 bits 11.0 -> 10.0 us), and no call needs the look-back.
template <class C, bool NARROW, bool WIDE_ST, bool MIXED>
__global__ void __launch_bounds__(kLaneThreads, 1) decode_lanes_kernel(const Args a) {
  using D = LaneCfg<C>;
  using S = DecodeLanes<C, NARROW>;
  constexpr int NT = kLaneThreads, E = D::E, P = D::P, TPR = D::TPR, NWORD = S::NWORD;
  constexpr uint32_t kTB = C::G / 8;   // bytes of a tile's codes per bit of width
  extern __shared__ __align__(128) uint8_t smem_dl[];
  __shared__ uint2 s_word[MIXED ? NT : 1];         // the segment's bit-map words, higher-width tiles of the CTA in front of each
  __shared__ uint32_t s_sum[2][32];    // per warp: set bits of its words of the segment, of its share of the words in front
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t sub = (uint32_t)lane % P;   // this lane's part of its tile
  const unsigned lt = (1u << lane) - 1u;
  uint32_t *const q_codes = reinterpret_cast<uint32_t *>(smem_dl + (size_t)warp * S::WARP);   // [NWORD / 2][64] pairs
  uint4 *const q_info = reinterpret_cast<uint4 *>(q_codes + 64 * NWORD);
  uint4 *const rows = q_info + 64;
  TraceScope trace(a.trace, 5);
  grid_dependency_wait();   // the packed buffer may be the work of the kernel in front (and so are cleared flags)
  trace.started();
  const uint32_t *bitmap = reinterpret_cast<const uint32_t *>(a.packed + a.off_bitmap);

  // the CTA's rounds, the bit-map words that hold their tiles
  const uint64_t n_rounds = (a.n_tiles + TPR - 1) / TPR;
  const uint64_t r0 = n_rounds * blockIdx.x / gridDim.x, r1 = n_rounds * (blockIdx.x + 1ull) / gridDim.x;
  const uint64_t u0 = r0 / P, u1 = (r1 + P - 1) / P;
  const uint64_t tile_cta = u0 * 32;

  // The prologue's loads -- the header, the bit-map words of the CTA's first segment, the words in front of its slice --
  // are all requested before the first barrier: one round trip to L2.
  const bool checks = blockIdx.x == 0 || a.own_prefix;
  const uint32_t hdr_w = (checks && threadIdx.x < 32) ? __ldg(reinterpret_cast<const uint32_t *>(a.packed) + threadIdx.x) : 0u;
  auto bm_word = [&](uint64_t i) -> uint32_t {   // bits beyond the last tile cleared
    const uint64_t left = a.n_tiles - i * 32;
    return __ldg(bitmap + i) & (left >= 32u ? 0xffffffffu : ((1u << (uint32_t)left) - 1u));
  };
  uint32_t word = MIXED && u0 + threadIdx.x < u1 ? bm_word(u0 + threadIdx.x) : 0u;
  uint32_t front = 0;   // a.own_prefix: this thread's share of the higher-width tiles in front of the CTA's words
  if (MIXED && a.own_prefix) {   // 128-bit loads, four in flight per thread, then the last few words one by one
    const uint4 *b4 = reinterpret_cast<const uint4 *>(bitmap);
    const uint32_t n4 = (uint32_t)(u0 / 4);
    for (uint32_t i = threadIdx.x; i < n4; i += 4u * NT) {
      uint4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = i + j * NT < n4 ? __ldg(b4 + i + j * NT) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int j = 0; j < 4; ++j) front += __popc(v[j].x) + __popc(v[j].y) + __popc(v[j].z) + __popc(v[j].w);
    }
    if (threadIdx.x < (uint32_t)(u0 & 3)) front += __popc(__ldg(bitmap + (uint64_t)n4 * 4 + threadIdx.x));
  }
  if (r0 == r1) {   // (never the first CTA, nor the last)
    bool stop;
    if (!a.own_prefix) cta_exclusive_prefix<NT>(a, 0, false, stop);
    return;
  }

  const bool wrong = checks && threadIdx.x < 32 && hdr_w != a.header[threadIdx.x];
  bool stop = false;
  uint32_t seg_hi = 0;   // higher-width tiles of this CTA's earlier segments
  uint32_t qhead = 0, qn = 0;
  const uint32_t *const sz_cta = reinterpret_cast<const uint32_t *>(a.packed + a.off_sz) + tile_cta;
  const uint8_t *const pv_cta = a.packed + a.off_pivot + tile_cta;
  uint8_t *const out_cta = a.out + tile_cta * (uint64_t)D::TB + sub * 64u;
  const uint32_t n_rel = a.n_tiles - tile_cta < 0xffffffffull ? (uint32_t)(a.n_tiles - tile_cta) : 0xffffffffu;

  const uint8_t *pay = a.packed + a.off_payload + (uint64_t)kTB * a.lo * tile_cta;   // the CTA's first code (less the higher widths' bits)
  uint32_t pay_left = 0;   // bytes of the payload from the CTA's first code (a corrupt bit map must not lead outside)
  // a warp's rounds take the same bits of their words
  uint32_t t = (uint32_t)((r0 + warp) % P) * TPR + (uint32_t)lane / P, bit = 1u << t, below = bit - 1u;
  uint32_t w[NWORD], sz, wp;   // the next round: codes; scale and zero-point; width + 16 * pivot byte, 0: no tile
  auto load = [&](uint32_t kk, uint32_t seg_tile) {   // round kk of the segment whose first word's tile `t` is seg_tile
    const uint2 bw = MIXED ? s_word[kk / P] : make_uint2(0u, 0u);
    const uint32_t tile = seg_tile + kk / P * 32u, W = a.lo + ((bw.x & bit) ? 1u : 0u);
    const uint32_t off = kTB * (a.lo * tile + bw.y + (uint32_t)__popc(bw.x & below));
    wp = 0;
    if (tile < n_rel) {
      load_codes<E, NWORD>(reinterpret_cast<const uint32_t *>(pay + off), sub, W, w);
      sz = __ldg(sz_cta + tile);
      wp = W | (uint32_t)__ldg(pv_cta + tile) << 4;
    }
  };
  if constexpr (!MIXED) {
    const uint32_t k = (uint32_t)(r0 - u0 * P) + warp;
    if (k < (uint32_t)(r1 - u0 * P)) load(k, t);
    const bool refuse = __syncthreads_or(wrong) != 0;   // every CTA for itself (a.own_prefix)
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *a.status = refuse ? 1u /* TAHQ_DEV_BAD_HEADER */ : 0u;
    if (refuse) return;
  }

  for (uint64_t s0 = u0, s1; s0 < u1; s0 = s1) {
    s1 = MIXED && s0 + NT < u1 ? s0 + NT : u1;
    uint32_t total = 0;
    if constexpr (MIXED) {
      if (s0 != u0) {
        word = s0 + threadIdx.x < u1 ? bm_word(s0 + threadIdx.x) : 0u;
        __syncthreads();   // every warp is done with the previous segment's words
      }
      // running count over the segment's words, one per thread; the words in front
      uint32_t incl = (uint32_t)__popc(word);
#pragma unroll
      for (int o = 1; o < 32; o *= 2) {
        const uint32_t v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
      }
      front = __reduce_add_sync(kFull, front);
      if (lane == 31) { s_sum[0][warp] = incl; s_sum[1][warp] = front; }
      const bool refuse = __syncthreads_or(wrong) != 0;
      const uint32_t sw = lane < kLaneWarps ? s_sum[0][lane] : 0u;
      const uint32_t before = __reduce_add_sync(kFull, lane < warp ? sw : 0u);
      total = __reduce_add_sync(kFull, sw);
      s_word[threadIdx.x] = make_uint2(word, seg_hi + before + incl - (uint32_t)__popc(word));
      if (s0 == u0) {   // Sec. 3.4: higher-width tiles in front of the CTA's words; what was found in the header
        // CTA 0 compares the received header with the one these parameters produce; what it finds travels with the
        // offset prefix, so a refused buffer leaves the output untouched.  (a.own_prefix: every CTA does this itself
        // and counts the bit map in front of its slice itself: nothing has to be cleared beforehand, and the last CTA,
        // which sees the whole count, writes the status.)
        const bool last = blockIdx.x == gridDim.x - 1 && threadIdx.x == 0;
        uint64_t base_hi;
        if (a.own_prefix) {
          base_hi = __reduce_add_sync(kFull, lane < kLaneWarps ? s_sum[1][lane] : 0u);
          stop = refuse;
          uint32_t rest = 0;   // (a device of fewer than 86 SMs: words of the CTA's later segments)
          if (s1 < u1) {
            for (uint64_t i = s1 + threadIdx.x; i < u1; i += NT) rest += __popc(bm_word(i));
            rest = block_sum<NT>(rest);
          }
          if (last)
            *a.status = (refuse ? 1u /* TAHQ_DEV_BAD_HEADER */ : 0u) |
                        ((!refuse && base_hi + total + rest != a.n_groups * a.k_hi) ? 2u /* TAHQ_DEV_BAD_BITMAP */ : 0u);
        } else {
          // a CTA publishes the count of the words that start in its range (one shared by two CTAs counts in the first)
          if (refuse && threadIdx.x == 0) atomicOr(a.status, 1u);
          const uint64_t uc0 = (r0 + P - 1) / P;
          uint32_t n = 0;
          for (uint64_t i = uc0 + threadIdx.x; i < u1; i += NT) n += __popc(bm_word(i));
          n = block_sum<NT>(n);
          base_hi = cta_exclusive_prefix<NT>(a, n, refuse, stop);
          if (last && !stop && base_hi + n != a.n_groups * a.k_hi) atomicOr(a.status, 2u);
          if (uc0 != u0) base_hi -= (uint32_t)__popc(bm_word(u0));
        }
        const uint64_t pay0 = (uint64_t)kTB * ((uint64_t)a.lo * tile_cta + base_hi);
        if (pay0 < a.payload_bytes) {
          pay += (uint64_t)kTB * base_hi;
          pay_left = a.payload_bytes - pay0 < 0xffffffffull ? (uint32_t)(a.payload_bytes - pay0) : 0xffffffffu;
        }
      }
      __syncthreads();
      if (stop) return;
      // does the segment's last code lie inside the payload?  If not, the bit map is corrupt and the rest is left out.
      const uint32_t tiles = (uint32_t)(s1 - u0) * 32u;
      if ((uint64_t)kTB * ((uint64_t)a.lo * (tiles < n_rel ? tiles : n_rel) + seg_hi + total) > pay_left) return;
    }

    // the warp's rounds
    const uint64_t rs0 = s0 * P > r0 ? s0 * P : r0, rs1 = s1 * P < r1 ? s1 * P : r1;
    const uint32_t k1 = (uint32_t)(rs1 - s0 * P);
    uint32_t k = (uint32_t)(rs0 - s0 * P) + warp;
    if (MIXED) { t = k % P * TPR + (uint32_t)lane / P; bit = 1u << t; below = bit - 1u; }
    const uint32_t seg_tile = (uint32_t)(s0 - u0) * 32u + t;   // from the CTA's first
    if (MIXED && k < k1) load(k, seg_tile);
    for (; k < k1; k += kLaneWarps) {
      uint32_t cw[NWORD];
#pragma unroll
      for (int j = 0; j < NWORD; ++j) cw[j] = w[j];
      const uint32_t csz = sz, cwp = wp, tile = seg_tile + k / P * 32u;
      if (k + kLaneWarps < k1) load(k + kLaneWarps, seg_tile);
      const bool flagged = (cwp & 0x800u) != 0;
      const unsigned held = __ballot_sync(kFull, flagged);
      if (flagged) {   // put aside
        const uint32_t at = (qhead + qn + (uint32_t)__popc(held & lt)) & 63u;
#pragma unroll
        for (int j = 0; j < NWORD / 2; ++j) reinterpret_cast<uint2 *>(q_codes)[64 * j + at] = make_uint2(cw[2 * j], cw[2 * j + 1]);
        q_info[at] = make_uint4(csz, tile, cwp, 0u);
      }
      qn += (uint32_t)__popc(held);
      if (held != kFull) {
        const float s = __half2float(__ushort_as_half((unsigned short)(csz & 0xffffu)));
        const float z = __half2float(__ushort_as_half((unsigned short)(csz >> 16)));
        float2 p[E / 2];
        dequant_lane<NARROW, E>(cw, sub, cwp & 15u, s, z, p);
        uint32_t o[16];
        lane_words<C>(p, o);
        if (cwp != 0u && !flagged) store_64_bytes<WIDE_ST>(out_cta + (uint64_t)tile * D::TB, o);
      }
      if (qn >= 32u) {
        __syncwarp();
        decode_flagged_round<C, NARROW, WIDE_ST>(q_codes, q_info, rows, qhead, 32u, out_cta);
        qhead = (qhead + 32u) & 63u;
        qn -= 32u;
        __syncwarp();
      }
    }
    seg_hi += total;
  }
  __syncwarp();
  if (qn) decode_flagged_round<C, NARROW, WIDE_ST>(q_codes, q_info, rows, qhead, qn, out_cta);
}

// A lane's 64 bytes of the tensor, aligned to 16 or (WIDE) 32 bytes.
template <bool WIDE>
__device__ __forceinline__ void load_64_bytes(const uint8_t *src, uint32_t (&w)[16]) {
  if constexpr (WIDE) {
#pragma unroll
    for (int i = 0; i < 16; i += 8)
      asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=r"(w[i]), "=r"(w[i + 1]), "=r"(w[i + 2]), "=r"(w[i + 3]), "=r"(w[i + 4]), "=r"(w[i + 5]), "=r"(w[i + 6]),
                     "=r"(w[i + 7])
                   : "l"(src + 4 * i));
  } else {
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
      const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src + 4 * i));
      w[i] = v.x; w[i + 1] = v.y; w[i + 2] = v.z; w[i + 3] = v.w;
    }
  }
}

// ------------------------------------------------------------------------------------------
// Eq. 1-2, screening scores (see tile_score_screen for the formula and its error)
// ------------------------------------------------------------------------------------------
constexpr int kScoreThreads = 512;   // two CTAs on an SM

// For bfloat16.  Bound by DRAM, with the logarithms (one MUFU instruction per element, 16 lanes a cycle and SM) close
// behind: what counts is that both run at once.  With a lane per tile, rows in shared memory and 8 warps on an SM they took
// turns: 8192 x 4096 15.4 -> 14.5 us, 65536 x 8192 201 -> 188 us, 4096 x 4096 in tiles of 128 8.4 -> 7.1 us, 16384 x 8192 in
// tiles of 32 57.4 -> 49.1 us.  Two rounds ahead instead of one, or three CTAs of 384 threads, are no faster; binary32,
// whose lanes lie 64 bytes apart at half the elements, is slower this way (33 MB 4.7 -> 7.4 us) and keeps score_kernel.
template <class C, bool WIDE>
__global__ void __launch_bounds__(kScoreThreads, 2) score_lanes_kernel(const Args a) {
  using D = LaneCfg<C>;
  static_assert(C::BF16, "binary32: score_kernel");
  constexpr int P = D::P, TPR = D::TPR;
  constexpr uint32_t WARPS = kScoreThreads / 32;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, sub = lane % P;
  TraceScope trace(a.trace, 1);
  const uint32_t n_tiles = (uint32_t)a.n_tiles, n_rounds = (n_tiles + TPR - 1) / TPR;
  const uint32_t r0 = (uint32_t)((uint64_t)n_rounds * blockIdx.x / gridDim.x);
  // The CTA's rounds are read back to front: the rows read last are the ones the encoder, which walks the tensor front to
  // back right afterwards, asks for first, while they are still in L2.
  const uint32_t r1 = (uint32_t)((uint64_t)n_rounds * (blockIdx.x + 1u) / gridDim.x);
  uint32_t raw[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) raw[i] = 0;
  auto load = [&](uint32_t r) {
    const uint32_t tile = r * TPR + lane / P;
    if (tile < n_tiles) load_64_bytes<WIDE>(a.in + (uint64_t)tile * D::TB + sub * 64u, raw);
  };
  grid_dependency_wait();   // the tensor may be the work of the kernel in front
  trace.started();
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.status = 0;   // nothing else of the workspace has to start at zero
  const uint32_t left0 = r1 - r0 > warp ? r1 - r0 - warp : 0u;
  uint32_t left = left0;   // the warp's next round is r0 + left - 1
  uint32_t range = 0;      // see screen_range
  if (left) load(r0 + left - 1u);
  while (left) {
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] = raw[i];
    const uint32_t r = r0 + left - 1u;
    left = left > WARPS ? left - WARPS : 0u;
    if (left) load(r0 + left - 1u);
    const float tiny = 1e-30f;
    constexpr int NP = D::E / 2, NC = 4;   // pairs; chains that sum them
    float2 L[NC], T[NC];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      float2 v;
      bf2_add_f32(w[i] & 0x7fff7fffu, tiny, v.x, v.y);
      const float2 l = f2(lg2_approx(v.x), lg2_approx(v.y));
      const int c = i % NC;
      if (i < NC) {
        L[c] = v;
        T[c] = f2(v.x * l.x, v.y * l.y);   // (scalar products: they feed the fused chain's addend)
      } else {
        L[c] = add2(L[c], v);
        T[c] = fma2(v, l, T[c]);
      }
    }
    const float2 L2 = add2(add2(L[0], L[1]), add2(L[2], L[3])), T2 = add2(add2(T[0], T[1]), add2(T[2], T[3]));
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
    const uint32_t tile = r * TPR + lane / P;
    if (sub == 0 && tile < n_tiles) a.scores[tile] = __fmaf_rn(lg2_approx(Lp), Ls, -Ts) * rc;
  }
  if (__any_sync(kFull, range > kScreenRange))
    for (left = left0; left; left = left > WARPS ? left - WARPS : 0u) {
      const uint32_t tile = (r0 + left - 1u) * TPR;
      exact_scores_of<C::G / 8, C::BF16>(a.in + (uint64_t)tile * D::TB, n_tiles - tile < TPR ? n_tiles - tile : TPR, a.eps_l1,
                                                a.eps_log, a.scores + tile, nullptr);
    }
}

// ------------------------------------------------------------------------------------------
// Quantise + pack (Eq. 3-4, Sec. 3.3-3.4)
//
// The quantiser of a tile and everything about its place are worked out by each of its lanes, and the butterfly crosses
// lanes by shuffles, so this kernel issues more instructions per tile than quant2_kernel, where a lane owns a tile (1190
// against 850 per 32 tiles of 64 bf16).  What it gains: 20 or 24 warps on an SM, no ring of slots to fill, and a warp's
// work comes in pieces of half a unit and less.  Binary32, where a tile fills 256 bytes and quant2_kernel has 8 warps on an
// SM: 12.2 -> 9.3 us for 8192 x 768, 28.2 -> 23.1 us for 10240 x 2240, 82 -> 78 us for 16384 x 6720.  For bf16 see
// quant_lanes_pays.
// ------------------------------------------------------------------------------------------
template <class C>
struct QuantLanes {
  static constexpr int NT = C::BF16 ? 640 : 768, WARPS = NT / 32;   // (32 elements to a lane need more registers than 16)
  static_assert(WARPS % LaneCfg<C>::P == 0, "a warp's rounds take the same part of their bit-map word");
  // per warp: the queue of lanes put aside, two times 32: their 64 bytes in four pieces; where the tile's codes go, tile
  // and width
  static constexpr int WARP = 64 * (64 + 8);
  static constexpr int SMEM = WARPS * WARP;
};

// Codes of a lane -> the tile's bit stream.  t(k) = q_k + 1.5*2^23 for a compile-time k; `dst` = the tile's first word.
// 16 codes of an odd width end in the middle of a word, which the lane shares with its neighbour: the even lane of the
// pair stores it.  All lanes of a warp call this; `mine`: the lane stores.
template <int E, bool NARROW, class F>
__device__ __forceinline__ void pack_lane(F &&t, uint32_t W, uint32_t sub, uint32_t *dst, bool mine) {
  if constexpr (NARROW) {   // the width is a lane's own value of 2, 3 or 4: see pack_store_narrow
    constexpr int NG = E / 8;
    constexpr uint32_t K2 = (uint32_t)((0x4B400000ull * group_ones(2, 8)) & 0xffffffffull);
    constexpr uint32_t K3 = (uint32_t)((0x4B400000ull * group_ones(3, 8)) & 0xffffffffull);
    constexpr uint32_t K4 = (uint32_t)((0x4B400000ull * group_ones(4, 8)) & 0xffffffffull);
    const bool four = W == 4u, three = W == 3u;
    uint32_t M = four ? 16u : three ? 8u : 4u;
    asm volatile("mov.u32 %0, %0;" : "+r"(M));   // opaque to the optimiser: keeps the multiply
    const uint32_t KW = four ? K4 : three ? K3 : K2;
    uint32_t g[NG];
#pragma unroll
    for (int j = 0; j < NG; ++j) {   // eight codes, W whole bytes
      uint32_t acc = __float_as_uint(t(8 * j + 7));
#pragma unroll
      for (int i = 6; i >= 0; --i) acc = acc * M + __float_as_uint(t(8 * j + i));
      g[j] = acc - KW;
    }
    const uint32_t s0 = four ? 0x3210u : three ? 0x4210u : 0x5410u;   // the first group, then bytes of the second
    if constexpr (E == 32) {
      const bool two = W == 2u;
      const uint32_t w0 = __byte_perm(g[0], g[1], s0);
      const uint32_t w1 = __byte_perm(two ? g[2] : g[1], two ? g[3] : g[2], four ? 0x3210u : three ? 0x5421u : 0x5410u);
      const uint32_t w2 = __byte_perm(g[2], g[3], four ? 0x3210u : 0x6542u);
      dst += sub * W;
      const uint32_t n = mine ? W : 0u;   // (four stores under conditions of their own: no branches)
      if (n > 0u) dst[0] = w0;
      if (n > 1u) dst[1] = w1;
      if (n > 2u) dst[2] = w2;
      if (n > 3u) dst[3] = g[3];
    } else {
      uint32_t v0 = __byte_perm(g[0], g[1], s0), v1 = three ? g[1] >> 8 : g[1];
      const uint32_t o = __shfl_xor_sync(kFull, v0, 1);
      const bool odd = sub & 1u;
      if (three) {
        if (odd) v0 = __funnelshift_r(v0, v1, 16);
        else v1 |= o << 16;
      }
      dst += (sub * W + 1u) >> 1;
      if (mine) dst[0] = v0;
      if (mine && (four || (three && !odd))) dst[1] = v1;
    }
  } else {
    // The lanes that take the branch of the odd width below: the two widths of a call are neighbours, so it is one branch.
    // (Asked for here, where the warp is together: in there a lane cannot know who else is.)
    const unsigned odd_width = __ballot_sync(kFull, (W & 1u) != 0u);
    auto width = [&](auto wc) {
      constexpr int CW = decltype(wc)::value, NW = (E * CW + 31) / 32;
      uint32_t w[NW + 1];
      w[NW] = 0;
      {
        uint32_t v[E * CW % 32 ? 2 * NW : NW];   // (pack_magic writes whole words)
        if constexpr (E * CW % 32) {
          float z[32];
#pragma unroll
          for (int k = 0; k < 32; ++k) z[k] = k < E ? t(k < E ? k : 0) : kMagic;
          pack_magic<CW, 32>([&](int k) { return z[k]; }, v);
        } else {
          pack_magic<CW, E>(t, v);
        }
#pragma unroll
        for (int j = 0; j < NW; ++j) w[j] = v[j];
      }
      const uint32_t first = E == 32 ? sub * (uint32_t)CW : (sub * (uint32_t)CW + 1u) >> 1;
      uint32_t n = NW;
      if constexpr (E * CW % 32) {
        const uint32_t o = __shfl_xor_sync(odd_width, w[0], 1);   // (the neighbour has the same width)
        if (sub & 1u) {
#pragma unroll
          for (int j = 0; j < NW; ++j) w[j] = __funnelshift_r(w[j], w[j + 1], 16);
          n = NW - 1;
        } else {
          w[NW - 1] |= o << 16;
        }
      }
      if (mine)
#pragma unroll
        for (int j = 0; j < NW; ++j)
          if ((uint32_t)j < n) dst[first + j] = w[j];
    };
    switch (W) {   // (the lower width is at least 4 here)
      case 4: width(std::integral_constant<int, 4>{}); break;
      case 5: width(std::integral_constant<int, 5>{}); break;
      case 6: width(std::integral_constant<int, 6>{}); break;
      case 7: width(std::integral_constant<int, 7>{}); break;
      default: width(std::integral_constant<int, 8>{}); break;
    }
    __syncwarp();
  }
}

// Where things of one tile go; the lower width, and what depends on it, for it and the next width.
struct QuantOut {
  uint32_t *payload, *sz;
  uint8_t *pivot;
  uint32_t lo;
  WidthConst wc;
};

// Codes from the differences to the zero-point: pair(i) = (x[2i] - z, x[2i+1] - z) for a compile-time i.  mn, mx: the
// range of the tile.  All lanes of a warp call this; `mine`: the lane has a tile to store.
template <class C, bool SR, bool NARROW, class F>
__device__ __forceinline__ void quantise_pack_lane(F &&pair, float mn, float mx, const Quantiser &q, uint32_t W, uint32_t sub,
                                                   uint32_t *dst, bool mine, unsigned long long seed, unsigned long long first) {
  constexpr int E = LaneCfg<C>::E;
  if constexpr (SR) {
    float d[E];
#pragma unroll
    for (int i = 0; i < E / 2; ++i) { const float2 p = pair(i); d[2 * i] = p.x; d[2 * i + 1] = p.y; }
    stochastic_codes<E>(d, q.inv_s, q.qmax, seed, first);
    pack_lane<E, NARROW>([&](int k) { return d[k]; }, W, sub, dst, mine);
  } else {
    // the clamp is left out when the whole warp's tiles provably stay inside: see quantise_pairs
    const float ymin = (mn - q.z) * q.inv_s, ymax = (mx - q.z) * q.inv_s;
    const bool safe = !mine || (ymin >= -0.4999f && ymax < q.qmax + 0.4999f);
    const float2 is = f2(q.inv_s), mg = f2(kMagic);
    if (__all_sync(kFull, safe)) {   // (the codes are formed where the packing asks for them)
      pack_lane<E, NARROW>([&](int k) { const float2 t = fma2(pair(k >> 1), is, mg); return (k & 1) ? t.y : t.x; }, W, sub, dst, mine);
    } else {
      const float top = kMagic + q.qmax;
      pack_lane<E, NARROW>([&](int k) {
        const float2 t = fma2(pair(k >> 1), is, mg);
        return fminf(fmaxf((k & 1) ? t.y : t.x, kMagic), top);
      }, W, sub, dst, mine);
    }
  }
}

// Smallest and largest element of the lane's 64 bytes.
template <class C>
__device__ __forceinline__ void lane_minmax(const uint32_t (&w)[16], float &mn, float &mx) {
  if constexpr (C::BF16) {
    uint32_t lo = bf2_min(bf2_min(w[0], w[1]), w[2]), hi = bf2_max(bf2_max(w[0], w[1]), w[2]);
    uint32_t lo2 = bf2_min(bf2_min(w[3], w[4]), w[5]), hi2 = bf2_max(bf2_max(w[3], w[4]), w[5]);
#pragma unroll
    for (int j = 6; j < 14; j += 4) {
      lo = bf2_min(bf2_min(lo, w[j]), w[j + 1]); hi = bf2_max(bf2_max(hi, w[j]), w[j + 1]);
      lo2 = bf2_min(bf2_min(lo2, w[j + 2]), w[j + 3]); hi2 = bf2_max(bf2_max(hi2, w[j + 2]), w[j + 3]);
    }
    lo = bf2_min(bf2_min(lo, w[14]), w[15]); hi = bf2_max(bf2_max(hi, w[14]), w[15]);
    lo = bf2_min(lo, lo2); hi = bf2_max(hi, hi2);
    mn = fminf(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u));
    mx = fmaxf(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
  } else {
    mn = __uint_as_float(w[0]);
    mx = mn;
    float mn2 = __uint_as_float(w[1]), mx2 = mn2;
#pragma unroll
    for (int j = 2; j < 16; j += 2) {
      mn = fminf(mn, __uint_as_float(w[j])); mx = fmaxf(mx, __uint_as_float(w[j]));
      mn2 = fminf(mn2, __uint_as_float(w[j + 1])); mx2 = fmaxf(mx2, __uint_as_float(w[j + 1]));
    }
    mn = fminf(mn, mn2);
    mx = fmaxf(mx, mx2);
  }
}

// Largest and second-largest magnitude of the lane's 64 bytes.
template <class C>
__device__ __forceinline__ void lane_top2(const uint32_t (&w)[16], float &a1, float &a2) {
  if constexpr (C::BF16) {
    uint32_t p1 = 0, p2 = 0, q1 = 0, q2 = 0;   // two independent (largest, second) pairs per 16-bit half
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
      p2 = bf2_max_abs(p2, bf2_min_abs(p1, w[j])); p1 = bf2_max_abs(p1, w[j]);
      q2 = bf2_max_abs(q2, bf2_min_abs(q1, w[j + 1])); q1 = bf2_max_abs(q1, w[j + 1]);
    }
    const uint32_t m1 = bf2_max_abs(p1, q1) & 0x7fff7fffu;
    const uint32_t m2 = bf2_max_abs(bf2_min_abs(p1, q1), bf2_max_abs(p2, q2)) & 0x7fff7fffu;
    const uint32_t e1 = m1 & 0xffffu, o1 = m1 >> 16, e2 = m2 & 0xffffu, o2 = m2 >> 16;
    a1 = __uint_as_float(max(e1, o1) << 16);
    a2 = __uint_as_float(max(min(e1, o1), max(e2, o2)) << 16);
  } else {
    float p1 = 0.0f, p2 = 0.0f, q1 = 0.0f, q2 = 0.0f;
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
      const float t0 = fabsf(__uint_as_float(w[j])), t1 = fabsf(__uint_as_float(w[j + 1]));
      p2 = fmaxf(p2, fminf(p1, t0)); p1 = fmaxf(p1, t0);
      q2 = fmaxf(q2, fminf(q1, t1)); q1 = fmaxf(q1, t1);
    }
    a1 = fmaxf(p1, q1);
    a2 = fmaxf(fminf(p1, q1), fmaxf(p2, q2));
  }
}

// Elements 2i and 2i+1 of the lane's 64 bytes, plus c.
template <class C>
__device__ __forceinline__ float2 lane_pair_plus(const uint32_t (&w)[16], int i, float c) {
  float2 d;
  if constexpr (C::BF16) bf2_add_f32(w[i], c, d.x, d.y);
  else d = add2(f2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1])), f2(c));
  return d;
}

// 32 lanes of the queue (the first n of them count), whole tiles with their lanes side by side: the exact pivot test
// (Eq. 3), the pivot swap in shared memory, the butterfly (Eq. 4), range, codes, bit stream.
template <class C, bool SR, bool NARROW>
__device__ __forceinline__ void encode_queued_round(float tau, float eps_ratio, uint4 *q_raw, const uint2 *q_info, uint32_t head,
                                                    uint32_t n, const QuantOut &out, unsigned long long seed) {
  using D = LaneCfg<C>;
  constexpr int E = D::E, P = D::P, EPC = 16 / C::ESZ;   // EPC: elements of a 16-byte piece
  const uint32_t lane = threadIdx.x & 31u, sub = lane % P;
  const uint32_t slot = (head + (lane < n ? lane : sub)) & 63u;
  const uint2 info = q_info[slot];
  uint32_t w[16];
  auto fetch = [&]() {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 v = q_raw[64 * q + slot];
      w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
    }
  };
  fetch();
  float a1, a2;
  lane_top2<C>(w, a1, a2);
#pragma unroll
  for (int h = 1; h < P; h *= 2) {
    const float o1 = __shfl_xor_sync(kFull, a1, h), o2 = __shfl_xor_sync(kFull, a2, h);
    a2 = fmaxf(fminf(a1, o1), fmaxf(a2, o2));
    a1 = fmaxf(a1, o1);
  }
  const float t1 = a2 + eps_ratio;
  const float t2 = tau * t1;
  const bool flag = a1 > t2;   // Eq. 3
  // the first position of the largest magnitude: the lane's first piece that holds it, its first element in there
  uint32_t d = 0xffu;
  {
    int hit = -1;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
      bool here;
      if constexpr (C::BF16) {
        const uint32_t t = bf2_max_abs(bf2_max_abs(w[4 * q], w[4 * q + 1]), bf2_max_abs(w[4 * q + 2], w[4 * q + 3])) & 0x7fff7fffu;
        here = max(t & 0xffffu, t >> 16) == __float_as_uint(a1) >> 16;
      } else {
        here = fmaxf(fmaxf(fabsf(__uint_as_float(w[4 * q])), fabsf(__uint_as_float(w[4 * q + 1]))),
                     fmaxf(fabsf(__uint_as_float(w[4 * q + 2])), fabsf(__uint_as_float(w[4 * q + 3])))) == a1;
      }
      hit = here ? q : hit;
    }
    if (hit >= 0) {
      const uint4 v = q_raw[64 * hit + slot];
      const uint32_t u[4] = {v.x, v.y, v.z, v.w};
      uint32_t kk = EPC - 1;
#pragma unroll
      for (int j = 3; j >= 0; --j) {
        if constexpr (C::BF16) {
          kk = ((u[j] >> 16) & 0x7fffu) == __float_as_uint(a1) >> 16 ? 2 * j + 1 : kk;
          kk = (u[j] & 0x7fffu) == __float_as_uint(a1) >> 16 ? 2 * j : kk;
        } else {
          kk = fabsf(__uint_as_float(u[j])) == a1 ? j : kk;
        }
      }
      d = sub * E + hit * EPC + kk;
    }
#pragma unroll
    for (int h = 1; h < P; h *= 2) d = min(d, __shfl_xor_sync(kFull, d, h));
  }
  __syncwarp();
  if (flag && sub == 0 && lane < n) {   // Eq. 4: the pivot swap P_d
    using T = typename std::conditional<C::BF16, uint16_t, uint32_t>::type;
    T *const p0 = reinterpret_cast<T *>(q_raw + slot);
    T *const pd = reinterpret_cast<T *>(q_raw + 64 * (d % E / EPC) + ((slot + d / E) & 63u)) + d % EPC;
    const T x0 = *p0, xd = *pd;
    *p0 = xd;
    *pd = x0;
  }
  __syncwarp();
  fetch();
  float2 p[E / 2];
  auto widen = [&]() {
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      if constexpr (C::BF16) p[i] = lane_pair_plus<C>(w, i, -0.0f);
      else p[i] = f2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1]));
    }
  };
  widen();
  // Eq. 4: (1/sqrt G) H_G.  For G = 64 the factor is a power of two: the products are exact, so the
  // factor is applied to the range and inside the quantiser's subtraction instead of element by element.
  constexpr bool kFold = C::G == 64;
  butterfly_lanes<E, P>(p, sub);   // (nearly every tile of the queue is flagged: all lanes go through it)
  if (!kFold) {
#pragma unroll
    for (int i = 0; i < E / 2; ++i)   // scalar products: they are added to right after
      p[i] = f2(p[i].x * hadamard_scale<C>(), p[i].y * hadamard_scale<C>());
  }
  if (!flag) {
    fetch();
    widen();
  }
  float mn = fminf(p[0].x, p[0].y), mx = fmaxf(p[0].x, p[0].y);
#pragma unroll
  for (int i = 1; i < E / 2; ++i) {
    mn = fminf(mn, fminf(p[i].x, p[i].y));
    mx = fmaxf(mx, fmaxf(p[i].x, p[i].y));
  }
#pragma unroll
  for (int h = 1; h < P; h *= 2) {
    mn = fminf(mn, __shfl_xor_sync(kFull, mn, h));
    mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, h));
  }
  const float pre = (kFold && flag) ? hadamard_scale<C>() : 1.0f;
  mn *= pre;
  mx *= pre;
  const bool hi = (info.y & 1u) != 0u;
  const uint64_t tile = info.y >> 1;
  const Quantiser q = make_quantiser(mn, mx, 0u, hi, out.wc);
  const float2 nz = f2(-q.z), pr = f2(pre);
  // (pre * x) - z as one fused multiply-add: the product is exact
  quantise_pack_lane<C, SR, NARROW>([&](int i) { return fma2(p[i], pr, nz); }, mn, mx, q, out.lo + (hi ? 1u : 0u), sub,
                                    out.payload + (uint64_t)(C::G / 32) * info.x, lane < n, seed,
                                    tile * (unsigned long long)C::G + sub * E);
  if (lane < n && sub == 0) {
    out.sz[tile] = q.sz;
    out.pivot[tile] = flag ? (uint8_t)(0x80u | d) : (uint8_t)0;
  }
}

template <class C, bool SR, bool NARROW, bool WIDE>
__global__ void __launch_bounds__(QuantLanes<C>::NT, 1) quant_lanes_kernel(const Args a) {
  using D = LaneCfg<C>;
  constexpr int E = D::E, P = D::P, TPR = D::TPR, WARPS = QuantLanes<C>::WARPS;
  extern __shared__ __align__(128) uint8_t smem_ql[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t sub = (uint32_t)lane % P;   // this lane's part of its tile
  const unsigned lt = (1u << lane) - 1u;
  uint4 *const q_raw = reinterpret_cast<uint4 *>(smem_ql + (size_t)warp * QuantLanes<C>::WARP);   // [4][64]
  uint2 *const q_info = reinterpret_cast<uint2 *>(q_raw + 4 * 64);
  TraceScope trace(a.trace, 3);
  grid_dependency_wait();   // bit map and running counts are the selection kernel's; the tensor may be a kernel's too
  trace.started();
  uint32_t *const bitmap = reinterpret_cast<uint32_t *>(a.packed + a.off_bitmap);
  const uint32_t n_tiles = (uint32_t)a.n_tiles, lo = a.lo;   // (at most 2^26)
  const QuantOut out = {reinterpret_cast<uint32_t *>(a.packed + a.off_payload), reinterpret_cast<uint32_t *>(a.packed + a.off_sz),
                        a.packed + a.off_pivot, lo, WidthConst(lo)};

  // the CTA's rounds, dealt out over its warps; a lane's tile always has the same bit in its bit-map word
  const uint32_t n_rounds = (n_tiles + TPR - 1) / TPR;
  const uint32_t r1 = (uint32_t)((uint64_t)n_rounds * (blockIdx.x + 1u) / gridDim.x);
  uint32_t r = (uint32_t)((uint64_t)n_rounds * blockIdx.x / gridDim.x) + warp;
  const uint32_t bit = r % P * TPR + (uint32_t)lane / P, below = (1u << bit) - 1u;
  uint32_t raw[16], word = 0, before = 0;   // the next round: 64 bytes of the tile; its bit-map word, higher-width tiles in front
  auto load = [&](uint32_t k) {
    const uint32_t tile = k / P * 32u + bit;
    if (tile < n_tiles) load_64_bytes<WIDE>(a.in + (uint64_t)tile * D::TB + sub * 64u, raw);
    if (a.mixed) { word = __ldg(bitmap + k / P); before = __ldg(a.pre + k / P); }
  };
#pragma unroll
  for (int i = 0; i < 16; ++i) raw[i] = 0;
  if (r < r1) load(r);

  if (blockIdx.x == 0) {   // header and the zero padding behind every section
    if (threadIdx.x == 0 && !a.mixed) *a.status = 0;   // (with two widths in use the score kernel has done it)
    if (threadIdx.x < 32) reinterpret_cast<uint32_t *>(a.packed)[threadIdx.x] = a.header[threadIdx.x];
    for (int s = 0; s < 4; ++s) {
      const uint64_t from = s == 0 ? a.off_bitmap + 4 * ((a.n_tiles + 31) / 32) : s == 1 ? a.off_sz + 4 * a.n_tiles
                          : s == 2 ? a.off_pivot + a.n_tiles : a.off_payload + a.payload_bytes;
      const uint64_t to = s == 0 ? a.off_sz : s == 1 ? a.off_pivot : s == 2 ? a.off_payload : a.total_bytes;
      for (uint64_t o = from + threadIdx.x; o < to; o += QuantLanes<C>::NT) a.packed[o] = 0;
    }
  }

  uint32_t qhead = 0, qn = 0;
  while (r < r1 || qn) {   // (one place for the queue's rounds: the last, partly filled one is run behind the others)
    if (r < r1) {
      uint32_t w[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) w[i] = raw[i];
      const uint32_t hi = (word >> bit) & 1u, tile = r / P * 32u + bit;
      const uint32_t n8 = lo * tile + before + (uint32_t)__popc(word & below);   // the tile's codes start G/8 times this many bytes in
      if (r + WARPS < r1) load(r + WARPS);
      if (!a.mixed && lane == 0 && r % P == 0) bitmap[r / P] = 0;
      const bool live = tile < n_tiles;

      // Eq. 3, first look: the second-largest magnitude is at least the smaller of |min| and |max| (they
      // sit at different positions, or every element is equal), so a tile whose largest magnitude does
      // not exceed tau * (that + varrho) cannot be flagged.  The others are put aside for the exact test.
      float mn, mx;
      lane_minmax<C>(w, mn, mx);
#pragma unroll
      for (int h = 1; h < P; h *= 2) {
        mn = fminf(mn, __shfl_xor_sync(kFull, mn, h));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, h));
      }
      const float m_big = fmaxf(fabsf(mn), fabsf(mx)), m_small = fminf(fabsf(mn), fabsf(mx));
      const bool maybe = live && m_big > a.tau * (m_small + a.eps_ratio);
      const unsigned held = __ballot_sync(kFull, maybe);
      if (maybe) {
        const uint32_t at = (qhead + qn + (uint32_t)__popc(held & lt)) & 63u;
#pragma unroll
        for (int q = 0; q < 4; ++q) q_raw[64 * q + at] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
        q_info[at] = make_uint2(n8, (tile << 1) | hi);
      }
      qn += (uint32_t)__popc(held);
      if (held != kFull) {
        const bool mine = live && !maybe;
        const Quantiser q = make_quantiser(mn, mx, 0u, hi != 0u, out.wc);
        const float nz = -q.z;   // x + (-z) is x - z
        quantise_pack_lane<C, SR, NARROW>([&](int i) { return lane_pair_plus<C>(w, i, nz); }, mn, mx, q, lo + hi, sub,
                                          out.payload + (uint64_t)(C::G / 32) * n8, mine, a.seed,
                                          tile * (unsigned long long)C::G + sub * E);
        if (mine && sub == 0) {
          out.sz[tile] = q.sz;
          out.pivot[tile] = 0;
        }
      }
      r += WARPS;
    }
    if (qn >= 32u || (r >= r1 && qn)) {
      const uint32_t n = qn < 32u ? qn : 32u;
      __syncwarp();
      encode_queued_round<C, SR, NARROW>(a.tau, a.eps_ratio, q_raw, q_info, qhead, n, out, a.seed);
      qhead = (qhead + n) & 63u;
      qn -= n;
      __syncwarp();
    }
  }
}

// Binary32 always; bfloat16 while the time is that of a warp's chain and not of the instructions: up to two rounds to a warp,
// and one where quant2_kernel is at its best (tiles of 64, widths up to 4 bits, rounding to nearest).  Encode, us, with
// quant2_kernel / with this one, at one, two and three rounds to a warp of 20 on 148 SMs:
//   tiles of 64     3.8 bits 16.3/15.8 19.3/19.5 22.4/25.1   6.8 bits 18.5/17.0 22.3/20.8 25.2/27.2   stochastic 22.2/20.6 28.6/26.6 33.8/37.0
//   tiles of 128    3.8 bits 16.5/15.6 21.2/20.9 25.3/24.8   6.8 bits 19.7/16.6 24.7/22.2 28.4/26.8   stochastic 23.5/20.7 34.2/30.7 40.4/37.0
//   tiles of 32     3.8 bits 18.5/18.5 21.9/22.1 27.8/26.9   6.8 bits 20.2/19.8 24.4/24.1 30.2/29.6   stochastic 22.4/23.3 28.0/29.4 38.4/36.3
// Tiles of 32 are even (within 5 % either way) and follow the rule of 128.  Binary32, 512 / 8192 x 4096: tiles of 64 at 3.5 bits
// 18.0/16.4 71.0/68.7, at 6.5 bits 20.6/17.2 87.5/76.4, stochastic 25.1/19.9 145/103; of 128 18.0/15.7 79.3/72.9; of 32
// 16.2/15.9 67.8/70.9, at 4 bits 5.0/5.1 30.7/32.4, stochastic 19.1/19.2 104.3/103.0 -- 4 % behind on large tensors of tiles of
// 32, which do not get a kernel of their own for that.
template <class C, bool SR>
bool quant_lanes_pays(uint64_t n_rounds, bool narrow, int sms) {
  const uint64_t per_warp = C::G == 64 && narrow && !SR ? 1 : 2;
  return C::G >= 32 && (!C::BF16 || n_rounds <= per_warp * QuantLanes<C>::WARPS * (unsigned)sms);
}

}  // namespace tahq
