// Fixed-point gradient compressor Q_Naive (Algorithm 1 lines 6-7; pre-scale g_hat = Q(c g) / c of
// the appendix) for sm_100a.
//   y = c * g;  s = max|y| / (2^(b-1) - 1);  q = clamp(round(y * (1/s)));  code = q + L
// with the product y * (1/s) rounded once (fused multiply-add with 1.5 * 2^23 as the addend).
//
// A lane owns 32 consecutive elements of a row, whose codes are b whole words (decoding binary32: 16 elements, so that
// a lane's 64 bytes leave by two 256-bit stores).  Encode: a row belongs to as many warps as it has stretches of 1024
// elements (short rows share a warp), so that a lane holds 32 elements however long the row is, the next row's
// elements are asked for before the current row is worked on, and the row's largest magnitude crosses the warps
// through shared memory.  Decode: pieces are independent and are dealt out to the lanes one by one.  Every width
// 2 ... 16 has code of its own (all shifts static).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "tahq_device.cuh"
#include "tahq_host.cuh"

namespace tahq {

constexpr int kQThreads = 256;
constexpr uint64_t kQPiecesPerLaunch = 1ull << 32;   // decode: less one step of the grid
constexpr float kQMagic = 12582912.0f;     // 1.5 * 2^23
constexpr uint32_t kQMagicBits = 0x4B400000u;

// A lane's 32 elements as loaded.
template <bool BF16>
struct QRaw {
  static constexpr int NW = BF16 ? 16 : 32;
  uint32_t w[NW];
  // `wide`: src is 32-byte aligned
  __device__ __forceinline__ void load(const uint8_t *src, bool wide) {
    if constexpr (!BF16) {
      if (wide) {   // (a lane's 128 bytes by 128-bit loads would take twice the passes over the L1 tags)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                       : "=r"(w[8 * i]), "=r"(w[8 * i + 1]), "=r"(w[8 * i + 2]), "=r"(w[8 * i + 3]), "=r"(w[8 * i + 4]),
                         "=r"(w[8 * i + 5]), "=r"(w[8 * i + 6]), "=r"(w[8 * i + 7])
                       : "l"(src + 32 * i));
        return;
      }
    }
#pragma unroll
    for (int i = 0; i < NW / 4; ++i) {
      const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src) + i);
      w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
    }
  }
  // the first n elements only (a multiple of 8), zeros behind them
  __device__ __forceinline__ void load_some(const uint8_t *src, uint32_t n) {
#pragma unroll
    for (int i = 0; i < NW / 4; ++i) {
      const uint4 v = (BF16 ? 8u : 4u) * i < n ? __ldg(reinterpret_cast<const uint4 *>(src) + i) : make_uint4(0, 0, 0, 0);
      w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
    }
  }
  // largest magnitude
  __device__ __forceinline__ float max_abs() const {
    if constexpr (BF16) {
      uint32_t m0 = w[0], m1 = w[1];
#pragma unroll
      for (int i = 2; i < NW; i += 2) { m0 = bf2_max_abs(m0, w[i]); m1 = bf2_max_abs(m1, w[i + 1]); }
      m0 = bf2_max_abs(m0, m1) & 0x7fff7fffu;
      return __uint_as_float(max(m0 & 0xffffu, m0 >> 16) << 16);
    } else {
      float m0 = fabsf(__uint_as_float(w[0])), m1 = fabsf(__uint_as_float(w[1]));
#pragma unroll
      for (int i = 2; i < NW; i += 2) {
        m0 = fmaxf(m0, fabsf(__uint_as_float(w[i])));
        m1 = fmaxf(m1, fabsf(__uint_as_float(w[i + 1])));
      }
      return fmaxf(m0, m1);
    }
  }
  // elements 2i and 2i + 1
  __device__ __forceinline__ float2 pair(int i) const {
    if constexpr (BF16) return f2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
    else return f2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1]));
  }
};

// Row scale and the reciprocal the codes are formed with, from the row's largest |g|: the largest |c g| is c times
// that, rounded (rounding keeps the order).
template <int B>
__device__ __forceinline__ float q_scale(float mg, float prescale, float &inv) {
  float s = __fdiv_rn(prescale * mg, (float)((1 << (B - 1)) - 1));
  s = s < 1.17549435e-38f ? 0.0f : s;   // below the normal range (its reciprocal may overflow): counts as zero
  inv = s > 0.0f ? __frcp_rn(s) : 0.0f;
  return s;
}

// 32 codes -> B words of the row's bit stream.  Four (b <= 8) or two codes are glued by a multiply-add chain on the
// raw bits of fma(y, 1/s, 1.5 * 2^23); the constant part of those bits, less L per code, is taken off once per chain.
// The clamp is left out: |y| <= m and s = m / L rounded give |y * (1/s)| < L + 1/2, so it never acts on a finite c g.
// (`prescale`: see the caller, where c g overflows.)
template <bool BF16, int B>
__device__ __forceinline__ void q_codes(const QRaw<BF16> &raw, float prescale, float inv, uint32_t (&w)[B]) {
  constexpr int GS = B <= 8 ? 4 : 2, GB = GS * B;   // codes and bits of a chain
  constexpr uint32_t Lq = (1u << (B - 1)) - 1u;
  constexpr uint32_t kOff = (uint32_t)(((unsigned long long)(kQMagicBits - Lq) * group_ones(B, GS)) & 0xffffffffull);
  uint32_t M = 1u << B;
  asm volatile("mov.u32 %0, %0;" : "+r"(M));   // opaque: the chain stays one multiply-add per code
#pragma unroll
  for (int j = 0; j < B; ++j) w[j] = 0;
#pragma unroll
  for (int j = 0; j < 32 / GS; ++j) {
    uint32_t acc = 0;
#pragma unroll
    for (int k = GS / 2 - 1; k >= 0; --k) {
      const float2 y = mul2(raw.pair(j * (GS / 2) + k), f2(prescale));
      const float2 t = fma2(y, f2(inv), f2(kQMagic));   // one rounding, ties to even
      acc = k == GS / 2 - 1 ? __float_as_uint(t.y) : acc * M + __float_as_uint(t.y);
      acc = acc * M + __float_as_uint(t.x);
    }
    const uint32_t g = acc - kOff;
    const int bit = j * GB, wi = bit >> 5, sh = bit & 31;
    w[wi] |= g << sh;
    if (sh + GB > 32) w[wi + 1] |= g >> (32 - sh);
  }
}

// The words of a lane's 32 codes, of which n belong to the row (the others are zero bits), to the lane's place `dst`;
// `room` = words of the row from there on (a multiple of the words of a store).
template <int B>
__device__ __forceinline__ void q_store(uint32_t *dst, uint32_t n, uint32_t room, uint32_t (&w)[B]) {
  constexpr int V = B % 4 == 0 ? 4 : B % 2 == 0 ? 2 : 1;   // words of a store
  if (n < 32u) {
    const int bits = (int)n * B;
#pragma unroll
    for (int j = 0; j < B; ++j) w[j] &= bits >= 32 * (j + 1) ? 0xffffffffu : bits <= 32 * j ? 0u : (1u << (bits - 32 * j)) - 1u;
#pragma unroll
    for (int j = 0; j < B; ++j)
      if ((uint32_t)j < room) dst[j] = w[j];
    return;
  }
#pragma unroll
  for (int j = 0; j < B; j += V) {
    if constexpr (V == 4) *reinterpret_cast<uint4 *>(dst + j) = make_uint4(w[j], w[j + 1], w[j + 2], w[j + 3]);
    else if constexpr (V == 2) *reinterpret_cast<uint2 *>(dst + j) = make_uint2(w[j], w[j + 1]);
    else dst[j] = w[j];
  }
}

// header and section padding (one CTA)
__device__ __forceinline__ void q_frame(const QArgs &a) {
  if (threadIdx.x == 0 && !a.per_tensor) *a.status = 0;   // (per tensor: cleared with the maximum in front)
  if (threadIdx.x < 32) reinterpret_cast<uint32_t *>(a.packed)[threadIdx.x] = threadIdx.x < 16 ? a.header[threadIdx.x] : 0u;
  const uint64_t n_s = a.per_tensor ? 1 : a.tokens;
  for (uint64_t o = a.off_scales + 4 * n_s + threadIdx.x; o < a.off_payload; o += blockDim.x) a.packed[o] = 0;
  for (uint64_t o = a.off_payload + a.tokens * a.row_bytes + threadIdx.x; o < a.total_bytes; o += blockDim.x) a.packed[o] = 0;
}

// per-tensor mode: max |g| over the whole tensor (non-negative floats order like their bit patterns)
template <bool BF16>
__global__ void __launch_bounds__(kQThreads) qnaive_max_kernel(const QArgs a) {
  grid_dependency_wait();   // launched as a programmatic dependent of the kernel in front
  constexpr int ESZ = BF16 ? 2 : 4;
  const uint64_t n = a.tokens * (uint64_t)a.hidden;
  const bool wide = (reinterpret_cast<uintptr_t>(a.in) & 31u) == 0;
  float m = 0.0f;
  for (uint64_t i = ((uint64_t)blockIdx.x * kQThreads + threadIdx.x) * 32; i < n; i += (uint64_t)gridDim.x * kQThreads * 32) {
    QRaw<BF16> raw;
    if (n - i >= 32) raw.load(a.in + i * ESZ, wide);
    else raw.load_some(a.in + i * ESZ, (uint32_t)(n - i));
    m = fmaxf(m, raw.max_abs());
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
  if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(a.gmax, __float_as_uint(m));
}

// 19 us for 8192 x 4096 bf16 at 6 bits (92 MB; with the decoder 43.0 -> 32.9 us per round trip, of which the launches that
// cleared 256 bytes took 4): bound half by memory, half by issue.  A warp to a row held 64 registers of raw data, which left 16
// warps on an SM and 3.5 waves of CTAs.
// LONG: rows beyond 8192 elements, which a CTA's eight warps take in several stretches (the later ones read twice).
template <bool BF16, int B, bool LONG>
__global__ void __launch_bounds__(kQThreads, BF16 ? 3 : 2) qnaive_encode_kernel(const QArgs a) {
  constexpr int ESZ = BF16 ? 2 : 4;
  __shared__ uint32_t s_max[2][8];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, C = a.hidden;
  const uint32_t n_warps = blockDim.x >> 5, row_words = (uint32_t)(a.row_bytes / 4), lanes_all = C / 32u + (C % 32u != 0u);
  float *scales = reinterpret_cast<float *>(a.packed + a.off_scales);
  const bool wide = (reinterpret_cast<uintptr_t>(a.in) & 31u) == 0;
  grid_dependency_wait();   // launched as a programmatic dependent of the kernel in front
  if (blockIdx.x == 0) q_frame(a);
  uint32_t mg = a.per_tensor ? *a.gmax : 0u;   // largest magnitude, as bits

  // rows of the CTA at a time, and this lane's place in one of them
  const bool shared_row = a.row_warps > 1;
  const uint32_t rows_at_once = shared_row ? n_warps / a.row_warps : n_warps * (32u / a.row_lanes);
  const uint32_t slot = shared_row ? warp / a.row_warps : warp * (32u / a.row_lanes) + lane / a.row_lanes;
  const uint32_t part = shared_row ? warp % a.row_warps * 32u + lane : lane % a.row_lanes;   // 32 elements each
  const uint32_t parts_at_once = shared_row ? a.row_warps * 32u : a.row_lanes;
  const uint64_t step = (uint64_t)gridDim.x * rows_at_once;
  auto elements = [&](uint32_t p) { return p >= lanes_all ? 0u : C - 32u * p < 32u ? C - 32u * p : 32u; };
  auto load_at = [&](QRaw<BF16> &raw, const uint8_t *src, uint32_t n) {
    if (n == 32u) raw.load(src, wide);
    else if (n) raw.load_some(src, n);
  };
  auto emit = [&](const QRaw<BF16> &raw, uint32_t *dst, uint32_t n, uint32_t room, float c, float inv) {
    uint32_t w[B];
    q_codes<BF16, B>(raw, c, inv, w);
    if (n) q_store<B>(dst, n, room, w);
  };
  const uint64_t r_cta = (uint64_t)blockIdx.x * rows_at_once;
  uint64_t r = r_cta + slot;
  const uint32_t n_mine = elements(part);
  const uint8_t *src = a.in + (r * (uint64_t)C + 32u * part) * ESZ;
  uint32_t *dst = reinterpret_cast<uint32_t *>(a.packed + a.off_payload + r * a.row_bytes) + part * (uint32_t)B;
  const uint64_t d_src = step * C * ESZ, d_dst = step * row_words;
  uint32_t parity = 0;

  // one row: its elements are here; those of the lane's row after it are asked for
  auto turn = [&](const QRaw<BF16> &cur, QRaw<BF16> &next) {
    const bool live = r < a.tokens;
    src += d_src;
    if (!LONG && r + step < a.tokens) load_at(next, src, n_mine);
    if (!a.per_tensor) {
      uint32_t m = __float_as_uint(cur.max_abs());   // (non-negative floats order like their bit patterns)
      if (LONG && live)
#pragma unroll 1
        for (uint32_t p = part + parts_at_once; p < lanes_all; p += parts_at_once) {
          QRaw<BF16> more;
          load_at(more, a.in + (r * (uint64_t)C + 32u * p) * ESZ, elements(p));
          m = max(m, __float_as_uint(more.max_abs()));
        }
      __syncwarp();
      if (a.row_lanes == 32u) {
        m = __reduce_max_sync(kFull, m);
        if (shared_row) {
          if (lane == 0) s_max[parity][warp] = m;
          asm volatile("bar.sync %0, %1;" ::"r"(slot + 1u), "r"(a.row_warps * 32u) : "memory");
          m = __reduce_max_sync(kFull, lane < a.row_warps ? s_max[parity][slot * a.row_warps + lane] : 0u);
          parity ^= 1u;   // (a warp writes this half again only after the next barrier, when all have read it)
        }
      } else {
        for (uint32_t o = a.row_lanes / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
      }
      mg = m;
    }
    float inv;
    const float s = q_scale<B>(__uint_as_float(mg), a.prescale, inv);
    // where c g overflows the scale is infinite, its reciprocal zero and, as with a scale of zero, every code that of zero; c g
    // itself would put codes that are no number into the chains of q_codes, which their neighbours share
    const float c = inv > 0.0f ? a.prescale : 0.0f;
    if (live) {
      if (part == 0) {
        if (!a.per_tensor || r == 0) scales[a.per_tensor ? 0 : r] = s;
        for (uint32_t o = lanes_all * (uint32_t)B; o < row_words; ++o) dst[o] = 0;   // the row's last words, behind its last lane's
      }
      emit(cur, dst, n_mine, row_words - part * (uint32_t)B, c, inv);
      if (LONG)
#pragma unroll 1
        for (uint32_t p = part + parts_at_once; p < lanes_all; p += parts_at_once) {
          QRaw<BF16> more;
          load_at(more, a.in + (r * (uint64_t)C + 32u * p) * ESZ, elements(p));
          emit(more, dst + (p - part) * (uint32_t)B, elements(p), row_words - p * (uint32_t)B, c, inv);
        }
    }
    dst += d_dst;
    r += step;
  };
  QRaw<BF16> ra, rb;
#pragma unroll
  for (int i = 0; i < QRaw<BF16>::NW; ++i) ra.w[i] = rb.w[i] = 0u;   // (lanes behind the row's end stay at zero)
  if (LONG) {
    for (uint64_t rc = r_cta; rc < a.tokens; rc += step) {   // (a row to the CTA)
      load_at(ra, src, n_mine);
      turn(ra, rb);
    }
  } else {
    if (r < a.tokens) load_at(ra, src, n_mine);
    for (uint64_t rc = r_cta; rc < a.tokens; rc += 2 * step) {   // (the same number of turns for every lane of the CTA)
      turn(ra, rb);
      if (rc + step < a.tokens) turn(rb, ra);
    }
  }
}

// t / c in binary32, correctly rounded, for several t by one c (rc = 1/c rounded): a quotient estimate is improved twice
// by its remainder, which a fused multiply-add gives exactly; the second step rounds correctly because the first one's
// result is within one unit in the last place (Markstein, IA-64 and Elementary Functions, ch. 8; Brisebarre, Muller and
// Raina, IEEE Trans. Computers 53(8), 2004).  No step may leave the normal range: see div_safe.  Half the instructions of
// __fdiv_rn, which cannot know that the divisor stays: 8192 x 4928 bf16 at 8 bits, c = 1000, encode + decode 74.8 -> 48.6 us.
__device__ __forceinline__ float2 div_by(float2 t, float2 nc, float2 rc) {
  const float2 q0 = f2(__fmul_rn(t.x, rc.x), __fmul_rn(t.y, rc.y));   // (scalar: they are addends below)
  const float2 q1 = fma2(fma2(q0, nc, t), rc, q0);
  return fma2(fma2(q1, nc, t), rc, q1);
}
// Every non-zero t = q * s of a row has s <= |t| < 2^16 s: t, its quotient and remainders (above 2^-50 |t|) stay normal.
__device__ __forceinline__ bool div_safe(float s, float c) {
  return (s == 0.0f || (s >= 0x1p-40f && s <= 0x1p60f)) && c >= 0x1p-30f && c <= 0x1p30f;
}

// Codes of a lane -> g_hat = (q * s) / c.  Dividing by a power of two is the same rounding as multiplying by its
// (exact) reciprocal.
template <bool BF16, int B, bool WIDE>
__global__ void __launch_bounds__(kQThreads, 4) qnaive_decode_kernel(const QArgs a) {
  constexpr int ESZ = BF16 ? 2 : 4, E = 64 / ESZ;
  constexpr int NW = (E * B + (E == 16 && B % 2 ? 16 : 0) + 31) / 32;   // words a lane's codes lie in
  constexpr int V = (E * B) % 128 == 0 ? 4 : (E * B) % 64 == 0 ? 2 : 1;  // words of a load
  constexpr float kOff = kQMagic + (float)((1 << (B - 1)) - 1);         // exact
  const uint32_t lane = threadIdx.x & 31u, C = a.hidden, row_words = (uint32_t)(a.row_bytes / 4);
  const uint32_t total = (uint32_t)a.tokens * a.pieces, step = gridDim.x * kQThreads;
  grid_dependency_wait();   // launched as a programmatic dependent of the kernel in front
  const float *scales = reinterpret_cast<const float *>(a.packed + a.off_scales);
  const uint8_t *payload = a.packed + a.off_payload;
  // the received header must describe these parameters; otherwise nothing is written
  const uint32_t hdr = lane < 16 ? __ldg(reinterpret_cast<const uint32_t *>(a.packed) + lane) : 0u;

  // piece i of the tensor: piece `pc` of row `row`; advanced without a division
  const uint32_t d_row = step / a.pieces, d_pc = step - d_row * a.pieces;
  uint32_t i = blockIdx.x * kQThreads + threadIdx.x;
  uint32_t row = i / a.pieces, pc = i - row * a.pieces;
  uint32_t w[NW];
  float s = 0.0f;
  auto load = [&](uint32_t rw, uint32_t p) {
    const uint32_t first = E == 32 ? p * (uint32_t)B : (p * (uint32_t)B) >> 1;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(payload + rw * a.row_bytes);
#pragma unroll
    for (int j = 0; j < NW; j += V) {
      if constexpr (V == 4) {
        const uint4 v = first + j < row_words ? __ldg(reinterpret_cast<const uint4 *>(src + first + j)) : make_uint4(0, 0, 0, 0);
        w[j] = v.x; w[j + 1] = v.y; w[j + 2] = v.z; w[j + 3] = v.w;
      } else if constexpr (V == 2) {
        const uint2 v = first + j < row_words ? __ldg(reinterpret_cast<const uint2 *>(src + first + j)) : make_uint2(0, 0);
        w[j] = v.x; w[j + 1] = v.y;
      } else {
        w[j] = first + j < row_words ? __ldg(src + first + j) : 0u;
      }
    }
    s = __ldg(scales + (a.per_tensor ? 0u : rw));
  };
  if (i < total) load(row, pc);
  const bool bad = __any_sync(kFull, lane < 16 && hdr != a.header[lane & 15u]);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.status = bad ? 1u /* TAHQ_DEV_BAD_HEADER */ : 0u;
  if (bad) return;
  const bool pow2 = (__float_as_uint(a.prescale) & 0x007fffffu) == 0u && (__float_as_uint(a.prescale) >> 23) - 2u < 250u;
  const float rc = __frcp_rn(a.prescale);

  for (; i < total; i += step) {
    uint32_t v[NW + 1];
#pragma unroll
    for (int j = 0; j < NW; ++j) v[j] = w[j];
    v[NW] = 0;
    const float sc = s;
    const uint32_t r0 = row, p0 = pc;
    row += d_row;
    pc += d_pc;
    if (pc >= a.pieces) { pc -= a.pieces; ++row; }
    if (i + step < total && i + step > i) load(row, pc);
    if constexpr (E == 16 && B % 2 == 1) {   // an odd piece starts in the middle of a word
      const uint32_t sh = (p0 & 1u) * 16u;
#pragma unroll
      for (int j = 0; j < NW; ++j) v[j] = __funnelshift_r(v[j], v[j + 1], sh);
    }
    float2 x[E / 2];
#pragma unroll
    for (int k = 0; k < E / 2; ++k) {
      uint32_t m[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // the code in the mantissa of 1.5 * 2^23
        const int bit = (2 * k + h) * B, wi = bit >> 5, sh = bit & 31;
        const uint32_t c = sh == 0 ? v[wi] : sh + B <= 32 ? v[wi] >> sh : __funnelshift_r(v[wi], v[wi + 1], sh);
        m[h] = (c & ((1u << B) - 1u)) | kQMagicBits;
      }
      const float2 q = add2(f2(__uint_as_float(m[0]), __uint_as_float(m[1])), f2(-kOff));   // code - L, exact
      x[k] = mul2(q, f2(sc));
    }
    if (pow2) {
#pragma unroll
      for (int k = 0; k < E / 2; ++k) x[k] = mul2(x[k], f2(rc));
    } else if (__all_sync(__activemask(), div_safe(sc, a.prescale))) {
#pragma unroll
      for (int k = 0; k < E / 2; ++k) x[k] = div_by(x[k], f2(-a.prescale), f2(rc));
    } else {
#pragma unroll
      for (int k = 0; k < E / 2; ++k) x[k] = f2(__fdiv_rn(x[k].x, a.prescale), __fdiv_rn(x[k].y, a.prescale));
    }
    uint32_t o[16];
#pragma unroll
    for (int k = 0; k < E / 2; ++k) {
      if constexpr (BF16) {
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(x[k].x, x[k].y);
        o[k] = *reinterpret_cast<const uint32_t *>(&h2);
      } else {
        o[2 * k] = __float_as_uint(x[k].x);
        o[2 * k + 1] = __float_as_uint(x[k].y);
      }
    }
    const uint32_t rest = C - p0 * (uint32_t)E, left = rest < (uint32_t)E ? rest * ESZ : 64u;   // bytes of the piece: a multiple of 16
    uint8_t *dst = a.out + ((uint64_t)r0 * C + p0 * (uint32_t)E) * ESZ;
#pragma unroll
    for (int j = 0; j < 16; j += WIDE ? 8 : 4) {
      if (4u * j < left) {
        if constexpr (WIDE)   // (rows of whole 32-byte pieces)
          asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 4 * j), "r"(o[j]), "r"(o[j + 1]),
                       "r"(o[j + 2]), "r"(o[j + 3]), "r"(o[j + 4]), "r"(o[j + 5]), "r"(o[j + 6]), "r"(o[j + 7])
                       : "memory");
        else
          *reinterpret_cast<uint4 *>(dst + 4 * j) = make_uint4(o[j], o[j + 1], o[j + 2], o[j + 3]);
      }
    }
  }
}

// ---- launches (one translation unit per element type: qnaive_*.cu) --------------------------------------
template <bool BF16, int B>
tahq_status qnaive_encode_b(QArgs a, const DevInfo &d, cudaStream_t st) {
  static std::atomic<int> occ[2][64];
  const uint32_t parts = a.hidden / 32 + (a.hidden % 32 != 0), stretches = (parts + 31) / 32;
  const bool lng = stretches > 8;
  void (*const kernel)(QArgs) = lng ? qnaive_encode_kernel<BF16, B, true> : qnaive_encode_kernel<BF16, B, false>;
  const int n = prepare(kernel, kQThreads, 0, d, occ[lng]);
  if (!n) return TAHQ_ERR_CUDA;
  a.row_warps = stretches < 8 ? stretches : 8;
  a.row_lanes = 32;
  while (a.row_warps == 1 && a.row_lanes / 2 >= parts) a.row_lanes /= 2;
  const uint32_t threads = a.row_warps > 1 ? 32 * a.row_warps * (8 / a.row_warps) : kQThreads;   // whole rows
  const uint32_t rows = a.row_warps > 1 ? 8 / a.row_warps : 8 * (32 / a.row_lanes);
  const uint64_t want = (a.tokens + rows - 1) / rows, cap = (uint64_t)d.sms * n;
  TAHQ_LAUNCH("qnaive_encode", st, launch_dependent(kernel, (unsigned)(want < cap ? want : cap), threads, 0, st, a));
  return cudaGetLastError() == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}
template <bool BF16, int B>
tahq_status qnaive_decode_b(QArgs a, const DevInfo &d, cudaStream_t st) {
  constexpr uint32_t E = BF16 ? 32 : 16;
  static std::atomic<int> occ[2][64];
  const bool wide = (reinterpret_cast<uintptr_t>(a.out) & 31u) == 0 && a.hidden % (E / 2) == 0;
  void (*const kernel)(QArgs) = wide ? qnaive_decode_kernel<BF16, B, true> : qnaive_decode_kernel<BF16, B, false>;
  const int n = prepare(kernel, kQThreads, 0, d, occ[wide]);
  if (!n) return TAHQ_ERR_CUDA;
  a.pieces = a.hidden / E + (a.hidden % E != 0);
  const uint64_t cap = (uint64_t)d.sms * n, tokens = a.tokens;
  // the kernel counts pieces in 32 bits: more of them (64 GiB, where a row is one piece of 16 bytes) go in several launches,
  // of an even number of rows each, which keeps the alignment
  const uint64_t rows = (kQPiecesPerLaunch - cap * kQThreads) / a.pieces / 2 * 2;
  for (uint64_t r = 0; r < tokens; r += rows) {
    a.tokens = tokens - r < rows ? tokens - r : rows;
    const uint64_t want = (a.tokens * a.pieces + kQThreads - 1) / kQThreads;
    TAHQ_LAUNCH("qnaive_decode", st, launch_dependent(kernel, (unsigned)(want < cap ? want : cap), kQThreads, 0, st, a));
    a.off_scales += a.per_tensor ? 0 : 4 * rows;
    a.off_payload += rows * a.row_bytes;
    a.out += rows * a.hidden * (BF16 ? 2 : 4);
  }
  return cudaGetLastError() == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}
template <bool BF16, bool ENC, int B = 2>
tahq_status qnaive_width(const QArgs &a, const DevInfo &d, cudaStream_t st) {
  if constexpr (B > 16) return TAHQ_ERR_INVALID_ARG;
  else if (a.bits != (uint32_t)B) return qnaive_width<BF16, ENC, B + 1>(a, d, st);
  else if constexpr (ENC) return qnaive_encode_b<BF16, B>(a, d, st);
  else return qnaive_decode_b<BF16, B>(a, d, st);
}
template <bool BF16>
tahq_status qnaive_encode_cfg(const QArgs &a, const DevInfo &d, cudaStream_t st) {
  if (a.per_tensor)
    TAHQ_LAUNCH("qnaive_max", st, launch_dependent(qnaive_max_kernel<BF16>, d.sms * 4, kQThreads, 0, st, a));
  return qnaive_width<BF16, true>(a, d, st);
}
template <bool BF16>
tahq_status qnaive_decode_cfg(const QArgs &a, const DevInfo &d, cudaStream_t st) {
  return qnaive_width<BF16, false>(a, d, st);
}
#define TAHQ_INSTANTIATE_QNAIVE(BF16)                                                          \
  template tahq_status qnaive_encode_cfg<BF16>(const QArgs &, const DevInfo &, cudaStream_t);  \
  template tahq_status qnaive_decode_cfg<BF16>(const QArgs &, const DevInfo &, cudaStream_t);

}  // namespace tahq
