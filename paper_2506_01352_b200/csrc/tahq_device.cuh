// Device-side building blocks of the TAH-Quant boundary codec for sm_100a.
//
// Two decompositions of the work build on them.  In one a thread owns a whole tile (quantisation group, Sec. 3.1) -- or
// half of a 128-wide tile -- in registers, so that the Hadamard butterfly (Eq. 4), the reductions of Eq. 1-3 and the bit
// packing need no cross-lane traffic; tiles reach it through an XOR-swizzled stage of 32 rows per warp, filled by 16-byte
// cp.async or tiled TMA with the 128-byte swizzle (tahq_stream.cuh).  In the other a lane owns 64 bytes of the tensor and
// neighbouring lanes share a tile (tahq_lanes.cuh).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace tahq {

constexpr int kThreads = 256;          // threads per CTA of the tile kernels
constexpr int kBins = 4096;            // histogram of the top-p% selection
constexpr unsigned kFull = 0xffffffffu;

// ------------------------------------------------------------------------------------------
// Geometry of one (tile width, dtype) instantiation
// ------------------------------------------------------------------------------------------
template <int G_, bool BF16_>
struct Cfg {
  static constexpr int G = G_;
  static constexpr bool BF16 = BF16_;
  static constexpr int LPT = (G == 128) ? 2 : 1;   // lanes (threads) per tile
  static constexpr int EPT = G / LPT;              // elements per thread: 8 ... 64
  static constexpr int ESZ = BF16 ? 2 : 4;
  static constexpr int ROWB = EPT * ESZ;           // bytes of one thread-row: 16 ... 256
  static constexpr int CPR = ROWB / 16;            // 16-byte chunks per row: 1 ... 16
  static constexpr int NOCT = EPT / 8;             // groups of 8 elements per thread
};

// XOR swizzle of 16-byte chunks: the eight threads of a quarter-warp, whose rows are ROWB bytes
// apart, land in eight different 16-byte bank groups for every chunk index q.
template <class C>
__device__ __forceinline__ int swz(int row) {
  return (C::CPR >= 8) ? (row & 7) : ((row >> 1) & 3);
}
template <class C>
__device__ __forceinline__ int phys_chunk(int row, int q) {
  return (row * C::CPR + q) ^ swz<C>(row);
}

// ------------------------------------------------------------------------------------------
// cp.async
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, int src_bytes) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(src_bytes)
               : "memory");
}
// Programmatic dependent launch: a kernel launched with the stream-serialisation attribute is set up while the
// kernel in front of it in the stream still runs; it must call this before it touches anything that kernel
// writes (it returns once that whole grid is done and its writes are visible).  A no-op in a kernel launched
// the ordinary way.  No kernel here signals its dependents early: measured, that only made things slower.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Optional timeline of a call (tahq_trace): per kernel, the earliest moment a CTA was resident, the earliest moment
// one got past its dependency wait, and the latest moment a warp finished, as global-timer nanoseconds.
struct TraceScope {
  unsigned long long *t;
  __device__ __forceinline__ static unsigned long long now() {
    unsigned long long v;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
    return v;
  }
  __device__ __forceinline__ TraceScope(unsigned long long *buf, int id) : t(buf ? buf + 4 * id : nullptr) {
    if (t && threadIdx.x == 0) atomicMin(t, now());
  }
  __device__ __forceinline__ void started() const {
    if (t && threadIdx.x == 0) atomicMin(t + 1, now());
  }
  __device__ __forceinline__ ~TraceScope() {
    if (t && (threadIdx.x & 31) == 0) atomicMax(t + 2, now());
  }
};

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ------------------------------------------------------------------------------------------
// TMA copies completing on an mbarrier.  Every wait is bounded.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// true when the phase with the given parity has completed; gives up after a bounded number of polls
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity) {
  for (unsigned spins = 0; spins < (1u << 22); ++spins) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// Tiled TMA copy of a [rows x 128-byte] box of a two-dimensional tensor map into shared memory,
// completing on an mbarrier.  x (the innermost coordinate) is always 0 here, so the 16-byte rule holds;
// rows past the end of the tensor are filled with zeros by the hardware.
__device__ __forceinline__ void tma_load_rows(void *dst, const void *tmap, int row0, unsigned long long *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_u32(dst)), "l"(tmap), "r"(0), "r"(row0), "r"(smem_u32(bar))
      : "memory");
}

// Eight consecutive elements (oct `o`) of this thread's row, widened to binary32.
template <class C>
__device__ __forceinline__ void load_oct(const uint8_t *stage, int row, int o, float (&v)[8]) {
  if constexpr (C::BF16) {
    const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, o) * 16);
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[2 * j] = __uint_as_float(u[j] << 16);
      v[2 * j + 1] = __uint_as_float(u[j] & 0xffff0000u);
    }
  } else {
    const float4 a = *reinterpret_cast<const float4 *>(stage + (size_t)phys_chunk<C>(row, 2 * o) * 16);
    const float4 b = *reinterpret_cast<const float4 *>(stage + (size_t)phys_chunk<C>(row, 2 * o + 1) * 16);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
}

// ------------------------------------------------------------------------------------------
// bf16 pairs handled in their packed form (sm_100a: packed bf16 min/max run on the ALU pipe, one
// instruction per two elements; a bf16 operand can feed an fp32 add on the FMA pipe directly)
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t bf2_max_abs(uint32_t a, uint32_t b) {   // magnitudes; sign bits are garbage
  uint32_t d;
  asm("max.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t bf2_min_abs(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("min.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t bf2_max(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t bf2_min(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("min.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
// (lo + c, hi + c) in binary32 for the two bf16 halves of w: the widening is exact, so this equals
// widening first and adding afterwards; with c = -0.0f it is the widening itself.
__device__ __forceinline__ void bf2_add_f32(uint32_t w, float c, float &lo, float &hi) {
  asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tadd.rn.f32.bf16 %0, l, %3;\n\tadd.rn.f32.bf16 %1, h, %3;\n\t}"
      : "=f"(lo), "=f"(hi)
      : "r"(w), "f"(c));
}

// ------------------------------------------------------------------------------------------
// Arithmetic of Eq. 1-2 (binary32, fixed order; the library is compiled with -fmad=false so that
// only the fused multiply-adds written here are fused)
// ------------------------------------------------------------------------------------------

// neighbours-first pairwise tree over 8 values
__device__ __forceinline__ float tree8(const float (&v)[8]) {
  const float a = v[0] + v[1], b = v[2] + v[3], c = v[4] + v[5], d = v[6] + v[7];
  return (a + b) + (c + d);
}
template <int N>
__device__ __forceinline__ float tree(float (&t)[N]) {
#pragma unroll
  for (int h = 1; h < N; h *= 2)
#pragma unroll
    for (int i = 0; i + h < N; i += 2 * h) t[i] = t[i] + t[i + h];
  return t[0];
}

// Pairs of binary32 values processed by one instruction (sm_100a add/mul/fma .f32x2: IEEE
// round-to-nearest per lane, so results equal the scalar operations bit for bit).  The assembler
// contracts a packed multiply that feeds a packed add into one packed fma even with explicit .rn
// and --fmad=false, which changes the rounding; so no result of mul2 may be an operand of add2
// (or the addend of fma2): such products are formed with scalar multiplies instead.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long &>(d))
      : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)));
  return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long &>(d))
      : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)));
  return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long &>(d))
      : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)),
        "l"(reinterpret_cast<const unsigned long long &>(c)));
  return d;
}

// log2 of a positive normal number as exponent + u*Q(u) (u = mantissa - 1, Q a fixed degree-5
// polynomial evaluated by Horner's rule with fused multiply-adds), with the exponent and the
// mantissa split done by multiply-adds so that everything runs on the FMA pipe (the ALU pipe has
// half its rate and is the busier one):  (x * 512) >> 32 is the biased exponent eb, placed into the
// mantissa of 2^23 by the addend of the same integer multiply-add; 2^-E is built as a bit pattern
// by one more integer multiply-add, and u = x * 2^-E - 1 is exact, as is every step before the
// polynomial.
__device__ __forceinline__ float lg2_fma(float x) {
  const uint32_t xi = __float_as_uint(x);
  uint32_t ebm;
  asm("mad.hi.u32 %0, %1, 512, 0x4B000000;" : "=r"(ebm) : "r"(xi));   // bits of 2^23 + eb
  const float e = __uint_as_float(ebm) - 8388735.0f;                   // eb - 127
  const uint32_t sb = ebm * 0xFF800000u + 0x7F000000u;                 // (254 - eb) << 23: bits of 2^-E
  const float u = __fmaf_rn(x, __uint_as_float(sb), -1.0f);
  float q = -0x1.a762d6p-6f;
  q = __fmaf_rn(q, u, 0x1.f2e252p-4f);
  q = __fmaf_rn(q, u, -0x1.1c9334p-2f);
  q = __fmaf_rn(q, u, 0x1.d487c6p-2f);
  q = __fmaf_rn(q, u, -0x1.6fb0bcp-1f);
  q = __fmaf_rn(q, u, 0x1.714aa0p+0f);
  return __fmaf_rn(u, q, e);
}

// The same for two numbers, two to an instruction where there is one (the same operations, the same bits).
__device__ __forceinline__ float2 lg2_fma2(float2 x) {
  uint32_t e0, e1;
  asm("mad.hi.u32 %0, %1, 512, 0x4B000000;" : "=r"(e0) : "r"(__float_as_uint(x.x)));
  asm("mad.hi.u32 %0, %1, 512, 0x4B000000;" : "=r"(e1) : "r"(__float_as_uint(x.y)));
  const float2 e = add2(f2(__uint_as_float(e0), __uint_as_float(e1)), f2(-8388735.0f));
  const uint32_t s0 = e0 * 0xFF800000u + 0x7F000000u, s1 = e1 * 0xFF800000u + 0x7F000000u;
  const float2 u = fma2(x, f2(__uint_as_float(s0), __uint_as_float(s1)), f2(-1.0f));
  float2 q = f2(-0x1.a762d6p-6f);
  q = fma2(q, u, f2(0x1.f2e252p-4f));
  q = fma2(q, u, f2(-0x1.1c9334p-2f));
  q = fma2(q, u, f2(0x1.d487c6p-2f));
  q = fma2(q, u, f2(-0x1.6fb0bcp-1f));
  q = fma2(q, u, f2(0x1.714aa0p+0f));
  return fma2(u, q, e);
}

// Magnitudes of eight consecutive elements of a row.
template <class C>
__device__ __forceinline__ void load_abs_oct(const uint8_t *stage, int row, int o, float (&v)[8]) {
  if constexpr (C::BF16) {
    const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, o) * 16);
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)   // clear both sign bits at once, widen on the FMA pipe
      bf2_add_f32(u[j] & 0x7fff7fffu, -0.0f, v[2 * j], v[2 * j + 1]);
  } else {
    load_oct<C>(stage, row, o, v);
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = fabsf(v[k]);
  }
}

// Entropy score of the tile this thread (pair) owns: -sum p log2(p + varsigma), p = |a| / (L1 + eps).
// Two streaming passes over the row in shared memory, eight elements at a time.
template <class C>
__device__ __forceinline__ float tile_score(const uint8_t *stage, int row, float eps_l1, float eps_log) {
  float part[C::NOCT];
#pragma unroll
  for (int o = 0; o < C::NOCT; ++o) {
    float v[8];
    load_abs_oct<C>(stage, row, o, v);
    part[o] = tree8(v);
  }
  float L1 = tree<C::NOCT>(part);
  if constexpr (C::LPT == 2) L1 = L1 + __shfl_xor_sync(kFull, L1, 1);
  const float inv = __fdiv_rn(1.0f, L1 + eps_l1);
#pragma unroll
  for (int o = 0; o < C::NOCT; ++o) {
    float v[8];
    load_abs_oct<C>(stage, row, o, v);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float p = v[k] * inv;
      v[k] = p * lg2_fma(p + eps_log);
    }
    part[o] = tree8(v);
  }
  float S = tree<C::NOCT>(part);
  if constexpr (C::LPT == 2) S = S + __shfl_xor_sync(kFull, S, 1);
  return 0.0f - S;
}

// ---- Screening score: an approximation of the score that costs one pass and one MUFU instruction per
// element.  With L' = L1 + eps and p = a / L', and leaving varsigma out of the logarithm,
//     -sum p log2 p  =  ( log2(L') * sum a  -  sum a log2 a ) / L',
// so the two sums are accumulated together and L' is needed only at the end.  Every magnitude gets
// 1e-30 added (for free, inside the widening addition) so that a zero contributes 0 * log2(1e-30) = 0.
// Distance from the exact score: what varsigma contributes, below G * varsigma / ln 2 (the host only
// selects this function when that is at most 1.5e-5); the hardware log2 (2^-22) and the rounding of
// the sums, each weighted by p or by |log2 a| <= 127 times a few units in the last place: under 1e-4
// in all.  It is only used to decide which tiles are far enough from a group's threshold to be
// classified without their exact score; see select_kernel.  All of this holds while L' is nowhere near the ends of binary32:
// see screen_range.
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Does the screening hold for a tile with L' = Lp?  Not below 2^-60, where the 1e-30 added to every magnitude would count (a
// varepsilon near zero and a tile of next to nothing), nor above 2^60, where the sums come near the largest numbers, nor where
// it is no number.  A warp that screens keeps the largest of these; beyond kScreenRange it goes back over its tiles when it is
// through (exact_scores_of).
constexpr uint32_t kScreenRange = 120u << 23;   // from 2^-60 to 2^60, in the bits of binary32
__device__ __forceinline__ uint32_t screen_range(float Lp) { return __float_as_uint(Lp) - 0x21800000u; }
// An exact score as it is stored and ranked: every one a number, of a size that the selection can calculate with.  (A tile of
// zeroes without epsilon has p = 0/0; it ranks first, as its key without this would.)
__device__ __forceinline__ float ranked_score(float s) { return s == s ? fminf(fmaxf(s, -1e30f), 1e30f) : 1e30f; }

template <class C>
__device__ __forceinline__ float tile_score_screen(const uint8_t *stage, int row, float eps_l1, uint32_t &range) {
  const float tiny = 1e-30f;
  float pl[C::NOCT], pt[C::NOCT];
#pragma unroll
  for (int o = 0; o < C::NOCT; ++o) {
    float v[8];
    if constexpr (C::BF16) {
      const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, o) * 16);
      const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) bf2_add_f32(u[j] & 0x7fff7fffu, tiny, v[2 * j], v[2 * j + 1]);
    } else {
      load_oct<C>(stage, row, o, v);
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = fabsf(v[k]) + tiny;
    }
    float t = v[0] * lg2_approx(v[0]);
#pragma unroll
    for (int k = 1; k < 8; ++k) t = __fmaf_rn(v[k], lg2_approx(v[k]), t);
    pt[o] = t;
    pl[o] = tree8(v);
  }
  float L = tree<C::NOCT>(pl), T = tree<C::NOCT>(pt);
  if constexpr (C::LPT == 2) {
    L = L + __shfl_xor_sync(kFull, L, 1);
    T = T + __shfl_xor_sync(kFull, T, 1);
  }
  const float Lp = L + eps_l1;
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(Lp));
  range = max(range, screen_range(Lp));
  return __fmaf_rn(lg2_approx(Lp), L, -T) * r;
}

// Exact score of one whole tile read straight from global memory by NOCT neighbouring lanes, lane o
// taking the o-th group of eight elements (used for the few tiles near a group's threshold).  Same
// arithmetic and summation tree as tile_score: the tree over the groups of eight runs as xor
// shuffles (neighbours first; addition is commutative, so every lane ends with the same bits).
// All 32 lanes of the warp must call it.
template <bool BF16>
__device__ __forceinline__ void load_abs_oct_global(const uint8_t *tile, int o, float (&v)[8]) {
  if constexpr (BF16) {
    const uint4 w = __ldg(reinterpret_cast<const uint4 *>(tile) + o);
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[2 * j] = __uint_as_float((u[j] << 16) & 0x7fffffffu);
      v[2 * j + 1] = __uint_as_float(u[j] & 0x7fff0000u);
    }
  } else {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(tile) + 2 * o);
    const float4 b = __ldg(reinterpret_cast<const float4 *>(tile) + 2 * o + 1);
    v[0] = fabsf(a.x); v[1] = fabsf(a.y); v[2] = fabsf(a.z); v[3] = fabsf(a.w);
    v[4] = fabsf(b.x); v[5] = fabsf(b.y); v[6] = fabsf(b.z); v[7] = fabsf(b.w);
  }
}
// ZEROES: many of the tiles are expected to hold nothing (padding comes by the thousand of equal scores).
template <int NOCT, bool ZEROES = false>
__device__ __forceinline__ float exact_score_of_octs(float (&v)[8], float eps_l1, float eps_log) {
  float L1 = tree8(v);
#pragma unroll
  for (int h = 1; h < NOCT; h *= 2) L1 = L1 + __shfl_xor_sync(kFull, L1, h);
  const float inv = __fdiv_rn(1.0f, L1 + eps_l1);
  if (ZEROES && __all_sync(kFull, L1 == 0.0f && inv <= 3.402823466e38f)) return 0.0f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float p = v[k] * inv;
    v[k] = p * lg2_fma(p + eps_log);
  }
  float S = tree8(v);
#pragma unroll
  for (int h = 1; h < NOCT; h *= 2) S = S + __shfl_xor_sync(kFull, S, h);
  return 0.0f - S;
}
template <int NOCT, bool BF16>
__device__ __forceinline__ float exact_score_coop(const uint8_t *tile, int o, float eps_l1, float eps_log) {
  float v[8];
  load_abs_oct_global<BF16>(tile, o, v);
  return exact_score_of_octs<NOCT>(v, eps_l1, eps_log);
}

// Exact scores of n consecutive tiles by a warp; `also`: a second copy of the scores, or null.  (Hardly ever run; out of line it
// costs every launch of its kernel 0.3 us all the same.)
template <int NOCT, bool BF16>
__device__ __forceinline__ void exact_scores_of(const uint8_t *tiles, uint32_t n, float eps_l1, float eps_log, float *scores, float *also) {
  const uint32_t lane = threadIdx.x & 31u, sub = lane % NOCT;
  __syncwarp();   // (other lanes have stored the screening scores)
  for (uint32_t t0 = 0; t0 < n; t0 += 32 / NOCT) {
    const uint32_t t = t0 + lane / NOCT;
    const bool live = t < n;
    const float ex = ranked_score(exact_score_coop<NOCT, BF16>(tiles + (live ? t : t0) * (uint32_t)(NOCT * 8 * (BF16 ? 2 : 4)), sub, eps_l1, eps_log));
    if (live && sub == 0) {
      scores[t] = ex;
      if (also) also[t] = ex;
    }
  }
}

// Order-preserving map binary32 -> uint32, and the 64-bit ranking key (score first, then the
// lower tile index wins): larger key = earlier in the ranking of Sec. 3.2.
__device__ __forceinline__ uint32_t score_key32(float s) {
  const uint32_t u = __float_as_uint(s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ uint64_t rank_key(float s, uint32_t idx_in_group) {
  return ((uint64_t)score_key32(s) << 32) | (uint64_t)(0xffffffffu - idx_in_group);
}
// ------------------------------------------------------------------------------------------
// Eq. 3-4 and the quantiser on a register-resident row
// ------------------------------------------------------------------------------------------

// In-thread butterfly (strides 1 .. EPT/2), neighbours first.
template <int N>
__device__ __forceinline__ void butterfly(float (&x)[N]) {
#pragma unroll
  for (int h = 1; h < N; h *= 2)
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (!(i & h)) {
        const float a = x[i], b = x[i + h];
        x[i] = a + b;
        x[i + h] = a - b;
      }
}

// The same butterfly on adjacent pairs p[i] = (x[2i], x[2i+1]): stride 1 works inside a pair, every
// larger stride adds and subtracts whole pairs (a - b is formed as fma(b, -1, a), which is exact).
template <int NPAIR>
__device__ __forceinline__ void butterfly2(float2 (&p)[NPAIR]) {
#pragma unroll
  for (int i = 0; i < NPAIR; ++i) p[i] = make_float2(p[i].x + p[i].y, p[i].x - p[i].y);
#pragma unroll
  for (int h = 1; h < NPAIR; h *= 2)
#pragma unroll
    for (int i = 0; i < NPAIR; ++i)
      if (!(i & h)) {
        const float2 a = p[i], b = p[i + h];
        p[i] = add2(a, b);
        p[i + h] = fma2(b, f2(-1.0f), a);
      }
}

// A row as adjacent pairs, widened to binary32.
template <class C>
__device__ __forceinline__ void load_row_pairs(const uint8_t *stage, int row, float2 (&p)[C::EPT / 2]) {
#pragma unroll
  for (int q = 0; q < C::CPR; ++q) {
    const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, q) * 16);
    if constexpr (C::BF16) {
      const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) bf2_add_f32(u[j], -0.0f, p[4 * q + j].x, p[4 * q + j].y);
    } else {
      p[2 * q] = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
      p[2 * q + 1] = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
    }
  }
}

// First index whose magnitude equals m (the row's largest magnitude), scanning the row in shared memory.
template <class C>
__device__ __forceinline__ int row_first_index_of(const uint8_t *stage, int row, float m) {
  int qhit = C::CPR - 1;
  if constexpr (C::BF16) {
    const uint32_t pat = __float_as_uint(m) >> 16;
#pragma unroll
    for (int q = C::CPR - 1; q >= 0; --q) {   // last assignment wins: the lowest chunk that holds the maximum
      const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, q) * 16);
      const uint32_t t = bf2_max_abs(bf2_max_abs(w.x, w.y), bf2_max_abs(w.z, w.w)) & 0x7fff7fffu;
      qhit = (max(t & 0xffffu, t >> 16) == pat) ? q : qhit;
    }
    const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, qhit) * 16);
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
    int k = 7;
#pragma unroll
    for (int j = 3; j >= 0; --j) {
      k = ((u[j] >> 16) & 0x7fffu) == pat ? 2 * j + 1 : k;
      k = (u[j] & 0x7fffu) == pat ? 2 * j : k;
    }
    return qhit * 8 + k;
  } else {
#pragma unroll
    for (int q = C::CPR - 1; q >= 0; --q) {
      const float4 v = *reinterpret_cast<const float4 *>(stage + (size_t)phys_chunk<C>(row, q) * 16);
      const float t = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
      qhit = (t == m) ? q : qhit;
    }
    const float4 v = *reinterpret_cast<const float4 *>(stage + (size_t)phys_chunk<C>(row, qhit) * 16);
    int k = 3;
    k = fabsf(v.z) == m ? 2 : k;
    k = fabsf(v.y) == m ? 1 : k;
    k = fabsf(v.x) == m ? 0 : k;
    return qhit * 4 + k;
  }
}

// Swap elements 0 and d of a row held in shared memory (the pivot swap P_d, its own inverse).
template <class C, bool F32>
__device__ __forceinline__ void row_swap_0_d(uint8_t *stage, int row, int d) {
  constexpr int ES = F32 ? 4 : 2, EPC = 16 / ES;
  uint8_t *p0 = stage + (size_t)phys_chunk<C>(row, 0) * 16;
  uint8_t *pd = stage + (size_t)phys_chunk<C>(row, d / EPC) * 16 + (size_t)(d % EPC) * ES;
  if constexpr (F32) {
    const uint32_t a = *reinterpret_cast<uint32_t *>(p0), b = *reinterpret_cast<uint32_t *>(pd);
    *reinterpret_cast<uint32_t *>(p0) = b;
    *reinterpret_cast<uint32_t *>(pd) = a;
  } else {
    const uint16_t a = *reinterpret_cast<uint16_t *>(p0), b = *reinterpret_cast<uint16_t *>(pd);
    *reinterpret_cast<uint16_t *>(p0) = b;
    *reinterpret_cast<uint16_t *>(pd) = a;
  }
}

// Largest and second-largest magnitude of a row (Eq. 3), no index.
template <class C>
__device__ __forceinline__ void row_top2(const uint8_t *stage, int row, float &a1, float &a2) {
  if constexpr (C::BF16) {
    uint32_t p1 = 0, p2 = 0, q1 = 0, q2 = 0;   // two independent (largest, second) pairs per 16-bit lane
#pragma unroll
    for (int q = 0; q < C::CPR; ++q) {
      const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)phys_chunk<C>(row, q) * 16);
      p2 = bf2_max_abs(p2, bf2_min_abs(p1, w.x)); p1 = bf2_max_abs(p1, w.x);
      q2 = bf2_max_abs(q2, bf2_min_abs(q1, w.y)); q1 = bf2_max_abs(q1, w.y);
      p2 = bf2_max_abs(p2, bf2_min_abs(p1, w.z)); p1 = bf2_max_abs(p1, w.z);
      q2 = bf2_max_abs(q2, bf2_min_abs(q1, w.w)); q1 = bf2_max_abs(q1, w.w);
    }
    const uint32_t m1 = bf2_max_abs(p1, q1) & 0x7fff7fffu;
    const uint32_t m2 = bf2_max_abs(bf2_min_abs(p1, q1), bf2_max_abs(p2, q2)) & 0x7fff7fffu;
    const uint32_t e1 = m1 & 0xffffu, o1 = m1 >> 16, e2 = m2 & 0xffffu, o2 = m2 >> 16;
    a1 = __uint_as_float(max(e1, o1) << 16);
    a2 = __uint_as_float(max(min(e1, o1), max(e2, o2)) << 16);
  } else {
    float p1 = 0.0f, p2 = 0.0f, q1 = 0.0f, q2 = 0.0f;
#pragma unroll
    for (int q = 0; q < C::CPR; ++q) {
      const float4 v = *reinterpret_cast<const float4 *>(stage + (size_t)phys_chunk<C>(row, q) * 16);
      const float t0 = fabsf(v.x), t1 = fabsf(v.y), t2 = fabsf(v.z), t3 = fabsf(v.w);
      p2 = fmaxf(p2, fminf(p1, t0)); p1 = fmaxf(p1, t0);
      q2 = fmaxf(q2, fminf(q1, t1)); q1 = fmaxf(q1, t1);
      p2 = fmaxf(p2, fminf(p1, t2)); p1 = fmaxf(p1, t2);
      q2 = fmaxf(q2, fminf(q1, t3)); q1 = fmaxf(q1, t3);
    }
    a1 = fmaxf(p1, q1);
    a2 = fmaxf(fminf(p1, q1), fmaxf(p2, q2));
  }
}

__host__ __device__ constexpr uint64_t group_ones(int W, int GS) {
  uint64_t v = 0;
  for (int i = 0; i < GS; ++i) v |= 1ull << (W * i);
  return v;
}

// Codes -> little-endian bit stream.  t[k] = q_k + 1.5*2^23 as binary32 (the rounding trick leaves
// the integer code in the low mantissa bits); groups of codes are combined by multiply-adds on the
// raw bit patterns and the constant's contribution is subtracted once per group.
template <int W, int N, class F>
__device__ __forceinline__ void pack_magic(F &&t, uint32_t *w) {
  constexpr int GS = (W <= 4) ? 8 : 4;   // codes per group
  constexpr int GB = GS * W;             // bits per group (<= 32)
  constexpr int NG = N / GS;
  constexpr uint64_t ONES = group_ones(W, GS);   // sum of 2^(W*i), i < GS
  constexpr uint32_t KW = (uint32_t)((0x4B400000ull * ONES) & 0xffffffffull);
#pragma unroll
  for (int j = 0; j < N * W / 32; ++j) w[j] = 0;
#pragma unroll
  for (int j = 0; j < NG; ++j) {
    uint32_t acc = __float_as_uint(t(j * GS + GS - 1));
#pragma unroll
    for (int i = GS - 2; i >= 0; --i) acc = acc * (1u << W) + __float_as_uint(t(j * GS + i));
    const uint32_t g = acc - KW;
    const int bit = j * GB, wi = bit >> 5, sh = bit & 31;
    w[wi] |= g << sh;
    if (sh + GB > 32) w[wi + 1] |= g >> (32 - sh);
  }
}

// Bit stream -> dequantised values z + q*s (one fused multiply-add per code).  A code is turned into
// a float without being shifted down: its bits, masked in place at bit p of a word (or of the word's
// upper half), are OR-ed into the mantissa of 2^23, giving 2^23 + q*2^p exactly; subtracting 2^23 and
// multiplying by s*2^-p inside the fused multiply-add gives the same real product q*s, so the result
// is bit-identical to fma((float)q, s, z).
template <int W, int N>
__device__ __forceinline__ void unpack_dequant(const uint32_t *w, float s, float z, float (&x)[N]) {
  constexpr uint32_t M = (1u << W) - 1u;
  uint32_t two23;   // 2^23 as a bit pattern, kept in a register so that (src & mask) | 2^23 is one instruction
  asm volatile("mov.u32 %0, 0x4B000000;" : "=r"(two23));
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const int bit = k * W, j = bit >> 5, sh = bit & 31;
    uint32_t src;
    int p;
    if (sh + W <= 23) { src = w[j]; p = sh; }
    else if (sh + W <= 32) { src = w[j] >> 16; p = sh - 16; }
    else { src = __funnelshift_r(w[j], w[j + 1], sh); p = 0; }
    uint32_t m;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(m) : "r"(src), "r"(M << p), "r"(two23));   // (src & mask) | 2^23
    const float f = __uint_as_float(m) - 8388608.0f;   // q * 2^p, exact
    x[k] = __fmaf_rn(f, s * (1.0f / (float)(1u << p)), z);
  }
}

}  // namespace tahq
