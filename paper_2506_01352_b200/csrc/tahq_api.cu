// Host side of the C ABI declared in include/tahq.h: parameter validation, layout of the packed
// buffer and of the workspace, kernel selection and launches on the caller's stream.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>

#include "tahq_host.cuh"
#include "tahq_kernels.cuh"

namespace tahq {

extern thread_local int g_launches;
extern unsigned long long *g_trace;

static uint64_t up(uint64_t x, uint64_t a) { return (x + a - 1) / a * a; }

static tahq_status make_plan(const tahq_params *p, Plan *pl) {
  if (!p || p->struct_size != sizeof(tahq_params)) return TAHQ_ERR_INVALID_ARG;
  const uint32_t G = p->tile;
  if (G < 8 || G > 128 || (G & (G - 1))) return TAHQ_ERR_INVALID_ARG;
  if (p->dtype > 1 || p->rounding > 1) return TAHQ_ERR_INVALID_ARG;
  if (p->tokens == 0 || p->hidden == 0 || p->hidden % G) return TAHQ_ERR_INVALID_ARG;
  const uint64_t S = p->group_tokens ? p->group_tokens : p->tokens;
  if (p->tokens % S) return TAHQ_ERR_INVALID_ARG;
  const uint32_t beta = p->budget_millibits;
  if (beta < 2000 || beta > 8000) return TAHQ_ERR_INVALID_ARG;
  // varsigma must be a positive normal number: p + varsigma is split into exponent and mantissa
  if (!(p->tau >= 0.0f) || !(p->eps_l1 >= 0.0f) || !(p->eps_log >= 1.17549435e-38f) || !(p->eps_ratio >= 0.0f))
    return TAHQ_ERR_INVALID_ARG;
  const uint64_t M = p->hidden / G;
  if (p->tokens > (1ull << 40) / M) return TAHQ_ERR_INVALID_ARG;
  const uint32_t A = p->alloc_tile ? p->alloc_tile : G;   // allocation-tile width (Sec. 3.2)
  if (A % G || A > p->hidden || p->hidden % A) return TAHQ_ERR_INVALID_ARG;
  pl->alloc_m = A / G;
  tahq_layout &L = pl->L;
  L.n_tiles = p->tokens * M;
  L.tiles_per_group = S * M;
  L.n_groups = p->tokens / S;
  if (L.tiles_per_group >= (1ull << 32) || L.n_tiles >= (1ull << 36)) return TAHQ_ERR_INVALID_ARG;
  if (L.n_tiles > (1ull << 26)) return TAHQ_ERR_UNSUPPORTED;   // one call: up to 2^26 tiles (32-bit offsets inside a CTA's share)
  pl->f = beta % 1000;
  L.lo_bits = beta / 1000;
  L.hi_bits = pl->f ? L.lo_bits + 1 : L.lo_bits;
  pl->rank_per_group = L.tiles_per_group / pl->alloc_m;
  pl->rank_k = pl->rank_per_group * (uint64_t)pl->f / 1000u;
  L.k_hi = pl->rank_k * pl->alloc_m;
  L.payload_bytes = L.n_groups * (uint64_t)(G / 8) * (L.tiles_per_group * L.lo_bits + L.k_hi);
  L.off_bitmap = 128;
  L.off_scale_zero = up(L.off_bitmap + (L.n_tiles + 7) / 8, 128);
  L.off_pivot = up(L.off_scale_zero + 4 * L.n_tiles, 128);
  L.off_payload = up(L.off_pivot + L.n_tiles, 128);
  L.total_bytes = up(L.off_payload + L.payload_bytes, 128);
  if (pl->alloc_m > 1 && A > 8192) return TAHQ_ERR_UNSUPPORTED;

  pl->mixed = L.k_hi > 0;
  pl->whole_words = pl->alloc_m == 1 && L.tiles_per_group % 32 == 0;
  uint64_t o = 256;                                         // status word
  pl->ws_flags = o;  o += 8ull * kMaxGrid;
  pl->ws_zero_end = o;                                      // [0, ws_zero_end) is cleared by a decode with a look-back
  pl->ws_scores = o; o = up(o + (pl->mixed ? 4 * (L.n_tiles / pl->alloc_m) : 0), 256);
  pl->ws_pre = o;    o = up(o + (pl->mixed ? 4 * ((L.n_tiles + 31) / 32) : 0), 256);
  pl->ws_total = o;
  return TAHQ_OK;
}

static void fill_header(const tahq_params *p, const Plan &pl, uint32_t *h) {
  std::memset(h, 0, 128);
  h[22] = pl.alloc_m > 1 ? pl.alloc_m * p->tile : 0u;   // allocation-tile width when it is not the tile
  auto f2u = [](float f) { uint32_t u; std::memcpy(&u, &f, 4); return u; };
  auto put64 = [&](int w, uint64_t v) { h[w] = (uint32_t)v; h[w + 1] = (uint32_t)(v >> 32); };
  h[0] = 0x51484154u;  // "TAHQ"
  h[1] = 1;
  h[2] = p->dtype;
  h[3] = p->rounding;
  put64(4, p->tokens);
  h[6] = p->hidden;
  h[7] = p->tile;
  h[8] = (uint32_t)(pl.L.tiles_per_group / (p->hidden / p->tile));
  h[9] = p->budget_millibits;
  h[10] = f2u(p->tau);
  h[11] = f2u(p->eps_l1);
  h[12] = f2u(p->eps_log);
  h[13] = f2u(p->eps_ratio);
  put64(14, p->seed);
  put64(16, pl.L.n_tiles);
  put64(18, pl.L.payload_bytes);
  put64(20, pl.L.total_bytes);
}

static void fill_args(const tahq_params *p, const Plan &pl, uint8_t *ws, Args *a) {
  std::memset(a, 0, sizeof(*a));
  a->n_tiles = pl.L.n_tiles;
  a->tiles_per_group = pl.L.tiles_per_group;
  a->k_hi = pl.L.k_hi;
  a->rank_per_group = pl.rank_per_group;
  a->rank_k = pl.rank_k;
  a->alloc_m = pl.alloc_m;
  a->n_groups = pl.L.n_groups;
  a->lo = pl.L.lo_bits;
  a->mixed = pl.mixed;
  a->off_bitmap = pl.L.off_bitmap;
  a->off_sz = pl.L.off_scale_zero;
  a->off_pivot = pl.L.off_pivot;
  a->off_payload = pl.L.off_payload;
  a->payload_bytes = pl.L.payload_bytes;
  a->total_bytes = pl.L.total_bytes;
  a->tau = p->tau;
  a->eps_l1 = p->eps_l1;
  a->eps_log = p->eps_log;
  a->seed = p->seed;
  a->eps_ratio = p->eps_ratio;
  a->status = reinterpret_cast<uint32_t *>(ws);
  a->trace = g_trace;
  a->whole_words = pl.whole_words;
  a->pre = reinterpret_cast<uint32_t *>(ws + pl.ws_pre);
  a->scores = reinterpret_cast<float *>(ws + pl.ws_scores);
  a->bf16 = p->dtype == TAHQ_BF16;
  a->tile = p->tile;
  a->flags = reinterpret_cast<unsigned long long *>(ws + pl.ws_flags);
  // the screening score leaves varsigma out; its share of the score is below G * varsigma / ln 2
  a->exact_scores = pl.alloc_m > 1 || (double)p->tile * (double)p->eps_log > 1e-5;
  {   // 1024 bins for the scores up to two below the largest possible, 3072 above
    const float knee = std::log2((float)(pl.alloc_m * p->tile)) - 2.0f;
    a->step_lo = 16.0f * 1024.0f / knee;
    a->step_hi = 8.0f * 3064.0f;   // (a few bins are left for rounding above the largest)
    a->step_off = a->step_hi * knee - 16.0f * 1024.0f;
  }
  fill_header(p, pl, a->header);
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Scratch for tahq_encode_noalloc: part of the library image, resident on every GPU that loads it.
// In host code this name is only a handle; the device address is looked up once per device.
// Room for TAHQ_NOALLOC_SCRATCH_BYTES, and behind that for the offset prefixes of calls whose ranking groups are no whole words
// (4 bytes per 32 tiles, 2^26 tiles at most): the accepted calls are those that fit without them.
constexpr uint64_t kNoallocPrefixes = 8ull << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[TAHQ_NOALLOC_SCRATCH_BYTES + kNoallocPrefixes + 256];
static void *g_noalloc_addr[64];
static std::atomic<int> g_noalloc_ready[64];

}  // namespace tahq

using namespace tahq;

extern "C" {

size_t tahq_packed_bound(const tahq_params *p) {
  Plan pl;
  return make_plan(p, &pl) == TAHQ_OK ? (size_t)pl.L.total_bytes : 0;
}

tahq_status tahq_packed_layout(const tahq_params *p, tahq_layout *out) {
  Plan pl;
  const tahq_status s = make_plan(p, &pl);
  if (s != TAHQ_OK) return s;
  if (!out) return TAHQ_ERR_INVALID_ARG;
  *out = pl.L;
  return TAHQ_OK;
}

size_t tahq_workspace_bound(const tahq_params *p) {
  Plan pl;
  return make_plan(p, &pl) == TAHQ_OK ? (size_t)pl.ws_total : 0;
}

tahq_status tahq_encode(const tahq_params *p, const void *d_in, void *d_packed, size_t packed_cap, void *d_ws,
                        size_t ws_cap, tahq_stream stream) {
  g_launches = 0;
  Plan pl;
  const tahq_status s = make_plan(p, &pl);
  if (s != TAHQ_OK) return s;
  if (!d_in || !d_packed || !d_ws) return TAHQ_ERR_INVALID_ARG;
  if (packed_cap < pl.L.total_bytes || ws_cap < pl.ws_total) return TAHQ_ERR_BUFFER_TOO_SMALL;
  if (!aligned16(d_in) || !aligned16(d_packed) || !aligned16(d_ws)) return TAHQ_ERR_MISALIGNED;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  Args a;
  fill_args(p, pl, static_cast<uint8_t *>(d_ws), &a);
  a.in = static_cast<const uint8_t *>(d_in);
  a.packed = static_cast<uint8_t *>(d_packed);
  // The selection of a group of more than 32 * kWordsShared tiles keeps the words of its slices, and their running counts,
  // where quantise + pack puts the codes afterwards: 8 bytes per 32 ranked tiles (and 16 words more), whose codes are 64 and up.
  a.words = reinterpret_cast<uint32_t *>(a.packed + a.off_payload);
  // groups that share words of the bit map: the selection puts those together on zeroes
  if (pl.mixed && !pl.whole_words && pl.alloc_m == 1 &&
      launch_clear(a.packed + a.off_bitmap, up((pl.L.n_tiles + 7) / 8, 128), st) != TAHQ_OK)
    return TAHQ_ERR_CUDA;
  const bool bf = p->dtype == TAHQ_BF16, sr = p->rounding == 1;
  switch (p->tile) {
    case 8: return bf ? encode_cfg<8, true>(pl, a, sr, st) : encode_cfg<8, false>(pl, a, sr, st);
    case 16: return bf ? encode_cfg<16, true>(pl, a, sr, st) : encode_cfg<16, false>(pl, a, sr, st);
    case 32: return bf ? encode_cfg<32, true>(pl, a, sr, st) : encode_cfg<32, false>(pl, a, sr, st);
    case 64: return bf ? encode_cfg<64, true>(pl, a, sr, st) : encode_cfg<64, false>(pl, a, sr, st);
    default: return bf ? encode_cfg<128, true>(pl, a, sr, st) : encode_cfg<128, false>(pl, a, sr, st);
  }
}

tahq_status tahq_decode(const tahq_params *p, const void *d_packed, size_t packed_bytes, void *d_out, void *d_ws,
                        size_t ws_cap, tahq_stream stream) {
  g_launches = 0;
  Plan pl;
  const tahq_status s = make_plan(p, &pl);
  if (s != TAHQ_OK) return s;
  if (!d_out || !d_packed || !d_ws) return TAHQ_ERR_INVALID_ARG;
  if (packed_bytes < pl.L.total_bytes || ws_cap < pl.ws_total) return TAHQ_ERR_BUFFER_TOO_SMALL;
  if (!aligned16(d_out) || !aligned16(d_packed) || !aligned16(d_ws)) return TAHQ_ERR_MISALIGNED;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  Args a;
  fill_args(p, pl, static_cast<uint8_t *>(d_ws), &a);
  a.packed = const_cast<uint8_t *>(static_cast<const uint8_t *>(d_packed));
  a.out = static_cast<uint8_t *>(d_out);
  // Up to 65536 bit-map words (256 KiB), and with one width, the kernels need no look-back and nothing cleared: one launch.
  a.own_prefix = (p->tile >= 32 && !pl.mixed) || (pl.L.n_tiles + 31) / 32 <= 65536;
  if (!a.own_prefix && launch_clear(d_ws, pl.ws_zero_end, st) != TAHQ_OK) return TAHQ_ERR_CUDA;   // status + flags
  const bool bf = p->dtype == TAHQ_BF16;
  switch (p->tile) {
    case 8: return bf ? decode_cfg<8, true>(pl, a, st) : decode_cfg<8, false>(pl, a, st);
    case 16: return bf ? decode_cfg<16, true>(pl, a, st) : decode_cfg<16, false>(pl, a, st);
    case 32: return bf ? decode_cfg<32, true>(pl, a, st) : decode_cfg<32, false>(pl, a, st);
    case 64: return bf ? decode_cfg<64, true>(pl, a, st) : decode_cfg<64, false>(pl, a, st);
    default: return bf ? decode_cfg<128, true>(pl, a, st) : decode_cfg<128, false>(pl, a, st);
  }
}

tahq_status tahq_encode_noalloc(const tahq_params *p, const void *d_in, void *d_packed, size_t packed_cap,
                                tahq_stream stream) {
  g_launches = 0;
  Plan pl;
  const tahq_status s = make_plan(p, &pl);
  if (s != TAHQ_OK) return s;
  if ((pl.whole_words ? pl.ws_total : pl.ws_pre) > (uint64_t)TAHQ_NOALLOC_SCRATCH_BYTES) return TAHQ_ERR_TOO_LARGE;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return TAHQ_ERR_CUDA;
  if (!g_noalloc_ready[dev].load(std::memory_order_acquire)) {
    // set-up, once per device, with that device current: the device address behind the symbol
    void *ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return TAHQ_ERR_CUDA;
    g_noalloc_addr[dev] = ptr;
    g_noalloc_ready[dev].store(1, std::memory_order_release);
  }
  return tahq_encode(p, d_in, d_packed, packed_cap, g_noalloc_addr[dev], sizeof(g_noalloc_scratch), stream);
}

// ---- fixed-point gradient compressor -------------------------------------------------------------------
namespace {
struct QPlan { uint64_t n_scales, off_scales, off_payload, row_bytes, total_bytes; };
tahq_status q_plan(const tahq_qnaive_params *p, QPlan *q) {
  if (!p || p->struct_size != sizeof(tahq_qnaive_params)) return TAHQ_ERR_INVALID_ARG;
  if (p->dtype > 1 || p->per_tensor > 1) return TAHQ_ERR_INVALID_ARG;
  if (p->tokens == 0 || p->hidden == 0 || p->hidden % 8) return TAHQ_ERR_INVALID_ARG;
  if (p->bits < 2 || p->bits > 16) return TAHQ_ERR_INVALID_ARG;
  if (!(p->prescale > 0.0f) || p->prescale > 3.402823466e38f) return TAHQ_ERR_INVALID_ARG;
  q->n_scales = p->per_tensor ? 1 : p->tokens;
  q->row_bytes = up(((uint64_t)p->hidden * p->bits + 7) / 8, 16);
  q->off_scales = 128;
  q->off_payload = up(q->off_scales + 4 * q->n_scales, 128);
  q->total_bytes = up(q->off_payload + p->tokens * q->row_bytes, 128);
  return TAHQ_OK;
}
void q_args(const tahq_qnaive_params *p, const QPlan &q, QArgs *a, void *ws) {
  std::memset(a, 0, sizeof(*a));
  a->tokens = p->tokens; a->hidden = p->hidden; a->bits = p->bits; a->per_tensor = p->per_tensor;
  a->prescale = p->prescale;
  a->off_scales = q.off_scales; a->off_payload = q.off_payload; a->row_bytes = q.row_bytes; a->total_bytes = q.total_bytes;
  a->status = reinterpret_cast<uint32_t *>(ws);
  a->gmax = reinterpret_cast<uint32_t *>(ws) + 16;
  uint32_t *h = a->header;
  std::memcpy(h, "TAHN", 4);
  h[1] = 1; h[2] = p->dtype; h[3] = p->bits;
  h[4] = (uint32_t)p->tokens; h[5] = (uint32_t)(p->tokens >> 32);
  h[6] = p->hidden; h[7] = p->per_tensor;
  std::memcpy(&h[8], &p->prescale, 4);
  h[10] = (uint32_t)q.row_bytes; h[11] = (uint32_t)(q.row_bytes >> 32);
  h[12] = (uint32_t)q.total_bytes; h[13] = (uint32_t)(q.total_bytes >> 32);
}
}  // namespace

size_t tahq_qnaive_packed_bound(const tahq_qnaive_params *p) {
  QPlan q;
  return q_plan(p, &q) == TAHQ_OK ? (size_t)q.total_bytes : 0;
}

size_t tahq_qnaive_workspace_bound(const tahq_qnaive_params *p) {
  QPlan q;
  return q_plan(p, &q) == TAHQ_OK ? 256 : 0;
}

tahq_status tahq_qnaive_encode(const tahq_qnaive_params *p, const void *d_in, void *d_packed, size_t packed_cap,
                               void *d_ws, size_t ws_cap, tahq_stream stream) {
  QPlan q;
  g_launches = 0;
  if (tahq_status rc = q_plan(p, &q)) return rc;
  if (!d_in || !d_packed || !d_ws) return TAHQ_ERR_INVALID_ARG;
  if (packed_cap < q.total_bytes || ws_cap < 256) return TAHQ_ERR_BUFFER_TOO_SMALL;
  if (!aligned16(d_in) || !aligned16(d_packed) || !aligned16(d_ws)) return TAHQ_ERR_MISALIGNED;
  DevInfo d;
  if (!dev_info(&d)) return TAHQ_ERR_CUDA;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  QArgs a;
  q_args(p, q, &a, d_ws);
  a.in = static_cast<const uint8_t *>(d_in);
  a.packed = static_cast<uint8_t *>(d_packed);
  if (p->per_tensor && launch_clear(d_ws, 256, st) != TAHQ_OK) return TAHQ_ERR_CUDA;   // the maximum is formed there
  return p->dtype == TAHQ_BF16 ? qnaive_encode_cfg<true>(a, d, st) : qnaive_encode_cfg<false>(a, d, st);
}

tahq_status tahq_qnaive_decode(const tahq_qnaive_params *p, const void *d_packed, size_t packed_bytes, void *d_out,
                               void *d_ws, size_t ws_cap, tahq_stream stream) {
  QPlan q;
  g_launches = 0;
  if (tahq_status rc = q_plan(p, &q)) return rc;
  if (!d_packed || !d_out || !d_ws) return TAHQ_ERR_INVALID_ARG;
  if (packed_bytes < q.total_bytes || ws_cap < 256) return TAHQ_ERR_BUFFER_TOO_SMALL;
  if (!aligned16(d_packed) || !aligned16(d_out) || !aligned16(d_ws)) return TAHQ_ERR_MISALIGNED;
  DevInfo d;
  if (!dev_info(&d)) return TAHQ_ERR_CUDA;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  QArgs a;
  q_args(p, q, &a, d_ws);
  a.packed = const_cast<uint8_t *>(static_cast<const uint8_t *>(d_packed));
  a.out = static_cast<uint8_t *>(d_out);
  return p->dtype == TAHQ_BF16 ? qnaive_decode_cfg<true>(a, d, st) : qnaive_decode_cfg<false>(a, d, st);
}

tahq_status tahq_selftest_wait_timeout(void *d_ws, size_t ws_cap, tahq_stream stream) {
  if (!d_ws) return TAHQ_ERR_INVALID_ARG;
  if (ws_cap < 256 + 8ull * kMaxGrid) return TAHQ_ERR_BUFFER_TOO_SMALL;
  if (!aligned16(d_ws)) return TAHQ_ERR_MISALIGNED;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(d_ws, 0, 256 + 8ull * kMaxGrid, st) != cudaSuccess) return TAHQ_ERR_CUDA;
  Args a;
  std::memset(&a, 0, sizeof(a));
  a.status = reinterpret_cast<uint32_t *>(d_ws);
  a.flags = reinterpret_cast<unsigned long long *>(static_cast<uint8_t *>(d_ws) + 256);
  return launch_wait_selftest(a, st);
}

const char *tahq_status_string(tahq_status s) {
  switch (s) {
    case TAHQ_OK: return "ok";
    case TAHQ_ERR_INVALID_ARG: return "invalid argument";
    case TAHQ_ERR_UNSUPPORTED: return "unsupported configuration";
    case TAHQ_ERR_BUFFER_TOO_SMALL: return "buffer too small";
    case TAHQ_ERR_MISALIGNED: return "pointer not 16-byte aligned";
    case TAHQ_ERR_CUDA: return "CUDA runtime error";
    case TAHQ_ERR_TOO_LARGE: return "tensor needs more scratch than the built-in buffer of tahq_encode_noalloc";
  }
  return "unknown status";
}

}  // extern "C"
