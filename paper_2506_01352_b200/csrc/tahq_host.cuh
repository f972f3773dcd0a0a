// Host-side declarations shared by the translation units of the library: the plan of a call (layout of the
// packed buffer and of the workspace), launch helpers, and the per-(tile width, element type) launchers that
// each instantiation unit defines.
#pragma once

#include <cuda.h>   // CUtensorMap (type only; the driver's encoder is looked up at run time)
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/tahq.h"
#include "../../include/tahq_testing.h"

namespace tahq {

struct Args;

struct Plan {
  tahq_layout L;
  uint32_t f;             // budget % 1000
  bool mixed;             // two widths in use (k_hi > 0)
  bool whole_words;       // ranking groups are whole words of the bit map and A = G
  uint32_t alloc_m;            // quantisation tiles per allocation tile (Sec. 3.2; 1 by default)
  uint64_t rank_per_group, rank_k;   // allocation tiles per ranking group, and how many of them get the higher width
  // workspace offsets
  uint64_t ws_flags, ws_zero_end, ws_scores, ws_pre, ws_total;   // (ws_pre: the last section)
};

// ---- launch bookkeeping --------------------------------------------------------------------------------
// Every launch of the library goes through TAHQ_LAUNCH: it counts the launch for the calling thread and,
// while tahq_profile is on, brackets it with two events on its stream.
void note_launch(const char *name, cudaStream_t st, bool begin);
struct LaunchScope {
  const char *name;
  cudaStream_t st;
  LaunchScope(const char *n, cudaStream_t s) : name(n), st(s) { note_launch(name, st, true); }
  ~LaunchScope() { note_launch(name, st, false); }
};
#define TAHQ_LAUNCH(name, st, ...) do { ::tahq::LaunchScope scope_(name, st); __VA_ARGS__; } while (0)

struct DevInfo { int dev, sms; };
bool dev_info(DevInfo *d);

// CTAs of a persistent tile kernel: every SM filled to the kernel's occupancy, never more than chunks.
unsigned persistent_grid(uint64_t n_chunks, const DevInfo &d, int occ);

// Tensor map of a row-major byte buffer seen as [n_rows x 128 bytes], boxes of 32 rows, 128-byte swizzle
// (`elem` = the element type the rows hold; it only labels the map).  False when TMA cannot be used here.
bool make_row_map(const void *base, uint64_t n_rows, bool bf16, CUtensorMap *tm);

// Opt a kernel into its dynamic shared memory once per device and return resident CTAs per SM (0: failed).
template <class K>
int prepare(K kernel, int threads, int smem, const DevInfo &d, std::atomic<int> *cache) {
  int v = cache[d.dev & 63].load(std::memory_order_acquire);
  if (v > 0) return v;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return 0;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem) != cudaSuccess || occ < 1) return 0;
  cache[d.dev & 63].store(occ, std::memory_order_release);
  return occ;
}

// Launch a kernel as a programmatic dependent of the kernel in front of it in the stream: the launch is set up
// while that kernel still runs (about 2 us less per kernel boundary, measured); the kernel starts with
// griddepcontrol.wait, so it reads nothing before that kernel is done.
template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                             A &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  if (e == cudaErrorNotSupported || e == cudaErrorInvalidValue) {   // attribute refused: an ordinary launch does
    (void)cudaGetLastError();
    cfg.numAttrs = 0;
    e = cudaLaunchKernelEx(&cfg, kernel, args...);
  }
  return e;
}

// ---- kernels that do not depend on the tile configuration (tahq_common.cu) ------------------------------
tahq_status launch_clear(void *p, uint64_t bytes, cudaStream_t st);
tahq_status launch_select(const Args &a, const DevInfo &d, cudaStream_t st);
tahq_status launch_alloc_score(const Args &a, const DevInfo &d, cudaStream_t st);
tahq_status launch_wait_selftest(const Args &a, cudaStream_t st);

// ---- per-configuration launchers: one explicit instantiation per translation unit (inst_*.cu) -----------
template <int G, bool BF16>
tahq_status encode_cfg(const Plan &pl, const Args &a, bool stochastic, cudaStream_t st);
template <int G, bool BF16>
tahq_status decode_cfg(const Plan &pl, const Args &a, cudaStream_t st);

// ---- fixed-point gradient compressor (qnaive.cuh; instantiated in qnaive_*.cu) -------------------------
struct QArgs {
  const uint8_t *in;      // encode: tensor
  uint8_t *packed;
  uint8_t *out;           // decode: tensor
  uint64_t tokens;
  uint32_t hidden, bits, per_tensor;
  float prescale;
  uint64_t off_scales, off_payload, row_bytes, total_bytes;
  uint32_t *gmax;         // per-tensor mode: bits of max |g| (zeroed per call)
  uint32_t *status;
  uint32_t pieces;        // decode: pieces of a row
  uint32_t row_warps;     // encode: warps that share a row (1: a warp takes one or more whole rows)
  uint32_t row_lanes;     // encode, row_warps = 1: lanes of a row, a power of two
  uint32_t header[16];
};

template <bool BF16>
tahq_status qnaive_encode_cfg(const QArgs &a, const DevInfo &d, cudaStream_t st);
template <bool BF16>
tahq_status qnaive_decode_cfg(const QArgs &a, const DevInfo &d, cudaStream_t st);

}  // namespace tahq
