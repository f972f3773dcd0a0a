// Parts of the library that are compiled once: launch bookkeeping, device queries, the tensor-map
// encoder, and the launches of the kernels that do not depend on the tile configuration.
#include <cstring>
#include <mutex>
#include <vector>

#include "tahq_host.cuh"
#include "tahq_select_launch.cuh"

namespace tahq {

// Zeroes 16-byte pieces; the call's first tile kernel is launched as its programmatic dependent.
__global__ void __launch_bounds__(kThreads) clear_kernel(uint4 *p, uint64_t n16, unsigned long long *trace_buf) {
  TraceScope trace(trace_buf, 0);
  grid_dependency_wait();
  for (uint64_t i = blockIdx.x * (uint64_t)kThreads + threadIdx.x; i < n16; i += (uint64_t)gridDim.x * kThreads)
    p[i] = make_uint4(0, 0, 0, 0);
}

// Self-test of the bounded waits: CTA 1 waits for a count that CTA 0 never publishes.  The wait gives
// up after kSpinLimit polls, the status word gets TAHQ_DEV_TIMEOUT, and the kernel returns.
__global__ void __launch_bounds__(kThreads) wait_selftest_kernel(const Args a) {
  if (blockIdx.x == 0) return;
  bool unused;
  cta_exclusive_prefix(a, 1, false, unused);
}

// ---- launch bookkeeping --------------------------------------------------------------------------------
thread_local int g_launches = 0;
unsigned long long *g_trace = nullptr;   // tahq_trace

// Optional per-kernel timing (tahq_profile): every launch is bracketed by two events on its stream.
struct ProfRec { const char *name; cudaEvent_t e0, e1; };
static std::atomic<bool> g_prof_on{false};
static std::mutex g_prof_mu;
static std::vector<ProfRec> g_prof;
static thread_local cudaEvent_t g_open_e1 = nullptr;   // end event of the launch this thread is inside

void note_launch(const char *name, cudaStream_t st, bool begin) {
  if (begin) {
    ++g_launches;
    if (!g_prof_on.load(std::memory_order_relaxed)) return;
    ProfRec r{name, nullptr, nullptr};
    cudaEventCreate(&r.e0);
    cudaEventCreate(&r.e1);
    cudaEventRecord(r.e0, st);
    g_open_e1 = r.e1;
    std::lock_guard<std::mutex> lk(g_prof_mu);
    g_prof.push_back(r);
  } else if (g_open_e1) {
    cudaEventRecord(g_open_e1, st);
    g_open_e1 = nullptr;
  }
}

bool dev_info(DevInfo *d) {
  if (cudaGetDevice(&d->dev) != cudaSuccess) return false;
  static std::atomic<int> sms[64];
  int v = sms[d->dev & 63].load(std::memory_order_acquire);
  if (v <= 0) {
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, d->dev) != cudaSuccess) return false;
    sms[d->dev & 63].store(v, std::memory_order_release);
  }
  d->sms = v;
  return true;
}

unsigned persistent_grid(uint64_t n_chunks, const DevInfo &d, int occ) {
  uint64_t cap = (uint64_t)d.sms * occ;
  if (cap > (uint64_t)kMaxGrid) cap = kMaxGrid;
  return (unsigned)(n_chunks < cap ? n_chunks : cap);
}

// The driver's encoder is looked up once through the runtime (no link-time dependency on libcuda).
bool make_row_map(const void *base, uint64_t n_rows, bool bf16, CUtensorMap *tm) {
  std::memset(tm, 0, sizeof(*tm));
  if (n_rows >= 0x7fffffe0ull) return false;   // row coordinates are 32-bit
  typedef CUresult (*encode_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static encode_fn enc = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<encode_fn>(f);
  }();
  if (!enc) { cudaGetLastError(); return false; }
  const cuuint32_t per_row = bf16 ? 64u : 32u;   // elements in 128 bytes
  const cuuint64_t dims[2] = {(cuuint64_t)per_row, (cuuint64_t)n_rows};
  const cuuint64_t strides[1] = {128};
  const cuuint32_t box[2] = {per_row, 32};
  const cuuint32_t estr[2] = {1, 1};
  return enc(tm, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
             const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- kernels that do not depend on the tile configuration ---------------------------------------------

// Zero `bytes` (a multiple of 16) with a kernel, so that the call's next kernel can be its programmatic dependent.
tahq_status launch_clear(void *p, uint64_t bytes, cudaStream_t st) {
  const uint64_t n16 = bytes / 16;
  uint64_t grid = (n16 + kThreads - 1) / kThreads;
  grid = grid < 1 ? 1 : grid > 592 ? 592 : grid;
  TAHQ_LAUNCH("clear", st, launch_dependent(clear_kernel, (unsigned)grid, kThreads, 0, st, static_cast<uint4 *>(p), n16, g_trace));
  return cudaGetLastError() == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}

tahq_status launch_select(const Args &a, const DevInfo &d, cudaStream_t st) { return launch_select_with<void>(a, d, st); }

tahq_status launch_alloc_score(const Args &a, const DevInfo &d, cudaStream_t st) {
  const uint64_t n_alloc = a.n_tiles / a.alloc_m;
  const uint64_t want = (n_alloc + kThreads / 32 - 1) / (kThreads / 32), cap = (uint64_t)d.sms * 8;
  const unsigned grid = (unsigned)(want < cap ? want : cap);
  // a tile of up to 256 or 512 channels has one or two rounds: more at a time would be padding
  const uint32_t A = a.alloc_m * a.tile;
  void (*const kernels[6])(Args) = {alloc_score_kernel<false, 1>, alloc_score_kernel<false, 2>, alloc_score_kernel<false, 4>,
                                    alloc_score_kernel<true, 1>,  alloc_score_kernel<true, 2>,  alloc_score_kernel<true, 4>};
  cudaError_t e;
  TAHQ_LAUNCH("alloc_score", st,
              e = launch_dependent(kernels[3 * a.bf16 + (A <= 256 ? 0 : A <= 512 ? 1 : 2)], grid, kThreads, 0, st, a));
  return e == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}

tahq_status launch_wait_selftest(const Args &a, cudaStream_t st) {
  wait_selftest_kernel<<<2, kThreads, 0, st>>>(a);
  return cudaGetLastError() == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}

}  // namespace tahq

using namespace tahq;

extern "C" {

int tahq_last_launch_count(void) { return g_launches; }

void tahq_trace(void *d_buf) { g_trace = static_cast<unsigned long long *>(d_buf); }

void tahq_profile(int enable) {
  std::lock_guard<std::mutex> lk(g_prof_mu);
  g_prof_on.store(enable != 0);
  if (enable) {
    for (auto &r : g_prof) { cudaEventDestroy(r.e0); cudaEventDestroy(r.e1); }
    g_prof.clear();
  }
}

int tahq_profile_read(char *names, float *ms, int max_records) {
  std::lock_guard<std::mutex> lk(g_prof_mu);
  int n = 0;
  for (auto &r : g_prof) {
    if (n < max_records) {
      cudaEventSynchronize(r.e1);
      float t = 0.0f;
      cudaEventElapsedTime(&t, r.e0, r.e1);
      if (ms) ms[n] = t;
      if (names) { std::strncpy(names + 32 * n, r.name, 31); names[32 * n + 31] = 0; }
      ++n;
    }
    cudaEventDestroy(r.e0);
    cudaEventDestroy(r.e1);
  }
  g_prof.clear();
  return n;
}

}  // extern "C"
