// Host side of the selection: cluster size, launch.  Included where a variant of the kernel is instantiated: once for scores
// that a kernel in front has formed (tahq_common.cu), once per tile configuration that forms them itself (inst_*.cu).
#pragma once

#include <type_traits>

#include "tahq_host.cuh"
#include "tahq_select.cuh"

namespace tahq {

constexpr size_t kSelSmem = (size_t)(kClKeys + kSelThreads) * 8 + (size_t)kBins * 4 + (size_t)kClKeys * 4 + (size_t)kWordsShared * 4;

// HELD of the second variant: where the scores are formed in the kernel (fuse_scores) every slice is held.
template <class C>
constexpr bool kLongSlices = !std::is_void<C>::value;

template <class C>
static bool select_ready(int dev) {
  static std::atomic<int> ready[64];
  if (ready[dev & 63].load(std::memory_order_acquire)) return true;
  for (auto kernel : {select_kernel<true, C>, select_kernel<kLongSlices<C>, C>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSelSmem) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
  ready[dev & 63].store(1, std::memory_order_release);
  return true;
}

static void cluster_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attr, unsigned grid, uint32_t cs, cudaStream_t st) {
  *cfg = {};
  cfg->gridDim = dim3(grid);
  cfg->blockDim = dim3(kSelThreads);
  cfg->dynamicSmemBytes = kSelSmem;
  cfg->stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

// Clusters of 2^lg CTAs of the selection kernel that the device holds at the same time (asked once per device and size).
// More ranking groups than that run in waves, each wave the whole chain of dependent steps.  0: cannot be asked.
template <class C>
static uint32_t select_capacity(int dev, int lg) {
  static std::atomic<int> cache[64][5];   // capacity + 1
  std::atomic<int> &slot = cache[dev & 63][lg];
  const int v = slot.load(std::memory_order_acquire);
  if (v > 0) return (uint32_t)(v - 1);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cluster_config(&cfg, attr, 1u << lg, 1u << lg, nullptr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, select_kernel<true, C>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); return 0; }
  slot.store(n + 1, std::memory_order_release);
  return (uint32_t)n;
}

// CTAs of a ranking group, as a power of two.  The smallest cluster whose threads can hold their scores in registers (8192 x
// 768 in 8 groups of 12288: 5.9 us in clusters of 4, 8 us in clusters of 16) -- or, where the scores are formed there, the
// largest that still has a warp's round for every warp --, at most 16 CTAs, and one of which the device holds one per group
// at once.
template <class C>
static int select_cluster_size(const Args &a, const DevInfo &d) {
  uint64_t slice = (uint64_t)kHeld * kSelThreads;
  if constexpr (!std::is_void<C>::value) slice = (uint64_t)LaneCfg<C>::TPR * (kSelThreads / 32);
  int lg = 4;
  while (lg > 0 && (a.rank_per_group <= slice << (lg - 1) || a.n_groups > select_capacity<C>(d.dev, lg))) --lg;
  return lg;
}

// Are the scores of this call formed in the selection kernel?  A launch less, and they are binned from shared memory; but a
// group's tensor then goes through the few SMs of its cluster, and the scores of many clusters crowd each other where a grid
// of score CTAs spreads evenly.  Encode (us), scores in front -> fused.  Elements per CTA: 3 x 256 x 640 fp32 (48 CTAs of
// 10240) 13.5 -> 12.0, 16 x 128 x 512 bf16 (64 CTAs of 16384) 12.1 -> 11.5; 1 x 512 x 768 bf16 (16 of 24576) 12.0 -> 12.2.
// CTAs: groups of 16 x 1024 bf16, which have one each, gain at every number (74: 12.4 -> 11.5, 148: 13.9 -> 12.7, 296: 17.0 ->
// 15.8), groups of two CTAs up to about half of the SMs (40 groups of 32 x 1024 12.7 -> 12.0, 80 groups 14.4 -> 15.0): the line is
// where both gain.  Groups that share words of the bit map have its clear in front anyway.
template <class C>
static bool fuse_scores(const Args &a, const DevInfo &d) {
  if (!a.whole_words || a.exact_scores || !select_ready<C>(d.dev)) return false;
  const uint32_t cs = 1u << select_cluster_size<C>(a, d);
  return a.rank_per_group * C::G <= 16384ull * cs && a.n_groups * cs <= (uint64_t)d.sms / 2;
}

// One cluster per ranking group, launched as a programmatic dependent of the score kernel.
template <class C>
tahq_status launch_select_with(const Args &a, const DevInfo &d, cudaStream_t st) {
  if (!select_ready<C>(d.dev)) return TAHQ_ERR_CUDA;
  const int lg = select_cluster_size<C>(a, d);
  const uint32_t cs = 1u << lg, per_cta = (uint32_t)(((a.rank_per_group + cs - 1) / cs + 31) / 32 * 32);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  cluster_config(&cfg, attr, (unsigned)(a.n_groups * cs), cs, st);
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  cudaError_t e;
  const auto kernel = per_cta <= (uint32_t)(kHeld * kSelThreads) ? select_kernel<true, C> : select_kernel<kLongSlices<C>, C>;
  TAHQ_LAUNCH("select", st, e = cudaLaunchKernelEx(&cfg, kernel, a, per_cta));
  return e == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}

}  // namespace tahq
