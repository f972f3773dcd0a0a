// Kernel selection and launches for one (tile width, element type): included by the instantiation units
// (inst_*.cu), each of which compiles the tile kernels of one configuration.
#pragma once

#include "tahq_host.cuh"
#include "tahq_lanes.cuh"
#include "tahq_select_launch.cuh"

namespace tahq {

template <class C, bool SR>
static tahq_status encode_t(const Plan &pl, const Args &a_in, cudaStream_t st) {
  DevInfo d;
  if (!dev_info(&d)) return TAHQ_ERR_CUDA;
  Args a = a_in;
  CUtensorMap tmap;
  a.use_tma = (C::ROWB == 128 && make_row_map(a.in, a.n_tiles * C::LPT, C::BF16, &tmap)) ? 1u : 0u;   // rows of 128 bytes
  bool fused = false;
  if constexpr (C::G >= 32) {
    if (pl.mixed && fuse_scores<C>(a, d)) {
      fused = true;
      if (launch_select_with<C>(a, d, st) != TAHQ_OK) return TAHQ_ERR_CUDA;
    }
  }
  if (pl.mixed && !fused) {
    if (pl.alloc_m > 1) {   // Sec. 3.2 with A = m * G: one warp per allocation tile, exact scores
      if (launch_alloc_score(a, d, st) != TAHQ_OK) return TAHQ_ERR_CUDA;
    } else if (C::G >= 32 && C::BF16 && !a.exact_scores) {
      if constexpr (C::G >= 32 && C::BF16) {
        const bool wide_ld = (reinterpret_cast<uintptr_t>(a.in) & 31u) == 0;   // 256-bit loads where the tensor is aligned to them
        const uint64_t n_rounds = (a.n_tiles + LaneCfg<C>::TPR - 1) / LaneCfg<C>::TPR;
        const unsigned grid = persistent_grid((n_rounds + 3) / 4, d, 2);
        if (wide_ld) TAHQ_LAUNCH("stats", st, launch_dependent(score_lanes_kernel<C, true>, grid, kScoreThreads, 0, st, a));
        else TAHQ_LAUNCH("stats", st, launch_dependent(score_lanes_kernel<C, false>, grid, kScoreThreads, 0, st, a));
      }
    } else {
      constexpr int NS = C::ROWB <= 128 ? 3 : 2;
      const int smem = kWarps * NS * StreamCfg<C>::UNIT_BYTES + 256;   // ring slots, then the warps' mbarriers
      static std::atomic<int> occ_sc[64], occ_sc_exact[64];
      const uint64_t n_units = (a.n_tiles * C::LPT + 31) / 32;
      // one CTA per SM: the kernel is bound by DRAM, and fewer, longer streams measured a little faster
      const unsigned grid = persistent_grid((n_units + kWarps - 1) / kWarps, d, 1);
      if (a.exact_scores) {
        if (!prepare(score_kernel<C, NS, true>, kThreads, smem, d, occ_sc_exact)) return TAHQ_ERR_CUDA;
        TAHQ_LAUNCH("stats", st, launch_dependent(score_kernel<C, NS, true>, grid, kThreads, smem, st, a, tmap));
      } else if constexpr (C::G < 32 || !C::BF16) {
        if (!prepare(score_kernel<C, NS, false>, kThreads, smem, d, occ_sc)) return TAHQ_ERR_CUDA;
        TAHQ_LAUNCH("stats", st, launch_dependent(score_kernel<C, NS, false>, grid, kThreads, smem, st, a, tmap));
      }
    }
    if (launch_select(a, d, st) != TAHQ_OK) return TAHQ_ERR_CUDA;
  }
  const bool narrow = a.lo + a.mixed <= 4u;   // no width above 4 bits: the kernel compiled for just that
  if constexpr (C::G >= 32) {
    const uint64_t n_rounds = (a.n_tiles + LaneCfg<C>::TPR - 1) / LaneCfg<C>::TPR;
    if (quant_lanes_pays<C, SR>(n_rounds, narrow, d.sms)) {
      const bool wide_ld = (reinterpret_cast<uintptr_t>(a.in) & 31u) == 0;   // 256-bit loads where the tensor is aligned to them
      void (*const kernels[4])(Args) = {quant_lanes_kernel<C, SR, false, false>, quant_lanes_kernel<C, SR, false, true>,
                                        quant_lanes_kernel<C, SR, true, false>, quant_lanes_kernel<C, SR, true, true>};
      static std::atomic<int> occ[4][64];
      const int k = 2 * narrow + wide_ld;
      if (!prepare(kernels[k], QuantLanes<C>::NT, QuantLanes<C>::SMEM, d, occ[k])) return TAHQ_ERR_CUDA;
      TAHQ_LAUNCH("quant_pack", st, launch_dependent(kernels[k], persistent_grid(n_rounds, d, 1), QuantLanes<C>::NT,
                                                     QuantLanes<C>::SMEM, st, a));
      return cudaGetLastError() == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
    }
  }
  if constexpr (C::G < 32 || C::BF16) {
    // Rows of 128 bytes (a TMA copy per unit): one slot, refilled as soon as its row is in registers; the second one's 64 KB
    // per SM serve better as L1 (65536 x 8192 bf16 358 -> 343 us, 16384 x 8192 in tiles of 128 123 -> 113 us).  Narrower rows
    // come by cp.async and want two (16384 x 8192 in tiles of 32 82.2 us, with one slot 84.6 us).
    constexpr int NQ = C::ROWB == 128 ? 1 : 2;
    const int smem = StreamCfg<C>::smem_bytes(NQ);
    static std::atomic<int> occ_narrow[64], occ_wide[64];
    const uint64_t n_units = (a.n_tiles * C::LPT + 31) / 32;
    const int occ = narrow ? prepare(quant2_kernel<C, NQ, SR, true>, kThreads, smem, d, occ_narrow)
                           : prepare(quant2_kernel<C, NQ, SR, false>, kThreads, smem, d, occ_wide);
    if (!occ) return TAHQ_ERR_CUDA;
    const unsigned grid = persistent_grid((n_units + kWarps - 1) / kWarps, d, occ);
    if (narrow)
      TAHQ_LAUNCH("quant_pack", st, launch_dependent(quant2_kernel<C, NQ, SR, true>, grid, kThreads, smem, st, a, tmap));
    else
      TAHQ_LAUNCH("quant_pack", st, launch_dependent(quant2_kernel<C, NQ, SR, false>, grid, kThreads, smem, st, a, tmap));
  }
  return cudaGetLastError() == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}

template <class C>
static tahq_status decode_t(const Plan &pl, const Args &a, cudaStream_t st) {
  DevInfo d;
  if (!dev_info(&d)) return TAHQ_ERR_CUDA;
  (void)pl;
  if constexpr (C::G >= 32) {
    // no width above 4 bits: the kernel compiled for just that; 256-bit stores where the tensor is aligned to them
    const bool narrow = a.lo + a.mixed <= 4u, wide_st = (reinterpret_cast<uintptr_t>(a.out) & 31u) == 0;
    void (*const kernels[8])(Args) = {
        decode_lanes_kernel<C, false, false, false>, decode_lanes_kernel<C, false, true, false>,
        decode_lanes_kernel<C, true, false, false>,  decode_lanes_kernel<C, true, true, false>,
        decode_lanes_kernel<C, false, false, true>,  decode_lanes_kernel<C, false, true, true>,
        decode_lanes_kernel<C, true, false, true>,   decode_lanes_kernel<C, true, true, true>};
    static std::atomic<int> occ[8][64];
    const int k = 4 * a.mixed + 2 * narrow + wide_st, smem = narrow ? DecodeLanes<C, true>::SMEM : DecodeLanes<C, false>::SMEM;
    if (!prepare(kernels[k], kLaneThreads, smem, d, occ[k])) return TAHQ_ERR_CUDA;
    const unsigned grid = persistent_grid((a.n_tiles + LaneCfg<C>::TPR - 1) / LaneCfg<C>::TPR, d, 1);
    TAHQ_LAUNCH("decode", st, launch_dependent(kernels[k], grid, kLaneThreads, smem, st, a));
  } else {
    static std::atomic<int> occ_dec[64];
    const int smem = DecStreamCfg<C>::TOTAL;
    const int occ = prepare(decode_stream_kernel<C>, kThreads, smem, d, occ_dec);
    if (!occ) return TAHQ_ERR_CUDA;
    const uint64_t n_units = (a.n_tiles * C::LPT + 31) / 32;   // units of 32 rows
    TAHQ_LAUNCH("decode", st,
                launch_dependent(decode_stream_kernel<C>, persistent_grid((n_units + kWarps - 1) / kWarps, d, occ),
                                 kThreads, smem, st, a));
  }
  return cudaGetLastError() == cudaSuccess ? TAHQ_OK : TAHQ_ERR_CUDA;
}

template <int G, bool BF16>
tahq_status encode_cfg(const Plan &pl, const Args &a, bool stochastic, cudaStream_t st) {
  // stochastic rounding has kernels of its own: the default path carries none of it
  return stochastic ? encode_t<Cfg<G, BF16>, true>(pl, a, st) : encode_t<Cfg<G, BF16>, false>(pl, a, st);
}
template <int G, bool BF16>
tahq_status decode_cfg(const Plan &pl, const Args &a, cudaStream_t st) {
  return decode_t<Cfg<G, BF16>>(pl, a, st);
}

#define TAHQ_INSTANTIATE(G, BF16)                                                                    \
  template tahq_status encode_cfg<G, BF16>(const Plan &, const Args &, bool, cudaStream_t);           \
  template tahq_status decode_cfg<G, BF16>(const Plan &, const Args &, cudaStream_t);

}  // namespace tahq
