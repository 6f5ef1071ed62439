// Definitions of SkewerUnit<N> (declared in mk_kernels.h): the launch and
// occupancy helpers of the fused skewer kernel and the statistics kernel for
// one FFT length.  Each length is explicitly instantiated in a translation
// unit of its own (mk_skewer_<N>.cu), so that the lengths compile in parallel.
#pragma once

#include <algorithm>

#include "mk_kernels.h"
#include "mk_segment.cuh"
#include "mk_skewer.cuh"
#include "mk_stats.cuh"

namespace mk {

namespace skewer_unit_detail {

// minb: register budget of the instance (from budget_of); psz: P_s tables at several
// redshifts
template <int NN, int L, int INTERP, typename F>
cudaError_t with_budget(bool psz, int minb, F &&fn) {
  if (psz) return fn(k_skewer<NN, L, budget_of(NN, L | kPsNodesVariant, 0), INTERP, true>);
  if (minb >= 4) return fn(k_skewer<NN, L, 4, INTERP, false>);
  if (minb == 3) return fn(k_skewer<NN, L, 3, INTERP, false>);
  return fn(k_skewer<NN, L, 2, INTERP, false>);
}

template <int NN, int L, typename F>
cudaError_t with_layout(bool psz, bool segment, int minb, F &&fn) {
  if (!segment) return with_budget<NN, L, MK_INTERP_TRILINEAR>(psz, minb, fn);
  constexpr int kBudget = budget_of(NN, L | kSegmentVariant, 0);
  return psz ? fn(k_segment<NN, L, kBudget, true>) : fn(k_segment<NN, L, kBudget, false>);
}

// Calls fn with the kernel instance for (kernel variant, register budget).
template <int NN, typename F>
cudaError_t with_skewer_kernel(int variant, int minb, F &&fn) {
  const bool psz = (variant & kPsNodesVariant) != 0, segment = (variant & kSegmentVariant) != 0;
  const int layout = variant & (kGauss7Variant - 1);
  if (variant & kGauss7Variant) return with_budget<NN, MK_BOX_HALO, MK_INTERP_GAUSS7>(psz, minb, fn);
  if (layout == MK_BOX_HALO) return with_layout<NN, MK_BOX_HALO>(psz, segment, minb, fn);
  if (layout == MK_BOX_TENSOR) return with_layout<NN, MK_BOX_TENSOR>(psz, segment, minb, fn);
  if (layout == MK_BOX_PADDED) return with_layout<NN, MK_BOX_PADDED>(psz, segment, minb, fn);
  if (layout == MK_BOX_INTERLEAVED) return with_layout<NN, MK_BOX_INTERLEAVED>(psz, segment, minb, fn);
  return with_layout<NN, MK_BOX_PLANAR>(psz, segment, minb, fn);
}

template <int NN>
size_t skewer_smem(int variant, int threads, int n_z, int n_k, bool stats, int cap) {
  return variant & kSegmentVariant ? SegmentSmem<NN>::bytes(threads, n_z, n_k, stats)
                                   : PairSmem<NN>::bytes(threads, n_z, n_k, stats, cap);
}

// Shared memory is what a large binning runs out of, team by team (8 n_z (10 +
// n_k) bytes of accumulators at N = 256), so that two CTAs of 256 threads may not
// fit where two of 224 do.  Of the multiples of a team up to 256 threads: the one
// that keeps the most threads resident, the largest of equals; regs: the threads
// that the register budget holds.  12 x 64 bins at N = 256: tuning pass 1.92 ms with
// one CTA of 256 threads, 1.53 with two of 224 (12 x 32 bins: 1.29; 300k skewers).
template <typename F>
int best_threads(int team, int regs, int sm_smem, F bytes) {
  constexpr int kReserved = 1024;  // of a CTA, for the system
  int best = 256, most = 0;
  for (int threads = 256; threads >= team; threads -= team) {
    const int ctas = std::min(regs / threads, static_cast<int>(sm_smem / (bytes(threads) + kReserved)));
    if (ctas * threads > most) {
      most = ctas * threads;
      best = threads;
    }
  }
  return best;
}

template <typename K>
int occupancy(K kern, int threads, size_t smem) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  int v = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, threads, smem) != cudaSuccess || v < 1) return 1;
  return v;
}
}  // namespace skewer_unit_detail

template <int NN>
int SkewerUnit<NN>::skewer_threads(int variant, int cap, int minb, int sm_smem, int n_z, int n_k, bool stats) {
  return skewer_unit_detail::best_threads(NN / 8, 256 * minb, sm_smem, [&](int threads) {
    return skewer_unit_detail::skewer_smem<NN>(variant, threads, n_z, n_k, stats, cap);
  });
}

// The same for both variants, which then agree bit for bit.
template <int NN>
int SkewerUnit<NN>::stats_threads(int sm_smem, int n_z, int n_k) {
  return skewer_unit_detail::best_threads(NN / 8, 512, sm_smem,
                                          [&](int threads) { return StatSmem<NN, true>::bytes(threads, n_z, n_k); });
}

template <int NN>
int SkewerUnit<NN>::blocks_per_sm(int variant, int cap, int minb, int threads, int n_z, int n_k, bool stats) {
  const size_t smem = skewer_unit_detail::skewer_smem<NN>(variant, threads, n_z, n_k, stats, cap);
  int b = 1;
  skewer_unit_detail::with_skewer_kernel<NN>(variant, minb, [&](auto kern) {
    b = skewer_unit_detail::occupancy(kern, threads, smem);
    return cudaSuccess;
  });
  return b;
}

template <int NN>
cudaError_t SkewerUnit<NN>::launch(const SkewerParams &P, int variant, int minb, int grid, int threads,
                                   cudaStream_t st) {
  const size_t smem = skewer_unit_detail::skewer_smem<NN>(variant, threads, P.n_z, P.n_k, P.do_stats != 0, P.cell_cap);
  return skewer_unit_detail::with_skewer_kernel<NN>(variant, minb, [&](auto kern) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    kern<<<grid, threads, smem, st>>>(P);
    return cudaGetLastError();
  });
}

template <int NN>
int SkewerUnit<NN>::stats_blocks_per_sm(int threads, int n_z, int n_k) {
  const int a = skewer_unit_detail::occupancy(k_stats<NN, true>, threads, StatSmem<NN, true>::bytes(threads, n_z, n_k));
  const int b = skewer_unit_detail::occupancy(k_stats<NN, false>, threads, StatSmem<NN, false>::bytes(threads, n_z, n_k));
  return a < b ? a : b;
}

template <int NN>
cudaError_t SkewerUnit<NN>::launch_stats(const StatParams &P, int grid, int threads, cudaStream_t st) {
  auto run = [&](auto kern, size_t smem) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    kern<<<grid, threads, smem, st>>>(P);
    return cudaGetLastError();
  };
  if (staged_pass(P.pixtab, P.delta, P.eta, P.rebin))
    return run(k_stats<NN, true>, StatSmem<NN, true>::bytes(threads, P.n_z, P.n_k));
  return run(k_stats<NN, false>, StatSmem<NN, false>::bytes(threads, P.n_z, P.n_k));
}

}  // namespace mk
