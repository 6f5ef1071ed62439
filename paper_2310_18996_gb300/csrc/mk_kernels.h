// Host-side launchers of the kernels in mk_kernels.cu.
#pragma once

#include <cuda_runtime.h>

#include "mk_params.h"

namespace mk {

constexpr int kGauss7Variant = 16;   // kernel variant bit of MK_INTERP_GAUSS7
constexpr int kPsNodesVariant = 32;  // kernel variant bit of P_s tables at several redshifts
constexpr int kSegmentVariant = 64;  // kernel variant bit of k_segment (see use_pairs)

// Default register budget of the fused kernel, in 256-thread CTAs per SM: three (80
// registers), or two (128 registers) on a tensor box up to N = 1024, where the
// cells' 64-byte corners need more loads in flight than three CTAs of 80 registers
// hold.  1.4e8 pixels of a 512^3 box at budgets 3 and 2: tensor N = 256 1.52 and
// 1.41 ms, N = 1024 2.35 and 2.18, N = 2048 3.02 and 3.31; padded N = 256 1.07 and
// 1.13, N = 2048 2.32 and 2.61 (budget 4 spills: 1.35 to 3.8 ms).
constexpr int default_budget(int n_fft, int layout) { return layout == MK_BOX_TENSOR && n_fft <= 1024 ? 2 : 3; }

// Register budget of the instance that runs when a variant is asked for budget
// `minb` (2, 3 or 4): k_segment and the P_s-node instances exist for one.
constexpr int budget_of(int n_fft, int variant, int minb) {
  return variant & kSegmentVariant   ? 3
         : variant & kPsNodesVariant ? default_budget(n_fft, variant & (kGauss7Variant - 1))
         : minb < 3                  ? 2
         : minb > 3                  ? 4
                                     : 3;
}

// Whether a trilinear run takes pairs of segments and the cells of its sight line
// (k_skewer) or single segments and a gather per pixel (k_segment).
// - Pixel length in cells: a pair's cells grow with it, and past these limits fewer
//   CTAs fit an SM (12 x 32 bins; the tensor box runs two CTAs anyway and gains more
//   from reading a corner once).  60k quasars of a 512^3 box, pairs and single
//   segments in ms: padded N = 256 0.66 and 0.76 at 0.111, 0.80 and 0.76 at 0.133;
//   N = 1024 1.06 and 1.10 at 0.133, 1.33 and 1.10 at 0.2; N = 2048 1.50 and 1.51 at
//   0.2; tensor N = 256 1.13 and 1.39 at 0.2, 1.30 and 1.42 at 0.25, 1.60 and 1.45 at
//   0.3.  (The paper's pixels are 0.091 cells.)
// - Skewers of one segment at most (n_max) leave half of every pair empty: padded
//   N = 512, n_max 400: 0.31 and 0.28, N = 1024, n_max 700: 0.61 and 0.54; planar and
//   tensor boxes, whose corners cost more, and N = 2048 still gain from the cells
//   (planar N = 1024: 0.63 and 0.66).
inline bool use_pairs(int n_fft, int layout, double dr_over_cell, int n_max) {
  if (n_max > 0 && n_max <= n_fft && n_fft <= 1024 && layout != MK_BOX_PLANAR && layout != MK_BOX_TENSOR)
    return false;
  const double limit = layout == MK_BOX_TENSOR ? (n_fft <= 1024 ? 0.25 : 0.2)
                                               : (n_fft == 256 ? 0.115 : n_fft <= 1024 ? 0.14 : 0.2);
  return dr_over_cell <= limit;
}

cudaError_t launch_geometry(const mk_qso *q, int64_t nq, const GeomParams &P, mk_skewer *sk, int64_t *cnt_px,
                            int64_t *cnt_seg, int *err, cudaStream_t st);
size_t scan_workspace_bytes(int64_t n);
// exclusive prefix sums (n + 1 outputs) of a (and b if not NULL); also
// stores the pixel offset into sk[i].offset when sk is not NULL
cudaError_t launch_scan(const int64_t *a, const int64_t *b, int64_t n, int64_t *out_a, int64_t *out_b,
                        mk_skewer *sk, void *ws, cudaStream_t st);
cudaError_t launch_pixtab(const double *zpix, const float *gpix, int32_t j_max, const NodeParams &nd,
                          float4 *pixtab, cudaStream_t st);
cudaError_t launch_zbin(const double *zpix, const double *cumz, int32_t j_max, double z_lo, double dz, int n_z,
                        int n_seg, int rebin, int16_t *zbin, int16_t *segzbin, cudaStream_t st);
cudaError_t launch_pack(const float *d, const float *e, int64_t n, float *out, int sms, cudaStream_t st);
cudaError_t launch_pack_tensor(const float *d, const float *e6, int lgn, float *out, int sms, cudaStream_t st);
cudaError_t launch_pack_halo(const float *d, const float *e, int lgn, float *out, int sms, cudaStream_t st);
cudaError_t launch_pack_padded(const float *d, const float *e, int lgn, float *out, int sms, cudaStream_t st);
cudaError_t launch_jcount(const mk_skewer *sk, int64_t n_sk, int32_t j_max, int32_t *diff, int sms, cudaStream_t st);
cudaError_t launch_zwin(const double *cumz, int32_t j_max, int n, float *zwin, cudaStream_t st);
cudaError_t launch_pick(const int64_t *off, int64_t n, int k, int64_t *out, cudaStream_t st);
cudaError_t launch_bin_end(const int16_t *zbin, int32_t j_max, int n_z, int32_t *bin_end, cudaStream_t st);
cudaError_t launch_out_counts(const mk_skewer *sk, int64_t n, int rebin, int64_t *cnt, cudaStream_t st);
cudaError_t launch_seg_counts(const int64_t *off, int64_t n, int n_fft, int64_t *cnt, cudaStream_t st);
// Threads of a CTA, at most 256, that keep the most warps on an SM of sm_smem bytes
// of shared memory: 256 unless the accumulators of a large binning leave fewer CTAs
// of them than the register budget would (see best_threads).
int skewer_threads(int n_fft, int variant, int cap, int minb, int sm_smem, int n_z, int n_k, bool stats);
int stats_threads(int n_fft, int sm_smem, int n_z, int n_k);
int skewer_blocks_per_sm(int n_fft, int variant, int cap, int minb, int threads, int n_z, int n_k, bool stats);
// Whether a statistics pass is a tuning pass whose fields can be staged with
// bulk copies (FGPA table set, rebin 1, 16-byte aligned fields).
inline bool staged_pass(const void *pixtab, const float *delta, const float *eta, int rebin) {
  return pixtab && delta && eta && rebin == 1 &&
         ((reinterpret_cast<uintptr_t>(delta) | reinterpret_cast<uintptr_t>(eta)) & 15) == 0;
}
int stats_blocks_per_sm(int n_fft, int threads, int n_z, int n_k);
// variant: box layout, plus kGauss7Variant for the Gaussian-kernel interpolation,
// plus kPsNodesVariant for z-dependent P_s, plus kSegmentVariant (k_segment); cap: cells
// of a run (P.cell_cap); minb: register budget asked for, that of minb 256-thread
// CTAs per SM (see budget_of)
cudaError_t launch_skewer(const SkewerParams &P, int n_fft, int variant, int minb, int grid, int threads,
                          cudaStream_t st);
// The fused skewer kernel and the statistics kernel for FFT length N: launch
// and occupancy helpers, defined in mk_skewer_unit.cuh and instantiated once
// per length (256, 512, 1024, 2048) in mk_skewer_<N>.cu.
template <int N>
struct SkewerUnit {
  static int blocks_per_sm(int variant, int cap, int minb, int threads, int n_z, int n_k, bool stats);
  static cudaError_t launch(const SkewerParams &P, int variant, int minb, int grid, int threads, cudaStream_t st);
  static int skewer_threads(int variant, int cap, int minb, int sm_smem, int n_z, int n_k, bool stats);
  static int stats_threads(int sm_smem, int n_z, int n_k);
  static int stats_blocks_per_sm(int threads, int n_z, int n_k);
  static cudaError_t launch_stats(const StatParams &P, int grid, int threads, cudaStream_t st);
};
extern template struct SkewerUnit<256>;
extern template struct SkewerUnit<512>;
extern template struct SkewerUnit<1024>;
extern template struct SkewerUnit<2048>;
cudaError_t launch_flux(const FluxParams &P, int sms, cudaStream_t st);
cudaError_t launch_stats(const StatParams &P, int n_fft, int grid, int threads, cudaStream_t st);
// One pass of the box synthesis: batched line FFTs along one axis, with the
// pass's extra step (noise, mode filter or output layout).
// Coordinate c of an axis of the work box sits at (c mod 64) lo + (c / 64) hi.
struct BoxAxis {
  int64_t lo, hi;
};
struct BoxPassParams {
  float2 *work;          // n^3: along x the modes kx < n/2 of one field, then those of the other
  float2 *spec;          // the filtered noise modes, in the places of the first field's (kept for further pairs) or NULL
  BoxAxis ax, ay, az;    // of work and spec
  const float2 *tw;      // e^{-2 pi i k / 2n}, k < 2n
  const float *pk;       // P(k) at k = i dk, i < n_pk
  int32_t n_pk;
  float inv_dk;
  float kf;              // 2 pi / (n cell)
  float amp;             // 1 / (cell^{3/2} n^3): sqrt(P / cell^3) and the inverse 1/n^3
  uint32_t key0, key1;   // Philox key of the white noise
  int32_t pair;          // filter pair 0..3: (1, eta_xx), (eta_yy, eta_zz), (eta_xy, eta_xz), (eta_yz, 0)
  int32_t lgn;
  float *out;            // output layout (last pass) or NULL
  int32_t out_side, out_margin, out_stride, out_slot;
};

// Box synthesis passes (mk_box.cu), modes in the order they run:
enum BoxPass : int {
  kBoxNoiseX = 0,  // white noise, forward FFT along x
  kBoxFwd = 1,     // forward FFT along y
  kBoxShapeZ = 2,  // forward FFT along z, filter (delta modes to spec if set), inverse along z of both fields
  kBoxSpecZ = 3,   // delta modes from spec, filter, inverse FFT along z of both fields
  kBoxInv = 4,     // inverse FFT along y of both fields
  kBoxInvXOut = 5  // inverse FFT along x, lines written into the output layout (or in place)
};
cudaError_t launch_box_pass(const BoxPassParams &P, int mode, int sms, cudaStream_t st);
// Sums the partials in a fixed order into *out and copies the error word to
// *err_out; both are page-locked host memory, valid once the stream is idle.
cudaError_t launch_finalize(const double *partials, int nparts, int n_z, int n_k, int n_fft, const int *err,
                            mk_stats_out *out, int *err_out, cudaStream_t st);

}  // namespace mk
