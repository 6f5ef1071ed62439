// Kernel parameter blocks shared by the host launch code and the kernels.
#pragma once

#include <stdint.h>

#include "../../include/mockskewer.h"

namespace mk {

// error bits of the device error word
enum : int { ERR_RANGE = 1, ERR_CAPACITY = 2, ERR_TIMEOUT = 4 };

// bin_end entry of a z bin that no tabulated pixel leaves
constexpr int32_t kBinEndNever = 1 << 30;

// Cubic-Hermite table of D_C(z) on z_i = i h: values and slopes c/(H0 E(z_i)).
struct DcTable {
  const double2 *dc;  // {D_C(z_i), dD_C/dz(z_i)}
  int n;              // entries
  double h, inv_h;    // z spacing (a power of two), and 1 / h
  double omega_m;     // for E(z) in the Newton inversion
  const double *zr;   // z(r_i) on r_i = i hr: the starting point of the inversion
  int n_r;            // entries
  double inv_hr;      // 1 / hr
};

struct GeomParams {
  DcTable tab;
  double lambda_lya, dr, lrf_min, lrf_max;
  double z_obs_min;  // Lyman-alpha redshift of the least observed wavelength, >= 0
  int32_t n_min, n_max;
  double origin[3], inv_cell;
  int32_t j_max;  // pixel tables cover J < j_max
  int32_t unit_px;  // pixels of a work unit of the skewer kernel (a pair of segments)
};

using NodeParams = mk_fgpa_nodes;

// FP64 accumulators of one team in shared memory:
//   sums[n_z][NSUM], p1d[n_z][n_k], nseg[n_z]
struct StatLayout {
  int n_z, n_k;
  __host__ __device__ int sums(int zb, int i) const { return zb * MK_NSUM + i; }
  __host__ __device__ int p1d(int zb, int k) const { return n_z * MK_NSUM + zb * n_k + k; }
  __host__ __device__ int nseg(int zb) const { return n_z * (MK_NSUM + n_k) + zb; }
  __host__ __device__ int size() const { return n_z * (MK_NSUM + n_k + 1); }
};

// One z bin of mk_stats_out.
struct mk_stats_bin {
  double sums[MK_NSUM], p1d_sum[MK_MAX_KBINS], n_seg;
  double mean_flux, sigma_f, b_f, beta_f;
  double p1d_f[MK_MAX_KBINS], p1d_df[MK_MAX_KBINS];
};

// Derived statistics of a z bin from its raw sums (sums, p1d_sum, n_seg), the
// rest of the bin being zero: F-bar, sigma_F, and b_F, beta_F from the
// least-squares fit F ~ F0 + k_d delta + k_e eta (Sec. 2.6, Sec. 4.1); then, per
// k bin, P1D_F per mode and P1D_F / F-bar^2.  per_bin: modes per k bin,
// (n_fft / 2) / n_k.  The finalize kernel and the host-side merge of per-rank
// sums (mk_stats_merge) both use them.
__host__ __device__ inline void finalize_bin_scalars(mk_stats_bin *b) {
  const double *s = b->sums;
  const double n = s[0];
  if (n <= 0.0) return;
  const double fbar = s[1] / n;
  b->mean_flux = fbar;
  const double varf = s[2] / n - fbar * fbar;
  b->sigma_f = varf > 0.0 ? sqrt(varf) : 0.0;
  const double md = s[3] / n, me = s[4] / n;
  const double cdd = s[5] / n - md * md, cee = s[6] / n - me * me, cde = s[7] / n - md * me;
  const double vfd = s[8] / n - fbar * md, vfe = s[9] / n - fbar * me;
  const double det = cdd * cee - cde * cde;
  if (det != 0.0) {
    const double kd = (cee * vfd - cde * vfe) / det;
    const double ke = (cdd * vfe - cde * vfd) / det;
    b->b_f = kd / fbar;
    b->beta_f = kd != 0.0 ? ke / kd : 0.0;
  }
}

__host__ __device__ inline void finalize_bin_p1d(mk_stats_bin *b, int k, double per_bin) {
  if (b->sums[0] <= 0.0 || b->n_seg <= 0.0) return;
  b->p1d_f[k] = b->p1d_sum[k] / (b->n_seg * per_bin);
  b->p1d_df[k] = b->p1d_f[k] / (b->mean_flux * b->mean_flux);
}

// Everything the fused / split skewer kernels read.
struct SkewerParams {
  const mk_skewer *sk;
  const int64_t *segoff;  // exclusive prefix of pairs of segments (k_segment: segments) per skewer, n_sk + 1
  int64_t n_sk;
  // box
  const float *box_d;  // planar delta, or (delta, eta) pairs (interleaved, padded)
  const float *box_e;  // planar eta or NULL
  int32_t lgn;
  int32_t cell_cap;  // cells a pair's sight line may cross (0: not by cells)
  // tables
  const float4 *pixtab;  // per global pixel J: {G, a log2e, b log2e, c}
  const int16_t *zbin;     // per J: z bin, -1 below, n_z above
  const int16_t *segzbin;  // per J: z bin of the mean z of pixels J .. J+N-1
  const int32_t *bin_end;  // [k + 1], k = -1 .. n_z: first J with zbin > k (large beyond the tables)
  const float *amp;        // A_m / N, m = 0..N/2; with ps_nodes >= 2: (A_m / N)^2 per node, node-major
  int32_t ps_nodes;        // z-dependent small-scale power: tables at ps_z (>= 2), else one
  float ps_z[MK_MAX_NODES];
  const float *zwin;       // per J: mean z of pixels J .. J+N-1 (with ps_nodes >= 2)
  const float2 *tw;      // e^{-2 pi i k/N}, k < N
  uint32_t seed;
  // outputs
  float *delta_out, *eta_out, *flux_out;
  int64_t capacity;
  // statistics
  int32_t do_stats;
  int32_t n_z, n_k;
  float p1d_scale;   // dr / N
  double *partials;  // [gridDim.x][layout size]
  int *err;
};

// Cells the sight line of a run of 2n pixels can cross, a multiple of 4: at most
// sqrt(3) dr/cell crossings a pixel (|ux| + |uy| + |uz| <= sqrt 3), one more
// per axis for the start, and the first cell.
inline int cell_capacity(int n, double dr_over_cell) {
  return (static_cast<int>(1.7320508076 * dr_over_cell * (2 * n - 1)) + 5 + 3) / 4 * 4;
}

// Statistics pass over stored flux (any rebin).
struct StatParams {
  const mk_skewer *sk;
  const int64_t *off_out;  // output offsets, n_sk + 1
  const int64_t *segoff;   // prefix of pairs of segments, ceil(n_out / 2N) per skewer
  int64_t n_sk;
  const float *flux;         // stored flux, or NULL with pixtab set
  const float *delta, *eta;  // fine fields or NULL
  const float4 *pixtab;      // tuning pass: FGPA table; the flux is computed from delta, eta
  int32_t rebin;
  const int16_t *zbin;     // per J: z bin of the output pixel (rebin fine pixels) starting there
  const int16_t *segzbin;  // per J: z bin of the segment of N output pixels starting there
  const int32_t *bin_end;  // first J past each z bin of zbin (index zbin + 1), as in SkewerParams
  const float2 *tw;
  int32_t j_max;
  int32_t n_z, n_k;
  float p1d_scale;  // rebin dr / N
  double *partials;
  int *err;
  int32_t wait_test;  // test hook: the tuning pass issues no bulk copies and waits ~2^20 cycles at most
};

struct FluxParams {
  const mk_skewer *sk;
  const int64_t *off_out;
  int64_t n_sk;
  const float *delta, *eta;
  const float4 *pixtab;
  int32_t rebin;
  int32_t j_max;
  float *flux;
  int64_t capacity;
  int *err;
};

}  // namespace mk
