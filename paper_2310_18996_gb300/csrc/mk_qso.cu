// Quasars from lognormal quasar-density fields (Sec. 2.2, App. A): the
// Hankel-transform pair that turns the matter spectrum into the spectrum of
// the Gaussian field delta_q, and the voxel draw from three delta_q boxes.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <exception>
#include <thread>
#include <vector>

#include "../../include/mockskewer.h"
#include "mk_device.cuh"
#include "mk_host.h"
#include "mk_kernels.h"
#include "mk_trace.h"

using namespace mk;

namespace {

int qfail(mk_ctx *ctx, int code, const char *msg) { return mkhost::ctx_fail(ctx, code, msg); }

#define CKQ(ctx, call)                                                                  \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) {                                                            \
      char b_[256];                                                                     \
      snprintf(b_, sizeof(b_), "%s: %s", #call, cudaGetErrorString(e_));                 \
      return qfail(ctx, MK_ECUDA, b_);                                                  \
    }                                                                                   \
  } while (0)

double sinc_j0(double x) {
  if (std::fabs(x) < 1e-4) return 1.0 - x * x / 6.0 + x * x * x * x / 120.0;
  return std::sin(x) / x;
}

// xi(r) of a tabulated P(k) (trapezoid rule on k_i = i dk)
double xi_at(const double *pk, int n, double dk, double r) {
  double s = 0.0;
  for (int i = 0; i < n; ++i) {
    const double k = i * dk, w = (i == 0 || i == n - 1) ? 0.5 : 1.0;
    s += w * pk[i] * k * k * sinc_j0(k * r);
  }
  return s * dk / (2.0 * M_PI * M_PI);
}

// -------------------------------------------------------------------------- draw kernels
// Coefficients of a table node that do not depend on the boxes: a_i, w_i, nbar.
struct DrawCoef {
  double a[3], w[3], nb;
};

// Over the table: the largest a_i, |norm| and |w_1| + |w_2| + |w_3| (the bits of
// non-negative floats order as integers), and whether a value is not finite.
struct DrawBound {
  int a, norm, w, not_finite;
};

struct DrawParams {
  const float *box[3];
  int32_t stride;
  int32_t n, lgn;  // n = 2^lgn
  float cell;
  float origin[3];
  const float4 *tab;  // per r node: (a_1, a_2, a_3, nbar cell^3 / E[p]), (w_1, w_2, w_3, 0)
  int32_t n_tab;
  float r0, inv_dr;
  uint32_t key0, key1;
  const DrawBound *bound;
  uint32_t *accepted;     // a bit per voxel
  int64_t *count;         // per sub-range (count pass)
  const int64_t *offset;  // per sub-range (write pass)
  mk_qso *out;
  int64_t capacity;
  double origin_d[3], cell_d;
};

__device__ __forceinline__ u32x4 voxel_words(const DrawParams &P, int64_t v) {
  return philox4x32_10(u32x4{static_cast<uint32_t>(v), static_cast<uint32_t>(static_cast<uint64_t>(v) >> 32), 0x51534Fu, 0u},
                       P.key0, P.key1);
}

// P(accept) of voxel v with the three fields d.
__device__ __forceinline__ float voxel_prob(const DrawParams &P, int64_t v, const float (&d)[3]) {
  const int mask = P.n - 1;
  const int x = static_cast<int>(v) & mask, y = static_cast<int>(v >> P.lgn) & mask,
            z = static_cast<int>(v >> (2 * P.lgn));
  const float cx = P.origin[0] + (x + 0.5f) * P.cell, cy = P.origin[1] + (y + 0.5f) * P.cell,
              cz = P.origin[2] + (z + 0.5f) * P.cell;
  const float r = sqrtf(cx * cx + cy * cy + cz * cz);
  float s = (r - P.r0) * P.inv_dr;
  s = fminf(fmaxf(s, 0.0f), static_cast<float>(P.n_tab - 1));
  int k = min(static_cast<int>(s), P.n_tab - 2);
  const float f = s - static_cast<float>(k);
  const float4 a0 = __ldg(P.tab + 2 * k), a1 = __ldg(P.tab + 2 * k + 2);
  const float4 w0 = __ldg(P.tab + 2 * k + 1), w1 = __ldg(P.tab + 2 * k + 3);
  const float aa[3] = {fmaf(f, a1.x - a0.x, a0.x), fmaf(f, a1.y - a0.y, a0.y), fmaf(f, a1.z - a0.z, a0.z)};
  const float ww[3] = {fmaf(f, w1.x - w0.x, w0.x), fmaf(f, w1.y - w0.y, w0.y), fmaf(f, w1.z - w0.z, w0.z)};
  const float norm = fmaf(f, a1.w - a0.w, a0.w);
  float p = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) p = fmaf(ww[i], expf(aa[i] * d[i]), p);
  return fminf(1.0f, norm * fmaxf(p, 0.0f));
}

constexpr int kDrawThreads = 256;
constexpr int kSub = 1024;  // voxels per warp sub-range: 32 words of accept bits

// One warp per sub-range of kSub voxels: a bit for each accepted voxel
// ((w0 + 1/2) 2^-32 < P in FP32) and their number.  The pass is bound by
// arithmetic (the Philox call, 60 instructions a voxel, beside 12 bytes).  A
// voxel's uniform is first held against an upper bound of P, of the table's
// largest coefficients and one exponential; only the lanes it leaves over (about
// one in a hundred at the benchmark's density) look up the table and take the
// three exponentials.  512^3: 0.61 ms, against 1.06 ms when every voxel took them
// (and 0.09 against 1.71 ms in the write pass, which decided everything again).
__global__ void __launch_bounds__(kDrawThreads) k_qso_count(DrawParams P) {
  const int64_t nv = static_cast<int64_t>(P.n) * P.n * P.n;
  const int64_t subs = (nv + kSub - 1) / kSub;
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (kDrawThreads / 32);
  // between the nodes norm, a and the weights are linear: they stay below the
  // largest; a table that is not finite takes every voxel to the full decision
  const DrawBound B = *P.bound;
  const float max_a = __int_as_float(B.a);
  const float max_p = B.not_finite ? __int_as_float(0x7f800000)
                                   : 1.01f * (__int_as_float(B.norm) * __int_as_float(B.w));
  constexpr int kBatch = 4;  // chunks of 32 voxels whose fields load together
  for (int64_t s = blockIdx.x * static_cast<int64_t>(kDrawThreads / 32) + (threadIdx.x >> 5); s < subs; s += warps) {
    const int64_t v0 = s * kSub;
    uint32_t mine = 0u;  // accept bits of chunk `lane`
    for (int c0 = 0; c0 < kSub / 32; c0 += kBatch) {
      float d[kBatch][3];
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int64_t v = v0 + 32 * (c0 + j) + lane;
#pragma unroll
        for (int i = 0; i < 3; ++i) d[j][i] = v < nv ? __ldg(P.box[i] + v * P.stride) : 0.f;
      }
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int64_t v = v0 + 32 * (c0 + j) + lane;
        bool acc = false;
        if (v < nv) {
          const float u = (__uint2float_rn(voxel_words(P, v).x) + 0.5f) * 0x1p-32f;
          // sum w_i exp(a_i d_i) <= sum |w_i| exp(max(0, max a max d)); 1 % over for the roundings
          const float top = fmaxf(fmaxf(fmaxf(d[j][0], d[j][1]), d[j][2]), 0.f);
          if (!(u >= max_p * __expf(max_a * top))) acc = u < voxel_prob(P, v, d[j]);
        }
        const uint32_t bits = __ballot_sync(0xffffffffu, acc);
        if (lane == c0 + j) mine = bits;
      }
    }
    P.accepted[s * (kSub / 32) + lane] = mine;
    const int c = __reduce_add_sync(0xffffffffu, __popc(mine));
    if (lane == 0) P.count[s] = c;
  }
}

// The records of the accepted voxels, in voxel order from each sub-range's
// offset: a lane per word of accept bits.
__global__ void __launch_bounds__(kDrawThreads) k_qso_write(DrawParams P) {
  const int64_t nv = static_cast<int64_t>(P.n) * P.n * P.n;
  const int64_t subs = (nv + kSub - 1) / kSub;
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (kDrawThreads / 32);
  for (int64_t s = blockIdx.x * static_cast<int64_t>(kDrawThreads / 32) + (threadIdx.x >> 5); s < subs; s += warps) {
    uint32_t bits = P.accepted[s * (kSub / 32) + lane];
    int before = __popc(bits);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += up;
    }
    int64_t o = P.offset[s] + before - __popc(bits);
    for (; bits && o < P.capacity; bits &= bits - 1, ++o) {
      const int64_t v = s * kSub + 32 * lane + (__ffs(bits) - 1);
      const int mask = P.n - 1;
      const u32x4 w = voxel_words(P, v);
      const int x = static_cast<int>(v) & mask, y = static_cast<int>(v >> P.lgn) & mask,
                z = static_cast<int>(v >> (2 * P.lgn));
      mk_qso q;
      q.pos[0] = P.origin_d[0] + (x + (static_cast<double>(w.y) + 0.5) * 0x1p-32) * P.cell_d;
      q.pos[1] = P.origin_d[1] + (y + (static_cast<double>(w.z) + 0.5) * 0x1p-32) * P.cell_d;
      q.pos[2] = P.origin_d[2] + (z + (static_cast<double>(w.w) + 0.5) * 0x1p-32) * P.cell_d;
      q.id = static_cast<uint64_t>(v);
      P.out[o] = q;
    }
  }
}

// Sums of delta_q,i^2 (FP32 over runs of 32 elements per thread, FP64 across
// runs and threads), one partial per block, summed on the host in order.
__global__ void __launch_bounds__(kDrawThreads) k_box_sq_sum(const float *b0, const float *b1, const float *b2,
                                                             int32_t stride, int64_t nv, double *partial) {
  __shared__ double red[3][kDrawThreads];
  double s[3] = {0.0, 0.0, 0.0};
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
  int64_t v = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  while (v < nv) {
    float f[3] = {0.f, 0.f, 0.f};
#pragma unroll 8
    for (int r = 0; r < 32 && v < nv; ++r, v += step) {
      const float a = __ldg(b0 + v * stride), b = __ldg(b1 + v * stride), c = __ldg(b2 + v * stride);
      f[0] = fmaf(a, a, f[0]);
      f[1] = fmaf(b, b, f[1]);
      f[2] = fmaf(c, c, f[2]);
    }
    for (int i = 0; i < 3; ++i) s[i] += f[i];
  }
  for (int i = 0; i < 3; ++i) red[i][threadIdx.x] = s[i];
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h)
      for (int i = 0; i < 3; ++i) red[i][threadIdx.x] += red[i][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int i = 0; i < 3; ++i) partial[3 * blockIdx.x + i] = red[i][0];
}

// The coefficient table: sigma_i^2 from the moments' partials (every CTA sums
// them all, in one order), then node k's E[p] and norm.
constexpr int kTabThreads = 128;

__global__ void __launch_bounds__(kTabThreads) k_qso_table(const double *__restrict__ partial, int n_part, double nv,
                                                           const DrawCoef *__restrict__ coef, int n_tab, double vol,
                                                           float4 *tab, DrawBound *bound) {
  __shared__ double red[3][kTabThreads];
  double s[3] = {0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < n_part; b += kTabThreads)
    for (int i = 0; i < 3; ++i) s[i] += partial[3 * b + i];
  for (int i = 0; i < 3; ++i) red[i][threadIdx.x] = s[i];
  __syncthreads();
  for (int h = kTabThreads / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h)
      for (int i = 0; i < 3; ++i) red[i][threadIdx.x] += red[i][threadIdx.x + h];
    __syncthreads();
  }
  const int k = blockIdx.x * kTabThreads + threadIdx.x;
  if (k >= n_tab) return;
  const DrawCoef C = coef[k];
  double ep = 0.0;
  for (int i = 0; i < 3; ++i) ep += C.w[i] * exp(0.5 * C.a[i] * C.a[i] * (red[i][0] / nv));
  const double norm = ep > 0.0 ? C.nb * vol / ep : 0.0;
  const float4 ta = make_float4(static_cast<float>(C.a[0]), static_cast<float>(C.a[1]), static_cast<float>(C.a[2]),
                                static_cast<float>(norm));
  const float4 tw = make_float4(static_cast<float>(C.w[0]), static_cast<float>(C.w[1]), static_cast<float>(C.w[2]), 0.f);
  tab[2 * k] = ta;
  tab[2 * k + 1] = tw;
  atomicMax(&bound->a, __float_as_int(fmaxf(fmaxf(fmaxf(ta.x, ta.y), ta.z), 0.f)));
  atomicMax(&bound->norm, __float_as_int(fabsf(ta.w)));
  atomicMax(&bound->w, __float_as_int(fabsf(tw.x) + fabsf(tw.y) + fabsf(tw.z)));
  if (!isfinite(ta.x + ta.y + ta.z + ta.w) || !isfinite(tw.x + tw.y + tw.z)) bound->not_finite = 1;
}

double bias_of(const double *bl, double z) { return bl[0] * std::pow((1.0 + z) / (1.0 + bl[1]), bl[2]); }

}  // namespace

extern "C" int mk_xi_of_pk(const double *h_pk, int32_t n_pk, double dk, const double *h_r, int32_t n_r,
                           double *h_xi) {
  if (!h_pk || n_pk < 2 || !(dk > 0.0) || (n_r > 0 && (!h_r || !h_xi)) || n_r < 0) return MK_EINVAL;
  for (int j = 0; j < n_r; ++j) h_xi[j] = xi_at(h_pk, n_pk, dk, h_r[j]);
  return MK_OK;
}

extern "C" int mk_lognormal_pk(const double *h_pk, int32_t n_pk, double dk, double B, double *h_pq) {
  if (!h_pk || !h_pq || n_pk < 2 || !(dk > 0.0) || !(B >= 0.0)) return MK_EINVAL;
  const int n = n_pk;
  const double dr = M_PI / (dk * (n - 1));
  std::vector<double> g(n);
  for (int j = 0; j < n; ++j) {
    const double r = j * dr, arg = 1.0 + B * xi_at(h_pk, n, dk, r);
    if (!(arg > 0.0)) return MK_EINVAL;
    const double w = (j == 0 || j == n - 1) ? 0.5 : 1.0;
    g[j] = w * dr * std::log(arg) * r * r;
  }
  for (int i = 0; i < n; ++i) {
    const double k = i * dk;
    double s = 0.0;
    for (int j = 0; j < n; ++j) s += g[j] * sinc_j0(k * j * dr);
    h_pq[i] = std::max(0.0, 4.0 * M_PI * s);  // ringing of the finite sums where P_q is small
  }
  return MK_OK;
}

extern "C" int mk_draw_qso(mk_ctx *ctx, const mk_qso_draw_params *q, const float *const d_box_q[3], int32_t box_stride,
                           mk_qso *d_qso, int64_t capacity, int64_t *h_count) {
  MK_TRACE("mk_draw_qso");
  if (!ctx) return MK_EINVAL;
  if (!q || !d_box_q || !d_box_q[0] || !d_box_q[1] || !d_box_q[2] || !h_count || (capacity > 0 && !d_qso) ||
      capacity < 0)
    return qfail(ctx, MK_EINVAL, "mk_draw_qso: NULL argument");
  int lgn = 0;
  while (lgn < 12 && (1 << lgn) < q->n) ++lgn;
  if (q->n < 2 || q->n > 2048 || (1 << lgn) != q->n || !(q->cell > 0.0) || (box_stride != 1 && box_stride != 2))
    return qfail(ctx, MK_EINVAL, "mk_draw_qso: box side must be a power of two in [2, 2048]; bad cell or stride");
  if (!(q->z_box[0] < q->z_box[1] && q->z_box[1] < q->z_box[2]) || !(q->bias[0] > 0.0))
    return qfail(ctx, MK_EINVAL, "mk_draw_qso: box redshifts must increase and the bias be > 0");
  if (!q->h_nbar || q->n_nbar < 2 || !(q->nbar_dz > 0.0)) return qfail(ctx, MK_EINVAL, "mk_draw_qso: bad nbar table");
  CKQ(ctx, cudaSetDevice(mkhost::ctx_device(ctx)));
  const cudaStream_t st = mkhost::ctx_stream(ctx);
  const int64_t n = q->n, nv = n * n * n;
  // device scratch: moments' partials, coefficient table, accept bits, counts and
  // offsets of the sub-ranges, scan tiles (0.14 bytes a voxel); the context keeps a
  // moderate one for the next call
  const int64_t subs = (nv + kSub - 1) / kSub;
  const int red_blocks = std::min<int64_t>(4 * mkhost::ctx_sms(ctx), (nv + kDrawThreads - 1) / kDrawThreads);
  const int n_tab = 8192;
  size_t at = 0;
  auto piece = [&at](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) / 256 * 256;
    return o;
  };
  const size_t o_part = piece(sizeof(double) * 3 * red_blocks), o_tab = piece(sizeof(float4) * 2 * n_tab);
  const size_t o_coef = piece(sizeof(DrawCoef) * n_tab), o_bound = piece(sizeof(DrawBound));
  const size_t o_bits = piece(sizeof(uint32_t) * subs * (kSub / 32)), o_cnt = piece(sizeof(int64_t) * subs);
  const size_t o_off = piece(sizeof(int64_t) * (subs + 1)), o_scan = piece(scan_workspace_bytes(subs));
  unsigned char *ws = nullptr;
  struct Trim {
    mk_ctx *ctx;
    ~Trim() { mkhost::ctx_trim_scratch(ctx); }
  } trim{ctx};
  if (int rc = mkhost::ctx_scratch(ctx, at, &ws)) return rc;
  double *d_part = reinterpret_cast<double *>(ws + o_part);
  float4 *d_tab = reinterpret_cast<float4 *>(ws + o_tab);
  int64_t *d_cnt = reinterpret_cast<int64_t *>(ws + o_cnt), *d_off = reinterpret_cast<int64_t *>(ws + o_off);

  // sigma_i^2 = mean delta_q,i^2 (fixed grid, partials summed in order); the
  // host works out what does not depend on it meanwhile (8192 nodes of two
  // roots and four powers each: 2 ms on one core, so a few threads share them)
  k_box_sq_sum<<<red_blocks, kDrawThreads, 0, st>>>(d_box_q[0], d_box_q[1], d_box_q[2], box_stride, nv, d_part);
  CKQ(ctx, cudaGetLastError());

  // coefficient table over the box's range of distances
  double rmin2 = 0.0, rmax2 = 0.0;
  for (int d = 0; d < 3; ++d) {
    const double lo = q->origin[d], hi = q->origin[d] + n * q->cell;
    const double near = (lo > 0.0) ? lo : (hi < 0.0 ? -hi : 0.0);
    const double far = std::max(std::fabs(lo), std::fabs(hi));
    rmin2 += near * near;
    rmax2 += far * far;
  }
  const double r0 = std::sqrt(rmin2), r1 = std::sqrt(rmax2) + 1e-6;
  const double dr = (r1 - r0) / (n_tab - 1);
  double bz[3], xi0[3];
  for (int i = 0; i < 3; ++i) {
    const double g = mkhost::ctx_growth(ctx, q->z_box[i]);
    bz[i] = bias_of(q->bias, q->z_box[i]);
    xi0[i] = bz[i] * bz[i] * g * g * q->xi_m5;
  }
  std::vector<DrawCoef> coef(n_tab);
  auto fill = [&](int k0, int k1) {
    for (int k = k0; k < k1; ++k) {
      DrawCoef &C = coef[k];
      const double r = r0 + k * dr, z = mkhost::ctx_z_of(ctx, r), g = mkhost::ctx_growth(ctx, z);
      const double b = bias_of(q->bias, z);
      double xi[3];
      for (int i = 0; i < 3; ++i) {
        C.a[i] = b * (1.0 + q->z_box[i]) / (bz[i] * (1.0 + z));
        xi[i] = std::pow(1.0 + xi0[i], C.a[i] * C.a[i]) - 1.0;
      }
      const double t12 = (z - q->z_box[0]) / (q->z_box[1] - q->z_box[0]);
      const double t23 = (z - q->z_box[1]) / (q->z_box[2] - q->z_box[1]);
      const double xi12 = (1.0 - t12) * xi[0] + t12 * xi[1], xi23 = (1.0 - t23) * xi[1] + t23 * xi[2];
      const double xmod = b * b * g * g * q->xi_m5;
      double lam = std::fabs(xi12 - xi23) > 0.0 ? (xmod - xi23) / (xi12 - xi23) : 0.5;
      lam = std::min(1.0, std::max(0.0, lam));
      C.w[0] = lam * (1.0 - t12);
      C.w[1] = lam * t12 + (1.0 - lam) * (1.0 - t23);
      C.w[2] = (1.0 - lam) * t23;
      C.nb = 0.0;
      const double s = (z - q->nbar_z0) / q->nbar_dz;
      if (s >= 0.0 && s <= q->n_nbar - 1) {
        const int j = std::min(static_cast<int>(std::floor(s)), q->n_nbar - 2);
        C.nb = q->h_nbar[j] + (s - j) * (q->h_nbar[j + 1] - q->h_nbar[j]);
      }
    }
  };
  constexpr int kShares = 8;
  std::thread helper[kShares - 1];
  for (int t = 0; t < kShares; ++t) {
    const int k0 = n_tab * t / kShares, k1 = n_tab * (t + 1) / kShares;
    try {
      if (t < kShares - 1) {
        helper[t] = std::thread(fill, k0, k1);
        continue;
      }
    } catch (const std::exception &) {  // no thread, or no memory for one: this one does the share
    }
    fill(k0, k1);
  }
  for (auto &h : helper)
    if (h.joinable()) h.join();
  DrawCoef *d_coef = reinterpret_cast<DrawCoef *>(ws + o_coef);
  DrawBound *d_bound = reinterpret_cast<DrawBound *>(ws + o_bound);
  CKQ(ctx, cudaMemsetAsync(d_bound, 0, sizeof(DrawBound), st));
  CKQ(ctx, cudaMemcpyAsync(d_coef, coef.data(), sizeof(DrawCoef) * n_tab, cudaMemcpyHostToDevice, st));
  k_qso_table<<<(n_tab + kTabThreads - 1) / kTabThreads, kTabThreads, 0, st>>>(
      d_part, red_blocks, static_cast<double>(nv), d_coef, n_tab, q->cell * q->cell * q->cell, d_tab, d_bound);
  CKQ(ctx, cudaGetLastError());
  DrawParams P{};
  for (int i = 0; i < 3; ++i) P.box[i] = d_box_q[i];
  P.stride = box_stride;
  P.n = q->n;
  P.lgn = lgn;
  P.cell = static_cast<float>(q->cell);
  for (int d = 0; d < 3; ++d) {
    P.origin[d] = static_cast<float>(q->origin[d]);
    P.origin_d[d] = q->origin[d];
  }
  P.cell_d = q->cell;
  P.n_tab = n_tab;
  P.r0 = static_cast<float>(r0);
  P.inv_dr = static_cast<float>(1.0 / dr);
  P.key0 = static_cast<uint32_t>(q->seed);
  P.key1 = static_cast<uint32_t>(q->seed >> 32);
  P.out = d_qso;
  P.capacity = capacity;
  P.tab = d_tab;
  P.bound = d_bound;
  P.accepted = reinterpret_cast<uint32_t *>(ws + o_bits);
  P.count = d_cnt;
  P.offset = d_off;
  const int64_t warps_per_block = kDrawThreads / 32;
  const int grid = static_cast<int>(
      std::min<int64_t>((subs + warps_per_block - 1) / warps_per_block, 8 * mkhost::ctx_sms(ctx)));
  k_qso_count<<<grid, kDrawThreads, 0, st>>>(P);
  CKQ(ctx, cudaGetLastError());
  CKQ(ctx, launch_scan(d_cnt, nullptr, subs, d_off, nullptr, nullptr, ws + o_scan, st));
  if (capacity > 0) {
    k_qso_write<<<grid, kDrawThreads, 0, st>>>(P);
    CKQ(ctx, cudaGetLastError());
  }
  int64_t total = 0;
  CKQ(ctx, cudaMemcpyAsync(&total, d_off + subs, sizeof(total), cudaMemcpyDeviceToHost, st));
  CKQ(ctx, cudaStreamSynchronize(st));
  *h_count = total;
  if (total > capacity) return qfail(ctx, MK_ERANGE, "mk_draw_qso: more quasars than capacity (count returned)");
  return MK_OK;
}
