// Gaussian box synthesis (Sec. 2.1, Eq. deltaL, Eq. eta): Philox white noise,
// a 3D FFT made of batched line FFTs in shared memory, the sqrt(P(k)) filter
// and the velocity-gradient filters -k_p k_q / k^2, written straight into the
// library's box layouts.
//
// Every field is real, so only the modes kx = 0 .. n/2 - 1 are kept (the Nyquist
// planes are zero): the work box holds rows of n complex values whose first half
// is one field's modes and whose second half is the other's.  Five passes make
// one (delta, eta_pq) pair of boxes:
//   noise + FFT x (two real lines per transform)       writes n^3/2 values
//   FFT y                                              reads and writes n^3/2
//   FFT z, filter, inverse FFT z of both fields        reads n^3/2, writes n^3
//   inverse y                                          reads and writes n^3
//   inverse x (both fields in one transform) + layout  reads n^3, writes the layout
// that is 60 GB at 1024^3 (8-byte values), 8.9 ms at the copy rate; with the full
// spectrum in the forward half and one complex line for both fields it was 77 GB
// and a third more line transforms.  The work box is kept in bricks of 64^3
// values (BoxAxis), so that a line touches few pages along every axis, and each
// group's rows are requested into L2 while the group before transforms.
// 1024^3 into the padded layout (per pass: noise + x, y, z, inverse y, inverse x):
//   full spectrum, plain box           25.3 ms  (3.4, 4.1, 9.9, 4.0, 3.8)
//   half spectrum, plain box           23.9 ms  (2.3, 2.1, 10.6, 4.3, 4.4)
//   half spectrum, bricks              20.8 ms  (2.4, 2.0, 7.4, 4.1, 4.9)
//   32-point DFTs as 8 x 4, twiddle table, L2 prefetch
//                                      18.5 ms  (2.1, 1.7, 6.7, 3.5, 4.5)
// Bound by the latency of its phases: two CTAs of 8 warps per SM (the register
// transform takes 128 registers) wait for copies, transform and store in turn.
#include <algorithm>
#include <type_traits>

#include "mk_device.cuh"
#include "mk_kernels.h"

namespace mk {
namespace {

constexpr int kLines = 8;     // lines per CTA group
constexpr int kLinePad = 2;   // complex slots of padding per line buffer
constexpr int kBoxThreads = 512;

// Lines of 1024 points take the warp-register FFT (REG): one warp per line,
// 256 threads, line buffers of 1024 + 34 slots (the 32 x 33 transpose fits).
template <int N2, bool REG>
struct BoxSmem {
  static constexpr int M = N2 / 2;  // line length n
  static constexpr int PAD = REG ? 34 : kLinePad;
  static constexpr int THREADS = REG ? 256 : kBoxThreads;
  static constexpr size_t TW = REG ? 32 * 32 * sizeof(float2) : TwTab<N2>::BYTES;  // REG: the four-step twiddles
  static constexpr size_t bytes() { return TW + sizeof(float2) * kLines * (M + PAD); }
};

// cos, sin of 2 pi m / 32 (FP64 rounded): literals, so that the unrolled
// butterflies take them as immediates
__device__ constexpr float kW32[22][2] = {
    {1.0f, 0.0f}, {0.980785251f, 0.195090324f}, {0.923879504f, 0.382683426f}, {0.831469595f, 0.555570245f},
    {0.707106769f, 0.707106769f}, {0.555570245f, 0.831469595f}, {0.382683426f, 0.923879504f},
    {0.195090324f, 0.980785251f}, {0.0f, 1.0f}, {-0.195090324f, 0.980785251f},
    {-0.382683426f, 0.923879504f}, {-0.555570245f, 0.831469595f}, {-0.707106769f, 0.707106769f},
    {-0.831469595f, 0.555570245f}, {-0.923879504f, 0.382683426f}, {-0.980785251f, 0.195090324f},
    {-1.0f, 0.0f}, {-0.980785251f, -0.195090324f}, {-0.923879504f, -0.382683426f},
    {-0.831469595f, -0.555570245f}, {-0.707106769f, -0.707106769f}, {-0.555570245f, -0.831469595f}};

// Place of X[k] after dft32.
__host__ __device__ constexpr int pos32(int k) { return 4 * (k & 7) + (k >> 3); }

// 32-point DFT in registers, natural order in, X[k] at x[pos32(k)] out: over n =
// 4 m + r four 8-point DFTs in m, the twiddles W_32^(r q), eight 4-point DFTs in
// r.  (Radix 2 with its twiddles read from shared memory took a third more
// instructions.)
template <int SIGN>
__device__ __forceinline__ void dft32(float2 (&x)[32]) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
    dft8<SIGN>(x[r], x[4 + r], x[8 + r], x[12 + r], x[16 + r], x[20 + r], x[24 + r], x[28 + r]);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
#pragma unroll
    for (int r = 1; r < 4; ++r)
      if (q > 0) x[4 * q + r] = cmul(x[4 * q + r], make_float2(kW32[r * q][0], SIGN * kW32[r * q][1]));
    dft4<SIGN>(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
  }
}

// 1024-point FFT of one line by one warp (four-step, 32 x 32): a 32-point DFT
// over n2 of x[lane + 32 n2], the twiddles mid[k2][lane] = e^{-2 pi i lane k2 /
// 1024}, a transpose through the line buffer (rows of 33), a 32-point DFT over
// n1; natural order in and out.
template <int SIGN>
__device__ __forceinline__ void fft1024_warp(float2 *b, const float2 *mid, int lane) {
  float2 x[32];
#pragma unroll
  for (int n2 = 0; n2 < 32; ++n2) x[n2] = b[lane + 32 * n2];
  dft32<SIGN>(x);
#pragma unroll
  for (int k2 = 1; k2 < 32; ++k2) {
    const float2 w = mid[32 * k2 + lane];
    x[pos32(k2)] = cmul(x[pos32(k2)], SIGN < 0 ? w : cconj(w));
  }
  __syncwarp();
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) b[k2 * 33 + lane] = x[pos32(k2)];
  __syncwarp();
#pragma unroll
  for (int n1 = 0; n1 < 32; ++n1) x[n1] = b[lane * 33 + n1];
  dft32<SIGN>(x);
  __syncwarp();
#pragma unroll
  for (int k1 = 0; k1 < 32; ++k1) b[lane + 32 * k1] = x[pos32(k1)];
  __syncwarp();
}

// Asynchronous global-to-shared copies (no register round trip, all of a
// thread's copies in flight at once).
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
  const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

__device__ __forceinline__ int wrap_index(int j, int n) { return j < n / 2 ? j : j - n; }

// Filter pair p of the Sec. 2.1 boxes at wave vector k (k2 = |k|^2 > 0):
// (f1, f2) with eta_pq = -k_p k_q / k^2 delta.
__device__ __forceinline__ float2 pair_filter(int pair, float kx, float ky, float kz, float inv_k2) {
  switch (pair) {
    case 0: return make_float2(1.0f, -kx * kx * inv_k2);
    case 1: return make_float2(-ky * ky * inv_k2, -kz * kz * inv_k2);
    case 2: return make_float2(-kx * ky * inv_k2, -kx * kz * inv_k2);
    default: return make_float2(-ky * kz * inv_k2, 0.0f);
  }
}

// Line groups.  Along x a group is kLines whole rows (the noise pass: kLines
// pairs of rows); along y kLines adjacent columns of the first P.cols; along z
// kCols columns of the first n/2, whose second field goes n/2 further.
constexpr int kCols = kLines / 2;

// Offset of coordinate c along an axis of the work box.
__device__ __forceinline__ int64_t off(const BoxAxis &A, int c) { return (c & 63) * A.lo + (c >> 6) * A.hi; }

template <int N2, int MODE, bool REG>
__global__ void __launch_bounds__(BoxSmem<N2, REG>::THREADS, 2) k_box_pass(BoxPassParams P) {
  constexpr int M = N2 / 2;  // box side
  constexpr int H = M / 2;   // modes kept along x
  constexpr int THREADS = BoxSmem<N2, REG>::THREADS;
  constexpr int T = Fft<N2>::T;
  constexpr int TEAMS = THREADS / T;
  static_assert(REG || T == 32 || TEAMS <= 15, "teams of more than one warp use named barriers 1..TEAMS");
  static_assert(!REG || (N2 == 2048 && THREADS == 32 * kLines), "the register FFT: 1024-point lines, a warp each");
  constexpr int LS = M + BoxSmem<N2, REG>::PAD;
  constexpr bool ZPASS = MODE == kBoxShapeZ || MODE == kBoxSpecZ;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *tws = reinterpret_cast<float2 *>(smem_raw);
  float2 *lines = reinterpret_cast<float2 *>(smem_raw + BoxSmem<N2, REG>::TW);
  if constexpr (REG) {
    for (int i = threadIdx.x; i < 32 * 32; i += THREADS) tws[i] = __ldg(P.tw + 2 * ((i / 32) * (i % 32)));  // W_1024
    __syncthreads();
  } else {
    fill_twiddles<N2>(tws, P.tw);
  }
  const int team = threadIdx.x / T, t = threadIdx.x % T;
  const int fields = P.pair == 3 ? 1 : 2;  // the last pair has one box
  // transforms of lines 0 .. count - 1
  auto transform = [&](auto sign, int count) {
    constexpr int SIGN = decltype(sign)::value;
    if constexpr (REG) {
      const int c = threadIdx.x >> 5;
      if (c < count) fft1024_warp<SIGN>(lines + c * LS, tws, threadIdx.x & 31);
    } else {
      for (int c = team; c < count; c += TEAMS) {
        float2 *b = lines + c * LS;
        float2 v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = b[t + r * T];
        dft4<SIGN>(v[0], v[1], v[2], v[3]);
        fft_finish<N2, SIGN, true>(b, v, tws, t, team);
      }
    }
    __syncthreads();
  };
  using Forward = std::integral_constant<int, -1>;
  using Inverse = std::integral_constant<int, 1>;
  constexpr int64_t NN = static_cast<int64_t>(M) * M;

  if constexpr (MODE == kBoxNoiseX) {
    // two real lines a, b as one complex line a + i b
    for (int64_t g = blockIdx.x; g < NN / (2 * kLines); g += gridDim.x) {
      const int64_t l0 = g * 2 * kLines;
      for (int i = 4 * threadIdx.x; i < kLines * M; i += 4 * THREADS) {
        const int c = i / M, e = i % M;  // 4 | M: the 4 voxels share a line
        float x[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // 4 voxels per Philox call: (w0, w1) and (w2, w3) through Box-Muller
          const uint64_t q = static_cast<uint64_t>((l0 + 2 * c + h) * M + e) >> 2;
          const u32x4 w = philox4x32_10(u32x4{static_cast<uint32_t>(q), static_cast<uint32_t>(q >> 32), 0u, 0u},
                                        P.key0, P.key1);
          const float2 nl = neg_log_uniform2(w.x, w.z);
          const float r0 = sqrt_pos(2.0f * nl.x), r1 = sqrt_pos(2.0f * nl.y);
          const float2 p0 = unit_phase(w.y), p1 = unit_phase(w.w);
          x[h][0] = r0 * p0.x;
          x[h][1] = r0 * p0.y;
          x[h][2] = r1 * p1.x;
          x[h][3] = r1 * p1.y;
        }
        float2 *b = lines + c * LS + e;
#pragma unroll
        for (int k = 0; k < 4; ++k) b[k] = make_float2(x[0][k], x[1][k]);
      }
      __syncthreads();
      transform(Forward{}, kLines);
      // A_k = (Z_k + conj Z_{n-k}) / 2, B_k = (Z_k - conj Z_{n-k}) / 2i, k < n/2
      for (int i = 2 * threadIdx.x; i < kLines * H; i += 2 * THREADS) {
        const int c = i / H, k = i % H;
        const float2 *z = lines + c * LS;
        float2 A[2], B[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float2 u = z[k + j], v = z[(M - k - j) & (M - 1)];
          A[j] = make_float2(0.5f * (u.x + v.x), 0.5f * (u.y - v.y));
          B[j] = make_float2(0.5f * (u.y + v.y), 0.5f * (v.x - u.x));
        }
        const int y = static_cast<int>((l0 + 2 * c) & (M - 1));  // rows y, y + 1 of plane l0 / n
        float2 *plane = P.work + off(P.az, static_cast<int>(l0 / M)) + off(P.ax, k);
        *reinterpret_cast<float4 *>(plane + off(P.ay, y)) = make_float4(A[0].x, A[0].y, A[1].x, A[1].y);
        *reinterpret_cast<float4 *>(plane + off(P.ay, y + 1)) = make_float4(B[0].x, B[0].y, B[1].x, B[1].y);
      }
      __syncthreads();
    }
  } else if constexpr (MODE == kBoxFwd || MODE == kBoxInv) {
    // along y: the first n/2 columns forward, both fields' inverse
    const int blocks = (MODE == kBoxFwd ? H : H * fields) / kLines;
    for (int64_t g = blockIdx.x; g < static_cast<int64_t>(M) * blocks; g += gridDim.x) {
      float2 *base = P.work + off(P.az, static_cast<int>(g / blocks)) + off(P.ax, static_cast<int>(g % blocks) * kLines);
      for (int i = threadIdx.x; i < kLines * M; i += THREADS)  // 8-byte copies, 64 B per row
        cp_async8(lines + (i % kLines) * LS + i / kLines, base + off(P.ay, i / kLines) + i % kLines);
      // the next group's rows are requested while this one transforms, so that its
      // copies then wait for L2, not for DRAM
      if (const int64_t gn = g + gridDim.x; gn < static_cast<int64_t>(M) * blocks) {
        const float2 *next = P.work + off(P.az, static_cast<int>(gn / blocks)) + off(P.ax, static_cast<int>(gn % blocks) * kLines);
        for (int e = threadIdx.x; e < M; e += THREADS) prefetch_l2(next + off(P.ay, e));
      }
      cp_async_wait_all();
      __syncthreads();
      if constexpr (MODE == kBoxFwd) transform(Forward{}, kLines); else transform(Inverse{}, kLines);
#pragma unroll 4
      for (int i = threadIdx.x; i < kLines * M; i += THREADS)
        base[off(P.ay, i / kLines) + i % kLines] = lines[(i % kLines) * LS + i / kLines];
      __syncthreads();
    }
  } else if constexpr (ZPASS) {
    // along z: element e is k_z
    for (int64_t g = blockIdx.x; g < static_cast<int64_t>(M) * (H / kCols); g += gridDim.x) {
      const int ky_i = static_cast<int>(g / (H / kCols)), x0 = static_cast<int>(g % (H / kCols)) * kCols;
      const int64_t col = off(P.ay, ky_i) + off(P.ax, x0), col2 = off(P.ay, ky_i) + off(P.ax, x0 + H);
      const float2 *src = (MODE == kBoxSpecZ ? P.spec : P.work) + col;
      for (int i = threadIdx.x; i < kCols * M; i += THREADS)
        cp_async8(lines + (i % kCols) * LS + i / kCols, src + off(P.az, i / kCols) + i % kCols);
      if (const int64_t gn = g + gridDim.x; gn < static_cast<int64_t>(M) * (H / kCols)) {
        const float2 *next = (MODE == kBoxSpecZ ? P.spec : P.work) + off(P.ay, static_cast<int>(gn / (H / kCols))) +
                             off(P.ax, static_cast<int>(gn % (H / kCols)) * kCols);
        for (int e = threadIdx.x; e < M; e += THREADS) prefetch_l2(next + off(P.az, e));
      }
      cp_async_wait_all();
      __syncthreads();
      if constexpr (MODE == kBoxShapeZ) transform(Forward{}, kCols);
      const float ky = P.kf * wrap_index(ky_i, M);
      for (int i = threadIdx.x; i < kCols * M; i += THREADS) {
        const int e = i / kCols, c = i % kCols, xi = x0 + c;
        float2 d = lines[c * LS + e];
        const float kx = P.kf * xi, kz = P.kf * wrap_index(e, M);
        const float k2 = kx * kx + ky * ky + kz * kz;
        if constexpr (MODE == kBoxShapeZ) {
          const bool zero = (ky_i == M / 2) || (e == M / 2) || k2 == 0.0f;
          float s = 0.0f;
          if (!zero) {
            // linear in the table, 0 beyond its last entry (n_pk <= 2^24: the
            // comparison is exact and j <= n_pk - 2 below); |k| and the roots
            // through rsqrt (a few ulp, far inside the synthesis tolerance)
            const float u = k2 * rsqrtf(k2) * P.inv_dk, last = static_cast<float>(P.n_pk - 1);
            float pk = -1.0f;
            if (u < last) {
              const int j = static_cast<int>(u);
              const float f = u - static_cast<float>(j);
              pk = fmaf(f, __ldg(P.pk + j + 1) - __ldg(P.pk + j), __ldg(P.pk + j));
            } else if (u == last) {
              pk = __ldg(P.pk + P.n_pk - 1);
            }
            s = pk > 0.0f ? pk * rsqrtf(pk) * P.amp : 0.0f;
          }
          d = make_float2(d.x * s, d.y * s);
          if (P.spec) P.spec[col + off(P.az, e) + c] = d;
        }
        const float2 f = k2 > 0.0f ? pair_filter(P.pair, kx, ky, kz, __frcp_rn(k2)) : make_float2(0.f, 0.f);
        lines[c * LS + e] = make_float2(d.x * f.x, d.y * f.x);
        lines[(kCols + c) * LS + e] = make_float2(d.x * f.y, d.y * f.y);
      }
      __syncthreads();
      transform(Inverse{}, kCols * fields);
      for (int h = 0; h < fields; ++h)
#pragma unroll 4
        for (int i = threadIdx.x; i < kCols * M; i += THREADS)
          P.work[(h ? col2 : col) + off(P.az, i / kCols) + i % kCols] = lines[(h * kCols + i % kCols) * LS + i / kCols];
      __syncthreads();
    }
  } else {  // kBoxInvXOut: both fields' half rows into one complex row, then the layout
    for (int64_t g = blockIdx.x; g < NN / kLines; g += gridDim.x) {
      // rows y0 .. y0 + 7 of plane g kLines / n
      float2 *plane = P.work + off(P.az, static_cast<int>(g * kLines / M));
      const int y0 = static_cast<int>(g * kLines & (M - 1));
      for (int i = 2 * threadIdx.x; i < kLines * M; i += 2 * THREADS) {  // 16-byte copies of element pairs
        const int c = i / M, e = i % M;
        if (fields == 2 || e < H) cp_async16(lines + c * LS + e, plane + off(P.ay, y0 + c) + off(P.ax, e));
      }
      if (const int64_t gn = g + gridDim.x; gn < NN / kLines) {
        const float2 *next = P.work + off(P.az, static_cast<int>(gn * kLines / M));
        const int y1 = static_cast<int>(gn * kLines & (M - 1));
        for (int i = threadIdx.x; i < kLines * (M / 16); i += THREADS)  // 128 bytes each
          prefetch_l2(next + off(P.ay, y1 + i / (M / 16)) + off(P.ax, (i % (M / 16)) * 16));
      }
      cp_async_wait_all();
      __syncthreads();
      // G_k = a_k + i b_k and G_{n-k} = conj a_k + i conj b_k: the four places k,
      // n/2 - k, n/2 + k, n - k exchange among themselves
      for (int i = threadIdx.x; i < kLines * (H / 2 + 1); i += THREADS) {
        const int c = i / (H / 2 + 1), k = i % (H / 2 + 1);
        float2 *z = lines + c * LS;
        const float2 none = make_float2(0.f, 0.f);
        const int k2 = H - k;  // k = 0: the Nyquist place, which holds b_0
        const float2 a1 = z[k], b1 = fields == 2 ? z[H + k] : none;
        if (k == 0) {
          z[0] = make_float2(a1.x - b1.y, a1.y + b1.x);
          z[H] = none;
        } else {
          const float2 a2 = z[k2], b2 = fields == 2 ? z[H + k2] : none;
          z[k] = make_float2(a1.x - b1.y, a1.y + b1.x);
          z[M - k] = make_float2(a1.x + b1.y, b1.x - a1.y);
          z[k2] = make_float2(a2.x - b2.y, a2.y + b2.x);
          z[M - k2] = make_float2(a2.x + b2.y, b2.x - a2.y);
        }
      }
      __syncthreads();
      transform(Inverse{}, kLines);
      if (P.out) {
        // lines l = g kLines + c of x at (y, z) = (l mod n, l / n); each goes to every
        // periodic copy of its row in the (side)^2 rows of the layout
        const int S = P.out_side, mg = P.out_margin;
        for (int c = 0; c < kLines; ++c) {
          const int64_t l = g * kLines + c;
          const int y = static_cast<int>(l % M), z = static_cast<int>(l / M);
          for (int rz = -1; rz <= 1; ++rz) {
            const int zp = z + mg + rz * M;
            if (zp < 0 || zp >= S) continue;
            for (int ry = -1; ry <= 1; ++ry) {
              const int yp = y + mg + ry * M;
              if (yp < 0 || yp >= S) continue;
              float *row = P.out + ((static_cast<int64_t>(zp) * S + yp) * S) * P.out_stride + P.out_slot;
              for (int xp = threadIdx.x; xp < S; xp += THREADS) {
                const int x = ((xp - mg) % M + M) % M;
                const float2 v = lines[c * LS + x];
                if (P.out_stride == 1) {  // delta alone
                  row[xp] = v.x;
                } else {
                  *reinterpret_cast<float2 *>(row + static_cast<int64_t>(xp) * P.out_stride) =
                      make_float2(v.x, (P.pair == 3) ? 0.0f : v.y);
                }
              }
            }
          }
        }
      } else {
        for (int i = threadIdx.x; i < kLines * M; i += THREADS)
          plane[off(P.ay, y0 + i / M) + off(P.ax, i % M)] = lines[(i / M) * LS + i % M];
      }
      __syncthreads();
    }
  }
}

template <int N2, int MODE>
cudaError_t launch_mode(const BoxPassParams &P, int sms, cudaStream_t st) {
  constexpr bool REG = N2 == 2048;
  constexpr int THREADS = BoxSmem<N2, REG>::THREADS;
  const size_t smem = BoxSmem<N2, REG>::bytes();
  cudaError_t e = cudaFuncSetAttribute(k_box_pass<N2, MODE, REG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  int per_sm = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_box_pass<N2, MODE, REG>, THREADS, smem) !=
          cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  constexpr int64_t n = N2 / 2;  // groups of the pass
  const int64_t groups = (MODE == kBoxNoiseX || MODE == kBoxFwd) ? n * n / (2 * kLines) : n * n / kLines;
  const int grid = static_cast<int>(std::min<int64_t>(groups, static_cast<int64_t>(sms) * per_sm));
  k_box_pass<N2, MODE, REG><<<grid, THREADS, smem, st>>>(P);
  return cudaGetLastError();
}

template <int N2>
cudaError_t launch_n(const BoxPassParams &P, int mode, int sms, cudaStream_t st) {
  switch (mode) {
    case kBoxNoiseX: return launch_mode<N2, kBoxNoiseX>(P, sms, st);
    case kBoxFwd: return launch_mode<N2, kBoxFwd>(P, sms, st);
    case kBoxShapeZ: return launch_mode<N2, kBoxShapeZ>(P, sms, st);
    case kBoxSpecZ: return launch_mode<N2, kBoxSpecZ>(P, sms, st);
    case kBoxInv: return launch_mode<N2, kBoxInv>(P, sms, st);
    default: return launch_mode<N2, kBoxInvXOut>(P, sms, st);
  }
}

}  // namespace

cudaError_t launch_box_pass(const BoxPassParams &P, int mode, int sms, cudaStream_t st) {
  switch (P.lgn) {
    case 7: return launch_n<256>(P, mode, sms, st);
    case 8: return launch_n<512>(P, mode, sms, st);
    case 9: return launch_n<1024>(P, mode, sms, st);
    case 10: return launch_n<2048>(P, mode, sms, st);
    case 11: return launch_n<4096>(P, mode, sms, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mk
