// Device building blocks of the skewer-synthesis kernels (sm_103a).
//
// A "team" of T = N/8 threads works on segments of N pixels: thread t handles
// pixels t + T k, k = 0..7.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mk_params.h"

namespace mk {

// ------------------------------------------------------------------ errors
__device__ __forceinline__ void raise_error(int *err, int bit) { atomicOr(err, bit); }

// ------------------------------------------------------------------ Philox4x32-10
// Salmon, Moraes, Dror & Shaw, SC'11: ten rounds of (hi, lo) = M * x on
// words 0 and 2, xor with words 1, 3 and the round key; the key advances by
// the Weyl constants between rounds.
struct u32x4 {
  uint32_t x, y, z, w;
};

__device__ __forceinline__ u32x4 philox4x32_10(u32x4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = u32x4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (cos, sin)(2 pi u), u = (x + 1/2) 2^-32: the angle is taken in (-pi, pi)
// and both outputs negated, cos(phi + pi) = -cos(phi).
__device__ __forceinline__ float2 unit_phase(uint32_t x) {
  const float phi =
      (static_cast<float>(static_cast<int32_t>(x ^ 0x80000000u)) + 0.5f) * 1.4629180792671596e-09f;
  float s, c;
  __sincosf(phi, &s, &c);
  return make_float2(-c, -s);
}

__device__ __forceinline__ float sqrt_pos(float x) { return x * rsqrtf(x); }  // x > 0

// ------------------------------------------------------------------ complex helpers
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
template <int SIGN>
__device__ __forceinline__ float2 cmul_i(float2 a) {  // times +i (SIGN > 0) or -i
  return SIGN > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// ------------------------------------------------------------------ packed FP32 pairs
// sm_100 and later execute add, sub, mul and fma on the two FP32 halves of a
// 64-bit register pair in one instruction; each half rounds exactly as the
// scalar instruction (round to nearest even, no flush to zero).
#define MK_F2_BINOP(name, op)                                                                  \
  __device__ __forceinline__ float2 name(float2 a, float2 b) {                                 \
    float2 r;                                                                                  \
    asm("{.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t" op        \
        " d, a, b;\n\tmov.b64 {%0, %1}, d;}"                                                  \
        : "=f"(r.x), "=f"(r.y)                                                                 \
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                                             \
    return r;                                                                                  \
  }
MK_F2_BINOP(f2add, "add.rn.f32x2")
MK_F2_BINOP(f2sub, "sub.rn.f32x2")
MK_F2_BINOP(f2mul, "mul.rn.f32x2")
#undef MK_F2_BINOP

// a * b + c per half, one rounding
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

// a + t (b - a) per half, t the same for both: the scalar lerp's rounding
__device__ __forceinline__ float2 f2lerp(float2 a, float2 b, float t) {
  return f2fma(make_float2(t, t), f2sub(b, a), a);
}

// ------------------------------------------------------------------ normals from Philox words
// -ln(u) for u = (x + 1/2) 2^-32 of two words, branch-free and accurate in
// relative terms over the whole range.  Below 1/2 the SFU log2 is accurate to
// ~2^-22 relative (|log2 u| >= 1).  Above, u = 1 - d with d = (~x + 1/2) 2^-32
// known exactly, and -ln(1 - d) = 2 atanh(s), s = d/(2 - d) <= 1/3, with
// atanh(s)/s a polynomial in s^2 of degree 5 interpolated at the Chebyshev
// points of [0, 1/9] (relative error 1e-9).  The two words run as packed pairs:
// the polynomial once for both.
__device__ __forceinline__ float2 neg_log_uniform2(uint32_t x0, uint32_t x1) {
  const float2 half = make_float2(0.5f, 0.5f), scale = make_float2(0x1p-32f, 0x1p-32f);
  const float2 u = f2mul(f2add(make_float2(__uint2float_rn(x0), __uint2float_rn(x1)), half), scale);
  const float2 d = f2mul(f2add(make_float2(__uint2float_rn(~x0), __uint2float_rn(~x1)), half), scale);
  const float2 s = make_float2(__fdividef(d.x, 2.0f - d.x), __fdividef(d.y, 2.0f - d.y));
  const float2 s2 = f2mul(s, s);
  float2 p = make_float2(0.12196954f, 0.12196954f);
  p = f2fma(p, s2, make_float2(0.10699280f, 0.10699280f));
  p = f2fma(p, s2, make_float2(0.14310104f, 0.14310104f));
  p = f2fma(p, s2, make_float2(0.19999355f, 0.19999355f));
  p = f2fma(p, s2, make_float2(0.33333340f, 0.33333340f));
  p = f2fma(p, s2, make_float2(1.0f, 1.0f));
  const float2 hi = f2mul(f2add(s, s), p);
  const float lo0 = -0.69314718055994531f * lg2_approx(u.x), lo1 = -0.69314718055994531f * lg2_approx(u.y);
  return make_float2((x0 & 0x80000000u) ? hi.x : lo0, (x1 & 0x80000000u) ? hi.y : lo1);
}

// ------------------------------------------------------------------ team barrier
template <int T>
__device__ __forceinline__ void team_sync(int team) {
  if constexpr (T == 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(T) : "memory");
  }
}

// true when pred holds on every thread of the team (a barrier of the team)
template <int T>
__device__ __forceinline__ bool team_all(int team, bool pred) {
  if constexpr (T == 32) {
    __syncwarp();
    return __all_sync(0xffffffffu, pred);
  } else {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred pi, po;\n\tsetp.ne.u32 pi, %1, 0;\n\tbar.red.and.pred po, %2, %3, pi;\n\t"
        "selp.u32 %0, 1, 0, po;\n\t}"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(pred)), "r"(team + 1), "r"(T)
        : "memory");
    return r != 0;
  }
}

// ------------------------------------------------------------------ FFT plan
template <int N>
struct Fft {
  static constexpr int M = N / 2;  // complex points
  static constexpr int T = N / 8;  // threads per team (M/4)
  static constexpr int LOGM = (M == 128) ? 7 : (M == 256) ? 8 : (M == 512) ? 9 : (M == 1024) ? 10 : 11;
  static constexpr int P4 = LOGM / 2;          // radix-4 passes
  static constexpr bool R2 = (LOGM & 1) != 0;  // one radix-2 pass at the end
  // 4096: complex lines of 2048 (box synthesis only)
  static_assert(N == 256 || N == 512 || N == 1024 || N == 2048 || N == 4096, "unsupported N");
};

// Shared-memory swizzle of complex index i: xor the low bits with 5 times
// bits 4-5.  Every Stockham access pattern (strided reads t + r T, writes at
// base + r Ns for Ns = 1, 4, 16, ..., the mode and power reads) then hits 16
// distinct 8-byte slots per half warp.
__device__ __forceinline__ int sw(int i) { return i ^ (5 * ((i >> 4) & 3)); }

// Per-thread twiddles, one shared-memory table per CTA (its teams share it):
// slot s of team thread t at tws[s T + t], so a warp's reads of one slot are
// conflict-free.  Stored for the forward sign e^{-i...}; the inverse uses
// conjugates.
//   slots 3 (p - 1) + r - 1, p = 1 .. P4 - 1, r = 1 .. 3: radix-4 pass p
//     (pass 0 has unit twiddles), e^{-2 pi i r (t mod 4^p) / 4^(p+1)}
//   slots R2 + q, q = 0, 1: radix-2 pass, butterflies t and t + T
template <int N>
struct TwTab {
  static constexpr int T = Fft<N>::T;
  static constexpr int R2 = 3 * (Fft<N>::P4 - 1);
  static constexpr int SLOTS = R2 + 2;
  static constexpr size_t BYTES = sizeof(float2) * SLOTS * T;
};

// tab[k] = e^{-2 pi i k/N}, k < N (FP64-rounded table in global memory).
// Called by every thread of the CTA; ends with a CTA barrier.
template <int N>
__device__ __forceinline__ void fill_twiddles(float2 *tws, const float2 *__restrict__ tab) {
  constexpr int T = Fft<N>::T;
  for (int i = threadIdx.x; i < TwTab<N>::SLOTS * T; i += blockDim.x) {
    const int s = i / T, t = i % T;
    int k;
    if (s < TwTab<N>::R2) {
      const int p = s / 3 + 1, r = s % 3 + 1, ns = 1 << (2 * p);
      k = (r * (t % ns) * (N / (4 * ns))) % N;
    } else {
      const int ns = 1 << (2 * Fft<N>::P4);
      k = (2 * ((t + (s - TwTab<N>::R2) * T) % ns)) % N;
    }
    tws[i] = tab[k];
  }
  __syncthreads();
}

// 4-point DFT in place (SIGN = -1 forward, +1 inverse); the sums run on
// packed pairs, the rotated difference b +- i^SIGN e on scalars.
template <int SIGN>
__device__ __forceinline__ void dft4(float2 &v0, float2 &v1, float2 &v2, float2 &v3) {
  const float2 a = f2add(v0, v2), b = f2sub(v0, v2), c = f2add(v1, v3), e = f2sub(v1, v3);
  v0 = f2add(a, c);
  v2 = f2sub(a, c);
  const float2 d = cmul_i<SIGN>(e);
  v1 = make_float2(b.x + d.x, b.y + d.y);
  v3 = make_float2(b.x - d.x, b.y - d.y);
}

// 8-point DFT in place, natural order
template <int SIGN>
__device__ __forceinline__ void dft8(float2 &v0, float2 &v1, float2 &v2, float2 &v3, float2 &v4, float2 &v5, float2 &v6,
                                     float2 &v7) {
  constexpr float kH = 0.70710678118654752f;
  float2 a0 = f2add(v0, v4), b0 = f2sub(v0, v4), a1 = f2add(v1, v5), b1 = f2sub(v1, v5);
  float2 a2 = f2add(v2, v6), b2 = f2sub(v2, v6), a3 = f2add(v3, v7), b3 = f2sub(v3, v7);
  // b1 (1 + SIGN i) / sqrt 2, SIGN i b2, b3 (-1 + SIGN i) / sqrt 2
  const float2 r1 = cmul_i<SIGN>(b1), r3 = cmul_i<SIGN>(b3);
  b1 = f2mul(make_float2(b1.x + r1.x, b1.y + r1.y), make_float2(kH, kH));
  b3 = f2mul(make_float2(r3.x - b3.x, r3.y - b3.y), make_float2(kH, kH));
  b2 = cmul_i<SIGN>(b2);
  dft4<SIGN>(a0, a1, a2, a3);
  dft4<SIGN>(b0, b1, b2, b3);
  v0 = a0; v2 = a1; v4 = a2; v6 = a3;
  v1 = b0; v3 = b1; v5 = b2; v7 = b3;
}

// Stockham passes after pass 0 (whose butterfly j = t outputs are in v[]).
// SIGN = -1 forward, +1 inverse.  On return buf holds the transform in
// natural order, through the swizzle, or with PLAIN at plain indices: the
// last pass writes t + r T (radix-4 ending: base t, stride T; radix-2
// ending: t, t + T, t + 2T, t + 3T), consecutive per lane, so the plain
// layout is conflict-free there.
template <int N, int SIGN, bool PLAIN = false>
__device__ __forceinline__ void fft_finish(float2 *buf, float2 (&v)[4], const float2 *tws, int t, int team) {
  constexpr int T = Fft<N>::T;
  constexpr int M = Fft<N>::M;
  team_sync<T>(team);
#pragma unroll
  for (int r = 0; r < 4; ++r) buf[sw(4 * t + r)] = v[r];
  int ns = 4;
#pragma unroll
  for (int p = 1; p < Fft<N>::P4; ++p) {
    team_sync<T>(team);
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = buf[sw(t + r * T)];
#pragma unroll
    for (int r = 1; r < 4; ++r) {
      const float2 w = tws[(3 * (p - 1) + r - 1) * T + t];
      v[r] = cmul(v[r], SIGN < 0 ? w : cconj(w));
    }
    dft4<SIGN>(v[0], v[1], v[2], v[3]);
    const int base = (t / ns) * ns * 4 + t % ns;
    const bool plain = PLAIN && !Fft<N>::R2 && p == Fft<N>::P4 - 1;
    team_sync<T>(team);
#pragma unroll
    for (int r = 0; r < 4; ++r) buf[plain ? base + r * ns : sw(base + r * ns)] = v[r];
    ns *= 4;
  }
  if constexpr (Fft<N>::R2) {
    team_sync<T>(team);
    float2 a0 = buf[sw(t)], b0 = buf[sw(t + M / 2)], a1 = buf[sw(t + T)], b1 = buf[sw(t + T + M / 2)];
    const float2 w0 = tws[TwTab<N>::R2 * T + t], w1 = tws[(TwTab<N>::R2 + 1) * T + t];
    b0 = cmul(b0, SIGN < 0 ? w0 : cconj(w0));
    b1 = cmul(b1, SIGN < 0 ? w1 : cconj(w1));
    team_sync<T>(team);
    buf[PLAIN ? t : sw(t)] = f2add(a0, b0);
    buf[PLAIN ? t + M / 2 : sw(t + M / 2)] = f2sub(a0, b0);
    buf[PLAIN ? t + T : sw(t + T)] = f2add(a1, b1);
    buf[PLAIN ? t + T + M / 2 : sw(t + T + M / 2)] = f2sub(a1, b1);
  }
  team_sync<T>(team);
}

// ------------------------------------------------------------------ fixed-point gather
// Positions are Q20.44 cell coordinates (minus 1/2, so that integer values
// fall on cell centres).  The kernels add kRoundQ to a skewer's start so that
// the weight below, the top 23 fraction bits, is the fraction rounded to
// nearest; a fraction that rounds up to 1 moves to the next cell with weight 0.
constexpr int64_t kRoundQ = int64_t(1) << 20;

// base cell index (periodic, n = mask + 1)
__device__ __forceinline__ int cell_of(int64_t p, int mask) { return static_cast<int>(p >> 44) & mask; }

// weight in [0, 1): 1.m - 1 with m the fraction bits 43..21 (exact)
__device__ __forceinline__ float weight_of(int64_t p) {
  const uint32_t m = static_cast<uint32_t>(static_cast<uint64_t>(p) >> 21) & 0x7FFFFFu;
  return __uint_as_float(0x3F800000u | m) - 1.0f;
}

// Normalised 1D weights of the Gaussian-kernel average (Sec. 2.3) along one
// axis: voxels c - 3 .. c + 3 around the voxel c containing the point, whose
// centre is at distance e = 1/2 - f (f the point's offset inside voxel c, in
// cells); voxel c + m sits at m + e, w_m ~ exp(-(m + e)^2 / 2).  With
// q = exp(-e), w_m ~ q^m C_m, C_m = exp(-m^2/2) (the common factor
// exp(-e^2/2) cancels in the normalisation): one exponential per axis.
static __constant__ float kGauss7C[7] = {0.011108996538242306f, 0.13533528323661270f, 0.60653065971263342f, 1.0f,
                                         0.60653065971263342f, 0.13533528323661270f, 0.011108996538242306f};

// q = exp(-e) of the point at f, and the reciprocal of sum_m q^(m+3) C_m by the
// steps that sum the voxels, so that the weights used add up to 1
__device__ __forceinline__ float gauss7_axis(float f, float &inv) {
  const float q = expf(f - 0.5f);
  float sum = kGauss7C[6];
#pragma unroll
  for (int m = 5; m >= 0; --m) sum = fmaf(sum, q, kGauss7C[m]);
  inv = 1.0f / sum;
  return q;
}

__device__ __forceinline__ float2 f2scale(float a, float2 b) { return f2mul(make_float2(a, a), b); }

// Gaussian-kernel average of (delta, eta) over 7^3 voxels (Sec. 2.3) from an
// MK_BOX_HALO box, for pixels 0 .. npx - 1 of a run whose pixel 0 is pixel j0 of
// the skewer; out[p] gets pixel p.  Warp w of nw; list: 256 entries of this warp.
//
// The 343 voxels of a pixel are what it costs: a thread a pixel waited for its
// 343 8-byte loads (the return path of L1 62 % busy, a third of the sectors from
// L2).  The pixels of a sight line that lie in one voxel (~7 at the paper's
// sizes) average the same voxels, so a task is up to kGaussRun consecutive
// pixels of one voxel, and a thread loads each voxel once for all of them, the
// next row of seven while it works on one.  Per axis sum_m q^m C_m v_m is a
// polynomial in q: C_m goes to the loaded value, once a task, and a pixel needs
// one packed multiply-add a voxel (Horner) and holds one number an axis instead
// of seven weights.  1.4e8 pixels of a 512^3 box, N = 256: 19.0 -> 11.4 ms with
// runs of 4, 12.0 with runs of 2, and half the error; now the latency of the loads again, behind 56 %
// of the FMA pipe and 57 % of L1.
constexpr int kGaussRun = 4;
__device__ __forceinline__ void gauss7_run(float2 *out, uint16_t *list, const float *__restrict__ d, int lgn,
                                           const mk_skewer *rec, int j0, int npx, int w, int nw, int lane) {
  constexpr int K = kGaussRun;
  const int mask = (1 << lgn) - 1;
  const int64_t n6 = mask + 7;
  // containing voxel: floor(p + 1/2) of the centre-based coordinate p
  const int64_t half = kRoundQ + (int64_t(1) << 43);
  const int groups = (npx + K - 1) / K, per = (groups + nw - 1) / nw;
  const int g0 = w * per, ng = min(per, groups - g0), pbase = K * g0;
  // tasks: the pieces of aligned groups of K pixels between changes of voxel
  int count = 0;
#pragma unroll 1
  for (int gg = 0; gg < ng; gg += 32) {
    const int g = gg + lane, p = pbase + K * g, last = min(K, npx - p);
    uint32_t m = g < ng ? 1u : 0u;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int64_t step = rec->step[a];
      int64_t h = rec->p0[a] + half + (j0 + p) * step;
#pragma unroll
      for (int r = 1; r < K; ++r) {
        const int64_t h1 = h + step;
        if (g < ng && r < last && (h1 >> 44) != (h >> 44)) m |= 1u << r;
        h = h1;
      }
    }
    int at = count;
#pragma unroll
    for (int r = 0; r < K; ++r) {
      const uint32_t b = __ballot_sync(0xffffffffu, m >> r & 1);
      at += __popc(b & ((1u << lane) - 1u));
      count += __popc(b);
    }
    for (; m; m &= m - 1) {  // in the order of the pixels: neighbouring lanes read neighbouring voxels
      const int r = __ffs(m) - 1, next = __ffs(m & (m - 1)) - 1;
      list[at++] = static_cast<uint16_t>((K * g + r) << 4 | ((next > 0 ? next : last) - r));
    }
  }
  __syncwarp();
#pragma unroll 1
  for (int k = lane; k < count; k += 32) {
    const int p = pbase + (list[k] >> 4), len = list[k] & 15;
    float qx[K], qy[K], qz[K], scale[K];
    int64_t h[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int64_t step = rec->step[a];
      h[a] = rec->p0[a] + half + (j0 + p) * step;
#pragma unroll
      for (int r = 0; r < K; ++r) {  // (past the task's end: some finite weight)
        float inv;
        (a == 0 ? qx : a == 1 ? qy : qz)[r] = gauss7_axis(weight_of(h[a] + r * step), inv);
        scale[r] = a ? scale[r] * inv : inv;
      }
    }
    // voxel (c - 3) per axis sits at halo index c
    const float2 *row = reinterpret_cast<const float2 *>(d) +
                        ((cell_of(h[2], mask) + 6) * n6 + cell_of(h[1], mask) + 6) * n6 + cell_of(h[0], mask);
    float2 sum[K];
#pragma unroll
    for (int r = 0; r < K; ++r) sum[r] = make_float2(0.f, 0.f);
    float2 v[7];  // the row at work; the next one is on its way
#pragma unroll
    for (int i = 0; i < 7; ++i) v[i] = __ldg(row + i);
#pragma unroll 1
    for (int z = 0; z < 7; ++z) {
      float2 ay[K];
#pragma unroll
      for (int r = 0; r < K; ++r) ay[r] = make_float2(0.f, 0.f);
#pragma unroll
      for (int y = 0; y < 7; ++y) {
        const float2 *x = y < 6 ? row - (y + 1) * n6 : (z < 6 ? row - n6 * n6 : row);
        float2 ax[K], nx[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) nx[i] = __ldg(x + i);
#pragma unroll
        for (int i = 6; i >= 0; --i) {
          const float2 c = f2scale(kGauss7C[i], v[i]);
#pragma unroll
          for (int r = 0; r < K; ++r) ax[r] = i == 6 ? c : f2fma(make_float2(qx[r], qx[r]), ax[r], c);
          v[i] = nx[i];
        }
#pragma unroll
        for (int r = 0; r < K; ++r) ay[r] = f2fma(make_float2(qy[r], qy[r]), ay[r], f2scale(kGauss7C[y], ax[r]));
      }
#pragma unroll
      for (int r = 0; r < K; ++r) sum[r] = f2fma(make_float2(qz[r], qz[r]), sum[r], f2scale(kGauss7C[z], ay[r]));
      row -= n6 * n6;
    }
#pragma unroll
    for (int r = 0; r < K; ++r)
      if (r < len) out[p + r] = f2scale(scale[r], sum[r]);
  }
}

// Start a line on its way to L2.
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Prefetch into L2 the four voxel rows (y0|y1, z0|z1) that the trilinear
// stencil at (px, py, pz) reads, for the paired layouts (each row's two
// corners x0, x0 + 1 are adjacent).
template <int LAYOUT>
__device__ __forceinline__ void prefetch_stencil(const float *__restrict__ d, int lgn, int64_t px, int64_t py,
                                                 int64_t pz) {
  if constexpr (LAYOUT == MK_BOX_PLANAR) return;
  const int mask = (1 << lgn) - 1;
  const int x0 = cell_of(px, mask), y0 = cell_of(py, mask), z0 = cell_of(pz, mask);
  constexpr int kRecord = LAYOUT == MK_BOX_TENSOR ? 32 : 8;  // bytes
  int64_t row[4];
  if constexpr (LAYOUT == MK_BOX_PADDED || LAYOUT == MK_BOX_HALO || LAYOUT == MK_BOX_TENSOR) {
    constexpr int h = LAYOUT == MK_BOX_HALO ? 3 : 0;
    const uint32_t n1 = mask + 1 + (LAYOUT == MK_BOX_HALO ? 6 : 1);
    row[0] = static_cast<uint64_t>((z0 + h) * n1 + (y0 + h)) * n1 + (x0 + h);
    row[1] = row[0] + n1;
    row[2] = row[0] + n1 * n1;
    row[3] = row[2] + n1;
  } else {
    const int y1 = (y0 + 1) & mask, z1 = (z0 + 1) & mask;
    const int64_t a = static_cast<int64_t>(z0) << (2 * lgn), b = static_cast<int64_t>(z1) << (2 * lgn);
    const int64_t c = static_cast<int64_t>(y0) << lgn, e = static_cast<int64_t>(y1) << lgn;
    row[0] = a | c | x0;
    row[1] = a | e | x0;
    row[2] = b | c | x0;
    row[3] = b | e | x0;
  }
  const char *base = reinterpret_cast<const char *>(d);
#pragma unroll
  for (int r = 0; r < 4; ++r) prefetch_l2(base + kRecord * row[r]);
}

// ------------------------------------------------------------------ FGPA
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// tab = {G, a log2 e, b log2 e, c}:  F = 2^(-a' 2^(b' (delta + c eta)))
__device__ __forceinline__ float fgpa(float4 tab, float delta, float eta) {
  return ex2_approx(-tab.y * ex2_approx(tab.z * fmaf(tab.w, eta, delta)));
}

// ------------------------------------------------------------------ statistics
// Accumulators of a team of N/256 warps in shared memory, FP32 with Kahan
// compensation (float2 {sum, compensation}; each slot has one writer lane),
// flushed to FP64 at the end of the kernel:
//   sums[warps][n_z][NSUM], p1d[n_z][slots], nseg[n_z] (uint32)
// A warp holds N/2 / warps = 128 of a segment's modes, so with n_k >= warps bins a
// bin's modes lie in one warp and the team shares one set of slots; with fewer
// bins every warp has a slot of its own.  (A set per warp took 8 n_z n_k bytes for
// every warp of the team: at N = 1024 and 16 x 32 bins that left one CTA per SM.)
template <int N>
struct TeamAcc {
  static constexpr int WARPS = N / 256;
  float2 *sums, *p1d;  // sums: this warp's
  uint32_t *nseg;
  __host__ __device__ static int slots(int n_k) { return WARPS == 1 || n_k > WARPS ? n_k : WARPS; }
  __host__ __device__ static size_t bytes(int n_z, int n_k) {
    return ((sizeof(float2) * n_z * (WARPS * MK_NSUM + slots(n_k)) + sizeof(uint32_t) * n_z) + 15) / 16 * 16;
  }
  __device__ static TeamAcc at(unsigned char *base, int warp_of_team, int n_z, int n_k) {
    TeamAcc a;
    float2 *s = reinterpret_cast<float2 *>(base);
    a.sums = s + warp_of_team * n_z * MK_NSUM;
    a.p1d = s + WARPS * n_z * MK_NSUM;
    a.nseg = reinterpret_cast<uint32_t *>(a.p1d + n_z * slots(n_k));
    return a;
  }
  // every thread of the team; a barrier has to follow
  __device__ static void zero(unsigned char *base, int n_z, int n_k, int t) {
    float *f = reinterpret_cast<float *>(base);
    for (size_t i = t; i < bytes(n_z, n_k) / sizeof(float); i += N / 8) f[i] = 0.f;
  }
};

__device__ __forceinline__ void kahan_add(float2 &acc, float x) {
  const float y = x - acc.y;
  const float t = acc.x + y;
  acc.y = (t - acc.x) - y;
  acc.x = t;
}

// Pairs of segments after which a thread's FP32 pixel sums go to the compensated
// accumulators even if its z bin goes on: 256 pixels a thread at most.  (One wide
// bin would otherwise collect 1e5 and more: errors of 1e-6 in the sums, and past
// 2^24 pixels a wrong count.)  With bins of ordinary width they went before that.
constexpr int kRunPairs = 16;

// Pixel sums of one thread for one z bin, in the StatLayout order
// n, F, F^2, d, e, d^2, e^2, d e, F d, F e; the (d, e) pairs run packed.
struct PixelSums {
  float n, f, ff, de;
  float2 m1, m2, fm;  // (d, e), (d^2, e^2), (F d, F e)
  __device__ __forceinline__ void zero() {
    n = f = ff = de = 0.f;
    m1 = m2 = fm = make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void add(float F, float2 x) {
    n += 1.f;
    add_sums(F, x);
  }
  // the sums without the count (a full segment adds its count once)
  __device__ __forceinline__ void add_sums(float F, float2 x) {
    f += F;
    ff = fmaf(F, F, ff);
    de = fmaf(x.x, x.y, de);
    m1 = f2add(m1, x);
    m2 = f2fma(x, x, m2);
    fm = f2fma(make_float2(F, F), x, fm);
  }
};

// Add the warp's PixelSums of bin zb to its accumulators (warp-uniform call; bins
// outside [0, n_z) are dropped).  It runs about once a pair of segments.  HALVE: two
// steps that halve the values a lane holds (10, 5, 3), then a rolled butterfly of
// three: 17 shuffles.  Otherwise a rolled butterfly of the ten sums, 50 shuffles in 60
// instructions.  Both add in the same order, bit for bit.  k_skewer, whose loop fills
// the instruction cache, loses more to fetches than it gains (11.10 -> 11.26 ms a
// step); the statistics kernels gain (tuning pass of 1M skewers 4.57 -> 4.36 ms,
// stored flux of 200k at N = 1024 2.24 -> 2.06), and k_segment from N = 512 on (N =
// 1024: 0.57 -> 0.54 ms).
template <bool HALVE, int N>
__device__ __forceinline__ void flush_bin_sums(const TeamAcc<N> &W, int n_z, int zb, const PixelSums &a, int lane) {
  float v[MK_NSUM] = {a.n, a.f, a.ff, a.m1.x, a.m1.y, a.m2.x, a.m2.y, a.de, a.fm.x, a.fm.y};
  if constexpr (HALVE) {
    static_assert(MK_NSUM == 10, "the halving steps");
    const bool hi = lane & 16, mid = lane & 8;
    float w[6], x[3];
#pragma unroll
    for (int i = 0; i < 5; ++i)
      w[i] = (hi ? v[i + 5] : v[i]) + __shfl_xor_sync(0xffffffffu, hi ? v[i] : v[i + 5], 16);
    w[5] = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      x[i] = (mid ? w[i + 3] : w[i]) + __shfl_xor_sync(0xffffffffu, mid ? w[i] : w[i + 3], 8);
#pragma unroll 1
    for (int s = 4; s >= 1; s >>= 1) {
#pragma unroll
      for (int i = 0; i < 3; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], s);
    }
    // lane 16 h + 8 m + k holds sum 5 h + 3 m + k
    const int k = lane & 7;
    const float sum = k == 0 ? x[0] : (k == 1 ? x[1] : x[2]);
    if (k < (mid ? 2 : 3) && zb >= 0 && zb < n_z)
      kahan_add(W.sums[zb * MK_NSUM + (hi ? 5 : 0) + (mid ? 3 : 0) + k], sum);
  } else {
#pragma unroll 1
    for (int s = 16; s >= 1; s >>= 1) {
#pragma unroll
      for (int i = 0; i < MK_NSUM; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], s);
    }
    float s = v[0];
#pragma unroll
    for (int i = 1; i < MK_NSUM; ++i) s = lane == i ? v[i] : s;
    if (lane < MK_NSUM && zb >= 0 && zb < n_z) kahan_add(W.sums[zb * MK_NSUM + lane], s);
  }
}

// Add the 4 mode powers of thread t (modes 4t+1..4t+4) to the P1D slots of z
// bin zb (warp-uniform call).  A bin holds N/2 / n_k modes and a slot at most the
// 128 of a warp, both powers of two.  Every slot has one writer.
template <int N>
__device__ __forceinline__ void accumulate_p1d(const TeamAcc<N> &W, int n_k, int t, const float (&pk)[4], float scale,
                                               int zb) {
  constexpr int kLgModes = N == 256 ? 7 : N == 512 ? 8 : N == 1024 ? 9 : 10;
  const int lg = min(kLgModes + 1 - __ffs(n_k), 7);  // of a slot's modes
  float2 *row = W.p1d + zb * TeamAcc<N>::slots(n_k) + ((4 * t) >> lg);
  if (lg >= 2) {
    float s = (pk[0] + pk[1]) + (pk[2] + pk[3]);
    const int group = 1 << (lg - 2);  // threads that share a slot
    for (int o = 1; o < group; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((t & (group - 1)) == 0) kahan_add(row[0], s * scale);
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r) kahan_add(row[r >> lg], pk[r] * scale);
  }
}

}  // namespace mk
