// The fused kernel for long pixels and short skewers: one segment a team at a time,
// a real FFT for it, and a gather of eight corners per pixel.
#pragma once

#include "mk_skewer.cuh"

namespace mk {

// ------------------------------------------------------------------ real FFT of a segment
// A segment of N reals as M = N/2 complex values, four a thread: radix-4 Stockham
// passes (fft_finish), and the untangling step at the mode end.
//
// With N = 256 (a team is one warp) the buffer is kept in two padded layouts instead
// of the swizzle: LA(i) = i + i/16 and LB(i) = i + 4 (i/16) for complex index i <= M.
// Every access is then a lane base plus a compile-time offset, and each half warp
// still hits 16 distinct 8-byte slots (apart from two 2-way conflicts among the
// mirror reads).  LA holds the modes, the outputs of the first write and of radix-4
// pass 2, and the forward result; LB the output of radix-4 pass 1.
template <int N>
struct SegmentFft {
  static constexpr int M = N / 2;
  static constexpr int BUF = N == 256 ? 156 : M + 2;  // complex slots (N = 256: LB(127) + 1)
  // per-thread twiddles: the table of fft_finish, then e^{-2 pi i (t + r T) / N}, r < 4
  static constexpr int U = TwTab<N>::SLOTS;
  static constexpr size_t TW_BYTES = sizeof(float2) * (U + 4) * (N / 8);
};
__device__ __forceinline__ int lay_a(int i) { return i + (i >> 4); }
__device__ __forceinline__ int lay_b(int i) { return i + 4 * (i >> 4); }

// fft_finish for N = 256 in the padded layouts (output plain with PLAIN, else LA)
template <int SIGN, bool PLAIN>
__device__ __forceinline__ void fft_finish256(float2 *buf, float2 (&v)[4], const float2 *tws, int t) {
  constexpr int T = 32, R2 = TwTab<256>::R2;
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 4; ++r) buf[lay_a(4 * t) + r] = v[r];
#pragma unroll
  for (int p = 1; p <= 2; ++p) {
    __syncwarp();
    // reads at t + 32 r: LA (pass 1) lay_a(t) + 34 r, LB (pass 2) lay_b(t) + 40 r
    const int rb = p == 1 ? lay_a(t) : lay_b(t);
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = buf[rb + (p == 1 ? 34 : 40) * r];
#pragma unroll
    for (int r = 1; r < 4; ++r) {
      const float2 w = tws[(3 * (p - 1) + r - 1) * T + t];
      v[r] = cmul(v[r], SIGN < 0 ? w : cconj(w));
    }
    dft4<SIGN>(v[0], v[1], v[2], v[3]);
    __syncwarp();
    // writes at base + r ns: pass 1 (ns 4) into LB, pass 2 (ns 16) into LA
    const int wb = p == 1 ? lay_b(16 * (t >> 2) + (t & 3)) : lay_a(64 * (t >> 4) + (t & 15));
#pragma unroll
    for (int r = 0; r < 4; ++r) buf[wb + (p == 1 ? 4 : 17) * r] = v[r];
  }
  __syncwarp();
  // radix-2 pass: t, t + M/2, t + T, t + T + M/2 in LA = lay_a(t) + 0, 68, 34, 102
  const int rb = lay_a(t);
  float2 a0 = buf[rb], b0 = buf[rb + 68], a1 = buf[rb + 34], b1 = buf[rb + 102];
  const float2 w0 = tws[R2 * T + t], w1 = tws[(R2 + 1) * T + t];
  b0 = cmul(b0, SIGN < 0 ? w0 : cconj(w0));
  b1 = cmul(b1, SIGN < 0 ? w1 : cconj(w1));
  __syncwarp();
  buf[PLAIN ? t : rb] = f2add(a0, b0);
  buf[PLAIN ? t + 64 : rb + 68] = f2sub(a0, b0);
  buf[PLAIN ? t + 32 : rb + 34] = f2add(a1, b1);
  buf[PLAIN ? t + 96 : rb + 102] = f2sub(a1, b1);
  __syncwarp();
}

// place of mode k in the buffer
template <int N>
__device__ __forceinline__ int mode_at(int k) {
  return N == 256 ? lay_a(k) : sw(k);
}

// Inverse real FFT of the Hermitian modes Y_0..Y_M held in buf (already scaled by
// 1/N); on return the float view holds the N real outputs, pixel p at float p.
template <int N>
__device__ __forceinline__ void inverse_real_fft(float2 *buf, const float2 *tws, int t, int team) {
  constexpr int T = N / 8, M = N / 2;
  float2 v[4];
  // N = 256: k = t + 32 r at lay_a(t) + 34 r, M - k at lay_a(32 - t) + 34 (3 - r)
  const int ka = N == 256 ? lay_a(t) : 0, kb = N == 256 ? lay_a(32 - t) : 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = t + r * T;
    const float2 yk = buf[N == 256 ? ka + 34 * r : sw(k)];
    const float2 ym = cconj(buf[N == 256 ? kb + 34 * (3 - r) : sw(M - k)]);
    // Z_k = (Y_k + conj Y_{M-k}) + i (Y_k - conj Y_{M-k}) e^{+2 pi i k/N}
    const float2 d = cmul_i<1>(cmul(f2sub(yk, ym), cconj(tws[(SegmentFft<N>::U + r) * T + t])));
    v[r] = f2add(f2add(yk, ym), d);
  }
  dft4<1>(v[0], v[1], v[2], v[3]);
  if constexpr (N == 256) fft_finish256<1, true>(buf, v, tws, t); else fft_finish<N, 1, true>(buf, v, tws, t, team);
}

// Forward complex FFT of the N reals in the float view of buf (pixel p at float p);
// on return buf holds Z_k at mode_at(k).
template <int N>
__device__ __forceinline__ void forward_packed_fft(float2 *buf, const float2 *tws, int t, int team) {
  constexpr int T = N / 8;
  float2 v[4];
  team_sync<T>(team);
#pragma unroll
  for (int r = 0; r < 4; ++r) v[r] = buf[t + r * T];
  dft4<-1>(v[0], v[1], v[2], v[3]);
  if constexpr (N == 256) fft_finish256<-1, false>(buf, v, tws, t); else fft_finish<N, -1, false>(buf, v, tws, t, team);
}

// |X_k|^2 of the real input for k = 4t+1 .. 4t+4 after forward_packed_fft:
// X_k = E_k + e^{-2 pi i k/N} O_k, E = (Z_k + conj Z_{M-k})/2,
// O = (Z_k - conj Z_{M-k})/(2i), Z_M = Z_0.
template <int N>
__device__ __forceinline__ void power_of_modes(const float2 *buf, const float2 *__restrict__ tab, int t,
                                               float (&pk)[4]) {
  constexpr int M = N / 2;
  // N = 256: k = 4t + 1 + r at lay_a(4t) + 1 + r (r < 3), M - k at lay_a(4 (31 - t)) + 3 - r
  const int pa = N == 256 ? lay_a(4 * t) : 0, pb = N == 256 ? lay_a(4 * (31 - t)) : 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = 4 * t + 1 + r;
    const float2 zk = buf[N == 256 && r < 3 ? pa + 1 + r : mode_at<N>(k & (M - 1))];
    const float2 zm = cconj(buf[N == 256 ? pb + 3 - r : sw((M - k) & (M - 1))]);
    const float2 e = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y + zm.y));
    const float2 d = f2sub(zk, zm);
    const float2 x = f2add(e, cmul(__ldg(tab + (k & (N - 1))), make_float2(0.5f * d.y, -0.5f * d.x)));
    pk[r] = fmaf(x.x, x.x, x.y * x.y);
  }
}

// ------------------------------------------------------------------ gather
// Trilinear (delta, eta) at one fixed-point position: lerps in x, then y, then z, the
// pair packed.
template <int LAYOUT>
__device__ __forceinline__ float2 gather(const float *__restrict__ d, const float *__restrict__ e, int lgn, int64_t px,
                                         int64_t py, int64_t pz, const float (&uu)[6]) {
  const int mask = (1 << lgn) - 1;
  float2 v[8];
  load_corners<LAYOUT>(d, e, lgn, cell_of(px, mask), cell_of(py, mask), cell_of(pz, mask), uu, v);
  const float tx = weight_of(px), ty = weight_of(py), tz = weight_of(pz);
  const float2 c0 = f2lerp(v[0], v[1], tx), c1 = f2lerp(v[2], v[3], tx);
  const float2 c2 = f2lerp(v[4], v[5], tx), c3 = f2lerp(v[6], v[7], tx);
  return f2lerp(f2lerp(c0, c1, ty), f2lerp(c2, c3, ty), tz);
}

// ------------------------------------------------------------------ kernel
template <int N>
struct SegmentSmem {
  static constexpr size_t TEAM = (sizeof(float2) * SegmentFft<N>::BUF + 15) / 16 * 16;
  static size_t bytes(int threads, int n_z, int n_k, bool stats) {
    return acc_bytes<N>(threads, n_z, n_k, stats) + SegmentFft<N>::TW_BYTES + static_cast<size_t>(threads / (N / 8)) * TEAM;
  }
};

// One team per segment of N pixels of a skewer (P.segoff counts segments): modes ->
// inverse real FFT -> per pixel the gather, growth, FGPA, stores and pixel sums ->
// forward FFT of the flux -> P1D.  The rest is as in k_skewer, which shares its
// transform between two segments and its corners between the pixels of a cell: that
// wins until a pair's cells need so much shared memory that fewer CTAs run (see
// use_pairs), and where every skewer has one segment the pair's second half is work
// for nothing.  Trilinear interpolation only.
template <int N, int LAYOUT, int MINB, bool PSZ>
__global__ void __launch_bounds__(256, MINB) k_segment(SkewerParams P) {
  constexpr int T = N / 8;
  const int teams = blockDim.x / T;
  const int team = threadIdx.x / T, t = threadIdx.x % T, lane = threadIdx.x & 31;
  const int wlo0 = t & ~31;  // first team pixel of this warp
  extern __shared__ __align__(16) unsigned char smem[];
  const size_t tbytes = P.do_stats ? TeamAcc<N>::bytes(P.n_z, P.n_k) : 0;
  float2 *tws = reinterpret_cast<float2 *>(smem + teams * tbytes);
  float2 *buf = reinterpret_cast<float2 *>(smem + teams * tbytes + SegmentFft<N>::TW_BYTES + team * SegmentSmem<N>::TEAM);
  float *fb = reinterpret_cast<float *>(buf);
  const TeamAcc<N> W = TeamAcc<N>::at(smem + team * tbytes, t >> 5, P.n_z, P.n_k);
  if (P.do_stats) W.zero(smem + team * tbytes, P.n_z, P.n_k, t);
  for (int i = threadIdx.x; i < 4 * T; i += blockDim.x) tws[SegmentFft<N>::U * T + i] = __ldg(P.tw + i);  // k = t + r T
  fill_twiddles<N>(tws, P.tw);  // (ends with a CTA barrier)

  // segments segoff[0] .. segoff[n_sk] (a slice of a larger catalogue may start at
  // segoff[0] > 0), in contiguous ranges: all cost the same
  const int64_t u0 = P.segoff[0], nunits = P.segoff[P.n_sk] - u0;
  const int64_t g = static_cast<int64_t>(blockIdx.x) * teams + team;
  const int64_t G = static_cast<int64_t>(gridDim.x) * teams;
  int64_t u = u0 + g * nunits / G;
  const int64_t uend = u0 + (g + 1) * nunits / G;
  int64_t i = u < uend ? upper_index(P.segoff, P.n_sk, u) : 0;

  PixelSums acc;
  acc.zero();
  int zc = -2;  // z bin of acc (warp-uniform), -2 before the first segment

  for (; u < uend; ++u) {
    while (P.segoff[i + 1] <= u) ++i;
    const int s = static_cast<int>(u - P.segoff[i]);
    const mk_skewer sk = P.sk[i];
    const int j0 = s * N, npx = min(N, sk.n - j0);
    if ((P.delta_out || P.flux_out) && sk.offset + sk.n > P.capacity) {
      if (t == 0) raise_error(P.err, ERR_CAPACITY);
      continue;
    }
    // ---- start the box rows of this segment's stencils on their way to L2: lane t
    // samples pixel 8t + 4 (the modes and the inverse FFT below hide the latency)
    {
      const int64_t q = j0 + min(npx - 1, 8 * t + 4);
      prefetch_stencil<LAYOUT>(P.box_d, P.lgn, sk.p0[0] + kRoundQ + q * sk.step[0], sk.p0[1] + kRoundQ + q * sk.step[1],
                               sk.p0[2] + kRoundQ + q * sk.step[2]);
    }
    // ---- small-scale field of this segment: modes 2c, 2c + 1, c = t + q T
    const float *amp = P.amp;
    float w_hi = 0.f;
    if constexpr (PSZ) {  // P_s at the mean z of the segment's window, linear between nodes
      const float zw = __ldg(P.zwin + sk.j_lo + j0);
      int n0 = 0;
      while (n0 + 2 < P.ps_nodes && zw >= P.ps_z[n0 + 1]) ++n0;
      w_hi = fminf(fmaxf((zw - P.ps_z[n0]) / (P.ps_z[n0 + 1] - P.ps_z[n0]), 0.f), 1.f);
      amp += n0 * (N / 2 + 1);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const uint32_t c = t + q * T;
      float2 y0, y1;
      small_scale_modes<N, PSZ>(c, amp, amp + (N / 2 + 1), w_hi, static_cast<uint32_t>(s), sk.id, P.seed, y0, y1);
      if (c == 0) buf[mode_at<N>(0)] = make_float2(0.f, 0.f);
      buf[mode_at<N>(c == 0 ? N / 2 : 2 * c)] = y0;
      buf[mode_at<N>(2 * c + 1)] = y1;
    }
    team_sync<T>(team);
    inverse_real_fft<N>(buf, tws, t, team);

    // ---- per pixel: gather, growth, FGPA, stores, pixel sums
    const int jb = sk.j_lo + j0;
    int pend = N;  // segment pixel where bin zc ends
    if (P.do_stats) {
      const int zs = __ldg(P.zbin + jb);
      if (zs != zc || u % (2 * kRunPairs) == 0) {
        if (zc != -2) flush_bin_sums<(N > 256)>(W, P.n_z, zc, acc, lane);
        acc.zero();
        zc = zs;
      }
      pend = __ldg(P.bin_end + zc + 1) - jb;
    }
    float uu[6];
    tensor_weights<LAYOUT>(static_cast<float>(sk.step[0]), static_cast<float>(sk.step[1]),
                           static_cast<float>(sk.step[2]), uu);
    int64_t px = sk.p0[0] + kRoundQ + (j0 + t) * sk.step[0];
    int64_t py = sk.p0[1] + kRoundQ + (j0 + t) * sk.step[1];
    int64_t pz = sk.p0[2] + kRoundQ + (j0 + t) * sk.step[2];
    const int64_t sx = T * sk.step[0], sy = T * sk.step[1], sz = T * sk.step[2];
    const int64_t out0 = sk.offset + j0;
    // warp-uniform: this warp's pixels of the segment all lie before pend
    const bool one_bin = !P.do_stats || min(T * 7 + wlo0 + 32, npx) <= pend;
    // pixel p: gather, growth, small-scale field, FGPA, stores; returns F
    auto synth = [&](int p, float2 &x) -> float {
      const float2 de = gather<LAYOUT>(P.box_d, P.box_e, P.lgn, px, py, pz, uu);
      const float4 tb = __ldg(P.pixtab + jb + p);
      x = make_float2(fmaf(tb.x, de.x, fb[p]), tb.x * de.y);
      const float f = fgpa(tb, x.x, x.y);
      if (P.delta_out) {
        P.delta_out[out0 + p] = x.x;
        P.eta_out[out0 + p] = x.y;
      }
      if (P.flux_out) P.flux_out[out0 + p] = f;
      return f;
    };
    auto step = [&]() {
      px += sx;
      py += sy;
      pz += sz;
    };
    // (the tensor's gather keeps one loop: its registers leave no room for a second)
    if (LAYOUT != MK_BOX_TENSOR && npx == N && one_bin) {
      // a full segment inside one z bin (most segments): no bounds or bin checks
#pragma unroll 2
      for (int k = 0; k < 8; ++k) {
        const int p = t + T * k;
        float2 x;
        const float f = synth(p, x);
        acc.add_sums(f, x);
        fb[p] = f;
        step();
      }
      acc.n += 8.f;  // this thread's pixels of the segment
    } else {
#pragma unroll 2
      for (int k = 0; k < 8; ++k) {
        const int p = t + T * k;
        float f = 0.f;
        float2 x = make_float2(0.f, 0.f);
        bool todo = p < npx;
        if (todo) f = synth(p, x);
        if (!one_bin) {
          // this warp's pixels at k: T k + wlo0 + lane; flush while they pass pend
          const int hi = min(T * k + wlo0 + 32, npx);
          while (hi > pend) {
            if (todo && p < pend) {
              acc.add(f, x);
              todo = false;
            }
            flush_bin_sums<(N > 256)>(W, P.n_z, zc, acc, lane);
            acc.zero();
            ++zc;
            pend = __ldg(P.bin_end + zc + 1) - jb;
          }
        }
        if (todo) acc.add(f, x);
        fb[p] = f;
        step();
      }
    }

    // ---- P1D of the segment
    if (P.do_stats && npx == N) {
      const int zs = __ldg(P.segzbin + jb);
      if (zs >= 0 && zs < P.n_z) {
        forward_packed_fft<N>(buf, tws, t, team);
        float pk[4];
        power_of_modes<N>(buf, P.tw, t, pk);
        accumulate_p1d(W, P.n_k, t, pk, P.p1d_scale, zs);
        if (t == 0) W.nseg[zs] += 1u;
      }
    }
    team_sync<T>(team);
  }
  if (P.do_stats) {
    if (zc != -2) flush_bin_sums<(N > 256)>(W, P.n_z, zc, acc, lane);
    flush_partials<N>(smem, teams, P.n_z, P.n_k, P.partials);
  }
}

}  // namespace mk
