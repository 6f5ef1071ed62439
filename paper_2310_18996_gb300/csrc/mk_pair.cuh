// Building blocks of the kernels that work on a pair of segments: the N-point
// complex FFT that carries two real segments, and the cells of a run of pixels.
//
// A team of T = N/8 threads owns the pair (2i, 2i + 1) of segments of N pixels
// of one skewer; thread t holds pixels t + T r, r = 0..7, of both.
#pragma once

#include "mk_device.cuh"

namespace mk {

// ------------------------------------------------------------------ FFT plan
// Radix-8 Stockham passes (sub-transform lengths 1, 8, 64) and one pass of
// radix F.  Eight points a thread stay in registers between the exchanges, and
// both ends of the transform sit at t + T r, the pixels of the thread: neither
// end needs shared memory.  Two real segments as the real and imaginary parts
// of one complex transform need no real-FFT untangling, and a radix-8 pass
// halves the exchanges of the radix-4 passes on N/2 points that went before:
// two for the pair at N = 256 instead of four for each segment.
template <int N>
struct PairFft {
  static constexpr int T = N / 8;
  static constexpr int P8 = N == 256 ? 2 : 3;
  static constexpr int F = N == 256 ? 4 : (N == 512 ? 1 : (N == 1024 ? 2 : 4));
  static_assert(N == 256 || N == 512 || N == 1024 || N == 2048, "unsupported N");
  // complex slots of the exchange buffer (layout LB: 8 of padding per 64)
  static constexpr int BUF = N + N / 8;
  // twiddles (forward sign), shared by the CTA's teams: pass 1 (7 x 8 entries,
  // e^{-2 pi i r j / 64}), pass 2 (7 x 64 entries, e^{-2 pi i r j / 512}, P8 = 3),
  // last pass (slot (i, q), i < 8 / F, q = 1..F-1: e^{-2 pi i q (t + T i) / N}, T
  // entries each; at N = 2048 these 12 KB would cost a CTA per SM, and the pass
  // reads the global table)
  static constexpr bool kGlobalLast = N == 2048;
  static constexpr int TW1 = 0;
  static constexpr int TW2 = 56;
  static constexpr int TWF = P8 == 3 ? TW2 + 7 * 64 : TW2;
  static constexpr int TWN = TWF + (kGlobalLast ? 0 : (8 / F) * (F - 1) * T);
  static constexpr size_t TW_BYTES = sizeof(float2) * TWN;
};

// tab[k] = e^{-2 pi i k/N}, k < N (FP64-rounded table in global memory).
// Called by every thread of the CTA; ends with a CTA barrier.
template <int N>
__device__ __forceinline__ void fill_pair_twiddles(float2 *tws, const float2 *__restrict__ tab) {
  using P = PairFft<N>;
  for (int i = threadIdx.x; i < P::TWN; i += blockDim.x) {
    int k;
    if (i < P::TW2) {
      k = (i / 8 + 1) * (i % 8) * (N / 64);
    } else if (i < P::TWF) {
      k = ((i - P::TW2) / 64 + 1) * ((i - P::TW2) % 64) * (N / 512);
    } else {
      const int s = (i - P::TWF) / P::T, t = (i - P::TWF) % P::T;
      k = (P::F > 1) ? (s % (P::F - 1) + 1) * (t + P::T * (s / (P::F > 1 ? P::F - 1 : 1))) : 0;
    }
    tws[i] = tab[k & (N - 1)];
  }
  __syncthreads();
}

// N-point forward complex FFT of a team, v[r] at index t + T r on both ends, natural
// order.  buf: BUF complex slots, free when the call starts after a team
// barrier; its contents are undefined on return, and a barrier is needed before
// others write it.  Layouts: LA(i) = i + i/16 after pass 0, LB(i) = i + 8 (i/64)
// after pass 1, plain after pass 2: every access is a lane base plus a
// compile-time offset and its half warps hit 16 distinct 8-byte slots.
template <int N>
__device__ __forceinline__ void pair_fft(float2 *buf, float2 (&v)[8], const float2 *tws,
                                         const float2 *__restrict__ tab, int t, int team) {
  using P = PairFft<N>;
  constexpr int T = P::T;
  dft8<-1>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
  {
    float2 *w = buf + 8 * t + (t >> 1);
#pragma unroll
    for (int r = 0; r < 8; ++r) w[r] = v[r];
  }
  team_sync<T>(team);
  {
    const float2 *p = buf + t + (t >> 4);
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = p[(T + T / 16) * r];
  }
#pragma unroll
  for (int r = 1; r < 8; ++r) {
    const float2 w = tws[P::TW1 + 8 * (r - 1) + (t & 7)];
    v[r] = cmul(v[r], w);
  }
  dft8<-1>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
  team_sync<T>(team);
  {
    float2 *w = buf + (t >> 3) * 72 + (t & 7);
#pragma unroll
    for (int r = 0; r < 8; ++r) w[8 * r] = v[r];
  }
  team_sync<T>(team);
  if constexpr (N == 256) {
    const float2 *p = buf + t;
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = p[32 * r + 8 * (r >> 1)];
  } else {
    const float2 *p = buf + t + 8 * (t >> 6);
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = p[(T + T / 8) * r];
  }
  if constexpr (P::P8 == 3) {
#pragma unroll
    for (int r = 1; r < 8; ++r) {
      const float2 w = tws[P::TW2 + 64 * (r - 1) + (t & 63)];
      v[r] = cmul(v[r], w);
    }
    dft8<-1>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);  // N = 512: index t + 64 r, done
    if constexpr (P::F > 1) {
      team_sync<T>(team);
      float2 *w = buf + (t >> 6) * 512 + (t & 63);
#pragma unroll
      for (int r = 0; r < 8; ++r) w[64 * r] = v[r];
      team_sync<T>(team);
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = buf[t + T * r];
    }
  }
  if constexpr (P::F == 2) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 w = tws[P::TWF + i * T + t];
      const float2 b = cmul(v[i + 4], w), a = v[i];
      v[i] = f2add(a, b);
      v[i + 4] = f2sub(a, b);
    }
  } else if constexpr (P::F == 4) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int q = 1; q < 4; ++q) {
        const float2 w = P::kGlobalLast ? __ldg(tab + q * (t + T * i)) : tws[P::TWF + (3 * i + q - 1) * T + t];
        v[i + 2 * q] = cmul(v[i + 2 * q], w);
      }
      dft4<-1>(v[i], v[i + 2], v[i + 4], v[i + 6]);
    }
  }
}

// Powers |X_k|^2 of the two real segments (real part: a, imaginary part: b) for
// k = 4t + 1 .. 4t + 4 from the transform v of a + i b: with Z_k and Z_{N-k},
// |A_k|^2 = |Z_k + conj Z_{N-k}|^2 / 4, |B_k|^2 = |Z_k - conj Z_{N-k}|^2 / 4.
// The factor 1/4 is left to the caller.  Starts and ends with a team barrier.
template <int N>
__device__ __forceinline__ void pair_powers(float2 *buf, const float2 (&v)[8], int t, int team, float (&pa)[4],
                                            float (&pb)[4]) {
  constexpr int T = PairFft<N>::T;
  team_sync<T>(team);
  {
    float2 *w = buf + t + (t >> 4);
#pragma unroll
    for (int r = 0; r < 8; ++r) w[(T + T / 16) * r] = v[r];
  }
  team_sync<T>(team);
  const float2 *up = buf + 4 * t + (t >> 2);                          // LA(4t)
  const float2 *dn = buf + 4 * (2 * T - t - 1) + ((2 * T - t - 1) >> 2);  // LA(N - 4t - 4)
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 zk = j < 3 ? up[1 + j] : buf[4 * (t + 1) + ((t + 1) >> 2)];
    const float2 zm = dn[3 - j];
    const float2 s = f2add(zk, zm), d = f2sub(zk, zm);
    pa[j] = fmaf(s.x, s.x, d.y * d.y);
    pb[j] = fmaf(d.x, d.x, s.y * s.y);
  }
  team_sync<T>(team);
}

// ------------------------------------------------------------------ what two segments must not share
// One transform carries both segments, so a value that is not finite would reach
// every mode of both, and a segment of much larger values would round its
// partner's modes away.  Each segment stands for itself.
//
// The z bin of a segment's power (za, zb of the kernels) carries a flag for it,
// which costs no register through the transform.
constexpr int kPartFlag = 64;
static_assert(MK_MAX_ZBINS <= kPartFlag, "the flag lies above the z bins");
__device__ __forceinline__ bool counted(int z, int n_z) {
  return static_cast<unsigned>(z & ~kPartFlag) < static_cast<unsigned>(n_z);
}

// The fused kernel's flux comes from the FGPA and lies in [0, 1] or is NaN: only the
// NaN has to be found (a packed sum of the thread's values and a vote; then,
// rarely, a vote per segment).  A segment that has one becomes zeros and its z bin
// is flagged.  A barrier of the team.
template <int T>
__device__ __forceinline__ void drop_nan(float2 (&v)[8], int &za, int &zb, int team) {
  float2 s = v[0];
#pragma unroll
  for (int k = 1; k < 8; ++k) s = f2add(s, v[k]);
  if (team_all<T>(team, s.x + s.y < INFINITY)) return;
  const bool a = !team_all<T>(team, s.x < INFINITY), b = !team_all<T>(team, s.y < INFINITY);
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = make_float2(a ? 0.f : v[k].x, b ? 0.f : v[k].y);
  za |= a ? kPartFlag : 0;
  zb |= b ? kPartFlag : 0;
}

// Stored flux may hold anything (and the tuning pass works as the statistics of its
// stored flux would).  Where every thread's square sums
// of the two lie within 2^8 of each other (amplitudes within 16: the transform's
// rounding stays at the level of the smaller one's own; only a counted segment can
// be too small), they pass as they are, for 16 instructions and a vote.  Otherwise
// each counted segment is scaled by the power of two that takes its largest value
// to [1, 2), one with a value that is not finite becomes zeros, both z bins are
// flagged and *factors gets what undoes the scale in the powers (twice each), NaN
// for what is not finite.  buf: the exchange buffer, whose readers are done at the
// next barrier.  A barrier of the team; the transform's barriers order *factors.
template <int T>
__device__ __forceinline__ void part_segments(float2 (&v)[8], int &za, int &zb, int n_z, float2 *buf, uint2 *factors,
                                              int t, int team) {
  constexpr uint32_t kInf = 0x7f800000u;
  float2 e = f2mul(v[0], v[0]);
#pragma unroll
  for (int k = 1; k < 8; ++k) e = f2fma(v[k], v[k], e);
  const uint32_t ea = __float_as_uint(e.x), eb = __float_as_uint(e.y);
  const int apart = static_cast<int>(ea >> 23) - static_cast<int>(eb >> 23);
  const bool pa = counted(za, n_z), pb = counted(zb, n_z);
  if (team_all<T>(team, max(ea, eb) < kInf && !(pb && apart > 8) && !(pa && apart < -8))) return;
  uint2 m = make_uint2(0u, 0u);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    m = make_uint2(max(m.x, __float_as_uint(v[k].x) & 0x7fffffffu), max(m.y, __float_as_uint(v[k].y) & 0x7fffffffu));
  m = make_uint2(__reduce_max_sync(0xffffffffu, m.x), __reduce_max_sync(0xffffffffu, m.y));
  if constexpr (T > 32) {
    uint2 *warps = reinterpret_cast<uint2 *>(buf);
    if ((t & 31) == 0) warps[t >> 5] = m;
    team_sync<T>(team);
#pragma unroll
    for (int w = 0; w < T / 32; ++w) m = make_uint2(max(m.x, warps[w].x), max(m.y, warps[w].y));
    team_sync<T>(team);  // (the transform writes there)
  }
  // 2^-e of the largest value's exponent e; zeros and subnormals stay (their
  // powers are 0 in either case)
  auto down = [](uint32_t w) {
    return w < 0x00800000u ? 1.f : __uint_as_float(max(254 - static_cast<int>(w >> 23), 1) << 23);
  };
  const float da = down(m.x), db = down(m.y);
  const bool a = pa && m.x < kInf, b = pb && m.y < kInf;
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = make_float2(a ? v[k].x * da : 0.f, b ? v[k].y * db : 0.f);
  if (t == 0) {
    const uint32_t nan = 0x7fffffffu;
    *factors = make_uint2(m.x < kInf ? __float_as_uint(1.f / da) : nan, m.y < kInf ? __float_as_uint(1.f / db) : nan);
  }
  za |= kPartFlag;
  zb |= kPartFlag;
}

// ------------------------------------------------------------------ small-scale modes
// Y_m = X_m / N of the modes 2c (y0) and 2c + 1 (y1) of one segment (Philox
// words -> Box-Muller): X_m = A_m sqrt(-ln u1) e^{2 pi i u2} (= A (e1 + i e2)/sqrt 2).
// Counter c serves modes 2c (words 0, 1) and 2c + 1 (words 2, 3); the words of
// counter 0 that mode 0 (X_0 = 0) would use serve the Nyquist mode, X = A e1,
// which y0 holds for c = 0.
// ZNODES: amp and amp_hi hold (A_m / N)^2 at two z nodes, mixed with weight
// w_hi; otherwise amp holds A_m / N and amp_hi is unused.
template <int N, bool ZNODES>
__device__ __forceinline__ void small_scale_modes(uint32_t c, const float *__restrict__ amp,
                                                  const float *__restrict__ amp_hi, float w_hi, uint32_t seg,
                                                  uint64_t id, uint32_t seed, float2 &y0, float2 &y1) {
  const u32x4 w = philox4x32_10(u32x4{c, seg, static_cast<uint32_t>(id >> 32), 0u}, seed, static_cast<uint32_t>(id));
  const bool nyq = (c == 0);
  const int m0 = nyq ? N / 2 : 2 * c, m1 = 2 * c + 1;
  const float s0 = __ldg(amp + m0), s1 = __ldg(amp + m1);
  const float2 p0 = unit_phase(w.y), p1 = unit_phase(w.w);
  const float2 nl = neg_log_uniform2(w.x, w.z);
  const float e0 = (nyq ? 2.0f : 1.0f) * nl.x, e1 = nl.y;
  float a0, a1;
  if (ZNODES) {  // interpolate P_s between the nodes; one root for amplitude and modulus
    const float x0 = fmaf(w_hi, __ldg(amp_hi + m0) - s0, s0) * e0, x1 = fmaf(w_hi, __ldg(amp_hi + m1) - s1, s1) * e1;
    a0 = x0 > 0.f ? sqrt_pos(x0) : 0.f;
    a1 = x1 > 0.f ? sqrt_pos(x1) : 0.f;
  } else {
    a0 = s0 * sqrt_pos(e0);
    a1 = s1 * sqrt_pos(e1);
  }
  y0 = make_float2(a0 * p0.x, nyq ? 0.f : a0 * p0.y);
  y1 = make_float2(a1 * p1.x, a1 * p1.y);
}

// The modes 2c, 2c + 1 of the pair (a, b) into the input of its transform.  The
// inverse FFT of Z = A + i B is the forward FFT of Z with its index reversed, so
// that one copy of the transform serves both directions: Z_m = A + i B goes to
// index N - m and Z_{N-m} = conj A + i conj B to index m.  The upper half sits one
// slot up, so that both pairs are stored 16 bytes at a time.
template <int N>
__device__ __forceinline__ void store_mode_pair(float2 *buf, int c, float2 a0, float2 a1, float2 b0, float2 b1) {
  float2 z0 = make_float2(a0.x - b0.y, a0.y + b0.x), y0 = make_float2(a0.x + b0.y, b0.x - a0.y);
  const float2 z1 = make_float2(a1.x - b1.y, a1.y + b1.x), y1 = make_float2(a1.x + b1.y, b1.x - a1.y);
  if (c == 0) {
    buf[N / 2 + 1] = make_float2(a0.x, b0.x);  // the Nyquist mode (real in each segment)
    z0 = y0 = make_float2(0.f, 0.f);
  }
  *reinterpret_cast<float4 *>(buf + 2 * c) = make_float4(y0.x, y0.y, y1.x, y1.y);
  *reinterpret_cast<float4 *>(buf + N - 2 * c) = make_float4(z1.x, z1.y, z0.x, z0.y);
}
template <int N>
__device__ __forceinline__ void load_modes(const float2 *buf, float2 (&v)[8], int t) {
  constexpr int T = N / 8;
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = buf[t + T * r + (r >= 4 ? 1 : 0)];
}

// ------------------------------------------------------------------ cells of a run of pixels
// A sight line crosses a cell in ~1/(dr/cell) pixels (11 at the paper's sizes),
// and inside a cell the trilinear interpolant along the line is a cubic in the
// pixel number.  So the team finds the cells of its run of up to 2N pixels,
// one thread per cell reads the 8 corners and expands the cubic of (delta,
// eta) about the cell's first pixel, and each pixel then takes two 16-byte
// shared-memory reads and three packed FMAs instead of eight global loads and
// seven lerps.
//
// Positions along a run are the record's own, 2^-44 cells: frac + step q at pixel
// q.  The same arithmetic decides which cell a pixel is in and where it is inside
// it.  A decreasing coordinate runs on its complement, which increases and crosses
// cells at the same pixels.  (2^-35 cells in 32 x 32-bit products were 65
// instructions a pair less, and let the step's rounding grow to 2^-24 cells, as
// much as the weight's own, by the end of a pair at N = 2048.)
struct alignas(16) LineAxis {
  uint64_t frac;  // position of pixel 0 inside its cell, in the direction of travel
  uint64_t step;  // |step|
  int32_t c0;     // cell of pixel 0
  float inv;      // 1 / step
  float slope;    // signed step in cells
  int32_t n;      // crossings up to the last pixel
};
struct CellPlan {
  float4 *a, *b;   // cubic: a = (c0, c1), b = (c2, c3), each (delta, eta)
  float *first;    // first pixel of the cell
  uint2 *mask;     // per 32 pixels: {a bit for each first pixel of a cell, bits before}
  LineAxis *line;  // x, y, z
  static constexpr size_t kLineBytes = 3 * sizeof(LineAxis);
};

// Cell plan of a run of npx pixels from pixel j0 of a skewer: lines, masks and
// first pixels; returns the number of cells (the same in every thread).  Starts
// with the plan's memory free and ends with a team barrier.  A run has at most
// cell_capacity() cells.
template <int N>
__device__ __forceinline__ int plan_cells(const CellPlan &C, const mk_skewer *rec, int j0, int npx, int t,
                                          int team) {
  constexpr int T = N / 8, WORDS = N / 16;
  if (t < WORDS) C.mask[t] = make_uint2(0u, 0u);
  if (t < 3) {
    const int64_t step = rec->step[t], p = rec->p0[t] + kRoundQ + j0 * step;
    const bool neg = step < 0;
    LineAxis A;
    A.frac = static_cast<uint64_t>(neg ? ~p : p) & ((uint64_t(1) << 44) - 1);
    A.step = static_cast<uint64_t>(neg ? -step : step);
    A.c0 = static_cast<int32_t>(p >> 44);
    A.inv = __fdividef(1.0f, __ull2float_rn(A.step));
    A.slope = static_cast<float>(step) * 0x1p-44f;
    A.n = static_cast<int>((A.frac + A.step * static_cast<uint32_t>(npx - 1)) >> 44);
    C.line[t] = A;
  }
  team_sync<T>(team);
  const int nx = C.line[0].n, nxy = nx + C.line[1].n, total = nxy + C.line[2].n;
  int *at = reinterpret_cast<int *>(C.a);  // (free until the cubics) first pixel past each crossing
#pragma unroll 1
  for (int i0 = 0; i0 < total; i0 += T) {
    const int i = t + i0;
    if (i < total) {
      const int ax = (i >= nx ? 1 : 0) + (i >= nxy ? 1 : 0);
      const uint32_t k = 1 + i - (i >= nxy ? nxy : (i >= nx ? nx : 0));
      const uint64_t frac = C.line[ax].frac;
      const uint64_t step = C.line[ax].step;
      // the smallest q with frac + q step >= k cells: the FP32 quotient is within
      // 1e-3 of it, so q is its integer part or one or two more
      const uint32_t q0 =
          static_cast<uint32_t>(__ull2float_rn((static_cast<uint64_t>(k) << 44) - frac) * C.line[ax].inv);
      const uint64_t v = frac + step * q0;
      const int q = static_cast<int>(q0) + (static_cast<uint32_t>(v >> 44) < k ? 1 : 0) +
                    (static_cast<uint32_t>((v + step) >> 44) < k ? 1 : 0);
      at[i] = q;
      atomicOr(&C.mask[q >> 5].x, 1u << (q & 31));
    }
  }
  team_sync<T>(team);
  if (t < 32) {  // prefix counts of the words, WORDS / 32 a lane
    constexpr int PER = WORDS < 32 ? 1 : WORDS / 32;
    int c[PER], s = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int w = t * PER + j;
      c[j] = w < WORDS ? __popc(C.mask[w].x) : 0;
      s += c[j];
    }
    int run = s;
#pragma unroll
    for (int o = 1; o < (WORDS < 32 ? WORDS : 32); o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, run, o);
      if (t >= o) run += v;
    }
    run -= s;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int w = t * PER + j;
      if (w < WORDS) C.mask[w].y = static_cast<uint32_t>(run);
      run += c[j];
    }
  }
  if (t == 0) C.first[0] = 0.f;
  team_sync<T>(team);
#pragma unroll 1
  for (int i0 = 0; i0 < total; i0 += T) {
    const int i = t + i0;
    if (i < total) {
      const int q = at[i];
      const uint2 m = C.mask[q >> 5];
      C.first[m.y + __popc(m.x & (0xffffffffu >> (31 - (q & 31))))] = static_cast<float>(q);
    }
  }
  const uint2 m = C.mask[WORDS - 1];
  const int cells = static_cast<int>(m.y) + __popc(m.x) + 1;
  team_sync<T>(team);
  return cells;
}

// Sight-line weights of the velocity-gradient tensor (Eq. eta) from the step in
// any unit: {ux^2, uy^2, uz^2, 2 ux uy, 2 ux uz, 2 uy uz} (MK_BOX_TENSOR only).
template <int LAYOUT>
__device__ __forceinline__ void tensor_weights(float ux, float uy, float uz, float (&uu)[6]) {
  if constexpr (LAYOUT == MK_BOX_TENSOR) {
    const float inv = rsqrtf(ux * ux + uy * uy + uz * uz);
    const float vx = ux * inv, vy = uy * inv, vz = uz * inv;
    uu[0] = vx * vx;
    uu[1] = vy * vy;
    uu[2] = vz * vz;
    uu[3] = 2.f * vx * vy;
    uu[4] = 2.f * vx * vz;
    uu[5] = 2.f * vy * vz;
  }
}

// (delta, eta) at the 8 corners of cell (x0, y0, z0); eta of MK_BOX_TENSOR is
// the velocity-gradient tensor contracted with the sight line, uu = {ux^2,
// uy^2, uz^2, 2 ux uy, 2 ux uz, 2 uy uz}.
template <int LAYOUT>
__device__ __forceinline__ void load_corners(const float *__restrict__ d, const float *__restrict__ e, int lgn, int x0,
                                             int y0, int z0, const float (&uu)[6], float2 (&v)[8]) {
  const int mask = (1 << lgn) - 1;
  if constexpr (LAYOUT == MK_BOX_PADDED || LAYOUT == MK_BOX_HALO || LAYOUT == MK_BOX_TENSOR) {
    constexpr int h = LAYOUT == MK_BOX_HALO ? 3 : 0;
    const uint32_t n1 = mask + 1 + (LAYOUT == MK_BOX_HALO ? 6 : 1);  // (one 32 x 32 + 64-bit product a point)
    const int64_t i00 = static_cast<uint64_t>((z0 + h) * n1 + (y0 + h)) * n1 + (x0 + h);
    const int64_t row[4] = {i00, i00 + n1, i00 + n1 * n1, i00 + n1 * n1 + n1};
    if constexpr (LAYOUT == MK_BOX_TENSOR) {
      const float4 *b = reinterpret_cast<const float4 *>(d);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float4 p = __ldg(b + 2 * (row[k >> 1] + (k & 1))), q = __ldg(b + 2 * (row[k >> 1] + (k & 1)) + 1);
        const float eta = fmaf(uu[0], p.y, fmaf(uu[1], p.z, fmaf(uu[2], p.w,
                          fmaf(uu[3], q.x, fmaf(uu[4], q.y, uu[5] * q.z)))));
        v[k] = make_float2(p.x, eta);
      }
    } else {
      const float2 *b = reinterpret_cast<const float2 *>(d);
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __ldg(b + row[k >> 1] + (k & 1));
    }
  } else {
    // (row pointers by a 32 x 32 + 64-bit product each)
    const uint32_t n = mask + 1, xa = x0, xb = (x0 + 1) & mask, y1 = (y0 + 1) & mask, z1 = (z0 + 1) & mask;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t zy = (k & 2 ? z1 : z0) * n + (k & 1 ? y1 : y0);
      if constexpr (LAYOUT == MK_BOX_INTERLEAVED) {
        const float2 *row = reinterpret_cast<const float2 *>(reinterpret_cast<const char *>(d) + static_cast<uint64_t>(zy) * (8u * n));
        v[2 * k] = __ldg(row + xa);
        v[2 * k + 1] = __ldg(row + xb);
      } else {
        const uint64_t i = static_cast<uint64_t>(zy) * n;
        v[2 * k] = make_float2(__ldg(d + (i | xa)), __ldg(e + (i | xa)));
        v[2 * k + 1] = make_float2(__ldg(d + (i | xb)), __ldg(e + (i | xb)));
      }
    }
  }
}

__device__ __forceinline__ float2 f2fma1(float a, float2 b, float2 c) { return f2fma(make_float2(a, a), b, c); }
__device__ __forceinline__ float2 f2mul1(float a, float2 b) { return f2mul(make_float2(a, a), b); }

// The cubic of cell c: the trilinear interpolant of the corners along the line,
// expanded in the pixel number from the cell's first pixel.  At that pixel it
// is the lerp in x, then y, then z.
template <int LAYOUT>
__device__ __forceinline__ void expand_cell(const CellPlan &C, int c, const float *__restrict__ d,
                                            const float *__restrict__ e, int lgn) {
  const int mask = (1 << lgn) - 1;
  const uint32_t q = static_cast<uint32_t>(C.first[c]);
  int cell[3];
  float w[3], sl[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const LineAxis A = C.line[k];
    const uint64_t v = A.frac + A.step * q;
    const int crossed = static_cast<int>(v >> 44);
    cell[k] = (A.slope < 0.f ? A.c0 - crossed : A.c0 + crossed) & mask;
    w[k] = weight_of(static_cast<int64_t>(A.slope < 0.f ? ~v : v));
    sl[k] = A.slope;
  }
  const float wx = w[0], wy = w[1], wz = w[2], sx = sl[0], sy = sl[1], sz = sl[2];
  float2 v[8];
  float uu[6];
  tensor_weights<LAYOUT>(sx, sy, sz, uu);
  load_corners<LAYOUT>(d, e, lgn, cell[0], cell[1], cell[2], uu, v);
  float2 f0[2], f1[2], f2[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float2 d0 = f2sub(v[4 * k + 1], v[4 * k]), d1 = f2sub(v[4 * k + 3], v[4 * k + 2]);
    const float2 a0 = f2fma1(wx, d0, v[4 * k]), a1 = f2fma1(wx, d1, v[4 * k + 2]);
    const float2 b0 = f2mul1(sx, d0), b1 = f2mul1(sx, d1);
    const float2 da = f2sub(a1, a0), db = f2sub(b1, b0);
    f0[k] = f2fma1(wy, da, a0);
    f1[k] = f2fma1(wy, db, f2fma1(sy, da, b0));
    f2[k] = f2mul1(sy, db);
  }
  const float2 g0 = f2sub(f0[1], f0[0]), g1 = f2sub(f1[1], f1[0]), g2 = f2sub(f2[1], f2[0]);
  const float2 c0 = f2fma1(wz, g0, f0[0]);
  const float2 c1 = f2fma1(wz, g1, f2fma1(sz, g0, f1[0]));
  const float2 c2 = f2fma1(wz, g2, f2fma1(sz, g1, f2[0]));
  const float2 c3 = f2mul1(sz, g2);
  C.a[c] = make_float4(c0.x, c0.y, c1.x, c1.y);
  C.b[c] = make_float4(c2.x, c2.y, c3.x, c3.y);
}

// (delta, eta) at pixel q of the run, m its mask word (uniform in the warp)
__device__ __forceinline__ float2 eval_cell(const CellPlan &C, uint2 m, float q, uint32_t lanes_le) {
  const int c = static_cast<int>(m.y) + __popc(m.x & lanes_le);
  const float4 a = C.a[c], b = C.b[c];
  const float x = q - C.first[c];
  const float2 r = f2fma1(x, make_float2(b.z, b.w), make_float2(b.x, b.y));
  return f2fma1(x, f2fma1(x, r, make_float2(a.z, a.w)), make_float2(a.x, a.y));
}

}  // namespace mk
