// Template of the fused skewer kernel and what it shares with the statistics
// (mk_stats.cuh) and single-segment (mk_segment.cuh) kernels; each FFT length is instantiated in its own translation
// unit (mk_skewer_<N>.cu).
#pragma once

#include "mk_pair.cuh"

namespace mk {

// =================================================================== shared-memory plan
template <int N>
__host__ __device__ inline size_t acc_bytes(int threads, int n_z, int n_k, bool stats) {
  return stats ? static_cast<size_t>(threads / (N / 8)) * TeamAcc<N>::bytes(n_z, n_k) : 0;
}

// Fused kernel, per CTA: the teams' accumulators (when statistics are on), the
// twiddles, the ends of the z bins, then per team one area that is the FFT's
// exchange buffer and, between the two transforms, the cubics of the pair's
// cells; a stash of N floats; the skewer's record; and the line, the masks and
// the cells' first pixels (cap, a multiple of 4, is 0 for the Gaussian kernel).
template <int N>
struct PairSmem {
  static constexpr int T = N / 8;
  __host__ __device__ static size_t area_bytes(int cap) {
    const size_t f = sizeof(float2) * PairFft<N>::BUF, c = 32 * static_cast<size_t>(cap);
    return f > c ? f : c;
  }
  static constexpr size_t HEAD = (PairFft<N>::TW_BYTES + 15) / 16 * 16 + (sizeof(int32_t) * (MK_MAX_ZBINS + 2) + 15) / 16 * 16;
  static constexpr int REC = 10;  // 8-byte words kept for the record
  __host__ __device__ static size_t team_bytes(int cap) {
    return area_bytes(cap) + sizeof(float) * N + sizeof(uint64_t) * REC +
           (cap > 0 ? CellPlan::kLineBytes + sizeof(uint2) * (N / 16) + sizeof(float) * cap : 0);
  }
  __host__ __device__ static size_t bytes(int threads, int n_z, int n_k, bool stats, int cap) {
    return acc_bytes<N>(threads, n_z, n_k, stats) + HEAD + static_cast<size_t>(threads / T) * team_bytes(cap);
  }
};

// largest i with a[i] <= v over a[0..n] (a non-decreasing)
__device__ __forceinline__ int64_t upper_index(const int64_t *a, int64_t n, int64_t v) {
  int64_t lo = 0, hi = n;
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (a[mid] <= v) lo = mid; else hi = mid;
  }
  return lo;
}

// Sum the CTA's compensated FP32 accumulators in FP64, warp after warp, and write
// its partials in the StatLayout order.
template <int N>
__device__ __forceinline__ void flush_partials(unsigned char *smem, int teams, int n_z, int n_k, double *partials) {
  using A = TeamAcc<N>;
  __syncthreads();
  const StatLayout L{n_z, n_k};
  const size_t tbytes = A::bytes(n_z, n_k);
  const int ns = n_z * MK_NSUM, np = n_z * n_k, slots = A::slots(n_k);
  auto value = [](float2 v) { return static_cast<double>(v.x) - static_cast<double>(v.y); };
  for (int idx = threadIdx.x; idx < L.size(); idx += blockDim.x) {
    double s = 0.0;
#pragma unroll 4
    for (int team = 0; team < teams; ++team) {
      const A a = A::at(smem + team * tbytes, 0, n_z, n_k);
      if (idx < ns) {
#pragma unroll 1
        for (int w = 0; w < A::WARPS; ++w) s += value(a.sums[w * ns + idx]);
      } else if (idx < ns + np) {
        const int z = (idx - ns) / n_k, k = (idx - ns) % n_k;
#pragma unroll 1
        for (int q = k * slots / n_k; q < (k + 1) * slots / n_k; ++q) s += value(a.p1d[z * slots + q]);
      } else {
        s += static_cast<double>(a.nseg[idx - ns - np]);
      }
    }
    partials[static_cast<size_t>(blockIdx.x) * L.size() + idx] = s;
  }
}

// =================================================================== fused skewer kernel
// One team per pair of segments of N pixels of a skewer: cells of the pair's
// sight line -> small-scale modes of both -> one inverse FFT -> per pixel the
// cell's cubic, growth, FGPA, stores and pixel sums -> one forward FFT of both
// fluxes -> P1D.  Pairs never straddle skewers, so a skewer's pixels do not
// depend on how a catalogue is cut into launches.  Teams take contiguous ranges
// of pairs.  Pixel sums stay in registers, across segments, for as long as the
// warp's pixels stay in one z bin: the warp flushes them to its shared
// accumulators when its pixels reach the end of the bin (bin_end) or a
// segment starts in another bin.
//
// Bound by instruction issue: 6.5 warp instructions a pixel at 67 % of the issue
// slots, DRAM ~10 B a pixel.  60k quasars (8.2e7 pixels, 512^3 box): one radix-8
// transform for two segments and one set of corner loads per cell of the sight line
// take 0.66 ms at N = 256 where a radix-4 transform per segment and a gather of
// eight corners per pixel took 0.74, 0.83 against 1.33 on a tensor box, 1.03 against
// 1.12 at N = 1024; a step of the 1024^3 box with 1M quasars went from 13.0 to 11.2 ms.
// The loop over pairs has to fit the instruction cache: variants of it whose
// pixel loops were unrolled further (4400 to 6000 instructions instead of 3600)
// ran 10 to 50 % slower, stalled on fetches.  Registers are as scarce: with the cells
// of one segment at a time (to hold fewer of them) it spilled and was 10 % slower.
//
// INTERP == MK_INTERP_TRILINEAR: from the cubics of the line's cells (needs
// P.cell_cap).  MK_INTERP_GAUSS7 (LAYOUT must be MK_BOX_HALO): the averages of a
// segment are computed ahead of its pixel loop into the exchange buffer
// (gauss7_run).  Long pixels and catalogues of single segments: k_segment.
// PSZ: P_s given at several redshifts (P.ps_nodes >= 2), interpolated per segment
template <int N, int LAYOUT, int MINB, int INTERP, bool PSZ>
__global__ void __launch_bounds__(256, MINB) k_skewer(SkewerParams P) {
  constexpr int T = N / 8;
  constexpr bool CELLS = INTERP == MK_INTERP_TRILINEAR;
  constexpr int kRows = 2;  // rows of T pixels per round of the pixel loop
  const int teams = blockDim.x / T;
  const int team = threadIdx.x / T, t = threadIdx.x % T, lane = threadIdx.x & 31;
  const int wlo0 = t & ~31;  // first team pixel of this warp
  extern __shared__ __align__(16) unsigned char smem[];
  const size_t tbytes = P.do_stats ? TeamAcc<N>::bytes(P.n_z, P.n_k) : 0;
  float2 *tws = reinterpret_cast<float2 *>(smem + teams * tbytes);
  int32_t *bin_end = reinterpret_cast<int32_t *>(tws + (PairFft<N>::TW_BYTES + 15) / 16 * 2);
  unsigned char *mine = smem + teams * tbytes + PairSmem<N>::HEAD + team * PairSmem<N>::team_bytes(P.cell_cap);
  float2 *buf = reinterpret_cast<float2 *>(mine);
  CellPlan C;
  C.a = reinterpret_cast<float4 *>(mine);
  C.b = C.a + P.cell_cap;
  float *stash = reinterpret_cast<float *>(mine + PairSmem<N>::area_bytes(P.cell_cap));
  uint64_t *recw = reinterpret_cast<uint64_t *>(stash + N);
  const mk_skewer *rec = reinterpret_cast<const mk_skewer *>(recw);
  C.line = reinterpret_cast<LineAxis *>(recw + PairSmem<N>::REC);
  C.mask = reinterpret_cast<uint2 *>(C.line + 3);
  C.first = reinterpret_cast<float *>(C.mask + N / 16);
  const TeamAcc<N> W = TeamAcc<N>::at(smem + team * tbytes, t >> 5, P.n_z, P.n_k);
  if (P.do_stats) {
    W.zero(smem + team * tbytes, P.n_z, P.n_k, t);
    for (int k = threadIdx.x; k < P.n_z + 2; k += blockDim.x) bin_end[k] = P.bin_end[k];
  }
  fill_pair_twiddles<N>(tws, P.tw);  // (ends with a CTA barrier)

  // pairs segoff[0] .. segoff[n_sk] (a slice of a larger catalogue may start
  // at segoff[0] > 0)
  const int64_t u0 = P.segoff[0], nunits = P.segoff[P.n_sk] - u0;
  const int64_t g = static_cast<int64_t>(blockIdx.x) * teams + team;
  const int64_t G = static_cast<int64_t>(gridDim.x) * teams;
  int64_t u = u0 + g * nunits / G;
  const int64_t uend = u0 + (g + 1) * nunits / G;
  int64_t i = u < uend ? upper_index(P.segoff, P.n_sk, u) : 0;

  // The skewer's record waits in shared memory, and the next skewer's in a
  // register of each of nine threads (thread t: word t), so that a new skewer costs
  // no round trip to memory.
  constexpr int kRecWords = 9;
  static_assert(sizeof(mk_skewer) == kRecWords * sizeof(uint64_t), "the record's words");
  auto fetch = [&](int64_t q) -> uint64_t {
    return q < P.n_sk && t < kRecWords ? reinterpret_cast<const uint64_t *>(P.sk + q)[t] : 0;
  };
  uint64_t next = fetch(i);
  int pair = static_cast<int>(u - P.segoff[i]), left = 0;  // next pair of the skewer, pairs left from it on
  --i;

  PixelSums acc;
  acc.zero();
  int zc = -2;  // z bin of acc (warp-uniform), -2 before the first segment
  const uint32_t lanes_le = 0xffffffffu >> (31 - lane);
  // inner node of this lane, for the search by ballot
  const float ps_node = PSZ && lane >= 1 && lane < P.ps_nodes - 1 ? P.ps_z[lane < MK_MAX_NODES ? lane : 0] : INFINITY;
  const bool put_fields = P.delta_out != nullptr, put_flux = P.flux_out != nullptr;

  for (; u < uend; ++u) {
    while (left == 0) {  // (the last pair ended with a barrier)
      ++i;
      if (t < kRecWords) recw[t] = next;
      next = fetch(i + 1);
      team_sync<T>(team);
      left = (rec->n + 2 * N - 1) / (2 * N) - pair;
      if (left == 0) team_sync<T>(team);  // an empty skewer
    }
    const int s = 2 * pair++;
    if (--left == 0) pair = 0;
    const int64_t offset = rec->offset;
    const int n = rec->n;
    const int j0 = s * N;              // first pixel of the pair
    const int npair = min(2 * N, n - j0);
    if ((put_fields || put_flux) && offset + n > P.capacity) {
      if (t == 0) raise_error(P.err, ERR_CAPACITY);
      team_sync<T>(team);
      continue;
    }
    const int jb0 = rec->j_lo + j0;
    const bool two = npair > N;
    // z bins of the two segments' first pixels and of the full segments
    int z0[2] = {0, 0}, zs[2] = {-1, -1};
    if (P.do_stats) {
      z0[0] = __ldg(P.zbin + jb0);
      if (two) z0[1] = __ldg(P.zbin + jb0 + N);
      if (npair >= N) zs[0] = __ldg(P.segzbin + jb0);
      if (npair == 2 * N) zs[1] = __ldg(P.segzbin + jb0 + N);
    }
    // ---- start the box rows of the pair's stencils on their way to L2, where
    // the loads are many (the tensor's 64 bytes a corner row, 1.57 -> 1.48 ms
    // per 1.4e8 pixels; the Gaussian kernel's): lane t samples pixel 16t + 8.  The
    // 8-byte layouts read each cell once and gain nothing from it.
    if constexpr (!CELLS || LAYOUT == MK_BOX_TENSOR) {
      const int64_t q = j0 + min(npair - 1, 16 * t + 8);
      prefetch_stencil<LAYOUT>(P.box_d, P.lgn, rec->p0[0] + kRoundQ + q * rec->step[0],
                               rec->p0[1] + kRoundQ + q * rec->step[1], rec->p0[2] + kRoundQ + q * rec->step[2]);
    }
    int cells = 0;
    if constexpr (CELLS) cells = plan_cells<N>(C, rec, j0, npair, t, team);

    float2 v[8];
    int za = zs[0], zb = zs[1];
    // Two rounds of one transform: modes to delta_S, then flux to its modes
    // (one copy of the code: the loop over pairs has to stay within what the
    // instruction cache holds; unrolled it stalled on fetches for a third of
    // its time)
#pragma unroll 1
    for (int round = 0; round < 2; ++round) {
      if (round == 0) {
        // ---- small-scale field of both segments: iteration (q, h) draws the
        // modes 2c, 2c + 1 (< N/2), c = t + q T, of segment h
        const uint64_t id = rec->id;
        // P_s at the mean z of each segment's window, linear between nodes (every
        // lane compares with one: 2.53 -> 2.40 ms a pass of 2e8 pixels with 12 nodes, N = 1024, with one root for both)
        int pn[2] = {0, 0};
        float pw[2] = {0.f, 0.f};
        if constexpr (PSZ) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (h == 0 || two) {
              const float zw = __ldg(P.zwin + jb0 + h * N);
              const int n0 = __popc(__ballot_sync(0xffffffffu, zw >= ps_node));
              pn[h] = n0;
              pw[h] = fminf(fmaxf((zw - P.ps_z[n0]) / (P.ps_z[n0 + 1] - P.ps_z[n0]), 0.f), 1.f);
            }
          }
        }
        float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
        for (int it = 0; it < 4; ++it) {
          const int h = it & 1;
          const uint32_t c = t + (it >> 1) * T;
          float2 y0 = make_float2(0.f, 0.f), y1 = y0;
          if (h == 0 || two) {
            const float *amp = P.amp;
            float w_hi = 0.f;
            if constexpr (PSZ) {
              amp += (h ? pn[1] : pn[0]) * (N / 2 + 1);
              w_hi = h ? pw[1] : pw[0];
            }
            small_scale_modes<N, PSZ>(c, amp, amp + (N / 2 + 1), w_hi, static_cast<uint32_t>(s + h), id, P.seed, y0,
                                      y1);
          }
          if (h == 0) {
            a0 = y0;
            a1 = y1;
          } else {
            store_mode_pair<N>(buf, c, a0, a1, y0, y1);
          }
        }
        team_sync<T>(team);
        load_modes<N>(buf, v, t);
      }
      // (a barrier: the modes are read; the cells are read)
      if (round == 0) team_sync<T>(team);
      else drop_nan<T>(v, za, zb, team);
      pair_fft<N>(buf, v, tws, P.tw, t, team);
      if (round == 1) break;

      // v[r].x, v[r].y: delta_S of pixel t + T r of the two segments
      // ---- the cells' cubics, over the exchange buffer
      if constexpr (CELLS) {
        team_sync<T>(team);
        for (int c = t; c < cells; c += T) expand_cell<LAYOUT>(C, c, P.box_d, P.box_e, P.lgn);
        team_sync<T>(team);
      }

      // ---- per pixel: interpolation, growth, FGPA, stores, pixel sums.  One pass
      // of the loop per segment, with the transform's parts swapped after each
      // (one copy of the code)
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        const int npx = min(N, npair - h * N);
        if constexpr (INTERP == MK_INTERP_GAUSS7) {  // (delta, eta) of the segment, over the exchange buffer
          static_assert(LAYOUT == MK_BOX_HALO, "the Gaussian kernel reads a halo box");
          team_sync<T>(team);
          if (npx > 0)
            gauss7_run(buf, reinterpret_cast<uint16_t *>(stash + 8 * wlo0), P.box_d, P.lgn, rec, j0 + h * N, npx, t >> 5,
                       T / 32, lane);
          team_sync<T>(team);
        }
        float f8[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) f8[k] = 0.f;
        if (npx > 0) {
          const int jb = jb0 + h * N;
          int pend = N;  // segment pixel where bin zc ends
          if (P.do_stats) {
            const int z = h ? z0[1] : z0[0];
            if (z != zc || (h == 0 && u % kRunPairs == 0)) {
              if (zc != -2) flush_bin_sums<false>(W, P.n_z, zc, acc, lane);
              acc.zero();
              zc = z;
            }
            pend = bin_end[zc + 1] - jb;
          }
          // Rows of T pixels go through the stash (a thread's own pixels: no
          // barrier), so that the loop stays rolled; everything points at the
          // thread's pixel of row d / T.
          const int64_t o = offset + j0 + h * N + t;
          const float4 *tp = P.pixtab + jb + t;
          const uint2 *mp = C.mask + ((h * N + wlo0) >> 5);
          float *sp = stash + t, *fp = P.flux_out + o;
          float qf = static_cast<float>(h * N + t);
          const int rem = npx - t, rem_flux = put_flux ? rem : 0;
#pragma unroll
          for (int k = 0; k < 8; ++k) sp[T * k] = v[k].x;
          // (delta, eta) at the thread's pixel of row d / T + k
          auto interpolate = [&](int d, int k) -> float2 {
            if constexpr (CELLS) {
              return eval_cell(C, mp[k * (T / 32)], qf + static_cast<float>(T * k), lanes_le);
            } else {
              return buf[t + d + T * k];
            }
          };
          auto flux_of = [&](float2 de, float4 tb, float ds, float2 &x) -> float {
            x = make_float2(fmaf(tb.x, de.x, ds), tb.x * de.y);
            return fgpa(tb, x.x, x.y);
          };
#pragma unroll 1
          for (int d = 0; d + wlo0 < npx; d += kRows * T) {
            if (d + (kRows - 1) * T + wlo0 + 32 <= pend || pend >= npx) {
              // rows inside one z bin: no branches, pixels past the segment's end
              // are computed and masked (their cells and table entries exist)
#pragma unroll
              for (int k = 0; k < kRows; ++k) {
                const bool on = d + T * k < rem;
                const float2 de = interpolate(d, k);
                float2 x;
                float f = flux_of(de, __ldg(tp + T * k), sp[T * k], x);
                if (d + T * k < rem_flux) fp[T * k] = f;
                if (put_fields && on) {
                  P.delta_out[o + d + T * k] = x.x;
                  P.eta_out[o + d + T * k] = x.y;
                }
                f = on ? f : 0.f;
                acc.n += on ? 1.f : 0.f;
                acc.add_sums(f, make_float2(on ? x.x : 0.f, on ? x.y : 0.f));
                sp[T * k] = f;
              }
            } else {
#pragma unroll 1
              for (int k = 0; k < kRows; ++k) {
                const int p = t + d + T * k;
                float f = 0.f;
                float2 x = make_float2(0.f, 0.f);
                bool todo = p < npx;
                if (todo) {
                  const float2 de = interpolate(d, k);
                  f = flux_of(de, __ldg(tp + T * k), sp[T * k], x);
                  if (put_fields) {
                    P.delta_out[o + d + T * k] = x.x;
                    P.eta_out[o + d + T * k] = x.y;
                  }
                  if (put_flux) fp[T * k] = f;
                }
                // this warp's pixels: d + T k + wlo0 + lane; flush while they pass pend
                const int hi = min(d + T * k + wlo0 + 32, npx);
                while (P.do_stats && hi > pend) {
                  if (todo && p < pend) {
                    acc.add(f, x);
                    todo = false;
                  }
                  flush_bin_sums<false>(W, P.n_z, zc, acc, lane);
                  acc.zero();
                  ++zc;
                  pend = bin_end[zc + 1] - jb;
                }
                if (todo) acc.add(f, x);
                sp[T * k] = f;
              }
            }
            tp += kRows * T;
            mp += kRows * (T / 32);
            sp += kRows * T;
            fp += kRows * T;
            qf += static_cast<float>(kRows * T);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) f8[k] = T * k < rem ? stash[T * k + t] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = make_float2(v[k].y, f8[k]);
      }
      // ---- P1D of the full segments
      if (!(counted(za, P.n_z) || counted(zb, P.n_z))) {  // (always without statistics)
        za = -2;
        break;
      }
    }
    if (za != -2) {
      float ka[4], kb[4];
      pair_powers<N>(buf, v, t, team, ka, kb);
      // (N = 512, 1024: the accumulators' place is worked out here; held through the
      // loop it costs registers, 88 bytes of spills and 3 % at N = 1024)
      int tm = team, wt = t >> 5;
      if constexpr (N == 512 || N == 1024) asm volatile("" : "+r"(tm), "+r"(wt));
      const TeamAcc<N> A = TeamAcc<N>::at(smem + tm * tbytes, wt, P.n_z, P.n_k);
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (counted(za, P.n_z)) {
          const int z = za & ~kPartFlag;
          accumulate_p1d(A, P.n_k, t, ka, za == z ? 0.25f * P.p1d_scale : __uint_as_float(0x7fffffffu), z);
          if (t == 0) A.nseg[z] += 1u;
        }
        za = zb;
#pragma unroll
        for (int j = 0; j < 4; ++j) ka[j] = kb[j];
      }
    } else {
      team_sync<T>(team);  // the cells are read
    }
  }
  if (P.do_stats) {
    if (zc != -2) flush_bin_sums<false>(W, P.n_z, zc, acc, lane);
    flush_partials<N>(smem, teams, P.n_z, P.n_k, P.partials);
  }
}

}  // namespace mk
