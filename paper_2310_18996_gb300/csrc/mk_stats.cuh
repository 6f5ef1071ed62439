// The statistics kernels: of stored flux at any rebin, or of the FGPA of stored
// delta, eta (the tuning pass), then with each team's next pair of segments
// staged in shared memory.
#pragma once

#include "mk_skewer.cuh"

namespace mk {

// =================================================================== shared memory
// Per CTA: the teams' accumulators, the twiddles, the ends of the z bins, then per
// team two stage buffers of delta and eta (a pair's transform runs in its own
// stage buffer once its fields are read) and one mbarrier per buffer, or, when
// nothing is staged, the transform's exchange buffer.
template <int N, bool STAGED>
struct StatSmem {
  static constexpr int STAGE = 2 * N + 4;  // floats per field and buffer (a pair plus its 16-byte misalignment)
  static_assert(2 * STAGE >= 2 * PairFft<N>::BUF, "a stage buffer holds the exchange buffer");
  static_assert((STAGE * sizeof(float)) % 16 == 0, "stage buffers start on 16 bytes");
  static constexpr size_t HEAD = PairSmem<N>::HEAD + 8 * sizeof(uint2);  // and the teams' factors of part_segments
  static constexpr size_t TEAM = STAGED ? 4 * STAGE * sizeof(float) + 2 * sizeof(uint64_t) : sizeof(float2) * PairFft<N>::BUF;
  static size_t bytes(int threads, int n_z, int n_k) {
    return acc_bytes<N>(threads, n_z, n_k, true) + HEAD + static_cast<size_t>(threads / (N / 8)) * TEAM;
  }
};

// ------------------------------------------------------------------ bulk copies
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
// the initialised barriers are visible to the bulk-copy engine
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
// the one expected arrival of a phase, with the bytes its copies will bring
__device__ __forceinline__ void mbar_arrive_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// Wait for the phase of the given parity for at most `limit` clock cycles
// (the copies of a segment take microseconds); false when the wait gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > limit) return false;
  return true;
}
// earlier generic accesses of shared memory are ordered before later bulk copies into it
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// bytes (a multiple of 16, both addresses 16-byte aligned) from global to shared memory
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Where the kernel finds a pair of segments: its first index in the stored
// arrays (fields, or flux), its output pixels, its first pixel-table index,
// whether its pixels lie inside the tables; and, staged, the last (shift + npx)
// mod 4 floats of delta and eta (thread t holds float t of them), which the whole
// 16-byte pieces of the bulk copies leave.
struct StatPair {
  int64_t field, flux;
  int npx, jb;
  bool ok;
  float td, te;
};

// =================================================================== statistics kernel
// Statistics of output pixels of R = P.rebin fine pixels.  A team takes pairs of
// segments of N output pixels of a skewer, in contiguous ranges; both segments'
// flux goes through one transform (mk_pair.cuh).  The pixel sums stay in
// registers across segments while the warp's pixels stay in one z bin and are
// flushed at the bin's end; an output pixel's z bin comes from the tables of mean
// z over R pixels (zbin, bin_end) for every R.  (With R > 1 the bin once came
// from an FP64 division per pixel, and this GPU's FP64 pipe was the bound: flux
// and statistics of 1.4e8 fine pixels at R = 3 took 3.28 ms then and 1.19 ms with
// the tables.)  Without staging, the next pair's lines are requested into L2 while
// one is processed: this kernel alone, 2.9e8 fine pixels at R = 3, 1.11 -> 0.82 ms,
// of it 0.12 from one copy of the bin loop's flush instead of eight.
//
// STAGED: a tuning pass (rebin 1, fields and FGPA table set; delta, eta 16-byte
// aligned): the next pair's fields are copied into shared memory by the bulk-copy
// (TMA) engine while the current one is processed.  It reads 8 bytes a pixel and
// is bound by latency and issue: 4.25 ms per 1.45e9 pixels, where one radix-4
// transform per segment took 5.67 ms; 16 warps an SM by registers.  (Buffers of a
// segment instead of a pair hold larger binnings at 16 warps, but 1.50 ms where
// these take 1.29: 300k skewers.)
// Both variants work through the same pairs in the same order with the same
// grid, so a tuning pass and the statistics of its stored flux agree bit for bit.
template <int N, bool STAGED>
__global__ void __launch_bounds__(256, 2) k_stats(StatParams P) {
  constexpr int T = N / 8;
  constexpr int STAGE = StatSmem<N, STAGED>::STAGE;
  const int teams = blockDim.x / T;
  const int team = threadIdx.x / T, t = threadIdx.x % T, lane = threadIdx.x & 31;
  const int wlo0 = t & ~31;  // first team pixel of this warp
  extern __shared__ __align__(16) unsigned char smem[];
  const size_t tbytes = TeamAcc<N>::bytes(P.n_z, P.n_k);
  float2 *tws = reinterpret_cast<float2 *>(smem + teams * tbytes);
  int32_t *bin_end = reinterpret_cast<int32_t *>(tws + (PairFft<N>::TW_BYTES + 15) / 16 * 2);
  unsigned char *areas = smem + teams * tbytes + StatSmem<N, STAGED>::HEAD;
  uint2 *factors = reinterpret_cast<uint2 *>(areas - 8 * sizeof(uint2)) + team;
  // stage buffers b = 0, 1: delta at stage_buf + 2 b STAGE, eta at stage_buf + (2 b + 1) STAGE
  float *stage_buf = reinterpret_cast<float *>(areas) + (STAGED ? team * 4 * STAGE : team * 2 * PairFft<N>::BUF);
  uint64_t *bars = reinterpret_cast<uint64_t *>(areas + static_cast<size_t>(teams) * 4 * STAGE * sizeof(float)) + 2 * team;
  const TeamAcc<N> W = TeamAcc<N>::at(smem + team * tbytes, t >> 5, P.n_z, P.n_k);
  W.zero(smem + team * tbytes, P.n_z, P.n_k, t);
  for (int k = threadIdx.x; k < P.n_z + 2; k += blockDim.x) bin_end[k] = P.bin_end[k];
  if (STAGED && t == 0) {
    mbar_init(bars);
    mbar_init(bars + 1);
    mbar_init_fence();
  }
  fill_pair_twiddles<N>(tws, P.tw);  // (ends with a CTA barrier)

  const int64_t nunits = P.segoff[P.n_sk];
  const int64_t g = static_cast<int64_t>(blockIdx.x) * teams + team;
  const int64_t G = static_cast<int64_t>(gridDim.x) * teams;
  const int64_t u_first = g * nunits / G, uend = (g + 1) * nunits / G;
  const int R = STAGED ? 1 : P.rebin;
  int64_t inext = u_first < uend ? upper_index(P.segoff, P.n_sk, u_first) : 0;  // skewer of the pair to describe next
  PixelSums acc;
  acc.zero();
  int zc = -2;  // z bin of acc (warp-uniform), -2 before the first segment

  // describe pair uu (of skewer inext, advanced as needed); team-uniform
  auto describe = [&](int64_t uu) -> StatPair {
    while (P.segoff[inext + 1] <= uu) ++inext;
    const int64_t o = P.off_out[inext], nout = P.off_out[inext + 1] - o;
    const int64_t k0 = (uu - P.segoff[inext]) * (2 * N);
    const int j_lo = P.sk[inext].j_lo;
    StatPair d;
    d.field = P.sk[inext].offset + k0 * R;
    d.flux = o + k0;
    d.npx = static_cast<int>(min(static_cast<int64_t>(2 * N), nout - k0));
    // records made for another pixel length may run past the pixel tables
    d.ok = j_lo >= 0 && j_lo + nout * R <= P.j_max;
    d.jb = d.ok ? j_lo + static_cast<int>(k0 * R) : 0;
    d.td = d.te = 0.f;
    return d;
  };
  // Copy pair d's fields into stage buffer b: thread 0 of the team issues two
  // bulk copies of the whole 16-byte pieces from d.field rounded down to 16 bytes
  // (pixel p lands at (field & 3) + p), completing on bars[b]; the threads
  // t < (shift + npx) mod 4 load the floats after the last piece.
  auto stage = [&](StatPair &d, int b) {
    const int shift = static_cast<int>(d.field & 3);
    const int nfl = (shift + d.npx) & ~3, tail = shift + d.npx - nfl;
    const float *bd = P.delta + (d.field - shift), *be = P.eta + (d.field - shift);
    d.td = t < tail ? __ldg(bd + nfl + t) : 0.f;
    d.te = t < tail ? __ldg(be + nfl + t) : 0.f;
    if (t == 0) {
      fence_async_shared();
      mbar_arrive_tx(bars + b, static_cast<uint32_t>(8 * nfl));
      if (nfl > 0 && !P.wait_test) {  // (the test hook leaves the expected bytes missing)
        bulk_g2s(stage_buf + 2 * b * STAGE, bd, static_cast<uint32_t>(4 * nfl), bars + b);
        bulk_g2s(stage_buf + (2 * b + 1) * STAGE, be, static_cast<uint32_t>(4 * nfl), bars + b);
      }
    }
  };
  auto prefetch = [&](const StatPair &d) {
    if (!d.ok) return;
    if (!P.pixtab)
      for (int i = 32 * t; i < d.npx; i += 32 * T) prefetch_l2(P.flux + d.flux + i);
    if (P.delta)
      for (int i = 32 * t; i < d.npx * R; i += 32 * T) {
        prefetch_l2(P.delta + d.field + i);
        prefetch_l2(P.eta + d.field + i);
      }
  };
  uint32_t parity = 0;  // bit b: parity of stage buffer b's next phase
  StatPair cur{0, 0, 0, 0, false, 0.f, 0.f};
  if (u_first < uend) {
    cur = describe(u_first);
    if (STAGED) stage(cur, 0);
  }
  team_sync<T>(team);

  for (int64_t u = u_first; u < uend; ++u) {
    const int b = STAGED ? static_cast<int>((u - u_first) & 1) : 0;
    StatPair nxt = cur;
    if (u + 1 < uend) {
      nxt = describe(u + 1);
      if (STAGED) stage(nxt, b ^ 1); else prefetch(nxt);
    }
    const int npair = cur.npx, jb0 = cur.jb;
    // z bins of the two segments' first pixels and of the full segments,
    // requested before the wait for the staged fields
    int z0[2] = {0, 0}, za = -1, zb = -1;
    if (cur.ok) {
      z0[0] = __ldg(P.zbin + jb0);
      if (npair > N) z0[1] = __ldg(P.zbin + jb0 + N * R);
      if (npair >= N) za = __ldg(P.segzbin + jb0);
      if (npair == 2 * N) zb = __ldg(P.segzbin + jb0 + N * R);
    }
    const int shift = static_cast<int>(cur.field & 3);
    if constexpr (STAGED) {
      // this pair's copies are in; its last floats join them from registers
      const long long limit = P.wait_test ? (1LL << 20) : (1LL << 31);  // cycles: ~0.5 ms, ~1 s
      const bool arrived = mbar_wait(bars + b, (parity >> b) & 1u, limit);
      parity ^= 1u << b;
      if (!team_all<T>(team, arrived)) {  // (team-uniform) the copies never completed
        if (t == 0) raise_error(P.err, ERR_TIMEOUT);
        if (u + 1 < uend) mbar_wait(bars + (b ^ 1), (parity >> (b ^ 1)) & 1u, limit);  // before leaving
        break;
      }
      const int nfl = (shift + npair) & ~3;
      if (t < shift + npair - nfl) {
        stage_buf[2 * b * STAGE + nfl + t] = cur.td;
        stage_buf[(2 * b + 1) * STAGE + nfl + t] = cur.te;
      }
      team_sync<T>(team);
    }
    if (!cur.ok) {  // (team-uniform: the whole team skips the pair)
      if (t == 0) raise_error(P.err, ERR_RANGE);
      team_sync<T>(team);
      cur = nxt;
      continue;
    }
    const float *sd = stage_buf + 2 * b * STAGE + shift + t, *se = sd + STAGE;
    float2 *buf = reinterpret_cast<float2 *>(stage_buf + (STAGED ? 2 * b * STAGE : 0));
    float2 v[8];  // the two segments' flux
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = make_float2(0.f, 0.f);
    // one segment a pass, with the transform's parts swapped after each (one copy of the code)
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int npx = min(N, npair - h * N), rem = npx - t;  // pixels t + T q of the segment exist for T q < rem
      float f8[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) f8[q] = 0.f;
      if (npx > 0) {
        const int jb = jb0 + h * N * R;
        float2 x8[8];
        if (STAGED || P.pixtab) {  // FGPA of the fields (pixels past the end: masked; the table has entries for them)
          float4 tb[8];
          const float4 *tp = P.pixtab + jb + t;
#pragma unroll
          for (int q = 0; q < 8; ++q) tb[q] = __ldg(tp + T * q);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const bool on = T * q < rem;
            if constexpr (STAGED) {
              x8[q] = on ? make_float2(sd[h * N + T * q], se[h * N + T * q]) : make_float2(0.f, 0.f);
            } else {
              const int64_t i = cur.field + h * N + t + T * q;
              x8[q] = on ? make_float2(__ldg(P.delta + i), __ldg(P.eta + i)) : make_float2(0.f, 0.f);
            }
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) f8[q] = T * q < rem ? fgpa(tb[q], x8[q].x, x8[q].y) : 0.f;
        } else if constexpr (!STAGED) {  // stored flux, and the mean of its fine pixels' fields
          const float *fp = P.flux + cur.flux + h * N + t;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            f8[q] = T * q < rem ? __ldg(fp + T * q) : 0.f;
            x8[q] = make_float2(0.f, 0.f);
          }
          if (P.delta) {
            const int64_t i = cur.field + static_cast<int64_t>(h * N + t) * R;
            const float *dp = P.delta + i, *ep = P.eta + i;
#pragma unroll 2
            for (int r = 0; r < R; ++r) {
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                if (T * q < rem) {
                  x8[q].x += __ldg(dp + T * q * R + r);
                  x8[q].y += __ldg(ep + T * q * R + r);
                }
              }
            }
            if (R > 1) {
              const float fr = static_cast<float>(R);
#pragma unroll
              for (int q = 0; q < 8; ++q) x8[q] = make_float2(x8[q].x / fr, x8[q].y / fr);
            }
          }
        }
        // pixel sums
        if (z0[0] != zc || (h == 0 && u % kRunPairs == 0)) {
          if (zc != -2) flush_bin_sums<true>(W, P.n_z, zc, acc, lane);
          acc.zero();
          zc = z0[0];
        }
        auto bin_stop = [&]() -> int {  // segment pixel where bin zc ends
          const int d = bin_end[zc + 1] - jb;
          return R == 1 ? d : (d + R - 1) / R;
        };
        int pend = bin_stop(), done = 0;
        const int whi = min(T * 7 + wlo0 + 32, npx);  // end of this warp's pixels
        if (whi <= pend) {  // (F and the fields of pixels past the end are 0)
#pragma unroll
          for (int q = 0; q < 8; ++q) acc.add_sums(f8[q], x8[q]);
          acc.n += static_cast<float>(max(0, min(8, (rem + T - 1) / T)));
        } else {  // bin after bin (one copy of the flush: unrolled over the pixels it was 900 instructions more)
#pragma unroll 1
          for (;;) {
            const int stop = min(pend, npx) - t;
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (T * q >= done - t && T * q < stop) acc.add(f8[q], x8[q]);
            if (whi <= pend) break;
            flush_bin_sums<true>(W, P.n_z, zc, acc, lane);
            acc.zero();
            ++zc;
            done = pend;
            pend = bin_stop();
          }
        }
      }
      z0[0] = z0[1];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = make_float2(v[q].y, f8[q]);
    }
    // ---- P1D of the full segments
    // a barrier on both ways: every field value is read before the transform overwrites the buffer
    if (!(counted(za, P.n_z) || counted(zb, P.n_z))) {
      team_sync<T>(team);
    } else {
      part_segments<T>(v, za, zb, P.n_z, buf, factors, t, team);
      pair_fft<N>(buf, v, tws, P.tw, t, team);
      float ka[4], kb[4];
      pair_powers<N>(buf, v, t, team, ka, kb);
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (counted(za, P.n_z)) {
          const int z = za & ~kPartFlag;
          const float up = za == z ? 1.f : __uint_as_float(h ? factors->y : factors->x);
          accumulate_p1d(W, P.n_k, t, ka, 0.25f * P.p1d_scale * up * up, z);
          if (t == 0) W.nseg[z] += 1u;
        }
        za = zb;
#pragma unroll
        for (int j = 0; j < 4; ++j) ka[j] = kb[j];
      }
      if (T > 32 && (zb & kPartFlag)) team_sync<T>(team);  // *factors is read
    }
    cur = nxt;
  }
  if (zc != -2) flush_bin_sums<true>(W, P.n_z, zc, acc, lane);
  flush_partials<N>(smem, teams, P.n_z, P.n_k, P.partials);
}

}  // namespace mk
