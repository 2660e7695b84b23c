// Compile-time form of the in-place FFT of fft_inplace.cuh (digit layout, DIT
// flow, paired radices) for 384 points: the index arithmetic of a stage folds
// into immediates.  The radix sequence is that of fft_radix (8, 4, 4, 3), the
// last two taken in registers one after the other.
//
// Tried at 256^3 as well: wider pairs (256 = 8 x 32, two trips through shared
// memory) take 90-128 registers and lose more to the missing warps than they
// save: z pass 420 us against 327 us, y pass 180 us against 150 us; single
// radices 391 and 150 us.
#pragma once

#include "fft_fast.cuh"

namespace rve {

// Stage s of length n: first and second factor (1: none).
template <int N> struct CtPlan;
#define RVE_CT_PLAN(N_, S_, ...)                                             \
  template <> struct CtPlan<N_> {                                            \
    static constexpr int S = S_;                                             \
    static constexpr int f[S_][2] = __VA_ARGS__;                             \
    static constexpr int r(int s) { return f[s][0] * f[s][1]; }              \
    static constexpr int span(int s) { return s == 0 ? 1 : span(s - 1) * r(s - 1); } \
    static constexpr int m(int s) { return N_ / (span(s) * r(s)); }          \
  };
RVE_CT_PLAN(384, 3, {{8, 1}, {4, 1}, {4, 3}})
#undef RVE_CT_PLAN

// Tile of NG line groups of TX columns: address of digit-0 value q0,
// remainder e, column t of group c.  The pitch of digit 0 is odd where a row
// of columns is narrower than the 128 bytes of all banks.
template <int N, int TX> struct CtTile {
  using P = CtPlan<N>;
  static constexpr int M0 = P::m(0);
  static constexpr int M0P = TX >= 16 ? M0 : (M0 | 1);
  static constexpr int LP = P::r(0) * M0P;
  __device__ __forceinline__ static constexpr int at(int c, int q0, int e, int t) { return (c * LP + q0 * M0P + e) * TX + t; }
  __device__ __forceinline__ static int natural(int x) { return (x / M0) * M0P + x % M0; }
  // position of frequency k (S <= 3; the plan's tables are read in constant
  // expressions only: they have no device storage)
  __device__ __forceinline__ static int freq(int k) {
    constexpr int S = P::S, R0 = P::r(0), R1 = P::r(1), M1 = P::m(1);
    const int q0 = k % R0, q = k / R0;
    int a = q0 * M0P + (S > 2 ? q % R1 : q) * M1;
    if constexpr (S > 2) {
      static_assert(S == 3, "three stages at most");
      a += q / R1;
    }
    return a;
  }
};

// DIT stage SI of a tile (tile_stage of fft_inplace.cuh); NT threads.
template <int N, int TX, int NG, int NT, bool INV, int SI, bool GIN, bool GOUT, typename C, typename LoadF,
          typename StoreF>
__device__ __forceinline__ void ct_stage(C* buf, const C* __restrict__ tw, LoadF load, StoreF store) {
  using P = CtPlan<N>;
  using T = CtTile<N, TX>;
  constexpr int RA = P::f[SI][0], RB = P::f[SI][1], R = RA * RB;
  constexpr int M = P::m(SI), SPAN = P::span(SI), R0 = P::r(0), M0 = T::M0;
  constexpr int NB = N / R;                       // butterflies per line
  constexpr int TOTAL = NB * NG * TX;
  constexpr int PER = (TOTAL + NT - 1) / NT;
  constexpr int MS = SI == 0 ? T::M0P : M;
  // butterflies whose inputs are loaded together: a thread's stores to shared
  // memory hold back its later loads, so the global loads of a batch go first
  constexpr int UB = GIN && PER * R <= 24 ? PER : (GIN && 24 / R > 0 ? 24 / R : 1);
  auto turn = [&](C& y, int k) {
    const C w = __ldg(&tw[k]);
    y = INV ? cmulc(y, w) : cmul(y, w);
  };
#pragma unroll
  for (int i0 = 0; i0 < PER; i0 += UB) {
    C xs[UB][R];
    int pos[UB], kps[UB], cs[UB];
#pragma unroll
    for (int i = 0; i < UB; ++i) {
      const int u = threadIdx.x + (i0 + i) * NT;
      if (i0 + i >= PER || (TOTAL % NT != 0 && u >= TOTAL)) continue;
      const int t = u % TX, b0 = u / TX;
      int lo;
      kps[i] = 0;
      if constexpr (SI == 0) {
        cs[i] = b0 / M0;
        lo = b0 - cs[i] * M0;
        pos[i] = lo;
      } else {
        constexpr int NW = M0 / R;
        const int x = b0 / R0, q0 = b0 - x * R0;
        cs[i] = x / NW;
        const int w = x - cs[i] * NW;
        const int hi = w / M;
        lo = w - hi * M;
        pos[i] = q0 * T::M0P + hi * M * R + lo;
        kps[i] = q0 + (SI == 2 ? hi * R0 : 0);
        static_assert(SI <= 2, "frequency of the done digits");
      }
      pos[i] = (cs[i] * T::LP + pos[i]) * TX + t;
#pragma unroll
      for (int a = 0; a < R; ++a) {
        if constexpr (GIN) xs[i][a] = load(cs[i], lo + a * M0, t);
        else xs[i][a] = buf[pos[i] + a * MS * TX];
      }
    }
#pragma unroll
    for (int i = 0; i < UB; ++i) {
      const int u = threadIdx.x + (i0 + i) * NT;
      if (i0 + i >= PER || (TOTAL % NT != 0 && u >= TOTAL)) continue;
      C* x = xs[i];
      const int kp = kps[i];
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        C y[RA];
#pragma unroll
        for (int a = 0; a < RA; ++a) y[a] = x[a * RB + b];
        if constexpr (SI > 0) {
#pragma unroll
          for (int a = 1; a < RA; ++a) turn(y[a], a * kp * (M * RB));
        }
        Dft<RA, INV, C>::run(y);
#pragma unroll
        for (int a = 0; a < RA; ++a) x[a * RB + b] = y[a];
      }
      if constexpr (RB > 1) {
#pragma unroll
        for (int a = 0; a < RA; ++a) {
          C y[RB];
#pragma unroll
          for (int b = 0; b < RB; ++b) y[b] = x[a * RB + b];
#pragma unroll
          for (int b = 1; b < RB; ++b) turn(y[b], b * (kp + SPAN * a) * M);
          Dft<RB, INV, C>::run(y);
#pragma unroll
          for (int b = 0; b < RB; ++b) x[a * RB + b] = y[b];
        }
      }
      // x[a RB + b] holds frequency a + RA b of the stage
#pragma unroll
      for (int b = 0; b < RB; ++b)
#pragma unroll
        for (int a = 0; a < RA; ++a) {
          if constexpr (GOUT) store(cs[i], kp + (a + RA * b) * SPAN, u % TX, x[a * RB + b]);
          else buf[pos[i] + (a + RA * b) * MS * TX] = x[a * RB + b];
        }
    }
  }
}

// Whole transform; barriers between the stages, none after the last.
template <int N, int TX, int NG, int NT, bool INV, bool GIN, bool GOUT, int SI = 0, typename C, typename LoadF,
          typename StoreF>
__device__ __forceinline__ void ct_dit(C* buf, const C* __restrict__ tw, LoadF load, StoreF store) {
  constexpr int S = CtPlan<N>::S;
  ct_stage<N, TX, NG, NT, INV, SI, GIN && SI == 0, GOUT && SI == S - 1>(buf, tw, load, store);
  if constexpr (SI + 1 < S) {
    __syncthreads();
    ct_dit<N, TX, NG, NT, INV, GIN, GOUT, SI + 1>(buf, tw, load, store);
  }
}

}  // namespace rve
