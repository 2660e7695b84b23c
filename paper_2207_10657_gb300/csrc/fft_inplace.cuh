// In-place mixed-radix FFT of lines held in shared memory, lengths and
// radices known at run time: the engine of the generic passes (FP64 fields,
// lengths without compiled passes, the batched solver, Kuhn tetrahedra).
// Products, with the self-sorting form it replaced -> with it and with what the
// passes gained since (tables of the x tiles, padded rows, chained launches):
// FP32 160x120x90 638 -> 187 us; FP64 128^3 2981 -> 1865 us; Kuhn tetrahedra
// 64^3 380 -> 176 us.  By itself it took them to 222, 1958 and 227 us.
//
// A line of n = r_0 r_1 ... r_{S-1} elements is a mixed-radix number: element
// x = d_0 m_0 + d_1 m_1 + ... with m_s = n / (r_0 ... r_s).  Stage s replaces
// digit d_s by its r_s-point DFT, in place: a butterfly reads and writes the
// same r_s elements, so one thread holds one butterfly at a time, a stage
// needs one barrier, and no second buffer.  A stage's radix is 2, 3, 4, 5, 8
// or a pair of those up to 20, taken in registers as two successive steps:
// most lengths up to 300 need two stages, i.e. two trips through shared
// memory.  (The self-sorting form this
// replaces permutes in every stage: all of a block's butterflies had to sit
// in registers between two barriers, 16-24 complex values a thread, spilled
// to local memory at the six blocks per SM the x and y passes ran with.)
// Two flows use it:
//
//  * DIT: input in natural order, stages 0 .. S-1, twiddles before each DFT;
//    the output frequency k = q_0 + r_0 q_1 + r_0 r_1 q_2 + ... sits at the
//    position of digits (q_0, q_1, ...).  Index arithmetic at the load or
//    store undoes the digit reversal.
//  * its transpose: input at those digit-reversed positions, stages S-1 ..
//    0, output in natural order.  A DIT transform followed by a transposed
//    inverse needs no reordering in between.
//
// Shared-memory address of digit d_0 and remainder e (e < m_0) of column t
// in line group c: (c LP + d_0 m0p + e) TX + t, where the pitch m0p is m_0
// rounded up to an odd number: stages after the first walk d_0 fastest, and
// an odd pitch spreads those accesses over the banks.
#pragma once

#include "common.cuh"

namespace rve {

// ------------------------------------------------------------- plans
// Division of a < 2^20 by a constant d <= 1024: one multiply-high.
struct FastDiv {
  unsigned mul;  // ceil(2^32 / d); 0: d = 1
  __host__ static FastDiv by(int d) { return {d <= 1 ? 0u : (unsigned)((0x100000000ull + d - 1) / d)}; }
  __device__ __forceinline__ int div(int a) const { return mul ? (int)__umulhi((unsigned)a, mul) : a; }
};

constexpr int kMaxStages = 7;

struct AxisPlan {
  int n, ns;
  int r[kMaxStages];           // radices
  int m[kMaxStages];           // digit strides: n / (r_0 ... r_s)
  int span[kMaxStages];        // r_0 ... r_{s-1}
  int m0p;                     // pitch of digit 0 (m_0 rounded up to odd)
  int lp;                      // elements of a padded line: r_0 m0p
  FastDiv dr[kMaxStages], dm[kMaxStages];
  int nw[kMaxStages];          // m_0 / r_s (s >= 1)
  FastDiv dw[kMaxStages];      // by nw
  FastDiv dn, dh;              // by n, by n/2 + 1
  FastDiv dc;                  // by the lines per voxel (the x axis)
  int keep_order;              // the inverse of a z pass keeps the forward's radix sequence (see zproj_body)

  // address of element x of a natural-order line
  __device__ __forceinline__ int at_natural(int x) const {
    const int d0 = dm[0].div(x);
    return d0 * m0p + (x - d0 * m[0]);
  }
  // address of frequency k after a DIT transform
  __device__ __forceinline__ int at_freq(int k) const {
    int q = dr[0].div(k);
    int a = (k - q * r[0]) * m0p;
    for (int s = 1; s < ns; ++s) {
      const int q2 = dr[s].div(q);
      a += (q - q2 * r[s]) * m[s];
      q = q2;
    }
    return a;
  }
  // frequency at digit-0 value q0 and remainder e after a DIT transform
  __device__ __forceinline__ int freq_of(int q0, int e) const {
    int k = q0;
    for (int s = 1; s < ns; ++s) {
      const int q = dm[s].div(e);
      e -= q * m[s];
      k += q * span[s];
    }
    return k;
  }
};

// A tile of lines: ng line groups of tx columns (tx a power of two; 1 for
// tiles of whole rows) at buf[(c lp + position) tx + t].
struct TileShape {
  int ng, tx, ltx;  // groups, columns, log2(columns)
};

// ------------------------------------------------------------- stages
// One stage of radix RA * RB.  TR = false: DIT; TR = true: the transposed
// flow.  S0: stage 0.  GIN: the inputs come from load(c, x, t), x in natural
// order (a DIT stage 0 only).  GOUT: the outputs go to store(c, k, t, v), k
// the frequency (a last DIT stage) or the natural index (TR, stage 0).
// Consecutive threads take consecutive columns, then (stage 0) consecutive
// elements or (later stages) consecutive values of digit 0: outputs that
// leave the tile are consecutive in both flows.
//
// Called, not inlined: a kernel holds a dozen radices, and inlined together
// they spill.  The plan's numbers come as scalars, in registers.
//  total: butterflies of the tile; m0, m0p, lp: AxisPlan; m: digit stride of
//  the stage; d0: by m_0 (stage 0) or r_0; nw, dw; dm: by m; span.
template <int RA, int RB, bool INV, bool TR, bool S0, bool GIN, bool GOUT, typename C, typename LoadF, typename StoreF>
__device__ __noinline__ void tile_stage(C* buf, const C* __restrict__ tw, const int total, const int ltx, const int lp,
                                        const int m0, const int m0p, const FastDiv d0, const int r0, const int nw,
                                        const FastDiv dw, const int m, const FastDiv dm, const int span, const int s,
                                        const AxisPlan* plan, LoadF load, StoreF store) {
  constexpr int R = RA * RB;
  // butterflies in flight per thread: small radices take several, so that
  // enough loads stay outstanding
  constexpr int U = R >= 8 ? 1 : (R >= 4 ? 2 : 4);
  const int ms = S0 ? m0p : m;  // distance of a butterfly's elements
  const int stride = blockDim.x, tmask = (1 << ltx) - 1;
  for (int u0 = threadIdx.x; u0 < total; u0 += U * stride) {
    C v[U][R];
    int base[U], kp[U], cc[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int u = u0 + i * stride;
      if (U > 1 && u >= total) continue;
      const int t = u & tmask, b0 = u >> ltx;
      int pos, lo;
      if (S0) {
        cc[i] = d0.div(b0);
        lo = b0 - cc[i] * m0;
        pos = lo;
        kp[i] = TR ? lo : 0;
      } else {
        // b0 = (c, w, q0): q0 fastest, w = the other digits in position order
        const int x = d0.div(b0), q0 = b0 - x * r0;
        cc[i] = dw.div(x);
        const int w = x - cc[i] * nw;
        const int hi = dm.div(w);  // digits q_1 .. q_{s-1}, the last least significant
        lo = w - hi * m;
        pos = q0 * m0p + hi * m * R + lo;
        if (TR) {
          kp[i] = lo;
        } else {
          int k = q0;
          if (s == 2) {
            k += hi * r0;
          } else if (s > 2) {
            int f = hi * m * R;
            for (int j = 1; j < s; ++j) {
              const int q = plan->dm[j].div(f);
              f -= q * plan->m[j];
              k += q * plan->span[j];
            }
          }
          kp[i] = k;
        }
      }
      base[i] = ((cc[i] * lp + pos) << ltx) + t;
      if constexpr (GIN) {
#pragma unroll
        for (int a = 0; a < R; ++a) v[i][a] = load(cc[i], lo + a * m0, t);
      } else {
#pragma unroll
        for (int a = 0; a < R; ++a) v[i][a] = buf[base[i] + ((a * ms) << ltx)];
      }
    }
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int u = u0 + i * stride;
      if (U > 1 && u >= total) continue;
      C* x = v[i];
      auto turn = [&](C& y, int k) {
        const C w = __ldg(&tw[k]);
        y = INV ? cmulc(y, w) : cmul(y, w);
      };
      C o[R];
      if constexpr (!TR) {
        // element a RB + b -> frequency a + RA b
#pragma unroll
        for (int b = 0; b < RB; ++b) {
          C y[RA];
#pragma unroll
          for (int a = 0; a < RA; ++a) y[a] = x[a * RB + b];
          if (!S0 && kp[i] > 0) {
#pragma unroll
            for (int a = 1; a < RA; ++a) turn(y[a], a * kp[i] * (m * RB));
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
            if (a > 0 || (!S0 && kp[i] > 0)) {
#pragma unroll
              for (int b = 1; b < RB; ++b) turn(y[b], b * (S0 ? a : kp[i] + span * a) * m);
            }
            Dft<RB, INV, C>::run(y);
#pragma unroll
            for (int b = 0; b < RB; ++b) o[a + RA * b] = y[b];
          }
        }
      } else {
        // frequency a + RA b -> element a RB + b
        if constexpr (RB > 1) {
#pragma unroll
          for (int a = 0; a < RA; ++a) {
            C y[RB];
#pragma unroll
            for (int b = 0; b < RB; ++b) y[b] = x[a + RA * b];
            if (kp[i] > 0) {
#pragma unroll
              for (int b = 1; b < RB; ++b) turn(y[b], b * kp[i] * (span * RA));
            }
            Dft<RB, INV, C>::run(y);
#pragma unroll
            for (int b = 0; b < RB; ++b) o[a * RB + b] = y[b];
          }
#pragma unroll
          for (int a = 0; a < R; ++a) x[a] = o[a];
        }
#pragma unroll
        for (int b = 0; b < RB; ++b) {
          C y[RA];
          const int k = kp[i] + (S0 ? m0 : m) * b;
#pragma unroll
          for (int a = 0; a < RA; ++a) y[a] = x[a * RB + b];
          if (b > 0 || k > 0) {
#pragma unroll
            for (int a = 1; a < RA; ++a) turn(y[a], a * k * span);
          }
          Dft<RA, INV, C>::run(y);
#pragma unroll
          for (int a = 0; a < RA; ++a) x[a * RB + b] = y[a];
        }
      }
      if constexpr (TR || RB == 1) {
#pragma unroll
        for (int a = 0; a < R; ++a) o[a] = x[a];
      }
      if constexpr (GOUT) {
        // element step of the outputs: m_0 (TR), the span of a last DIT stage
        const int step = TR ? m0 : span;
#pragma unroll
        for (int a = 0; a < R; ++a) store(cc[i], kp[i] + a * step, u & tmask, o[a]);
      } else {
#pragma unroll
        for (int a = 0; a < R; ++a) buf[base[i] + ((a * ms) << ltx)] = o[a];
      }
    }
  }
}

struct NoIo {
  template <typename... A> __device__ __forceinline__ int operator()(A...) const { return 0; }
};

template <bool INV, bool TR, bool S0, bool GIN, bool GOUT, typename C, typename LoadF, typename StoreF>
__device__ __forceinline__ void tile_stage_any(C* buf, const AxisPlan& p, const int s, const TileShape& ts,
                                               const C* __restrict__ tw, LoadF load, StoreF store) {
  const int r0 = p.r[0], nw = S0 ? 1 : p.nw[s], m = p.m[s];
  const int total = (S0 ? p.m[0] * ts.ng : r0 * nw * ts.ng) << ts.ltx;
  const FastDiv d0 = S0 ? p.dm[0] : p.dr[0];
#define RVE_STAGE(A, B)                                                                                              \
  case A * B:                                                                                                        \
    tile_stage<A, B, INV, TR, S0, GIN, GOUT>(buf, tw, total, ts.ltx, p.lp, p.m[0], p.m0p, d0, r0, nw, p.dw[s], m,   \
                                             p.dm[s], p.span[s], s, &p, load, store);                                \
    break;
  switch (p.r[s]) {
    RVE_STAGE(2, 1) RVE_STAGE(3, 1) RVE_STAGE(4, 1) RVE_STAGE(5, 1) RVE_STAGE(8, 1) RVE_STAGE(2, 3) RVE_STAGE(2, 5)
    RVE_STAGE(3, 3) RVE_STAGE(3, 5) RVE_STAGE(4, 3) RVE_STAGE(4, 4) RVE_STAGE(4, 5)
    default: break;
  }
#undef RVE_STAGE
}

// Whole DIT transform of a tile.  GIN / GOUT: input from load, output to
// store; otherwise in place.  Ends with a barrier unless GOUT.  The caller
// has synchronised after filling buf (GIN: buf is free).
template <bool INV, bool GIN, bool GOUT, typename C, typename LoadF, typename StoreF>
__device__ __forceinline__ void tile_dit(C* buf, const AxisPlan& p, const TileShape& ts, const C* __restrict__ tw,
                                         LoadF load, StoreF store) {
  if constexpr (GOUT) if (p.ns == 1) {
    tile_stage_any<INV, false, true, GIN, GOUT>(buf, p, 0, ts, tw, load, store);
    return;
  }
  tile_stage_any<INV, false, true, GIN, false>(buf, p, 0, ts, tw, load, NoIo{});
  __syncthreads();
  const int last = GOUT ? p.ns - 1 : p.ns;
  for (int s = 1; s < last; ++s) {
    tile_stage_any<INV, false, false, false, false>(buf, p, s, ts, tw, NoIo{}, NoIo{});
    __syncthreads();
  }
  if constexpr (GOUT) tile_stage_any<INV, false, false, false, true>(buf, p, p.ns - 1, ts, tw, NoIo{}, store);
}

// Transposed inverse of a tile from digit-reversed positions, natural-order
// output to store.  No barrier at the end.
template <typename C, typename StoreF>
__device__ __forceinline__ void tile_transposed_inverse(C* buf, const AxisPlan& p, const TileShape& ts,
                                                        const C* __restrict__ tw, StoreF store) {
  for (int s = p.ns - 1; s > 0; --s) {
    tile_stage_any<true, true, false, false, false>(buf, p, s, ts, tw, NoIo{}, NoIo{});
    __syncthreads();
  }
  tile_stage_any<true, true, true, false, true>(buf, p, 0, ts, tw, NoIo{}, store);
}

// ------------------------------------------------------ column tiles
// Tiles of tx consecutive kx columns over `planes` planes of nxh columns.
// The remainder columns of a plane (a half spectrum has n/2 + 1) share tiles
// with those of the next planes, so that no tile is nearly empty.
struct ColTiles {
  int planes, nxh, tx, main, rem, per;  // main: full tiles per plane; per: planes sharing a remainder tile
  __host__ __device__ ColTiles(int planes_, int nxh_, int tx_)
      : planes(planes_), nxh(nxh_), tx(tx_), main(nxh_ / tx_), rem(nxh_ % tx_), per(nxh_ % tx_ ? tx_ / (nxh_ % tx_) : 1) {}
  __host__ __device__ int count() const { return planes * main + (rem ? (planes + per - 1) / per : 0); }
  // plane and column of column t of tile b; false: none
  __device__ __forceinline__ bool at(int b, int t, int* plane, int* kx) const {
    if (b < planes * main) {
      *plane = b / main;
      *kx = (b - *plane * main) * tx + t;
      return true;
    }
    const int g = t / (rem ? rem : 1);
    *plane = (b - planes * main) * per + g;
    *kx = main * tx + (t - g * rem);
    return g < per && *plane < planes;
  }
};

}  // namespace rve
