// Generic (runtime-length) spectral pass bodies and their single-grid
// kernels.  A body processes one tile of one grid; the kernels call it with
// their block index, batched kernels with an index taken from a work list.
#pragma once

#include "fft_inplace.cuh"
#include "hv_passes.cuh"
#include "launch.cuh"
#include "project.cuh"

namespace rve {

constexpr int kSmemCap = 112 * 1024;  // dynamic shared memory cap per block: two blocks fit an SM
constexpr int kGT = 128;                  // threads of the x, y and 2D passes
constexpr int kGZ = 256;              // threads of the z pass
constexpr int kHold = 4, kHold2 = 8;  // frequencies a z-pass / 2D y-pass thread holds while its tile is reordered

// One butterfly per thread in registers (radix <= 20: 40 reals) leaves no
// reason to cap the registers hard: 24 resident warps of FP32 at 80 registers
// and 16 of FP64 at 128 (whose passes are bound by the FP64 pipe, 2 lanes per
// SM and clock, not by latency) are asked for.
template <typename R> constexpr int xy_blocks() { return sizeof(R) == 4 ? 6 : 4; }
template <typename R> constexpr int z_blocks() { return sizeof(R) == 4 ? 3 : 2; }

// ------------------------------------------------------------ x tiles
// Tables of an x tile behind its lines in shared memory: the grid row
// (component and voxel row) of every real row of the tile, and the address of
// every frequency of a transformed line.  Formed once per tile; without them
// the x passes spend two thirds of their instructions on row / component
// splits and digit reversals (product at 160x120x90 222 -> 199 us, Kuhn
// tetrahedra at 64^3 220 -> 184 us).
struct XTables {
  int* row;            // [2 npair]: c nrows + voxel row; -1: none
  unsigned short* at;  // [nx]: address of frequency k after a DIT transform
  static __host__ __device__ size_t bytes(int npair, int nx) { return (size_t)npair * 8 + (size_t)nx * 2; }

  template <typename C>
  __device__ __forceinline__ XTables(C* buf, const GridDesc& g, const AxisPlan& px, int Q, int npair,
                                     long long row0, bool freq) {
    row = reinterpret_cast<int*>(buf + npair * px.lp);
    at = reinterpret_cast<unsigned short*>(row + 2 * npair);
    for (int r = threadIdx.x; r < 2 * npair; r += blockDim.x) {
      const int q = px.dc.div(r);
      row[r] = q < Q && row0 + q < g.nrows ? (int)((r - q * g.ncomp) * g.nrows + row0 + q) : -1;
    }
    if (freq)
      for (int k = threadIdx.x; k < g.nx; k += blockDim.x) at[k] = (unsigned short)px.at_freq(k);
  }
};

// ------------------------------------------------------------ x forward
// Q voxel rows per block, all ncomp components of each row.  MODE 0: plain;
// 1: the damaged isotropic tangent (1-D)(lambda tr(v) 1 + 2 mu v) applied on
// load (Eq. (13), secant reading); 2: with the rank-one part of the symmetric
// consistent tangent (`ct`).  NC: components per voxel, 0 for Kuhn simplices.
// Real rows are packed in pairs into one complex FFT (real + i*imag) and
// separated with the Hermitian symmetry of real-input spectra.
template <typename R, int MODE, int NC>
__device__ __forceinline__ void xfwd_load(Cx<R>* buf, const R* __restrict__ in, const uint8_t* __restrict__ phase,
                                          const R* __restrict__ dmg, const MatTable<R>& mt, const GridDesc& g,
                                          const int Q, const AxisPlan& px, const long long row0,
                                          const ConsTan<R>& ct) {
  const int nx = g.nx, lp = px.lp;
  const int left = (int)(g.nrows - row0 < Q ? g.nrows - row0 : Q);  // rows of the tile that exist
  for (int idx = threadIdx.x; idx < Q * nx; idx += blockDim.x) {
    const int q = px.dn.div(idx), x = idx - q * nx;
    const long long vox = row0 * nx + idx;
    // line (rho >> 1) of row rho = q ncomp + c, element x
    R* slot = reinterpret_cast<R*>(buf + px.at_natural(x));
    if constexpr (NC == 0) {
      // line c * nq + p is Mandel component c of simplex p, whose damage is
      // dmg[p * nvox + vox]; the tangent acts per simplex
      const int nqp = g.nq, nd = g.ndim, nm = nd == 3 ? 6 : 3;
      for (int p = 0; p < nqp; ++p) {
        R m[6] = {0, 0, 0, 0, 0, 0};
        if (q < left) {
#pragma unroll
          for (int c = 0; c < 6; ++c)
            if (c < nm) m[c] = in[(c * nqp + p) * g.nvox + vox];
          if (MODE >= 1) {
            const int ph = phase[vox];
            const R keep = (R)1 - dmg[p * g.nvox + vox];
            const R lam = mt.lam[ph] * keep, two_mu = (R)2 * mt.mu[ph] * keep;
            R tr = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i)
              if (i < nd) tr += m[i];
#pragma unroll
            for (int c = 0; c < 6; ++c) m[c] = two_mu * m[c] + (c < nd ? lam * tr : (R)0);
          }
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          if (c < nm) {
            const int rho = q * g.ncomp + c * nqp + p;
            slot[2 * (rho >> 1) * lp + (rho & 1)] = m[c];
          }
        }
      }
    } else {
      constexpr int ND = NC == 6 ? 3 : 2;
      R val[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) val[c] = q < left ? in[c * g.nvox + vox] : (R)0;
      if (MODE >= 1 && q < left) {
        const int ph = phase[vox];
        const R keep = (R)1 - dmg[vox];
        const R lam = mt.lam[ph] * keep, two_mu = (R)2 * mt.mu[ph] * keep;
        R tr = 0;
#pragma unroll
        for (int i = 0; i < ND; ++i) tr += val[i];
        const R ltr = mul_rn(lam, tr);  // rounded by itself, whichever product the compiler would contract
        const R hdp = MODE == 2 ? (R)0.5 * ct.dp[vox] : (R)0;
        R nv = 0, av = 0;
        if (MODE == 2 && hdp != (R)0) {
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            nv += ct.n[c * g.nvox + vox] * val[c];
            av += ct.a[c * g.nvox + vox] * val[c];
          }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          val[c] = c < ND ? fma_rn(two_mu, val[c], ltr) : two_mu * val[c];
          if (MODE == 2 && hdp != (R)0) val[c] -= hdp * (ct.a[c * g.nvox + vox] * nv + ct.n[c * g.nvox + vox] * av);
        }
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int rho = q * NC + c;
        slot[2 * (rho >> 1) * lp + (rho & 1)] = val[c];
      }
    }
  }
}

template <typename R, int MODE>
__device__ __forceinline__ void xfwd_body(const R* __restrict__ in, const uint8_t* __restrict__ phase,
                                          const R* __restrict__ dmg, const MatTable<R>& mt,
                                          Cx<R>* __restrict__ spec, const GridDesc& g, const int Q,
                                          const AxisPlan& px, const Cx<R>* __restrict__ tw, const int bx,
                                          const ConsTan<R> ct = ConsTan<R>{}) {
  using C = Cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  const long long row0 = (long long)bx * Q;
  const int npair = (g.ncomp * Q) >> 1, nx = g.nx, nxh = g.nxh, nxs = g.nxs, lp = px.lp;
  const XTables tab(buf, g, px, Q, npair, row0, true);
  if (g.nq > 1) xfwd_load<R, MODE, 0>(buf, in, phase, dmg, mt, g, Q, px, row0, ct);
  else if (g.ndim == 3) xfwd_load<R, MODE, 6>(buf, in, phase, dmg, mt, g, Q, px, row0, ct);
  else xfwd_load<R, MODE, 3>(buf, in, phase, dmg, mt, g, Q, px, row0, ct);
  __syncthreads();
  tile_dit<false, false, false>(buf, px, TileShape{npair, 1, 0}, tw, NoIo{}, NoIo{});
  for (int idx = threadIdx.x; idx < npair * nxh; idx += blockDim.x) {
    const int p = px.dh.div(idx), k = idx - p * nxh;
    const C* line = buf + p * lp;
    const C zk = line[tab.at[k]], zm = line[tab.at[k == 0 ? 0 : nx - k]];
    const int ra = tab.row[2 * p], rb = tab.row[2 * p + 1];
    if (ra >= 0) spec[(long long)ra * nxs + k] = C{(zk.x + zm.x) * (R)0.5, (zk.y - zm.y) * (R)0.5};
    if (rb >= 0) spec[(long long)rb * nxs + k] = C{(zk.y + zm.y) * (R)0.5, (zm.x - zk.x) * (R)0.5};
  }
}

template <typename R, int MODE>
__global__ void __launch_bounds__(kGT, xy_blocks<R>())
    k_xfwd(const R* __restrict__ in, const uint8_t* __restrict__ phase, const R* __restrict__ dmg,
           const MatTable<R> mt, Cx<R>* __restrict__ spec, const GridDesc g, const int Q,
           const __grid_constant__ AxisPlan px, const Cx<R>* __restrict__ tw, const ConsTan<R> ct) {
  chain_begin();
  xfwd_body<R, MODE>(in, phase, dmg, mt, spec, g, Q, px, tw, blockIdx.x, ct);
}

// ------------------------------------------------------------ y columns
// One tile of TX kx columns of the planes (component, z), transformed in
// global memory.
template <typename R, bool INV>
__device__ __forceinline__ void ycols_body(Cx<R>* __restrict__ spec, const GridDesc& g, const int ltx,
                                           const AxisPlan& py, const Cx<R>* __restrict__ tw, const int b) {
  using C = Cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  const int tx = 1 << ltx, nxs = g.nxs;
  // the threads are a multiple of the columns: a thread keeps one column
  int plane, kx;
  const bool ok = ColTiles(g.ncomp * g.nz, g.nxh, tx).at(b, threadIdx.x & (tx - 1), &plane, &kx);
  C* col = spec + (long long)plane * g.ny * nxs + kx;
  auto load = [=](int, int y, int) -> C { return ok ? col[(long long)y * nxs] : C{0, 0}; };
  auto store = [=](int, int y, int, C v) {
    if (ok) col[(long long)y * nxs] = v;
  };
  tile_dit<INV, true, true>(buf, py, TileShape{1, tx, ltx}, tw, load, store);
}

template <typename R, bool INV>
__global__ void __launch_bounds__(kGT, xy_blocks<R>())
    k_ycols(Cx<R>* __restrict__ spec, const GridDesc g, const int ltx, const __grid_constant__ AxisPlan py,
            const Cx<R>* __restrict__ tw) {
  chain_begin();
  ycols_body<R, INV>(spec, g, ltx, py, tw, blockIdx.x);
}

// ------------------------------------------------- z + projection (3D)
// One tile of kx columns at ky, all components: z transform, projection,
// inverse z transform.
//
// pz.keep_order (FP32 cells of one element per voxel): the inverse runs the
// forward's radix sequence from natural order, so that every value is formed
// by the same operations in the same order as in earlier releases of this
// pass (an FP32 load path follows its roundings).  The tile is reordered
// through registers with the projection (kHold frequencies per thread).
// Otherwise the inverse is the transposed flow and nothing is reordered.
template <typename R>
__device__ __forceinline__ void zproj_body(Cx<R>* __restrict__ spec, const GridDesc& g, const int ltx,
                                           const AxisPlan& pz, const Cx<R>* __restrict__ tw, const AxisSyms<R>& sy,
                                           const unsigned free_mask, const int b) {
  using C = Cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  const int nz = g.nz, ny = g.ny, nxs = g.nxs, tx = 1 << ltx;
  const int ncl = g.ncomp;  // lines per column: 6, or 36 for Kuhn tetrahedra
  const int t = threadIdx.x & (tx - 1);
  int ky, kx;
  const bool ok = ColTiles(ny, g.nxh, tx).at(b, t, &ky, &kx);
  const long long zs = (long long)ny * nxs;
  C* col = spec + (long long)ky * nxs + kx;
  auto load = [=](int c, int z, int) -> C { return ok ? col[(c * nz + z) * zs] : C{0, 0}; };
  auto store = [=](int c, int z, int, C v) {
    if (ok) col[(c * nz + z) * zs] = v;
  };
  const TileShape ts{ncl, tx, ltx};
  tile_dit<false, true, false>(buf, pz, ts, tw, load, NoIo{});
  const bool kxy0 = kx == 0 && ky == 0;
  const int lp = pz.lp << ltx;
  if (ncl == 36) {
    if (ok) {
      for (int i = threadIdx.x >> ltx; i < nz; i += blockDim.x >> ltx) {
        const int e = pz.dr[0].div(i), q0 = i - e * pz.r[0], z = pz.freq_of(q0, e);
        const C d[3] = {sy.d[0][kx], sy.d[1][ky], sy.d[2][z]};
        const C ex[3] = {C{(R)1 + d[0].x, d[0].y}, C{(R)1 + d[1].x, d[1].y}, C{(R)1 + d[2].x, d[2].y}};
        project_simplex3<R>(buf + ((q0 * pz.m0p + e) << ltx) + t, lp, ex, d, kxy0 && z == 0, free_mask);
      }
    }
    __syncthreads();
    tile_transposed_inverse(buf, pz, ts, tw, store);
    return;
  }
  const ColSym3<R> cs = ok ? ColSym3<R>(sy, kx, ky) : ColSym3<R>();
  if (!pz.keep_order) {
    if (ok) {
      for (int i = threadIdx.x >> ltx; i < nz; i += blockDim.x >> ltx) {
        const int e = pz.dr[0].div(i), q0 = i - e * pz.r[0], z = pz.freq_of(q0, e);
        C* at = buf + ((q0 * pz.m0p + e) << ltx) + t;
        C m[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) m[c] = at[c * lp];
        cs.project(m, sy, z, kxy0 && z == 0, free_mask);
#pragma unroll
        for (int c = 0; c < 6; ++c) at[c * lp] = m[c];
      }
    }
    __syncthreads();
    tile_transposed_inverse(buf, pz, ts, tw, store);
    return;
  }
  if constexpr (sizeof(R) == 4) {
    C m[kHold][6];
#pragma unroll
    for (int h = 0; h < kHold; ++h) {
      const int z = (threadIdx.x >> ltx) + h * (blockDim.x >> ltx);
      if (ok && z < nz) {
        const C* at = buf + (pz.at_freq(z) << ltx) + t;
#pragma unroll
        for (int c = 0; c < 6; ++c) m[h][c] = at[c * lp];
        cs.project(m[h], sy, z, kxy0 && z == 0, free_mask);
      }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < kHold; ++h) {
      const int z = (threadIdx.x >> ltx) + h * (blockDim.x >> ltx);
      if (ok && z < nz) {
        C* at = buf + (pz.at_natural(z) << ltx) + t;
#pragma unroll
        for (int c = 0; c < 6; ++c) at[c * lp] = m[h][c];
      }
    }
    __syncthreads();
    tile_dit<true, false, true>(buf, pz, ts, tw, NoIo{}, store);
  }
}

template <typename R>
__global__ void __launch_bounds__(kGZ, z_blocks<R>())
    k_zproj(Cx<R>* __restrict__ spec, const GridDesc g, const int ltx, const __grid_constant__ AxisPlan pz,
            const Cx<R>* __restrict__ tw, const AxisSyms<R> sy, const unsigned free_mask) {
  chain_begin();
  zproj_body<R>(spec, g, ltx, pz, tw, sy, free_mask, blockIdx.x);
}

// ------------------------------------------------- y + projection (2D)
template <typename R>
__device__ __forceinline__ void yproj2d_body(Cx<R>* __restrict__ spec, const GridDesc& g, const int ltx,
                                             const AxisPlan& py, const Cx<R>* __restrict__ tw,
                                             const AxisSyms<R>& sy, const unsigned free_mask, const int b) {
  using C = Cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  const int ny = g.ny, nxs = g.nxs, ncl = g.ncomp, tx = 1 << ltx;  // 3 lines per column, or 6 (Kuhn triangles)
  const int t = threadIdx.x & (tx - 1);
  int zero, kx;
  const bool ok = ColTiles(1, g.nxh, tx).at(b, t, &zero, &kx);
  C* col = spec + kx;
  auto load = [=](int c, int y, int) -> C { return ok ? col[((long long)c * ny + y) * nxs] : C{0, 0}; };
  auto store = [=](int c, int y, int, C v) {
    if (ok) col[((long long)c * ny + y) * nxs] = v;
  };
  const TileShape ts{ncl, tx, ltx};
  tile_dit<false, true, false>(buf, py, ts, tw, load, NoIo{});
  const int lp = py.lp << ltx;
  if constexpr (sizeof(R) == 4) {
    if (py.keep_order) {  // as in zproj_body
      C m[kHold2][3];
#pragma unroll
      for (int h = 0; h < kHold2; ++h) {
        const int y = (threadIdx.x >> ltx) + h * (blockDim.x >> ltx);
        if (ok && y < ny) {
          const C* at = buf + (py.at_freq(y) << ltx) + t;
#pragma unroll
          for (int c = 0; c < 3; ++c) m[h][c] = at[c * lp];
          project2_at<R>(m[h], sy, kx, y, kx == 0 && y == 0, free_mask);
        }
      }
      __syncthreads();
#pragma unroll
      for (int h = 0; h < kHold2; ++h) {
        const int y = (threadIdx.x >> ltx) + h * (blockDim.x >> ltx);
        if (ok && y < ny) {
          C* at = buf + (py.at_natural(y) << ltx) + t;
#pragma unroll
          for (int c = 0; c < 3; ++c) at[c * lp] = m[h][c];
        }
      }
      __syncthreads();
      tile_dit<true, false, true>(buf, py, ts, tw, NoIo{}, store);
      return;
    }
  }
  if (ok) {
    for (int i = threadIdx.x >> ltx; i < ny; i += blockDim.x >> ltx) {
      const int e = py.dr[0].div(i), q0 = i - e * py.r[0], y = py.freq_of(q0, e);
      C* at = buf + ((q0 * py.m0p + e) << ltx) + t;
      if (ncl == 6) {
        C m[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) m[c] = at[c * lp];
        const C dx = sy.d[0][kx], dy = sy.d[1][y];
        project_simplex2<R>(m, C{(R)1 + dx.x, dx.y}, dx, C{(R)1 + dy.x, dy.y}, dy, kx == 0 && y == 0, free_mask);
#pragma unroll
        for (int c = 0; c < 6; ++c) at[c * lp] = m[c];
      } else {
        C m[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) m[c] = at[c * lp];
        project2_at<R>(m, sy, kx, y, kx == 0 && y == 0, free_mask);
#pragma unroll
        for (int c = 0; c < 3; ++c) at[c * lp] = m[c];
      }
    }
  }
  __syncthreads();
  tile_transposed_inverse(buf, py, ts, tw, store);
}

template <typename R>
__global__ void __launch_bounds__(kGT, xy_blocks<R>())
    k_yproj2d(Cx<R>* __restrict__ spec, const GridDesc g, const int ltx, const __grid_constant__ AxisPlan py,
              const Cx<R>* __restrict__ tw, const AxisSyms<R> sy, const unsigned free_mask) {
  chain_begin();
  yproj2d_body<R>(spec, g, ltx, py, tw, sy, free_mask, blockIdx.x);
}

// ------------------------------------------------------------ x inverse
// Pairs of half spectra are recombined as Z = Xa + i Xb over the full
// length (Hermitian extension; the imaginary parts of the k = 0 and
// Nyquist bins are dropped, as for any complex-to-real transform), one
// inverse complex FFT gives both real rows.  DOT adds sum(out * w) in FP64.
template <typename R, bool DOT>
__device__ __forceinline__ void xinv_body(const Cx<R>* __restrict__ spec, R* __restrict__ out,
                                          const R* __restrict__ dotw, double* __restrict__ partial,
                                          const GridDesc& g, const int Q, const AxisPlan& px,
                                          const Cx<R>* __restrict__ tw, const R scale, const bool self_dot,
                                          const int bx) {
  using C = Cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  __shared__ double red[32];
  const int nx = g.nx, nxh = g.nxh, nxs = g.nxs, half = nx >> 1, lp = px.lp;
  const int npair = (g.ncomp * Q) >> 1;
  const XTables tab(buf, g, px, Q, npair, (long long)bx * Q, DOT);
  __syncthreads();
  for (int idx = threadIdx.x; idx < npair * nxh; idx += blockDim.x) {
    const int p = px.dh.div(idx), k = idx - p * nxh;
    const int ra = tab.row[2 * p], rb = tab.row[2 * p + 1];
    C a = ra >= 0 ? spec[(long long)ra * nxs + k] : C{0, 0};
    C c = rb >= 0 ? spec[(long long)rb * nxs + k] : C{0, 0};
    if (k == 0 || k == half) a.y = c.y = 0;
    buf[p * lp + px.at_natural(k)] = C{a.x - c.y, a.y + c.x};
    if (k != 0 && k != half) buf[p * lp + px.at_natural(nx - k)] = C{a.x + c.y, c.x - a.y};
  }
  __syncthreads();
  const TileShape ts{npair, 1, 0};
  if constexpr (DOT) {
    // the sums want one accumulator per thread: transform in place, then one
    // sweep over the rows
    tile_dit<true, false, false>(buf, px, ts, tw, NoIo{}, NoIo{});
    KSum<R> acc;
    for (int idx = threadIdx.x; idx < 2 * npair * nx; idx += blockDim.x) {
      const int rho = px.dn.div(idx), x = idx - rho * nx;
      const int row = tab.row[rho];
      if (row >= 0) {
        const C z = buf[(rho >> 1) * lp + tab.at[x]];
        const R val = ((rho & 1) ? z.y : z.x) * scale;
        const long long off = (long long)row * nx + x;
        out[off] = val;
        acc.add(val * (self_dot ? val : dotw[off]));
      }
    }
    double v[1] = {acc.value()};
    block_sum<1>(v, red);
    if (threadIdx.x == 0) *partial = v[0];
  } else {
    const int* rows = tab.row;
    auto store = [=](int p, int x, int, C v) {
      const int ra = rows[2 * p], rb = rows[2 * p + 1];
      if (ra >= 0) out[(long long)ra * nx + x] = v.x * scale;
      if (rb >= 0) out[(long long)rb * nx + x] = v.y * scale;
    };
    tile_dit<true, false, true>(buf, px, ts, tw, NoIo{}, store);
  }
}

template <typename R, bool DOT>
__global__ void __launch_bounds__(kGT, xy_blocks<R>())
    k_xinv(const Cx<R>* __restrict__ spec, R* __restrict__ out, const R* __restrict__ dotw,
           double* __restrict__ partials, const GridDesc g, const int Q, const __grid_constant__ AxisPlan px,
           const Cx<R>* __restrict__ tw, const R scale, const bool self_dot) {
  chain_begin();
  xinv_body<R, DOT>(spec, out, dotw, DOT ? partials + blockIdx.x : nullptr, g, Q, px, tw, scale, self_dot,
                    blockIdx.x);
}

}  // namespace rve
