// Spectral passes of the Hessian-vector product and of the projection:
//   x-forward (tangent fused) -> y-forward -> z-forward + projection +
//   z-inverse -> y-inverse -> x-inverse (+ fused FP64 dot product).
// 2D: x-forward -> y-forward + projection + y-inverse -> x-inverse.
//
// Sec. 2.1: G : zeta = F^-1{ Ghat(k) : F{zeta} } (Eq. (5)), Ghat from the
// linear finite-element gradient symbol through Eq. (9); the Hessian-vector
// product of Eq. (8) applies the tangent first, then the projection.
#include <algorithm>
#include <cmath>
#include <vector>

#include <type_traits>

#include "hv_cluster.cuh"
#include "hv_fast.cuh"
#include "hv_passes.cuh"
#include "hv_tma.cuh"
#include "passes_generic.cuh"
#include "project.cuh"
#include "scalar_logic.cuh"
#include "solver_kernels.cuh"

namespace rve {


// ------------------------------------------------------------ reduction
__global__ void k_reduce_partials(const double* __restrict__ part, int nb, int ns, double* __restrict__ out) {
  __shared__ double red[32];
  const int s = blockIdx.x;
  double acc = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) acc += part[(long long)b * ns + s];
  double v[1] = {acc};
  block_sum<1>(v, red);
  if (threadIdx.x == 0) out[s] = v[0];
}

cudaError_t reduce_partials(const double* part, int nblocks, int ns, double* out, cudaStream_t st,
                            long long* nlaunch) {
  k_reduce_partials<<<ns, 256, 0, st>>>(part, nblocks, ns, out);
  if (nlaunch) ++*nlaunch;
  return cudaGetLastError();
}

// ================================================================ host side
void finish_plan(AxisPlan& p) {
  int span = 1;
  for (int s = 0; s < p.ns; ++s) {
    p.span[s] = span;
    span *= p.r[s];
    p.m[s] = p.n / span;
    p.dr[s] = FastDiv::by(p.r[s]);
    p.dm[s] = FastDiv::by(p.m[s]);
  }
  for (int s = 0; s < p.ns; ++s) {
    p.nw[s] = std::max(1, p.m[0] / p.r[s]);
    p.dw[s] = FastDiv::by(p.nw[s]);
  }
  p.m0p = p.m[0] | 1;
  p.lp = p.r[0] * p.m0p;
  p.dn = FastDiv::by(p.n);
  p.dh = FastDiv::by(p.n / 2 + 1);
}

// The radix sequence of the compiled passes (8s, 4s, 2, 3s, 5s), successive
// factors below 8 joined in pairs so that the fewest stages result; `narrow`:
// 4s in place of the 8s and no pairs (kNarrowMax).
static void make_plan(int n, AxisPlan& p, bool keep, bool narrow) {
  p = AxisPlan{};
  p.n = n;
  p.keep_order = keep ? 1 : 0;
  int f[16], nf = 0, m = n, twos = 0;
  while (m % 2 == 0) { m /= 2; ++twos; }
  int n8 = twos / 3, rem = twos % 3;
  int n4 = 0, n2 = 0;
  if (rem == 2) n4 = 1;
  else if (rem == 1) {
    if (n8 > 0) { --n8; n4 = 2; } else n2 = 1;
  }
  if (narrow) {
    n8 = 0;
    n4 = twos / 2;
    n2 = twos % 2;
  }
  for (int i = 0; i < n8; ++i) f[nf++] = 8;
  for (int i = 0; i < n4; ++i) f[nf++] = 4;
  for (int i = 0; i < n2; ++i) f[nf++] = 2;
  while (m % 3 == 0) { m /= 3; f[nf++] = 3; }
  while (m % 5 == 0) { m /= 5; f[nf++] = 5; }
  auto pairs = [&](int i) { return !narrow && i >= 0 && i + 1 < nf && f[i] < 8 && f[i] * f[i + 1] <= 20; };
  // from the back, and from the front: keep the shorter, then the one with
  // the smaller largest radix
  int best[16], nb = 99, mx = 99;
  for (int side = 0; side < 2; ++side) {
    int r[16], k = 0;
    if (side == 0) {
      for (int i = 0; i < nf; ++i) {
        if (pairs(i)) { r[k++] = f[i] * f[i + 1]; ++i; }
        else r[k++] = f[i];
      }
    } else {
      for (int i = nf - 1; i >= 0; --i) {
        if (pairs(i - 1)) { r[k++] = f[i] * f[i - 1]; --i; }
        else r[k++] = f[i];
      }
      std::reverse(r, r + k);
    }
    const int rm = k ? *std::max_element(r, r + k) : 1;
    if (k < nb || (k == nb && rm < mx)) {
      nb = k;
      mx = rm;
      std::copy(r, r + k, best);
    }
  }
  p.ns = nb;
  std::copy(best, best + nb, p.r);
  if (n == 1) {  // an absent axis
    p.ns = 1;
    p.r[0] = 1;
  }
  finish_plan(p);
}

// Angles from long double libm calls, rounded once to R.  Two calls an entry:
// on the Grace host long double is software quad arithmetic, and four of them
// made an FP64 context of 512^2 take 2.8 ms to create instead of 1.9 ms.  FP64
// wants the half angle too, so it calls for that and doubles it.
template <typename R>
void axis_tables(int n, Cx<R>* tw, Cx<R>* gdiff, Cx<R>* gavg) {
  for (int k = 0; k < n; ++k) {
    const long double th = 2.0L * 3.14159265358979323846264338327950288L * (long double)k / (long double)n;
    if constexpr (std::is_same<R, double>::value) {
      const long double sh = sinl(0.5L * th), ch = cosl(0.5L * th);
      const long double s = 2.0L * sh * ch, c1 = -2.0L * sh * sh;  // sin th, cos th - 1
      tw[k] = Cx<R>{(R)(c1 + 1.0L), (R)(-s)};
      gdiff[k] = (k == 0) ? Cx<R>{0, 0} : Cx<R>{(R)c1, (R)s};
      gavg[k] = Cx<R>{k == 0 ? (R)0 : (R)sh, 2 * k == n ? (R)0 : (R)ch};
    } else {
      const long double c = cosl(th), s = sinl(th);
      tw[k] = Cx<R>{(R)c, (R)(-s)};
      gdiff[k] = (k == 0) ? Cx<R>{0, 0} : Cx<R>{(R)(c - 1.0L), (R)s};
      gavg[k] = (2 * k == n) ? Cx<R>{0, 0} : Cx<R>{(R)((1.0L + c) * 0.5L), (R)(s * 0.5L)};
    }
  }
}
template void axis_tables<float>(int, float2*, float2*, float2*);
template void axis_tables<double>(int, double2*, double2*, double2*);

template <typename R>
static cudaError_t upload_tables(int n, Cx<R>** tw, Cx<R>** gdiff, Cx<R>** gavg) {
  std::vector<Cx<R>> t(n), d(n), a(n);
  axis_tables<R>(n, t.data(), d.data(), a.data());
  cudaError_t e;
  if ((e = cudaMalloc(tw, n * sizeof(Cx<R>))) != cudaSuccess) return e;
  if ((e = cudaMalloc(gdiff, n * sizeof(Cx<R>))) != cudaSuccess) return e;
  if ((e = cudaMalloc(gavg, n * sizeof(Cx<R>))) != cudaSuccess) return e;
  if ((e = cudaMemcpy(*tw, t.data(), n * sizeof(Cx<R>), cudaMemcpyHostToDevice)) != cudaSuccess) return e;
  if ((e = cudaMemcpy(*gdiff, d.data(), n * sizeof(Cx<R>), cudaMemcpyHostToDevice)) != cudaSuccess) return e;
  return cudaMemcpy(*gavg, a.data(), n * sizeof(Cx<R>), cudaMemcpyHostToDevice);
}

template <typename R>
GenericTiles<R>::GenericTiles(const GridDesc& g, int qx, int lty, int ltz, const AxisPlan& px, const AxisPlan& py,
                              const AxisPlan& pz) {
  using C = Cx<R>;
  xblocks = (int)((g.nrows + qx - 1) / qx);
  xsmem = (size_t)((g.ncomp * qx) / 2) * px.lp * sizeof(C) + XTables::bytes((g.ncomp * qx) / 2, g.nx);
  if (g.ndim == 3) {
    yblocks = ColTiles(g.ncomp * g.nz, g.nxh, 1 << lty).count();
    ysmem = (size_t)(py.lp << lty) * sizeof(C);
    zblocks = ColTiles(g.ny, g.nxh, 1 << ltz).count();
    zsmem = (size_t)g.ncomp * (pz.lp << ltz) * sizeof(C);
  } else {
    yblocks = 0;
    ysmem = 0;
    zblocks = ColTiles(1, g.nxh, 1 << ltz).count();
    zsmem = (size_t)g.ncomp * (py.lp << ltz) * sizeof(C);
  }
}
template struct GenericTiles<float>;
template struct GenericTiles<double>;

// FP64 cells of up to this many field values take radices 2, 3, 4 and 5 only.
// Such a grid leaves most SMs a warp or two, and an FP64 instruction occupies
// its scheduler for 64 cycles however few lanes it has: a stage's time is the
// number of instructions of ONE butterfly, so small butterflies spread over
// more warps win.  Products, wide -> narrow: 16^2 33.6 -> 21.9 us, 90x60 50.1 ->
// 40.3, 128^2 (49152 values) 53.9 -> 37.7, 16^3 51.9 -> 35.5.  Once the pipe is
// full the extra trips through shared memory lose: 192^2 (110592 values) 48.5
// -> 59.4, 256^2 52.3 -> 62.6, 32^3 62.6 -> 67.3.  Around the line the lengths
// decide: 144x150 (64800) 50.1 -> 51.9, 18x20x30 (64800) 55.0 -> 47.5, 150^2
// (67500) 44.5 -> 52.6, 24x24x20 (69120) 76.0 -> 54.0, 160^2 73.6 -> 46.8, 24^3
// (82944) 56.0 -> 58.9.
constexpr long long kNarrowMax = 65536;

// Plans and tiles.  A tile is as large as keeps its threads busy (about one
// butterfly each, 128-byte column segments) and as small as gives the grid
// `wave` blocks, which alone on the chip leaves every SM work: with one tile size for all grids, each pass of a 32^2 cell ran on ONE
// SM (FP64 product 129 -> 35 us with 16-17 blocks per pass).  The element
// budgets leave the 32 bytes of a memory sector to a tile's columns; three
// limits go below that: what fits a block, the blocks wanted of a small grid,
// and the frequencies a block can hold while an FP32 tile is reordered (kHold:
// two columns at z lengths above 256, one above 512).
template <typename R>
void plan_tiles(const GridDesc& g, SpecWork<R>& w, int wave) {
  using C = Cx<R>;
  // FP32 cells of one element per voxel keep their roundings (zproj_body)
  const bool keep = std::is_same<R, float>::value && g.nq == 1;
  const bool narrow = std::is_same<R, double>::value && g.nvox * g.ncomp <= kNarrowMax;
  make_plan(g.nx, w.px, keep, narrow);
  make_plan(g.ny, w.py, keep, narrow);
  make_plan(g.ndim == 3 ? g.nz : 1, w.pz, keep, narrow);
  w.px.dc = FastDiv::by(g.ncomp);
  const int q1 = (g.ncomp & 1) ? 2 : 1;  // rows come in pairs where ncomp is odd
  // x: about 2048 elements (16 KB in FP32) per block
  long long q = std::max<long long>(q1, 2 * 2048 / ((long long)g.ncomp * g.nx));
  q = std::min<long long>(q, std::max<long long>(q1, g.nrows / wave));
  w.qx = (int)((g.ncomp & 1) ? std::max<long long>(2, q & ~1LL) : q);
  const int lseg = sizeof(C) == 8 ? 4 : 3, lsec = lseg - 2;  // columns of 128 and of 32 bytes (log2)
  // hold: elements per line group that one block's threads can reorder
  auto columns = [&](const AxisPlan& p, int groups, int planes, int elems, int hold) {
    int l = 7;  // short lines: up to 128 columns, so that a tile keeps its threads busy
    while (l > lseg && ((long long)groups * p.n << l) > 2048) --l;
    while (l > 0 && (((size_t)groups * (p.lp << l) * sizeof(C) > (size_t)kSmemCap) || (keep && (p.n << l) > hold))) --l;
    while (l > lsec && ((long long)groups * p.n << l) > elems) --l;
    while (l > 0 && ColTiles(planes, g.nxh, 1 << l).count() < wave) --l;
    return l;
  };
  w.lty = g.ndim == 3 ? columns(w.py, 1, g.ncomp * g.nz, 4096, 1 << 30) : 0;
  if (g.ndim == 3) w.ltz = columns(w.pz, g.ncomp, g.ny, sizeof(C) == 8 ? 6144 : 3072, kHold * kGZ);
  else w.ltz = columns(w.py, g.ncomp, 1, 3072, kHold2 * kGT);
}

template <typename R>
cudaError_t spectral_plan(const GridDesc& g, SpecWork<R>& w, int wave) {
  plan_tiles<R>(g, w, wave);
  // a tile that no block can hold is an error here, not a failed launch later
  // (the sizes that the entry points take all fit)
  const GenericTiles<R> t(g, w.qx, w.lty, w.ltz, w.px, w.py, w.pz);
  if (std::max({t.xsmem, t.ysmem, t.zsmem}) > (size_t)kSmemCap) return cudaErrorInvalidValue;
  // opt in to large dynamic shared memory
  cudaFuncSetAttribute(k_xfwd<R, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_xfwd<R, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_xfwd<R, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_ycols<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_ycols<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_zproj<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_yproj2d<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_xinv<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_xinv<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  return cudaGetLastError();
}

template <typename R>
cudaError_t spectral_setup(const GridDesc& g, SpecWork<R>& w, int wave) {
  using C = Cx<R>;
  cudaError_t e = spectral_plan<R>(g, w, wave);
  if (e != cudaSuccess) return e;
  const int ns[3] = {g.nx, g.ny, g.nz};
  for (int a = 0; a < g.ndim; ++a)
    if ((e = upload_tables<R>(ns[a], &w.tw[a], &w.gdiff[a], &w.gavg[a])) != cudaSuccess) return e;
  const size_t nspec = (size_t)g.ncomp * g.nrows * g.nxs;
  if ((e = cudaMalloc(&w.spec, nspec * sizeof(C))) != cudaSuccess) return e;
  if (std::is_same<R, float>::value && cluster_size_ok(g)) {
    // twiddles of the cluster passes' M-point y sub-transform (M = Nx / 4)
    const int m = g.nx / 4;
    std::vector<C> t(m);
    for (int k = 0; k < m; ++k) {
      const long double th = 2.0L * 3.14159265358979323846264338327950288L * (long double)k / (long double)m;
      t[k] = C{(R)cosl(th), (R)(-sinl(th))};
    }
    if ((e = cudaMalloc(&w.twq, m * sizeof(C))) != cudaSuccess) return e;
    if ((e = cudaMemcpy(w.twq, t.data(), m * sizeof(C), cudaMemcpyHostToDevice)) != cudaSuccess) return e;
  }
  // up to three partial sums per x block (the fused CG x-inverse), and an x
  // block may hold a single row
  w.max_partials = (int)std::max<long long>(3 * g.nrows + 8, 4096 * 8);
  return cudaMalloc(&w.partials, (size_t)w.max_partials * sizeof(double));
}

template <typename R>
void spectral_free(SpecWork<R>& w) {
  for (int a = 0; a < 3; ++a) {
    if (w.tw[a]) cudaFree(w.tw[a]);
    if (w.gdiff[a]) cudaFree(w.gdiff[a]);
    if (w.gavg[a]) cudaFree(w.gavg[a]);
    w.tw[a] = w.gdiff[a] = w.gavg[a] = nullptr;
  }
  if (w.spec) cudaFree(w.spec);
  if (w.partials) cudaFree(w.partials);
  if (w.twq) cudaFree(w.twq);
  w.spec = nullptr;
  w.partials = nullptr;
  w.twq = nullptr;
}

// y / z passes with the projection (3D) or the y pass with the projection
// (2D), between the x-forward and the x-inverse passes.
template <typename R>
static cudaError_t spectral_middle(const GridDesc& g, SpecWork<R>& w, cudaStream_t st, long long* nlp,
                                   bool skip_yfwd = false, bool skip_yinv = false) {
  using C = Cx<R>;
  constexpr bool F32 = std::is_same<R, float>::value;
  long long nl = 0;
  cudaError_t e;
  const GenericTiles<R> gt(g, w.qx, w.lty, w.ltz, w.px, w.py, w.pz);
  const AxisSyms<R> sy{{w.gdiff[0], w.gdiff[1], w.gdiff[2]}, {w.gavg[0], w.gavg[1], w.gavg[2]}};
  if (g.ndim == 3) {
    for (int pass = 0; pass < 3; ++pass) {
      if ((pass == 0 && skip_yfwd) || (pass == 2 && skip_yinv)) continue;  // done by the cluster x+y passes
      e = cudaErrorNotSupported;
      PassScope ps(w.timer, st, pass == 0 ? PASS_YFWD : (pass == 1 ? PASS_ZPROJ : PASS_YINV));
      if constexpr (F32) {
        if (!w.generic && pass != 1 && fast_size(g.ny)) e = fast_ycols(g, w.spec, w.tw[1], pass == 2, st);
        if (!w.generic && pass == 1 && fast_size(g.nz)) e = fast_zproj(g, w.spec, w, st);
      }
      if (e == cudaErrorNotSupported) {
        if (pass == 0) launch_chained(k_ycols<R, false>, gt.yblocks, kGT, gt.ysmem, st, w.spec, g, w.lty, w.py, w.tw[1]);
        else if (pass == 2) launch_chained(k_ycols<R, true>, gt.yblocks, kGT, gt.ysmem, st, w.spec, g, w.lty, w.py, w.tw[1]);
        else launch_chained(k_zproj<R>, gt.zblocks, kGZ, gt.zsmem, st, w.spec, g, w.ltz, w.pz, w.tw[2], sy, w.free_mask);
        e = cudaGetLastError();
      }
      if (e != cudaSuccess) return e;
      ++nl;
    }
  } else {
    e = cudaErrorNotSupported;
    PassScope ps(w.timer, st, PASS_YPROJ2D);
    if constexpr (F32) {
      if (!w.generic && fast_size(g.ny)) e = fast_yproj2d(g, w.spec, w, st);
    }
    if (e == cudaErrorNotSupported) {
      launch_chained(k_yproj2d<R>, gt.zblocks, kGT, gt.zsmem, st, w.spec, g, w.ltz, w.py, w.tw[1], sy, w.free_mask);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    ++nl;
  }
  *nlp += nl;
  return cudaSuccess;
}

// the cluster x+y passes were asked for and apply (3D FP32, Nx = Ny of a
// cluster length)
template <typename R>
static bool use_cluster(const GridDesc& g, const SpecWork<R>& w) {
  return std::is_same<R, float>::value && w.cluster && !w.generic && w.twq != nullptr && cluster_size_ok(g);
}

template <typename R>
cudaError_t spectral_apply(const GridDesc& g, SpecWork<R>& w, const MatTable<R>& mt, const R* in,
                           const uint8_t* phase, const R* damage, XIn mode, R* out,
                           const R* dot_with, double* dot_out, cudaStream_t st, long long* nlaunch) {
  using C = Cx<R>;
  constexpr bool F32 = std::is_same<R, float>::value;
  long long nl = 0;
  cudaError_t e;
  const GenericTiles<R> gt(g, w.qx, w.lty, w.ltz, w.px, w.py, w.pz);
  const int xblocks = gt.xblocks;
  const size_t xsm = gt.xsmem;
  // dot(in, G:B:in) for a compatible input (in = G:in, as every CG direction
  // is) equals dot(in, B:in): the compiled x-forward pass forms it from the
  // tangent it already computes, so the x-inverse need not read `in` again
  bool fwd_dot = false;
  int fwd_blocks = 0;
  // the cluster passes take the x and y transforms together (not the
  // consistent tangent's forward pass)
  const bool cl = use_cluster(g, w);
  const bool cl_fwd = cl && !(mode == XIn::Tangent && w.cons.dp != nullptr);
  // x forward (tangent fused)
  e = cudaErrorNotSupported;
  {
  PassScope ps(w.timer, st, PASS_XFWD);
  if constexpr (F32) {
    if (cl_fwd) {
      const bool want = mode == XIn::Tangent && dot_with != nullptr && dot_with == in && !w.unfused;
      e = cluster_xyfwd(g, in, phase, damage, mt, w.spec, w.tw[0], w.twq, mode == XIn::Tangent,
                        want ? w.partials : nullptr, st);
      fwd_blocks = cluster_blocks(g);
      fwd_dot = want && e == cudaSuccess;
    } else if (!w.generic && fast_size(g.nx)) {
      const bool want = mode == XIn::Tangent && dot_with != nullptr && dot_with == in && !w.unfused;
      if (!(mode == XIn::Tangent && w.cons.dp != nullptr))
        e = tma_xfwd(g, in, phase, damage, mt, w.spec, w.tw[0], mode == XIn::Tangent, want ? w.partials : nullptr,
                     &fwd_blocks, st, w.wait_err);
      if (e == cudaErrorNotSupported)
        e = fast_xfwd(g, in, phase, damage, mt, w.spec, w.tw[0], mode == XIn::Tangent, want ? w.partials : nullptr,
                      &fwd_blocks, st, &w.cons);
      fwd_dot = want && e == cudaSuccess;
    }
  }
  if (e == cudaErrorNotSupported) {
    if (mode == XIn::Tangent && w.cons.dp)
      launch_chained(k_xfwd<R, 2>, xblocks, kGT, xsm, st, in, phase, damage, mt, w.spec, g, w.qx, w.px, w.tw[0], w.cons);
    else if (mode == XIn::Tangent)
      launch_chained(k_xfwd<R, 1>, xblocks, kGT, xsm, st, in, phase, damage, mt, w.spec, g, w.qx, w.px, w.tw[0], w.cons);
    else
      launch_chained(k_xfwd<R, 0>, xblocks, kGT, xsm, st, in, phase, damage, mt, w.spec, g, w.qx, w.px, w.tw[0],
                                                    ConsTan<R>{});
    e = cudaGetLastError();
  }
  }
  if (e != cudaSuccess) return e;
  ++nl;
  if ((e = spectral_middle<R>(g, w, st, &nl, cl_fwd, cl)) != cudaSuccess) return e;
  const R scale = (R)(1.0 / (double)g.nvox);
  const bool dot = dot_with != nullptr && !fwd_dot;
  const bool self = dot && (dot_with == out);
  int nblocks = xblocks;
  e = cudaErrorNotSupported;
  {
  PassScope ps(w.timer, st, PASS_XINV);
  if constexpr (F32) {
    if (cl) {
      e = cluster_yxinv(g, w.spec, out, self ? nullptr : dot_with, w.partials, w.tw[0], w.twq, dot, self, st);
      nblocks = cluster_blocks(g);
    } else if (!w.generic && fast_size(g.nx)) {
      e = fast_xinv(g, w.spec, out, self ? nullptr : dot_with, w.partials, w.tw[0], dot, self, &nblocks, st);
    }
  }
  if (e == cudaErrorNotSupported) {
    nblocks = xblocks;
    if (dot)
      launch_chained(k_xinv<R, true>, xblocks, kGT, xsm, st, w.spec, out, self ? nullptr : dot_with, w.partials, g, w.qx,
                                                       w.px, w.tw[0], scale, self);
    else
      launch_chained(k_xinv<R, false>, xblocks, kGT, xsm, st, w.spec, out, nullptr, nullptr, g, w.qx, w.px, w.tw[0],
                                                        scale, false);
    e = cudaGetLastError();
  }
  }
  if (e != cudaSuccess) return e;
  ++nl;
  if (dot || fwd_dot) {
    e = reduce_partials(w.partials, fwd_dot ? fwd_blocks : nblocks, 1, dot_out, st, &nl);
    if (e != cudaSuccess) return e;
  }
  if (nlaunch) *nlaunch += nl;
  return cudaSuccess;
}

// Single-block launches (256 threads): a CG pass's block sums reduced into
// the device scalars, then the scalar step of Algorithm 1 that needs them.
__global__ void __launch_bounds__(256) k_reduce_alpha(const double* __restrict__ part, int nb, DevScalars* S) {
  __shared__ double sh[32];
  block_reduce_partials<1>(part, nb, &S->dHd, sh);
  if (threadIdx.x == 0) cg_alpha_scalars(S);
}

__global__ void __launch_bounds__(256) k_reduce_beta(const double* __restrict__ part, int nb, DevScalars* S) {
  __shared__ double sh[3 * 32];
  block_reduce_partials<3>(part, nb, &S->rr_new, sh);
  if (threadIdx.x == 0) cg_beta_scalars(S);
}

cudaError_t spectral_hv_cg(const GridDesc& g, SpecWork<float>& w, const MatTable<float>& mt, const float* d,
                           const uint8_t* phase, const float* damage, float* z, float* r, DevScalars* S,
                           cudaStream_t st, long long* nlaunch) {
  if (w.generic || w.unfused || !fast_size(g.nx)) return cudaErrorNotSupported;
  long long nl = 0;
  cudaError_t e;
  int fb = 0, ib = 0;
  const bool cl = use_cluster(g, w), cl_fwd = cl && w.cons.dp == nullptr;
  bool fwd_reduced = false;  // d:H:d and the step length done by the x-forward launch
  {
    PassScope ps(w.timer, st, PASS_XFWD);
    if (cl_fwd) {
      e = cluster_xyfwd(g, d, phase, damage, mt, w.spec, w.tw[0], w.twq, true, w.partials, st);
      fb = cluster_blocks(g);
    } else {
      e = w.cons.dp == nullptr ? tma_xfwd(g, d, phase, damage, mt, w.spec, w.tw[0], true, w.partials, &fb, st,
                                          w.wait_err, S)
                               : cudaErrorNotSupported;
      fwd_reduced = e == cudaSuccess;
      if (e == cudaErrorNotSupported)
        e = fast_xfwd(g, d, phase, damage, mt, w.spec, w.tw[0], true, w.partials, &fb, st, &w.cons);
    }
  }
  if (e != cudaSuccess) return e;
  ++nl;
  if (!fwd_reduced) {
    k_reduce_alpha<<<1, 256, 0, st>>>(w.partials, fb, S);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ++nl;
  }
  if ((e = spectral_middle<float>(g, w, st, &nl, cl_fwd, cl)) != cudaSuccess) return e;
  {
    PassScope ps(w.timer, st, PASS_XINV);
    if (cl) {
      e = cluster_yxinv_cg(g, w.spec, z, r, d, &S->status, &S->alpha, &S->tau, w.partials, w.tw[0], w.twq, st);
      ib = cluster_blocks(g);
    } else {
      e = fast_xinv_cg(g, w.spec, z, r, d, &S->status, &S->alpha, &S->tau, w.partials, w.tw[0], &ib, st);
    }
  }
  if (e != cudaSuccess) return e;
  ++nl;
  k_reduce_beta<<<1, 256, 0, st>>>(w.partials, ib, S);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  ++nl;
  if (nlaunch) *nlaunch += nl;
  return cudaSuccess;
}

template cudaError_t spectral_setup<float>(const GridDesc&, SpecWork<float>&, int);
template cudaError_t spectral_setup<double>(const GridDesc&, SpecWork<double>&, int);
template cudaError_t spectral_plan<float>(const GridDesc&, SpecWork<float>&, int);
template void plan_tiles<float>(const GridDesc&, SpecWork<float>&, int);
template void plan_tiles<double>(const GridDesc&, SpecWork<double>&, int);
template void spectral_free<float>(SpecWork<float>&);
template void spectral_free<double>(SpecWork<double>&);
template cudaError_t spectral_apply<float>(const GridDesc&, SpecWork<float>&, const MatTable<float>&, const float*,
                                           const uint8_t*, const float*, XIn, float*, const float*, double*,
                                           cudaStream_t, long long*);
template cudaError_t spectral_apply<double>(const GridDesc&, SpecWork<double>&, const MatTable<double>&,
                                            const double*, const uint8_t*, const double*, XIn, double*,
                                            const double*, double*, cudaStream_t, long long*);

}  // namespace rve
