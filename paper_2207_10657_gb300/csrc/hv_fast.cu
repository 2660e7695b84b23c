// FP32 spectral passes specialised at compile time for the common axis
// lengths (powers of two from 32 to 512 and 3 * 2^k up to 384).  Same data
// layout and the same arithmetic as the generic passes in hv_passes.cu;
// only the FFT engine (fft_fast.cuh) and the staging differ: global loads
// are batched in registers before they are written to shared memory, and
// the x passes give consecutive threads consecutive x so that the
// line-interleaved shared-memory accesses stay (nearly) conflict free.
#include "fft_ct.cuh"
#include "hv_fast.cuh"
#include "hv_tiles.cuh"
#include "launch.cuh"
#include "project.cuh"

namespace rve {

// MODE 0: plain; 1: secant tangent; 2: symmetric consistent tangent (the
// secant plus the rank-one correction of ConsTan on loading voxels).
template <int N, int NC, int MODE>
__global__ void __launch_bounds__(kFT)
    kf_xfwd(const float* __restrict__ in, const uint8_t* __restrict__ phase, const float* __restrict__ dmg,
            const MatTable<float> mt, float2* __restrict__ spec, const long long nrows, const int nxs, const long long nvox,
            const float2* __restrict__ tw, double* __restrict__ partials, const float* __restrict__ cdp,
            const float* __restrict__ ca, const float* __restrict__ cn) {
  chain_begin();
  constexpr int Q = xq<N, NC>();
  __shared__ __align__(16) float2 buf[xlines<N, NC * Q / 2>()];
  __shared__ double red[32];
  const long long row0 = (long long)blockIdx.x * Q;
  const float acc = xfwd_rows<N, NC, MODE>(buf, in, phase, dmg, mt, spec, nrows, nxs, nvox, tw, row0, nrows, cdp, ca, cn);
  if (MODE >= 1 && partials) {
    double val[1] = {(double)acc};
    block_sum<1>(val, red);
    if (threadIdx.x == 0) partials[blockIdx.x] = val[0];
  }
}

template <int N, int NC, bool DOT, bool CG = false>
__global__ void __launch_bounds__(kFT, 4)
    kf_xinv(const float2* __restrict__ spec, float* __restrict__ out, const float* __restrict__ dotw,
            double* __restrict__ partials, const long long nrows, const int nxs, const long long nvox,
            const float2* __restrict__ tw, const float scale, const bool self_dot, float* __restrict__ cz,
            float* __restrict__ cr, const float* __restrict__ cd, const int* __restrict__ cstatus,
            const double* __restrict__ calpha, const double* __restrict__ ctau) {
  chain_begin();
  constexpr int Q = xq<N, NC>();
  __shared__ __align__(16) float2 buf[NC * Q / 2 * N];
  __shared__ double red[3 * 32];
  const long long row0 = (long long)blockIdx.x * Q;
  xinv_rows<N, NC, DOT, CG>(buf, red, spec, out, dotw, partials, nrows, nxs, nvox, tw, scale, self_dot, cz, cr, cd,
                                   cstatus, calpha, ctau, row0, nrows, blockIdx.x);
}

template <int N, bool INV>
__global__ void __launch_bounds__(kFT)
    kf_ycols(float2* __restrict__ spec, const int nxh, const int nxs, const float2* __restrict__ tw) {
  chain_begin();
  constexpr int TX = ytx<N>();
  __shared__ __align__(16) float2 buf[TX * N];
  const int kx = blockIdx.x * TX + threadIdx.x % TX;
  ycols_tile<N, INV>(buf, spec + (long long)blockIdx.y * N * nxs + kx, kx < nxh, nxs, tw);
}

// The in-place form, for the length whose Stockham tile takes ten columns (80
// of the 128 bytes of a segment): 16 columns, 606 -> 481 us per pass at 384^3.
template <int N> constexpr bool yinplace() { return N == 384; }

template <int N, bool INV>
__global__ void __launch_bounds__(kFT)
    kf_ycols_ip(float2* __restrict__ spec, const int nxh, const int nxs, const float2* __restrict__ tw) {
  chain_begin();
  constexpr int TX = 16;
  __shared__ __align__(16) float2 buf[CtTile<N, TX>::LP * TX];
  const int kx = blockIdx.x * TX + threadIdx.x % TX;
  const bool ok = kx < nxh;
  float2* col = spec + (long long)blockIdx.y * N * nxs + kx;
  auto load = [=](int, int y, int) -> float2 { return ok ? col[(long long)y * nxs] : make_float2(0.f, 0.f); };
  auto store = [=](int, int y, int, float2 v) {
    if (ok) col[(long long)y * nxs] = v;
  };
  ct_dit<N, TX, 1, kFT, INV, true, true>(buf, tw, load, store);
}

// ------------------------------------------------- z + projection (3D)
template <int N>
__global__ void __launch_bounds__(zthreads<N>(), zminblocks<N>())
    kf_zproj(float2* __restrict__ spec, const int ny, const int nxh, const int nxs, const float2* __restrict__ tw,
             const AxisSyms<float> sy, const unsigned free_mask) {
  chain_begin();
  constexpr int TX = ztx<N>();
  constexpr int NL = 6 * TX;
  constexpr int NT = zthreads<N>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* buf = reinterpret_cast<float2*>(smem_raw);
  // line l = c * TX + t: component c, column t.  NT is a multiple of TX, so a
  // thread keeps its column in the projection, not in the transforms, whose
  // lines run over 6 TX threads
  static_assert(NT % TX == 0, "z-pass threads must be a multiple of its columns");
  const int kx0 = blockIdx.x * TX, ky = blockIdx.y, tv = min(TX, nxh - kx0);
  const long long zs = (long long)ny * nxs;
  float2* col = spec + (long long)ky * nxs + kx0;
  auto load = [&](int l, int z) -> float2 {
    const int c = l / TX, t = l - (l / TX) * TX;
    return t < tv ? col[(c * N + z) * zs + t] : make_float2(0.f, 0.f);
  };
  auto store = [&](int l, int z, float2 v) {
    const int c = l / TX, t = l - (l / TX) * TX;
    if (t < tv) col[(c * N + z) * zs + t] = v;
  };
  // The first forward stage reads straight from global memory and the last
  // inverse stage writes straight back.
  fft_stage0_from<N, NL, NT, false>(buf, load);
  fft_ct_range<N, NL, NT, false, 1, fft_nstages(N)>(buf, tw);
  // every point of a thread has the same column t: the x and y factors of the
  // symbol are formed once
  const int t = threadIdx.x % TX;
  if (t < tv) {
    const int kx = kx0 + t;
    const float2 ay = sy.h[1][ky], dy = sy.d[1][ky], ax = sy.h[0][kx], dx = sy.d[0][kx];
    const float2 fx = cmul(dx, ay), fy = cmul(ax, dy), fz = cmul(ax, ay);
    const bool kxy0 = kx == 0 && ky == 0;
    for (int z = threadIdx.x / TX; z < N; z += NT / TX) {
      float2 m[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) m[c] = buf[z * NL + c * TX + t];
      const float2 az = sy.h[2][z];
      project3<float>(m, cmul(fx, az), cmul(fy, az), cmul(fz, sy.d[2][z]), kxy0 && z == 0, free_mask);
#pragma unroll
      for (int c = 0; c < 6; ++c) buf[z * NL + c * TX + t] = m[c];
    }
  }
  __syncthreads();
  // inverse z transform
  fft_ct_range<N, NL, NT, true, 0, fft_nstages(N) - 1>(buf, tw);
  fft_stage_last_to<N, NL, NT, true>(buf, tw, store);
}

// The in-place form (fft_ct.cuh), for the length whose Stockham tile (72
// butterfly values a thread) had to be staged through shared memory: 2141 ->
// 1357 us per pass at 384^3.  The powers of two and 192 stay on the Stockham
// form, which needs no reordering between the projection and the inverse
// (256^3: 321 us against 391 us in place).
template <int N> constexpr bool zinplace() { return N == 384; }
constexpr int kZipTX = 4;  // columns of a tile: 75 KB, two blocks per SM
// 256 threads at 128 registers 4241 us per 384^3 product, 512 at 64 registers 4291 us
constexpr int kZipThreads = 256;

template <int N>
__global__ void __launch_bounds__(kZipThreads, 2)
    kf_zproj_ip(float2* __restrict__ spec, const int ny, const int nxh, const int nxs, const float2* __restrict__ tw,
             const AxisSyms<float> sy, const unsigned free_mask) {
  chain_begin();
  constexpr int TX = kZipTX, NT = kZipThreads;
  using T = CtTile<N, TX>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* buf = reinterpret_cast<float2*>(smem_raw);
  static_assert(NT % TX == 0, "a thread keeps one column");
  const int t = threadIdx.x % TX, kx = blockIdx.x * TX + t, ky = blockIdx.y;
  const bool ok = kx < nxh;
  float2* col = spec + (long long)ky * nxs + kx;
  const long long zs = (long long)ny * nxs;
  auto load = [=](int c, int z, int) -> float2 { return ok ? col[(c * N + z) * zs] : make_float2(0.f, 0.f); };
  auto store = [=](int c, int z, int, float2 v) {
    if (ok) col[(c * N + z) * zs] = v;
  };
  ct_dit<N, TX, 6, NT, false, true, false>(buf, tw, load, store);
  __syncthreads();
  // projection: read at the frequencies' digit-reversed places, written back
  // in natural order for the inverse
  constexpr int NP = (N * TX + NT - 1) / NT;
  constexpr int D = NT / TX;
  float2 m[NP][6];
  if (ok) {
    const float2 ay = sy.h[1][ky], dy = sy.d[1][ky], ax = sy.h[0][kx], dx = sy.d[0][kx];
    const float2 fx = cmul(dx, ay), fy = cmul(ax, dy), fz = cmul(ax, ay);
    const bool kxy0 = kx == 0 && ky == 0;
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      const int z = threadIdx.x / TX + h * D;
      if (N % D == 0 || z < N) {
        const float2* at = buf + T::freq(z) * TX + t;
#pragma unroll
        for (int c = 0; c < 6; ++c) m[h][c] = at[c * T::LP * TX];
        const float2 az = sy.h[2][z];
        project3<float>(m[h], cmul(fx, az), cmul(fy, az), cmul(fz, sy.d[2][z]), kxy0 && z == 0, free_mask);
      }
    }
  }
  __syncthreads();
  if (ok) {
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      const int z = threadIdx.x / TX + h * D;
      if (N % D == 0 || z < N) {
        float2* at = buf + T::natural(z) * TX + t;
#pragma unroll
        for (int c = 0; c < 6; ++c) at[c * T::LP * TX] = m[h][c];
      }
    }
  }
  __syncthreads();
  ct_dit<N, TX, 6, NT, true, false, true>(buf, tw, load, store);
}

// ------------------------------------------------- y + projection (2D)
// NCL = 3: one element per pixel (Mandel components); NCL = 6: the two Kuhn
// triangles of every pixel (lines c * 2 + q).
template <int N, int NCL> constexpr int p2tx_l() {
  return (kFBudget / (NCL * N)) < 16 ? ((kFBudget / (NCL * N)) < 1 ? 1 : kFBudget / (NCL * N)) : 16;
}

template <int N, int NCL>
__global__ void __launch_bounds__(kFT)
    kf_yproj2d(float2* __restrict__ spec, const int nxh, const int nxs, const float2* __restrict__ tw,
               const float2* __restrict__ gdx, const float2* __restrict__ gax, const float2* __restrict__ gdy,
               const float2* __restrict__ gay, const unsigned free_mask) {
  chain_begin();
  constexpr int TX = p2tx_l<N, NCL>();
  constexpr int NL = NCL * TX;
  __shared__ __align__(16) float2 buf[N * NL];
  const int kx0 = blockIdx.x * TX;
  const int tv = min(TX, nxh - kx0);
  for (int idx = threadIdx.x; idx < N * NL; idx += kFT) {
    const int y = idx / NL, rem = idx - (idx / NL) * NL;
    const int c = rem / TX, t = rem - (rem / TX) * TX;
    buf[idx] = t < tv ? spec[((long long)c * N + y) * nxs + kx0 + t] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  fft_ct<N, NL, kFT, false>(buf, tw);
  for (int pt = threadIdx.x; pt < N * TX; pt += kFT) {
    const int y = pt / TX, t = pt - (pt / TX) * TX;
    const int kx = kx0 + t;
    if (t >= tv) continue;
    float2 m[NCL];
#pragma unroll
    for (int c = 0; c < NCL; ++c) m[c] = buf[y * NL + c * TX + t];
    if constexpr (NCL == 3) {
      project2<float>(m, cmul(gdx[kx], gay[y]), cmul(gax[kx], gdy[y]), kx == 0 && y == 0, free_mask);
    } else {
      const float2 dx = gdx[kx], dy = gdy[y];
      project_simplex2<float>(m, make_float2(1.f + dx.x, dx.y), dx, make_float2(1.f + dy.x, dy.y), dy,
                              kx == 0 && y == 0, free_mask);
    }
#pragma unroll
    for (int c = 0; c < NCL; ++c) buf[y * NL + c * TX + t] = m[c];
  }
  __syncthreads();
  fft_ct<N, NL, kFT, true>(buf, tw);
  for (int idx = threadIdx.x; idx < N * NL; idx += kFT) {
    const int y = idx / NL, rem = idx - (idx / NL) * NL;
    const int c = rem / TX, t = rem - (rem / TX) * TX;
    if (t < tv) spec[((long long)c * N + y) * nxs + kx0 + t] = buf[idx];
  }
}

// ================================================================ dispatch
#define RVE_FAST_SIZES(X) X(32) X(64) X(128) X(256) X(512) X(96) X(192) X(384)

bool fast_size(int n) {
#define RVE_CASE(n_) if (n == n_) return true;
  RVE_FAST_SIZES(RVE_CASE)
#undef RVE_CASE
  return false;
}

template <int N>
static cudaError_t xfwd_n(const GridDesc& g, const float* in, const uint8_t* phase, const float* dmg,
                          const MatTable<float>& mt, float2* spec, const float2* tw, bool tangent, double* partials,
                          int* nblocks, cudaStream_t st, const ConsTan<float>* ct) {
  double* pd = tangent ? partials : nullptr;
  const bool cons = tangent && ct && ct->dp;
  if (g.ncomp == 6) {
    constexpr int Q = xq<N, 6>();
    const int blocks = (int)((g.nrows + Q - 1) / Q);
    *nblocks = blocks;
    if (tangent && g.nq == 2)
      launch_chained(kf_xfwd<N, 6, 3>, blocks, kFT, 0, st, in, phase, dmg, mt, spec, g.nrows, g.nxs, g.nvox, tw, pd, nullptr, nullptr, nullptr);
    else if (cons)
      launch_chained(kf_xfwd<N, 6, 2>, blocks, kFT, 0, st, in, phase, dmg, mt, spec, g.nrows, g.nxs, g.nvox, tw, pd, ct->dp, ct->a,
                                                ct->n);
    else if (tangent) launch_chained(kf_xfwd<N, 6, 1>, blocks, kFT, 0, st, in, phase, dmg, mt, spec, g.nrows, g.nxs, g.nvox, tw, pd, nullptr, nullptr, nullptr);
    else launch_chained(kf_xfwd<N, 6, 0>, blocks, kFT, 0, st, in, phase, dmg, mt, spec, g.nrows, g.nxs, g.nvox, tw, nullptr, nullptr, nullptr, nullptr);
  } else {
    constexpr int Q = xq<N, 3>();
    const int blocks = (int)((g.nrows + Q - 1) / Q);
    *nblocks = blocks;
    if (cons)
      launch_chained(kf_xfwd<N, 3, 2>, blocks, kFT, 0, st, in, phase, dmg, mt, spec, g.nrows, g.nxs, g.nvox, tw, pd, ct->dp, ct->a,
                                                ct->n);
    else if (tangent) launch_chained(kf_xfwd<N, 3, 1>, blocks, kFT, 0, st, in, phase, dmg, mt, spec, g.nrows, g.nxs, g.nvox, tw, pd, nullptr, nullptr, nullptr);
    else launch_chained(kf_xfwd<N, 3, 0>, blocks, kFT, 0, st, in, phase, dmg, mt, spec, g.nrows, g.nxs, g.nvox, tw, nullptr, nullptr, nullptr, nullptr);
  }
  return cudaGetLastError();
}

template <int N>
static cudaError_t xinv_n(const GridDesc& g, const float2* spec, float* out, const float* dotw, double* partials,
                          const float2* tw, bool dot, bool self, int* nblocks, cudaStream_t st) {
  const float scale = (float)(1.0 / (double)g.nvox);
  if (g.ncomp == 6) {
    constexpr int Q = xq<N, 6>();
    const int blocks = (int)((g.nrows + Q - 1) / Q);
    *nblocks = blocks;
    if (dot) launch_chained(kf_xinv<N, 6, true, false>, blocks, kFT, 0, st, spec, out, dotw, partials, g.nrows, g.nxs, g.nvox, tw, scale, self, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
    else launch_chained(kf_xinv<N, 6, false, false>, blocks, kFT, 0, st, spec, out, dotw, partials, g.nrows, g.nxs, g.nvox, tw, scale, self, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
  } else {
    constexpr int Q = xq<N, 3>();
    const int blocks = (int)((g.nrows + Q - 1) / Q);
    *nblocks = blocks;
    if (dot) launch_chained(kf_xinv<N, 3, true, false>, blocks, kFT, 0, st, spec, out, dotw, partials, g.nrows, g.nxs, g.nvox, tw, scale, self, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
    else launch_chained(kf_xinv<N, 3, false, false>, blocks, kFT, 0, st, spec, out, dotw, partials, g.nrows, g.nxs, g.nvox, tw, scale, self, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
  }
  return cudaGetLastError();
}

template <int N>
static cudaError_t ycols_n(const GridDesc& g, float2* spec, const float2* tw, bool inv, cudaStream_t st) {
  const int planes = g.ncomp * g.nz;
  if constexpr (yinplace<N>()) {
    const dim3 grid((g.nxh + 15) / 16, planes);
    if (inv) launch_chained(kf_ycols_ip<N, true>, grid, kFT, 0, st, spec, g.nxh, g.nxs, tw);
    else launch_chained(kf_ycols_ip<N, false>, grid, kFT, 0, st, spec, g.nxh, g.nxs, tw);
  } else {
    const dim3 grid((g.nxh + ytx<N>() - 1) / ytx<N>(), planes);
    if (inv) launch_chained(kf_ycols<N, true>, grid, kFT, 0, st, spec, g.nxh, g.nxs, tw);
    else launch_chained(kf_ycols<N, false>, grid, kFT, 0, st, spec, g.nxh, g.nxs, tw);
  }
  return cudaGetLastError();
}

template <int N>
static cudaError_t zproj_n(const GridDesc& g, float2* spec, const SpecWork<float>& w, cudaStream_t st) {
  constexpr bool IP = zinplace<N>();
  constexpr int TX = IP ? kZipTX : ztx<N>();
  constexpr int NT = IP ? kZipThreads : zthreads<N>();
  size_t smem = (size_t)6 * N * TX * sizeof(float2);
  if constexpr (IP) smem = (size_t)6 * CtTile<N, TX>::LP * TX * sizeof(float2);
  auto kernel = [] {
    if constexpr (IP) return kf_zproj_ip<N>;
    else return kf_zproj<N>;
  }();
  // the attribute is per device: set it once on every device that runs the pass
  constexpr int kDevs = 64;
  static bool attr[kDevs] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kDevs || !attr[dev]) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kDevs) attr[dev] = true;
  }
  const AxisSyms<float> sy{{w.gdiff[0], w.gdiff[1], w.gdiff[2]}, {w.gavg[0], w.gavg[1], w.gavg[2]}};
  launch_chained(kernel, dim3((g.nxh + TX - 1) / TX, g.ny), NT, smem, st, spec, g.ny, g.nxh, g.nxs, w.tw[2], sy, w.free_mask);
  return cudaGetLastError();
}

template <int N>
static cudaError_t yproj2d_n(const GridDesc& g, float2* spec, const SpecWork<float>& w, cudaStream_t st) {
  if (g.ncomp == 6) {
    constexpr int TX = p2tx_l<N, 6>();
    launch_chained(kf_yproj2d<N, 6>, (g.nxh + TX - 1) / TX, kFT, 0, st, spec, g.nxh, g.nxs, w.tw[1], w.gdiff[0], w.gavg[0],
                                                             w.gdiff[1], w.gavg[1], w.free_mask);
  } else {
    constexpr int TX = p2tx_l<N, 3>();
    launch_chained(kf_yproj2d<N, 3>, (g.nxh + TX - 1) / TX, kFT, 0, st, spec, g.nxh, g.nxs, w.tw[1], w.gdiff[0], w.gavg[0],
                                                             w.gdiff[1], w.gavg[1], w.free_mask);
  }
  return cudaGetLastError();
}

cudaError_t fast_xfwd(const GridDesc& g, const float* in, const uint8_t* phase, const float* dmg,
                      const MatTable<float>& mt, float2* spec, const float2* tw, bool tangent, double* partials,
                      int* nblocks, cudaStream_t st, const ConsTan<float>* ct) {
#define RVE_CASE(n_) \
  if (g.nx == n_) return xfwd_n<n_>(g, in, phase, dmg, mt, spec, tw, tangent, partials, nblocks, st, ct);
  RVE_FAST_SIZES(RVE_CASE)
#undef RVE_CASE
  return cudaErrorNotSupported;
}

cudaError_t fast_xinv(const GridDesc& g, const float2* spec, float* out, const float* dotw, double* partials,
                      const float2* tw, bool dot, bool self, int* nblocks, cudaStream_t st) {
#define RVE_CASE(n_) \
  if (g.nx == n_) return xinv_n<n_>(g, spec, out, dotw, partials, tw, dot, self, nblocks, st);
  RVE_FAST_SIZES(RVE_CASE)
#undef RVE_CASE
  return cudaErrorNotSupported;
}

template <int N>
static cudaError_t xinv_cg_n(const GridDesc& g, const float2* spec, float* z, float* r, const float* d,
                             const int* status, const double* alpha, const double* tau, double* partials,
                             const float2* tw, int* nblocks, cudaStream_t st) {
  const float scale = (float)(1.0 / (double)g.nvox);
  if (g.ncomp == 6) {
    constexpr int Q = xq<N, 6>();
    const int blocks = (int)((g.nrows + Q - 1) / Q);
    *nblocks = blocks;
    launch_chained(kf_xinv<N, 6, false, true>, blocks, kFT, 0, st, spec, nullptr, nullptr, partials, g.nrows, g.nxs, g.nvox, tw, scale,
                                                       false, z, r, d, status, alpha, tau);
  } else {
    constexpr int Q = xq<N, 3>();
    const int blocks = (int)((g.nrows + Q - 1) / Q);
    *nblocks = blocks;
    launch_chained(kf_xinv<N, 3, false, true>, blocks, kFT, 0, st, spec, nullptr, nullptr, partials, g.nrows, g.nxs, g.nvox, tw, scale,
                                                       false, z, r, d, status, alpha, tau);
  }
  return cudaGetLastError();
}

cudaError_t fast_xinv_cg(const GridDesc& g, const float2* spec, float* z, float* r, const float* d, const int* status,
                         const double* alpha, const double* tau, double* partials, const float2* tw, int* nblocks,
                         cudaStream_t st) {
#define RVE_CASE(n_) \
  if (g.nx == n_) return xinv_cg_n<n_>(g, spec, z, r, d, status, alpha, tau, partials, tw, nblocks, st);
  RVE_FAST_SIZES(RVE_CASE)
#undef RVE_CASE
  return cudaErrorNotSupported;
}

cudaError_t fast_ycols(const GridDesc& g, float2* spec, const float2* tw, bool inv, cudaStream_t st) {
#define RVE_CASE(n_) \
  if (g.ny == n_) return ycols_n<n_>(g, spec, tw, inv, st);
  RVE_FAST_SIZES(RVE_CASE)
#undef RVE_CASE
  return cudaErrorNotSupported;
}

cudaError_t fast_zproj(const GridDesc& g, float2* spec, const SpecWork<float>& w, cudaStream_t st) {
#define RVE_CASE(n_) \
  if (g.nz == n_) return zproj_n<n_>(g, spec, w, st);
  RVE_FAST_SIZES(RVE_CASE)
#undef RVE_CASE
  return cudaErrorNotSupported;
}

cudaError_t fast_yproj2d(const GridDesc& g, float2* spec, const SpecWork<float>& w, cudaStream_t st) {
#define RVE_CASE(n_) \
  if (g.ny == n_) return yproj2d_n<n_>(g, spec, w, st);
  RVE_FAST_SIZES(RVE_CASE)
#undef RVE_CASE
  return cudaErrorNotSupported;
}

}  // namespace rve
