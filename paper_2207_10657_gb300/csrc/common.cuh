// Shared device-side definitions: complex helpers, radix butterflies,
// material tables and block reductions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rve {

// ---------------------------------------------------------------- complex
template <typename R> struct CxT;
template <> struct CxT<float> { using T = float2; };
template <> struct CxT<double> { using T = double2; };
template <typename R> using Cx = typename CxT<R>::T;

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return C{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename C> __device__ __forceinline__ C cconj(C a) { return C{a.x, -a.y}; }
// a * conj(b)
template <typename C> __device__ __forceinline__ C cmulc(C a, C b) {
  return C{a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y};
}
template <typename C, typename R> __device__ __forceinline__ C cscale(C a, R s) { return C{a.x * s, a.y * s}; }
// multiply by -i (forward) or +i (inverse)
template <bool INV, typename C> __device__ __forceinline__ C rot90(C a) {
  return INV ? C{-a.y, a.x} : C{a.y, -a.x};
}

constexpr int kMaxPhases = 16;

// single-rounding product and fused multiply-add: where the result must not
// depend on which product of a sum the compiler contracts
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// ------------------------------------------------------ radix butterflies
// Small DFTs with the constants of the R-th roots of unity written out.
template <int R, bool INV, typename C> struct Dft;

template <bool INV, typename C> struct Dft<2, INV, C> {
  __device__ __forceinline__ static void run(C* a) {
    C t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
  }
};

template <bool INV, typename C> struct Dft<4, INV, C> {
  __device__ __forceinline__ static void run(C* a) {
    C t0 = cadd(a[0], a[2]), t1 = csub(a[0], a[2]);
    C t2 = cadd(a[1], a[3]), t3 = rot90<INV>(csub(a[1], a[3]));
    a[0] = cadd(t0, t2);
    a[2] = csub(t0, t2);
    a[1] = cadd(t1, t3);
    a[3] = csub(t1, t3);
  }
};

template <bool INV, typename C> struct Dft<8, INV, C> {
  __device__ __forceinline__ static void run(C* a) {
    using R = decltype(a[0].x);
    const R h = (R)0.70710678118654752440;  // sqrt(2)/2
    C e[4] = {a[0], a[2], a[4], a[6]};
    C o[4] = {a[1], a[3], a[5], a[7]};
    Dft<4, INV, C>::run(e);
    Dft<4, INV, C>::run(o);
    // twiddles w8^k, k = 0..3 (w8 = e^{-i pi/4} forward)
    C o1 = INV ? C{h * (o[1].x - o[1].y), h * (o[1].x + o[1].y)}
               : C{h * (o[1].x + o[1].y), h * (o[1].y - o[1].x)};
    C o2 = rot90<INV>(o[2]);
    C o3 = INV ? C{-h * (o[3].x + o[3].y), h * (o[3].x - o[3].y)}
               : C{h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y)};
    a[0] = cadd(e[0], o[0]);
    a[4] = csub(e[0], o[0]);
    a[1] = cadd(e[1], o1);
    a[5] = csub(e[1], o1);
    a[2] = cadd(e[2], o2);
    a[6] = csub(e[2], o2);
    a[3] = cadd(e[3], o3);
    a[7] = csub(e[3], o3);
  }
};

template <bool INV, typename C> struct Dft<3, INV, C> {
  __device__ __forceinline__ static void run(C* a) {
    using R = decltype(a[0].x);
    const R c = (R)-0.5;
    const R s = (R)0.86602540378443864676;  // sin(2 pi / 3)
    C t = cadd(a[1], a[2]);
    C u = csub(a[1], a[2]);
    C m = C{a[0].x + c * t.x, a[0].y + c * t.y};
    C w = rot90<INV>(C{s * u.x, s * u.y});
    a[0] = cadd(a[0], t);
    a[1] = cadd(m, w);
    a[2] = csub(m, w);
  }
};

template <bool INV, typename C> struct Dft<5, INV, C> {
  __device__ __forceinline__ static void run(C* a) {
    using R = decltype(a[0].x);
    const R c1 = (R)0.30901699437494742410, s1 = (R)0.95105651629515357212;
    const R c2 = (R)-0.80901699437494742410, s2 = (R)0.58778525229247312917;
    C t1 = cadd(a[1], a[4]), u1 = csub(a[1], a[4]);
    C t2 = cadd(a[2], a[3]), u2 = csub(a[2], a[3]);
    C m1 = C{a[0].x + c1 * t1.x + c2 * t2.x, a[0].y + c1 * t1.y + c2 * t2.y};
    C m2 = C{a[0].x + c2 * t1.x + c1 * t2.x, a[0].y + c2 * t1.y + c1 * t2.y};
    C w1 = rot90<INV>(C{s1 * u1.x + s2 * u2.x, s1 * u1.y + s2 * u2.y});
    C w2 = rot90<INV>(C{s2 * u1.x - s1 * u2.x, s2 * u1.y - s1 * u2.y});
    a[0] = cadd(a[0], cadd(t1, t2));
    a[1] = cadd(m1, w1);
    a[4] = csub(m1, w1);
    a[2] = cadd(m2, w2);
    a[3] = csub(m2, w2);
  }
};

// ------------------------------------------------------- material tables
template <typename R> struct MatTable {
  int nphase;
  R lam[kMaxPhases], mu[kMaxPhases];
  R kappa0[kMaxPhases], kappaf[kMaxPhases];
  int damaging[kMaxPhases];
};

// --------------------------------------------------------- reductions
// Neumaier-compensated FP32/FP64 per-thread sums, FP64 across threads.
template <typename R> struct KSum {
  R s = 0, c = 0;
  __device__ __forceinline__ void add(R x) {
    R t = s + x;
    if (fabs(s) >= fabs(x)) c += (s - t) + x;
    else c += (x - t) + s;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// Block-wide FP64 sum of NS values; result valid in thread 0.  `sh` must
// hold NS * 32 doubles.
template <int NS>
__device__ __forceinline__ void block_sum(double (&v)[NS], double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    double x = v[s];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) sh[s * 32 + warp] = x;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      double x = lane < nw ? sh[s * 32 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      v[s] = x;
    }
  }
  __syncthreads();
}

// out[s] = sum_b part[b * NS + s], s < NS, summed by one block as the
// separate reduction kernel k_reduce_partials does -- thread t < 256 (every
// thread of a smaller block) adds blocks t, t + 256, ... in that order, then
// the block-wide FP64 sum -- so the results agree bit for bit.  The NS sums
// share one sweep whose loads are issued U blocks at a time: ten thousand
// partials cost a few L2 round trips rather than one per partial.  The
// partials are read through L2 (other blocks of the grid wrote them).
// Called by every thread of the block; `sh` holds NS * 32 doubles, free on
// entry; thread 0 writes out.
template <int NS>
__device__ void block_reduce_partials(const double* part, int nblocks, double* out, double* sh) {
  constexpr int U = 8;
  const int stride = blockDim.x < 256 ? (int)blockDim.x : 256;
  double acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0.0;
  if ((int)threadIdx.x < stride) {
    int b = threadIdx.x;
#pragma unroll 1
    for (; b + (U - 1) * stride < nblocks; b += U * stride) {
      double v[U][NS];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int s = 0; s < NS; ++s) v[u][s] = __ldcg(part + (long long)(b + u * stride) * NS + s);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int s = 0; s < NS; ++s) acc[s] += v[u][s];
    }
#pragma unroll 1
    for (; b < nblocks; b += stride)
#pragma unroll
      for (int s = 0; s < NS; ++s) acc[s] += __ldcg(part + (long long)b * NS + s);
  }
  block_sum<NS>(acc, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int s = 0; s < NS; ++s) out[s] = acc[s];
  }
}

// Called by every thread of every block once thread 0 has written the
// block's NS partial sums to part[block * NS + s].  The last block to arrive
// (thread 0 fences its partials, then one atomic on `counter`) sums them with
// block_reduce_partials, resets the counter for the next launch and returns
// true; the other blocks return false.  No block waits on another.  Meant
// for grids of a few hundred blocks: the fence holds thread 0 until its
// stores are visible, which a grid of many short-lived blocks would pay once
// per block.  `sh` holds NS * 32 doubles, free on entry.
template <int NS>
__device__ bool reduce_in_last_block(const double* part, int nblocks, double* out, unsigned* counter, double* sh) {
  __shared__ unsigned s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(counter, 1u) == (unsigned)nblocks - 1u ? 1u : 0u;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  block_reduce_partials<NS>(part, nblocks, out, sh);
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

}  // namespace rve
