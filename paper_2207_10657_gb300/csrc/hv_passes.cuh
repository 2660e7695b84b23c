// Host-side description of the FFT / projection passes of one grid.
#pragma once

#include "common.cuh"
#include "fft_inplace.cuh"
#include "pass_timer.cuh"

namespace rve {

struct GridDesc {
  int ndim;       // 2 or 3
  int nx, ny, nz; // nz = 1 in 2D
  int nxh;        // nx/2 + 1 (half spectrum along x)
  int nxs;        // row stride of the spectrum (spectrum_stride)
  int ncomp;      // 3 or 6
  long long nvox;
  long long nrows;  // ny * nz voxel rows along x
  int nq = 1;       // strain points per voxel: 1 (one element per voxel), 2 (2D Kuhn
                    // triangles) or 6 (3D Kuhn tetrahedra); the spectral lines are then
                    // c * nq + q, ncomp = 6 or 36
};

// Row stride of a half spectrum: rows start on 32-byte sectors (64 bytes in
// FP64), so that the column segments of the y and z passes touch no sector in
// vain; nx/2 + 1 itself is odd for most lengths, and a 128-byte segment then
// straddles five sectors instead of four (product at 128^3 161.6 -> 159.8 us, 64^3
// 43.0 -> 41.2 us; 128-byte rows instead: 256^3 1046 -> 1084 us).  Short rows
// stay as they are: the padding is a larger part of them, and such grids are
// small (products, as they are / padded: 36x32x32 (19 values a row) 18.0 / 18.8
// us, 40x64x64 (21) 29.0 / 28.2; 48x64x64 (25) 29.5 / 28.7, 54x64x64 (28) 28.7 /
// 28.7).
__host__ __device__ constexpr int spectrum_stride(int nxh) { return nxh <= 24 ? nxh : (nxh + 3) & ~3; }

// Rank-one part of the symmetric consistent damage tangent, per voxel: the
// tangent applied to v is (1-D) C : v - dp/2 (a (n.v) + n (a.v)) with
// a = C : eps, n = eps^(t) / kappa and dp = D'(kappa) on loading voxels
// (0 elsewhere; a and n are read only where dp != 0).  All NULL: secant.
template <typename R> struct ConsTan {
  const R* dp = nullptr;  // Nvox
  const R* a = nullptr;   // ncomp x Nvox
  const R* n = nullptr;   // ncomp x Nvox
};

// Tables and workspace for the spectral passes at precision R.
template <typename R> struct SpecWork {
  AxisPlan px{}, py{}, pz{};
  Cx<R>* tw[3] = {nullptr, nullptr, nullptr};    // e^{-2 pi i t / n_axis}
  Cx<R>* gdiff[3] = {nullptr, nullptr, nullptr}; // e^{i th} - 1 (exact 0 at k=0)
  Cx<R>* gavg[3] = {nullptr, nullptr, nullptr};  // FP32: (1 + e^{i th})/2; FP64: (sin, cos)(th/2) (AxisSyms)
  Cx<R>* spec = nullptr;                          // ncomp * nz * ny * nxs
  unsigned free_mask = 0;                         // bit c: Mandel comp c stress-controlled
  // tiling of the generic passes
  int qx;        // voxel rows per x-pass block
  int lty, ltz;  // log2 of the kx columns per y-pass block, per z-pass / 2D y-pass block
  double* partials = nullptr;  // per-block FP64 partial sums (epilogues)
  int max_partials = 0;
  PassTimer* timer = nullptr;  // optional per-pass event timing
  ConsTan<R> cons;             // set: tangent passes apply the consistent tangent
  bool generic = false;        // true: never take the compiled FP32 passes
  bool unfused = false;        // true: compiled passes, but CG scalars and updates as the generic path
  bool cluster = false;        // true: the cluster x+y passes where they apply (opt-in: slower, see hv_cluster.cu)
  Cx<R>* twq = nullptr;        // e^{-2 pi i t / (Nx/4)}: the cluster passes' y sub-transform
  int* wait_err = nullptr;     // device word a kernel sets when a bounded wait runs out (NULL: no TMA passes)
};

enum class XIn { Plain = 0, Tangent = 1 };

// Launch helpers (hv_passes.cu).  Every pass runs on `st`; the number of
// launches issued is added to *nlaunch.
template <typename R>
cudaError_t spectral_apply(const GridDesc& g, SpecWork<R>& w, const MatTable<R>& mt, const R* in,
                           const uint8_t* phase, const R* damage, XIn mode, R* out,
                           const R* dot_with, double* dot_out, cudaStream_t st, long long* nlaunch);

struct DevScalars;  // solver_kernels.cuh

// One Steihaug-CG iteration's product on the compiled FP32 x passes, on the
// device scalars S: the forward passes with d:H:d formed in the x-forward
// pass (into S->dHd), then Algorithm 1's step length, then the x-inverse
// applying z += alpha d, r += alpha Hd (or z += tau d on an exit) with
// r'.r', r'.r, z'.z into S->rr_new, S->rnr, S->zz_new, then the convergence
// / beta decision.  Hd is never stored.  The persistent x-forward pass
// reduces d:H:d and takes the step-length decision in its last block; else
// one single-block kernel does both, as one does after the x-inverse.
// Returns cudaErrorNotSupported (nothing launched) when Nx has no compiled
// pass.
cudaError_t spectral_hv_cg(const GridDesc& g, SpecWork<float>& w, const MatTable<float>& mt, const float* d,
                           const uint8_t* phase, const float* damage, float* z, float* r, DevScalars* S,
                           cudaStream_t st, long long* nlaunch);

constexpr int kWave = 2 * 152;  // blocks that give every SM two

// wave: blocks that this grid's generic passes should have at least, where
// its size allows (kWave: the grid has a launch to itself; a member of a
// batch: its share of the batch's launches).
template <typename R>
cudaError_t spectral_setup(const GridDesc& g, SpecWork<R>& w, int wave = kWave);
template <typename R>
void spectral_free(SpecWork<R>& w);
// Plans and tile sizes of the generic passes; host work only.
template <typename R>
void plan_tiles(const GridDesc& g, SpecWork<R>& w, int wave = kWave);
// plan_tiles and the kernels' shared-memory attributes, no device allocation
// (the caller provides the tables and the spectrum storage in SpecWork).
template <typename R>
cudaError_t spectral_plan(const GridDesc& g, SpecWork<R>& w, int wave = kWave);
// Tile sizes and the blocks / dynamic shared memory they give, for the
// generic passes with these plans.
template <typename R> struct GenericTiles {
  int xblocks, yblocks, zblocks;  // zblocks: the 2D y pass in 2D
  size_t xsmem, ysmem, zsmem;
  GenericTiles(const GridDesc& g, int qx, int lty, int ltz, const AxisPlan& px, const AxisPlan& py,
               const AxisPlan& pz);
};
// Twiddles and gradient factors of an axis of n points (the host arrays of
// SpecWork's tw, gdiff and gavg).
template <typename R>
void axis_tables(int n, Cx<R>* tw, Cx<R>* gdiff, Cx<R>* gavg);
// Stage tables of a plan from its radices.
void finish_plan(AxisPlan& p);

// FP64 final reduction of per-block partials: out[s] = sum_b part[b*ns + s]
// (out: ns contiguous device doubles).  Fixed summation order.
cudaError_t reduce_partials(const double* part, int nblocks, int ns, double* out, cudaStream_t st,
                            long long* nlaunch);

}  // namespace rve
