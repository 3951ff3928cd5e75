// Matrix-free gridded operators: Q acts on fields on an nx x ny grid (row
// index y * nx + x) as
//   Q[(y, x), (y', x')] = W(|y - y'|, |x - x'|)   for |y - y'|, |x - x'| <= R,
// and 0 otherwise (a compactly supported stationary covariance restricted to
// the grid, e.g. the Wendland covariance of the paper's GRF study, Sec. 4).
// W is a quadrant table of (R + 1)^2 values.  The operator is applied by a
// register-tiled convolution over shared-memory rows (grid.cu) or, for wide
// supports, by 2D Fourier transforms (gridfft.cu); nothing of size
// n x (stencil) is stored.
#pragma once

#include "handle.cuh"

namespace ld {

constexpr int kMaxGridRadius = 96;
constexpr int kGridP = 8;          // outputs per thread along x
constexpr int kGridTX = 32;        // threads along x: an x segment of 256 outputs
constexpr int kGridTY = 8;         // output rows per CTA (one warp each)
constexpr int kGridThreads = kGridTX * kGridTY;

// Row length of the expanded table: W(dy, dx) at [dy * L + dx + R], dx in
// [-R, R], followed by kGridP zeros.
inline int grid_row_len(int R) { return 2 * R + 1 + kGridP; }

int create_grid_handle(int nx, int ny, int R, const double* w, logdet_handle* out);

// Expanded table of W / c in the compute type CT (double or float).
template <typename CT>
int grid_table(const logdet_ctx* h, double c, CT* out, cudaStream_t st);
size_t grid_table_count(const logdet_ctx* h);

// y = Q x (+ colshift[p] x[:, p]) on a block (n x ld), tab from grid_table.
template <typename T>
int grid_apply(const logdet_ctx* h, const typename Compute<T>::type* tab, const T* x, T* y,
               int ld, const double* colshift, cudaStream_t st);

// ---- fast convolution (gridfft.cu) ----
// A cover of the grid by tx x ty windows of 2^lnx x 2^lny points, taken in
// pairs; pairs == 0: the direct convolution.
struct GridFft {
  int pairs = 0;
  int lnx = 0, lny = 0, lnt = 0;  // lnt = max(lnx, lny): the root table's length
  int tx = 0, ty = 0;             // windows along x and y
  int bx = 0, by = 0;             // results per window along x and y
  int hx = 0, hy = 0;             // points of a window before its first result
};
// Workspace of one unit: the complex points of a pair of windows for the V
// block columns of a 16-byte vector (32 bytes a point for FP32 and FP64).
template <typename T>
inline size_t grid_fft_unit_bytes(const GridFft& p) {
  return ((size_t)1 << (p.lnx + p.lny)) * Vec16<T>::N * 2 * sizeof(T);
}
// A unit is limited to this or to the size of a block, whichever is larger.  A
// Krylov step lends the block that its update pass writes next as workspace,
// and a run has one of its own only where its blocks are smaller than this
// (33 x 30 points, FP64: one unit at a time took 524 us, all of them at once
// 56), so the memory estimate of a solve stays what it was.
constexpr size_t kGridFftFree = (size_t)8 << 20;
template <typename T>
inline size_t grid_fft_own_bytes(const GridFft& p, int ld) {
  const size_t unit = grid_fft_unit_bytes<T>(p), all = unit * p.pairs * (ld / Vec16<T>::N);
  return std::max(unit, std::min(all, kGridFftFree));
}
// Workspace used at a time: what stays in the 129 MB L2 between the kernels.
constexpr size_t kGridFftGroup = (size_t)64 << 20;
// Which of the two a solve uses: estimates in microseconds for a block of ld
// columns, fitted to both measured on GB300 over grids from 33 x 30 to 1200 x
// 900 and supports from 2 to 60 cells (20 columns).  Direct: a launch, then
// the larger of one CTA's serial walk over the taps and the whole grid's taps
// (plus the staging of each input row, worth `stage` taps) at the FMA rate.
// Transforms: three launches, then the points times log2 of the window's
// size.  FP32, 1200 x 900: support 4 cells 268 us direct, 266 transformed;
// 10 cells 640 and 312; 25 cells 2315 and 304; 64 x 64, 25 cells 142 and 21.
// FP64, 1200 x 900: 3 cells 1762 and 1745, 10 cells 15568 and 2712; 301 x
// 240, 17 cells 5201 and 350.  The margin leaves near ties to the direct
// convolution, which needs no tables.
struct GridCost {
  double start, tap, stage, taps_per_us, unit;
};
template <typename T>
constexpr GridCost grid_cost() {
  return std::is_same<T, double>::value ? GridCost{40.0, 1.6, 13.0, 4.35e5, 1.25e-5}
                                        : GridCost{13.0, 0.09, 180.0, 1.97e7, 1.3e-6};
}
constexpr double kGridFftMargin = 1.15;

// The cover for blocks of leading dimension ld (the narrowest of a solve).
template <typename T>
GridFft grid_fft_plan(const logdet_ctx* h, int ld);
// Tables of W / c for that cover (roots and symbol; count in elements of T).
template <typename T>
size_t grid_fft_table_count(const GridFft& p);
template <typename T>
int grid_fft_table(const logdet_ctx* h, const GridFft& p, double c, T* out, cudaStream_t st);
// y = Q x (+ colshift[p] x[:, p]) as grid_apply; scratch: workspace the call
// may overwrite (16-byte aligned; allocated here when too small).  Every
// value of a block column must be finite: a transform spreads others over it.
template <typename T>
int grid_fft_apply(const logdet_ctx* h, const GridFft& p, const T* tab, const T* x, T* y, int ld,
                   const double* colshift, void* scratch, size_t scratch_bytes, cudaStream_t st);

// Partials [d][ld][ntiles] of dotv_d . y over uniform tiles (the pass-1
// dots of a Krylov step whose SpMM is grid_apply).
template <typename T>
int dots_pass(const T* y, const T* const* dotv, int ndots, typename PartOf<T>::type* part, int n,
              int ld, int tile_rows, int ntiles, int threads, cudaStream_t st);

}  // namespace ld
