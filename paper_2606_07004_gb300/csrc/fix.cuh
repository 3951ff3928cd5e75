// Fixed-point form of the FP64 SpMM pass for grid stencil matrices (see
// fix.cu).
#pragma once

#include "handle.cuh"
#include "krylov.cuh"

namespace ld {

// Blocks smaller than this keep the CSR pass: their steps are bound by the
// latency of dependent launches, not by the FP64 pipe (a 64 x 64 grid's pass
// takes 4 us of which the pipe is busy 0.8).  Solves of 20 steps, us, CSR pass /
// this one, by the MB of the narrower block: 3D Laplacian OSLQ 4 MB 1184/1451,
// 8 2012/1826, 16 3445/2485, 34 5199/4191; OSA-IOP window 4 8 4246/4164, 16
// 7357/5785; 2D Laplacian window 4 8 3904/3992, 16 6644/5899; Matern OSLQ 8
// 2703/2421, window 4 8 5266/5899, 16 9493/7440.
constexpr size_t kFixMinBlock = (size_t)16 << 20;

// Geometry of a slice of `width` columns of an FP64 block; false when the matrix has no
// grid structure or the slice does not fit.
struct FixGeom {
  int T, kc, nseg, nlines, units, tx, ty, txs;
};
bool fix_geom(const logdet_ctx* h, int width, int ld, FixGeom* g);

// Whether every row's absolute sum is within 8 of the largest.  The results'
// unit follows the largest row, so a much smaller row would lose that many
// bits: with one row 4e5 times heavier than the others the forms moved by
// 1e-9.
inline bool fix_balanced(const logdet_ctx* h, double shift) {
  return std::max(h->g_hi, -h->g_lo) + shift <= 8.0 * (h->row_min + shift);
}

// Values of (Q + shift I) / c per row and diagonal, [n][ndiag], as fixed-point
// numbers A 2^(ka - 60), A = hi 2^30 + lo with |lo| <= 2^29; ka from fix_scale.
int fix_scale(const logdet_ctx* h, double c, double shift);
int fix_values(const logdet_ctx* h, double c, double shift, int ka, int2* out, cudaStream_t st);

// A job's fixed-point fields (fix, ka, hn, err, bad) and tensor map from its x,
// ld, col_off and width; sig / sig_stride / xexp are the caller's.  *bad is the
// job's own: set when its columns leave the range, and from the next launch on
// the fixed-point pass leaves the job to the general kernel.
int fix_job(SpmmJob<double>& J, const logdet_ctx* h, const FixGeom& g, const int2* fix, int ka,
            int* err, int* bad);
// One product y = A x over a block whose entries are below 2^xexp in
// magnitude (no dots).  *err_host (pinned) is written in stream order: nonzero
// if a staged copy's wait gave up, and y is not complete then.
int fix_spmm_block(const logdet_ctx* h, const int2* fix, int ka, const double* x, double* y, int ld,
                   int xexp, int* err_host, cudaStream_t st);
// Batched launch (all jobs with fix != nullptr and one grid dimension).
int launch_spmm_fix(const SpmmBatch<double>& b, cudaStream_t s);

}  // namespace ld
