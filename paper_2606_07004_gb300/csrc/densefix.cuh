// Fixed-point forms of the Hutch++ split's dense products (see densefix.cu).
#pragma once

#include "common.cuh"

namespace ld {

// Whether the projection of a block of n rows and s columns takes the
// fixed-point products (FP32 blocks from a larger size), and whether its
// orthogonalisation does (a part of those).
bool densefix_ok(int n, int s, bool fp32 = false);
bool densefix_orth_ok(int n, int s, bool fp32);
// Workspace (doubles) of column_scales for s columns.
size_t densefix_workspace_doubles(int s);
// Partial slots of gram_fix and atg_fix: at most one per 256 rows.
int densefix_slots(int n);

// Per-column exponents f (|x| < 2^f) of a block, and the flag that sends the
// products to the FP64 (or compensated FP32) kernels instead: set where a
// column is not finite, or 2^f is above 16 times (FP32 blocks: 64 times) its
// mean magnitude.
struct ColScales {
  int* exp = nullptr;  // [s]
  int* bad = nullptr;  // [1]
};
template <typename TY>
int column_scales(const TY* Y, int ldy, int n, int s, double* ws, ColScales* out, cudaStream_t st);

// Partials [pair][densefix_slots(n)] of Y^T Y (pairs i <= j, row by row) and
// of A^T G (pair i r + j; G the +-1 probe block of the key); nothing is
// written when the flag is set.
template <typename TY>
int gram_fix(const TY* Y, int ldy, int n, int s, const ColScales& c, double* part, cudaStream_t st);
template <typename TY>
int atg_fix(const TY* A, int lda, int n, int s, int r, uint64_t key, const uint64_t* keyp,
            const ColScales& c, double* part, cudaStream_t st);

// A = Y Rinv (upper triangular s x s; A may alias Y), and
// X[:, 0:r] = G - A B; nothing is written when the flag is set.
int apply_fix(const double* Y, int ldy, int n, int s, const double* Rinv, double* A, int lda,
              const ColScales& c, cudaStream_t st);
int project_fix(const double* A, int lda, int n, int s, int r, uint64_t key, const uint64_t* keyp,
                const double* B, double* X, int ldx, const ColScales& c, cudaStream_t st);

}  // namespace ld
