// What the translation units of the subspace refresh share: a batch of matrices travels as pointer tables passed to the
// kernels by value.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "qg_common.cuh"

namespace qg {

constexpr int kMaxBatch = 8;  // matrices refreshed together

// One pointer per matrix of a batch.
template <class T>
struct Ptrs {
  T* p[kMaxBatch];
};

// A cooperative launch whose CTAs wait for one another.  Two such grids must never be half resident each (refreshes may run
// on several streams), so every one waits on the device for the previous one of this process, whatever its stream.
int launch_cooperative(const void* kern, unsigned grid, unsigned block, void** args, size_t smem, cudaStream_t st);

// ---- sym_eig.cu: the leading eigenvectors of symmetric positive semi-definite N x N matrices (2 <= N <= kEigMax)
constexpr int64_t kEigMax = 4096;
inline int64_t eig_pitch(int64_t N) { return round_up(N, 128); }   // row pitch of A and V (floats)

// Buffers of one matrix, carved by carve_eig: A and V first, back to back.  After launch_sym_eig all but Z is free for use.
struct EigBuffers {
  float* A;            // N rows of eig_pitch(N) floats, symmetric: the matrix, destroyed
  float* V;            // same extents: row k holds Householder vector v_k
  float *tau, *d, *e;  // N floats each: the reflectors' factors, the tridiagonal matrix
  float* cross;        // N floats: v_k . v_{k-1}
  float* scale;        // the power of two A is scaled by
  double *lam, *inv;   // r doubles each: the leading eigenvalues (of the scaled matrix), 1 / norm of the vectors of step 3
  double *plus, *minus;  // the pivots of the two factorisations of step 3 for some of the vectors (plus over A)
  float* Z;            // N x r (pitch r): eigenvectors of the tridiagonal matrix, then of A
  uint4* xchg;         // 2 x eig_pitch(N): exchange between the CTAs of a matrix
};
size_t carve_eig(void* base, int64_t N, int64_t r, EigBuffers* out);
// On return (stream order) Z[i][j] holds the eigenvector of the j-th largest eigenvalue, j < r, of every matrix.
// QG_DEV_BAD_FACTOR is raised in *status where the `wanted`-th eigenvalue (wanted <= r) is so small against the first that its
// vector is lost in rounding.
int launch_sym_eig(const EigBuffers* w, int nb, int64_t N, int64_t r, int64_t wanted, int32_t* status, cudaStream_t st);

// ---- refresh_tc.cu
// A[i] (N x N fp32, pitch lda) = X X^T for every matrix of a batch; X(i, k) = G[i * ldg + k] (N rows of K), or, if `columns`,
// X(i, k) = G[k * ldg + i] (the gradient has K rows of N).
int launch_gram(const uint16_t* const* G, int nmat, int64_t ldg, bool columns, int64_t N, int64_t K, float* const* A, int64_t lda,
                int32_t* status, cudaStream_t st);

}  // namespace qg
