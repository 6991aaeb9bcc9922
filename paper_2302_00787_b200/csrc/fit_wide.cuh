// Fits that need an eigen-decomposition (ADERF, SDERF) for d = 64 and 128: a chain of kernels (fit_wide.cu).
#pragma once
#include "common.cuh"

namespace fitw {

// Scratch of one group in doubles.
struct Layout {
  int d;
  __host__ __device__ size_t dd() const { return (size_t)d * d; }
  __host__ __device__ size_t LT() const { return 0; }              // L^T, row k: column k of L (zero left of the diagonal)
  __host__ __device__ size_t L() const { return dd(); }            // L by rows
  __host__ __device__ size_t Li() const { return 2 * dd(); }       // L^-1 by rows
  __host__ __device__ size_t A0() const { return 3 * dd(); }       // the matrix of the eigenproblem
  __host__ __device__ size_t RF() const { return 4 * dd(); }       // Householder vectors, one per row; later V' (orthonormal)
  __host__ __device__ size_t V() const { return 5 * dd(); }        // eigenvectors, one per row
  __host__ __device__ size_t U1() const { return 6 * dd(); }       // V' L^-1
  __host__ __device__ size_t U2() const { return 7 * dd(); }       // V' L^T
  __host__ __device__ size_t diag() const { return 8 * dd(); }     // tridiagonal matrix: diagonal, off-diagonal, reflector scales
  __host__ __device__ size_t lam() const { return diag() + 3 * d; }
  __host__ __device__ size_t scal() const { return lam() + d; }    // see FS_*
  __host__ __device__ size_t total() const { return scal() + 8; }
};
enum { FS_T1 = 0, FS_T2 = 1, FS_MM = 2, FS_TOT = 3, FS_FLAG = 4 };  // traces, mu4 . mu5, |A0|^2, 1: the fall-back solver is needed

// Everything but the fall-back; groups whose vectors failed the checks have flag FS_FLAG set.
int run(fsharp_ctx* ctx, const double* stats, int G, int d, int variant, double ridge, double* params, double* scratch);

}  // namespace fitw
