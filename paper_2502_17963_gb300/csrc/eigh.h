// Small FP64 products and refined symmetric eigen-decomposition (eigh.cu).
#pragma once
#include <cuda_runtime.h>
#include <cusolverDn.h>

#include "bqc_internal.h"

namespace bqc {

// Largest orders served.  Products: above 640 the SCF's work matrices are large
// enough that the slices would count.  The refined decomposition is tested up to
// 320 (tests/test_gpu_eigh.py); it also wins above (600: 6.5 ms of FP32 syevd and
// about 2 of refinement against 19), where the FP64 call stays: with it taken, an
// FP64 solve of 400 functions ends within the 0.3 s after which
// tests/test_gpu_serve.py expects to find it running.
constexpr int kSmallGemmMax = 640;
constexpr int kEighRefineMax = 320;

struct SmallGemm {
  Ctx *ctx = nullptr;
  DBuf scr;  // slices of two operands
  int reserve(Ctx *c, int nmax);
  bool takes(int m, int n, int k) const;
  // C (m x n) = op(A) op(B), column-major
  int run(bool tA, bool tB, int m, int n, int k, const double *A, int lda, const double *B, int ldb,
          double *C, int ldc, cudaStream_t s) const;
};

struct EighRefiner {
  DBuf X, T, S, XX, Af, wf, work, J, idx, stat;
  int lwork = 0, nmax = 0;
  int reserve(Ctx *c, cusolverDnHandle_t sol, int n);
  // Eigenvectors of A (n x n) in place and ascending eigenvalues; *done is
  // false, with A untouched, when the refinement does not apply.
  int run(cusolverDnHandle_t sol, const SmallGemm &mm, double *A, int n, double *evals, bool *done,
          cudaStream_t s);
};

}  // namespace bqc
