// FP64 dense kernels of the DF pipeline: blocked Cholesky of the Coulomb metric
// V = L L^T, and the in-place triangular solve B = L^{-1} (Q|mu nu) that
// turns raw three-centre integrals into the Cholesky-decomposed ERIs (CD-ERIs) of
// Sec. 2.2.
//
// On GB300 FP64 runs at ~1.2 TFLOP/s (about 2 DFMA per clock per SM, a quarter
// of that for a lone warp).  The factorisation (Naux^3 / 3) runs there; the
// solve's products run as sliced FP16 products on the tensor cores (oz.cu) where
// the caller gives scratch for the slices, which a handle without split shadows
// does, and on the 64x64 register-blocked DFMA GEMM (gemm64.cuh) elsewhere.
// Set-up of (H2O)_24 (Naux = 1800): 73 ms sliced, 570 on the DFMA pipe.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "bqc_internal.h"
#include "gemm64.cuh"
#include "oz.h"

namespace bqc {

int dgemm(bool tA, bool tB, int M, int N, int K, double alpha, const double *A, int64_t lda,
          const double *B, int64_t ldb, double beta, double *C, int64_t ldc, cudaStream_t s) {
  Gemm64Args g;
  g.M = M;
  g.N = N;
  g.K1 = 1;
  g.K2 = K;
  g.alpha = alpha;
  g.beta = beta;
  g.A = A;
  g.lda = lda;
  g.sA1 = 0;
  g.B = B;
  g.ldb = ldb;
  g.sB1 = 0;
  g.C = C;
  g.ldc = ldc;
  return launch_gemm64(tA ? kAT : kAN, tB, g, s);
}

// ----------------------------------------------------------- Cholesky ---

constexpr int kNB = 64;

// Unblocked Cholesky of the kNB x kNB diagonal block at (k0, k0), in shared
// memory; writes L (lower) and zeros above.  flag <- 1 when not positive.
__global__ void __launch_bounds__(256) k_potrf_diag(double *A, int n, int k0, int *flag) {
  __shared__ double a[kNB][kNB + 1];
  const int nb = min(kNB, n - k0);
  for (int i = threadIdx.x; i < kNB * kNB; i += blockDim.x) {
    const int r = i / kNB, c = i % kNB;
    a[r][c] = (r < nb && c < nb) ? A[(int64_t)(k0 + r) * n + k0 + c] : 0.0;
  }
  __syncthreads();
  for (int j = 0; j < nb; ++j) {
    if (threadIdx.x == 0) {
      const double d = a[j][j];
      if (!(d > 0.0)) {
        atomicExch(flag, 1);
        a[j][j] = 1.0;
      } else {
        a[j][j] = sqrt(d);
      }
    }
    __syncthreads();
    const double djj = a[j][j];
    for (int i = j + 1 + threadIdx.x; i < nb; i += blockDim.x) a[i][j] /= djj;
    __syncthreads();
    const int m = nb - j - 1;
    for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
      const int r = j + 1 + t / m, c = j + 1 + t % m;
      if (c <= r) a[r][c] -= a[r][j] * a[c][j];
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < nb * nb; i += blockDim.x) {
    const int r = i / nb, c = i % nb;
    A[(int64_t)(k0 + r) * n + k0 + c] = (c <= r) ? a[r][c] : 0.0;
  }
}

// Rows below the diagonal block: A_rk := A_rk L_kk^{-T} (forward substitution
// per row, one thread per row); also zeroes the block above the diagonal.
__global__ void __launch_bounds__(128) k_chol_panel(double *A, int n, int k0) {
  __shared__ double L[kNB][kNB + 1];
  const int nb = min(kNB, n - k0);
  for (int i = threadIdx.x; i < kNB * kNB; i += blockDim.x) {
    const int r = i / kNB, c = i % kNB;
    L[r][c] = (r < nb && c < nb) ? A[(int64_t)(k0 + r) * n + k0 + c] : 0.0;
  }
  __syncthreads();
  const int row = k0 + nb + blockIdx.x * blockDim.x + threadIdx.x;
  if (row < n) {
    double x[kNB];
    double *ar = A + (int64_t)row * n + k0;
    for (int j = 0; j < nb; ++j) {
      double v = ar[j];
      for (int l = 0; l < j; ++l) v -= x[l] * L[j][l];
      x[j] = v / L[j][j];
    }
    for (int j = 0; j < nb; ++j) ar[j] = x[j];
    // upper block (row k0 + j, column `row`) = 0
    for (int j = 0; j < nb; ++j) A[(int64_t)(k0 + j) * n + row] = 0.0;
  }
}

int cholesky_lower(Ctx *ctx, double *A, int n, cudaStream_t s) {
  for (int k0 = 0; k0 < n; k0 += kNB) {
    const int nb = std::min(kNB, n - k0);
    k_potrf_diag<<<1, 256, 0, s>>>(A, n, k0, ctx->flag);
    BQC_LAUNCH_CHECK();
    const int rem = n - k0 - nb;
    if (rem <= 0) break;
    k_chol_panel<<<(rem + 127) / 128, 128, 0, s>>>(A, n, k0);
    BQC_LAUNCH_CHECK();
    // trailing update, lower triangle only: A22 -= L21 L21^T
    Gemm64Args g;
    g.M = rem;
    g.N = rem;
    g.K1 = 1;
    g.K2 = nb;
    g.alpha = -1.0;
    g.beta = 1.0;
    g.A = A + (int64_t)(k0 + nb) * n + k0;
    g.lda = n;
    g.sA1 = 0;
    g.B = g.A;
    g.ldb = n;
    g.sB1 = 0;
    g.C = A + (int64_t)(k0 + nb) * n + k0 + nb;
    g.ldc = n;
    g.lower_only = 1;
    BQC_TRY(launch_gemm64(kAN, true, g, s));
  }
  return BQC_OK;
}

// ------------------------------------------------------ triangular solve ---

// X_k := L_kk^{-1} X_k for the kNB rows of block k, one thread per column.
__global__ void __launch_bounds__(128) k_trsm_diag(const double *L, int n, int k0, double *X,
                                                   int64_t ncol, int64_t ld) {
  __shared__ double Lk[kNB][kNB + 1];
  const int nb = min(kNB, n - k0);
  for (int i = threadIdx.x; i < kNB * kNB; i += blockDim.x) {
    const int r = i / kNB, c = i % kNB;
    Lk[r][c] = (r < nb && c < nb) ? L[(int64_t)(k0 + r) * n + k0 + c] : 0.0;
  }
  __syncthreads();
  const int64_t col = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= ncol) return;
  double x[kNB];
  double *xc = X + (int64_t)k0 * ld + col;
  for (int j = 0; j < nb; ++j) {
    double v = xc[(int64_t)j * ld];
    for (int l = 0; l < j; ++l) v -= Lk[j][l] * x[l];
    x[j] = v / Lk[j][j];
    xc[(int64_t)j * ld] = x[j];
  }
}

// Explicit inverses of the kNB x kNB diagonal blocks of L, out[block][kNB][kNB]
// row-major with zeros above the diagonal (and the identity past the end of a
// ragged last block).  One block per diagonal block, one thread per column:
// forward substitution of a unit vector held in registers.
__global__ void __launch_bounds__(kNB) k_tri_inv(const double *L, int n, double *out) {
  __shared__ double a[kNB][kNB + 1];
  __shared__ double dinv[kNB];
  const int k0 = blockIdx.x * kNB, nb = min(kNB, n - k0), j = threadIdx.x;
  for (int r = 0; r < kNB; ++r)
    a[r][j] = (r < nb && j < nb) ? (j <= r ? L[(int64_t)(k0 + r) * n + k0 + j] : 0.0)
                                 : (r == j ? 1.0 : 0.0);
  __syncthreads();
  dinv[j] = 1.0 / a[j][j];
  __syncthreads();
  double x[kNB];
#pragma unroll
  for (int r = 0; r < kNB; ++r) x[r] = r == j ? 1.0 : 0.0;
  double *o = out + (int64_t)blockIdx.x * kNB * kNB + j;
#pragma unroll
  for (int r = 0; r < kNB; ++r) {
    x[r] *= dinv[r];
#pragma unroll
    for (int l = r + 1; l < kNB; ++l) x[l] = fma(-x[r], a[l][r], x[l]);
    o[r * kNB] = x[r];
  }
}

// The metric solve as tensor-core products (oz.cu): recursive halving,
//   X_1 := L_11^{-1} X_1;  X_2 -= L_21 X_1;  X_2 := L_22^{-1} X_2,
// down to 64-row diagonal blocks, which are multiplied by their explicit
// inverses.  Every product reads sliced copies, so all of them run in place.
// L's slices are made once; X is solved in column panels whose slices (half
// of X's rows at the top of the recursion) fit the scratch.
struct OzTrsmOp {
  int r0, nr, k0, nk;  // X[r0 .. r0 + nr) from X[k0 .. k0 + nk); r0 == k0: diagonal block
  size_t slices, exps;  // offsets of L's operand in the scratch
};

static void oz_trsm_ops(int n, int b0, int b1, std::vector<OzTrsmOp> &ops) {
  const int r0 = b0 * kNB;
  if (b1 - b0 == 1) {
    const int nb = std::min(kNB, n - r0);
    ops.push_back({r0, nb, r0, nb, 0, 0});
    return;
  }
  const int mid = (b0 + b1 + 1) / 2, rm = mid * kNB;
  oz_trsm_ops(n, b0, mid, ops);
  ops.push_back({rm, std::min(n, b1 * kNB) - rm, r0, rm - r0, 0, 0});
  oz_trsm_ops(n, mid, b1, ops);
}

// Columns of X a panel can hold in the scratch (0: not worth it).
static int64_t oz_trsm_plan(int n, int64_t ncol, size_t bytes, std::vector<OzTrsmOp> &ops,
                            size_t *inv, size_t *panel) {
  const int nblk = (n + kNB - 1) / kNB;
  oz_trsm_ops(n, 0, nblk, ops);
  size_t off = 0;
  int kmax = 0;
  for (auto &o : ops) {
    o.slices = off;
    off += oz_slice_bytes(o.nr, o.nk);
    o.exps = off;
    off += oz_exp_bytes(o.nr, 1);
    kmax = std::max(kmax, o.nk);
  }
  *inv = off;
  off += oz_align((size_t)nblk * kNB * kNB * 8);
  *panel = off;
  if (off >= bytes) return 0;
  const size_t per_col = (size_t)oz_kblocks(kmax) * kOzSlices * kOzKb * 2 + sizeof(int);
  int64_t cols = (int64_t)((bytes - off) / per_col) - 512;  // alignment of the two arrays
  if (cols >= ncol) return ncol;
  cols = cols / 128 * 128;
  if (cols < 4096) return 0;
  const int64_t np = (ncol + cols - 1) / cols;  // equal panels
  return std::min(cols, ((ncol + np - 1) / np + 127) / 128 * 128);
}

static int oz_trsm(Ctx *ctx, const double *L, int n, double *X, int64_t ncol, int64_t ld,
                   const std::vector<OzTrsmOp> &ops, int64_t cols, size_t inv, size_t panel,
                   char *scr, cudaStream_t s) {
  const int nblk = (n + kNB - 1) / kNB;
  double *li = reinterpret_cast<double *>(scr + inv);
  k_tri_inv<<<(unsigned)nblk, kNB, 0, s>>>(L, n, li);
  BQC_LAUNCH_CHECK();
  for (const auto &o : ops) {
    OzSrc a;
    a.kind = kOzRows;
    a.rows = o.nr;
    a.K = o.nk;
    if (o.r0 == o.k0) {
      a.p = li + (int64_t)(o.r0 / kNB) * kNB * kNB;
      a.ld = kNB;
    } else {
      a.p = L + (int64_t)o.r0 * n + o.k0;
      a.ld = n;
    }
    BQC_TRY(oz_slice(a, oz_kblocks(o.nk), scr + o.slices, reinterpret_cast<int *>(scr + o.exps), s));
  }
  for (int64_t c0 = 0; c0 < ncol; c0 += cols) {
    const int64_t nc = std::min(cols, ncol - c0);
    for (const auto &o : ops) {
      OzSrc x;
      x.kind = kOzCols;
      x.p = X + (int64_t)o.k0 * ld + c0;
      x.rows = nc;
      x.K = o.nk;
      x.ld = ld;
      void *xs = scr + panel;
      int *xe = reinterpret_cast<int *>(scr + panel + oz_slice_bytes(nc, o.nk));
      BQC_TRY(oz_slice(x, oz_kblocks(o.nk), xs, xe, s));
      OzOperand A, B;
      A.slices = xs;
      A.exps = xe;
      A.rows = nc;
      A.K = o.nk;
      B.slices = scr + o.slices;
      B.exps = reinterpret_cast<int *>(scr + o.exps);
      B.rows = o.nr;
      B.K = o.nk;
      const bool diag = o.r0 == o.k0;
      BQC_TRY(oz_gemm(A, B, oz_kblocks(o.nk), diag ? 1 : -1, diag ? 0 : 1,
                      X + (int64_t)o.r0 * ld + c0, ld, 0, 0, ctx->flag, s));
    }
  }
  return BQC_OK;
}

int trsm_lower_left(Ctx *ctx, const double *L, int n, double *X, int64_t ncol, int64_t ld,
                    void *scratch, size_t scratch_bytes, cudaStream_t s) {
  if (ncol <= 0) return BQC_OK;
  if (scratch && n > kNB) {
    std::vector<OzTrsmOp> ops;
    size_t inv = 0, panel = 0;
    const int64_t cols = oz_trsm_plan(n, ncol, scratch_bytes, ops, &inv, &panel);
    if (cols > 0)
      return oz_trsm(ctx, L, n, X, ncol, ld, ops, cols, inv, panel, static_cast<char *>(scratch),
                     s);
  }
  for (int k0 = 0; k0 < n; k0 += kNB) {
    const int nb = std::min(kNB, n - k0);
    k_trsm_diag<<<(unsigned)((ncol + 127) / 128), 128, 0, s>>>(L, n, k0, X, ncol, ld);
    BQC_LAUNCH_CHECK();
    const int rem = n - k0 - nb;
    if (rem <= 0) break;
    // X[k0+nb:, :] -= L[k0+nb:, k0:k0+nb] X[k0:k0+nb, :]
    Gemm64Args g;
    g.M = rem;
    g.N = (int)std::min<int64_t>(ncol, (int64_t)1 << 30);
    g.K1 = 1;
    g.K2 = nb;
    g.alpha = -1.0;
    g.beta = 1.0;
    g.A = L + (int64_t)(k0 + nb) * n + k0;
    g.lda = n;
    g.sA1 = 0;
    g.B = X + (int64_t)k0 * ld;
    g.ldb = ld;
    g.sB1 = 0;
    g.C = X + (int64_t)(k0 + nb) * ld;
    g.ldc = ld;
    BQC_TRY(launch_gemm64(kAN, false, g, s));
  }
  return BQC_OK;
}

}  // namespace bqc
