// Symmetric eigen-decomposition and small FP64 products of the SCF.
//
// A full FP64 eigen-decomposition of a Fock matrix is latency-bound for a few
// hundred functions and was most of an SCF there (n = 150: 5.3 ms of cuSOLVER's
// syevd an iteration, against 1.1 ms for the same call in FP32).  Here the
// FP32 decomposition is refined to FP64 by products (Ogita and Aishima 2018,
// iterative refinement for symmetric eigenvectors; clusters of close
// eigenvalues are diagonalised exactly first):
//   with X the current vectors, S = X^T A X, Rt = X^T X - 1 and the
//   orthonormalised H = S - (Rt S + S Rt) / 2 (S near diagonal there),
//   J = block-diagonal eigenvectors of H in each cluster,
//   E_ij = (J^T H J)_ij / (l_j - l_i) between clusters,
//   X := X (1 - Rt / 2) J (1 + E).
// A cluster is a run of eigenvalues with gaps below 128 times the largest
// off-diagonal g of H, so |E| < 1/128 and a round squares the error, or below
// 1e-8 of the largest eigenvalue: three rounds take g from FP32's 1e-6 to FP64's
// rounding (1e-15), and E between two levels that such a g still couples would
// leave E^2 in X^T X - 1 (with a gap limit of 1e-12, 1e-10 and more for levels
// 1e-11 to 1e-10 apart).  From the third round on the vectors are then made
// orthonormal, X (3 - X^T X) / 2, and the result is accepted when g had fallen
// below 1e-12 of the largest eigenvalue and the R = X^T X - 1 measured before
// that step below 1e-9, which leaves 3/4 R^2.  Otherwise (a cluster of more than
// eight, no convergence) the caller falls back to the FP64 decomposition.
#include <cublas_v2.h>
#include <cuda_runtime.h>
#include <cusolverDn.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "bqc_internal.h"
#include "eigh.h"
#include "oz.h"

namespace bqc {

// C (m x n, column-major) = op(A) op(B): 16 x 16 tiles, one element a thread.
// A 64 x 64 tile would leave a 150 x 150 product on 9 SMs, each bound by its
// FP64 pipe (2 DFMA a clock); 100 small tiles take 10 us (cuBLAS: 41 us).
template <bool TA, bool TB>
__global__ void __launch_bounds__(256) k_dgemm_small(int m, int n, int k, const double *__restrict__ A,
                                                     int lda, const double *__restrict__ B, int ldb,
                                                     double *__restrict__ C, int ldc) {
  __shared__ double As[16][17], Bs[16][17];  // [k][i], [k][j]
  const int i0 = blockIdx.x * 16, j0 = blockIdx.y * 16, lo = threadIdx.x & 15, hi = threadIdx.x >> 4;
  auto la = [&](int k0) {
    const int i = i0 + (TA ? hi : lo), q = k0 + (TA ? lo : hi);
    return i < m && q < k ? __ldg(A + (TA ? q + (int64_t)i * lda : i + (int64_t)q * lda)) : 0.0;
  };
  auto lb = [&](int k0) {
    const int j = j0 + (TB ? lo : hi), q = k0 + (TB ? hi : lo);
    return j < n && q < k ? __ldg(B + (TB ? j + (int64_t)q * ldb : q + (int64_t)j * ldb)) : 0.0;
  };
  double a = la(0), b = lb(0), c = 0.0;
  for (int k0 = 0; k0 < k; k0 += 16) {
    __syncthreads();
    As[TA ? lo : hi][TA ? hi : lo] = a;
    Bs[TB ? hi : lo][TB ? lo : hi] = b;
    __syncthreads();
    a = la(k0 + 16);
    b = lb(k0 + 16);
#pragma unroll
    for (int q = 0; q < 16; ++q) c = fma(As[q][lo], Bs[q][hi], c);
  }
  if (i0 + lo < m && j0 + hi < n) C[i0 + lo + (int64_t)(j0 + hi) * ldc] = c;
}

// Sliced tensor-core products from 256 on: their launches (two slicings and a
// product, about 25 us together) are above a small DFMA product's time, and
// below it from about 250 functions (300: 47 us at the DFMA rate).
constexpr int kOzGemmMin = 256;

int SmallGemm::reserve(Ctx *c, int nmax) {
  ctx = c;
  if (nmax < kOzGemmMin || nmax > kSmallGemmMax) return BQC_OK;
  const size_t one = oz_slice_bytes(nmax, nmax) + oz_exp_bytes(nmax, 1);
  if (scr.alloc(c, 2 * one) != BQC_OK) scr.release();
  return BQC_OK;
}

bool SmallGemm::takes(int m, int n, int k) const {
  return std::max({m, n, k}) <= kSmallGemmMax;
}

int SmallGemm::run(bool tA, bool tB, int m, int n, int k, const double *A, int lda, const double *B,
                   int ldb, double *C, int ldc, cudaStream_t s) const {
  const size_t sa = oz_slice_bytes(m, k), ea = oz_exp_bytes(m, 1), sb = oz_slice_bytes(n, k);
  if (std::min({m, n, k}) >= kOzGemmMin / 2 && std::max({m, n, k}) >= kOzGemmMin && scr.p &&
      sa + ea + sb + oz_exp_bytes(n, 1) <= scr.n) {
    char *p = scr.as<char>();
    OzOperand o[2];
    for (int q = 0; q < 2; ++q) {
      OzSrc x;
      x.kind = (q == 0) != tA ? kOzCols : kOzRows;
      if (q == 1) x.kind = tB ? kOzCols : kOzRows;
      x.p = q ? B : A;
      x.rows = q ? n : m;
      x.K = k;
      x.ld = q ? ldb : lda;
      o[q].slices = p;
      int *e = reinterpret_cast<int *>(p + (q ? sb : sa));
      o[q].exps = e;
      o[q].rows = x.rows;
      o[q].K = k;
      BQC_TRY(oz_slice(x, oz_kblocks(k), p, e, s));
      p += sa + ea;
    }
    return oz_gemm(o[0], o[1], oz_kblocks(k), 1, 0, C, ldc, 0, kOzFull, ctx->flag, s);
  }
  const dim3 g((unsigned)((m + 15) / 16), (unsigned)((n + 15) / 16));
  if (tA) {
    if (tB) k_dgemm_small<true, true><<<g, 256, 0, s>>>(m, n, k, A, lda, B, ldb, C, ldc);
    else k_dgemm_small<true, false><<<g, 256, 0, s>>>(m, n, k, A, lda, B, ldb, C, ldc);
  } else {
    if (tB) k_dgemm_small<false, true><<<g, 256, 0, s>>>(m, n, k, A, lda, B, ldb, C, ldc);
    else k_dgemm_small<false, false><<<g, 256, 0, s>>>(m, n, k, A, lda, B, ldb, C, ldc);
  }
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

// ------------------------------------------------------------- refinement --

constexpr int kClusterMax = 8;

struct RefineStat {
  unsigned long long g, top;  // bits of the largest |off-diagonal| and |diagonal| of H, by round
  unsigned long long res;     // bits of the largest |X^T X - 1| after it
  int fail;                   // of any round
};

__global__ void k_to_f32(int64_t n, const double *a, float *b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (float)a[i];
}

__global__ void k_to_f64(int64_t n, const float *a, double *b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (double)a[i];
}

// H_ij = S_ij - (l_i + l_j) (X^T X - 1)_ij / 2 with l = diag(S); its largest
// elements.  (Non-negative doubles order like their bits; a NaN is above all.)
__global__ void __launch_bounds__(256) k_refine_h(int n, const double *__restrict__ S,
                                                  const double *__restrict__ XX,
                                                  double *__restrict__ H, RefineStat *st) {
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  unsigned long long g = 0, d = 0;
  if (e < (int64_t)n * n) {
    const int i = (int)(e % n), j = (int)(e / n);
    const double rt = XX[e] - (i == j ? 1.0 : 0.0);
    const double h =
        0.5 * (S[e] + S[(int64_t)i * n + j]) -
        0.5 * rt * (S[(int64_t)i * n + i] + S[(int64_t)j * n + j]);
    H[e] = h;
    const unsigned long long b =
        (unsigned long long)__double_as_longlong(h) & 0x7fffffffffffffffULL;
    if (i == j) d = b; else g = b;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
    d = max(d, __shfl_xor_sync(0xffffffffu, d, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&st->g, g);
    atomicMax(&st->top, d);
  }
}

// The thread of a cluster's first index diagonalises the cluster's block of H
// (cyclic Jacobi, Golub and Van Loan Sec. 8.5): J[q * n + j] is element
// (start + q, j) of J, lam ascending.
__global__ void __launch_bounds__(64) k_refine_clusters(int n, const double *__restrict__ H,
                                                        RefineStat *st, double *J, double *lam,
                                                        int *start, int *size) {
  const int i = blockIdx.x * 64 + threadIdx.x;
  if (i >= n) return;
  auto diag = [&](int k) { return H[(int64_t)k * n + k]; };
  const double top = __longlong_as_double((long long)st->top);
  const double thr =
      fmax(128.0 * __longlong_as_double((long long)st->g), 1e-8 * top);
  if (i > 0 && diag(i) - diag(i - 1) < -thr) st->fail = 1;  // not in order
  if (i > 0 && !(diag(i) - diag(i - 1) > thr)) return;      // not the first of a cluster
  int m = 1;
  while (i + m < n && !(diag(i + m) - diag(i + m - 1) > thr)) ++m;
  if (m == 1) {
    J[i] = 1.0;
    lam[i] = diag(i);
    start[i] = i;
    size[i] = 1;
    return;
  }
  if (m > kClusterMax) {
    st->fail = 1;
    m = kClusterMax;
  }
  double a[kClusterMax][kClusterMax], v[kClusterMax][kClusterMax];
  for (int p = 0; p < m; ++p)
    for (int q = 0; q < m; ++q) {
      a[p][q] = H[(int64_t)(i + q) * n + i + p];
      v[p][q] = p == q ? 1.0 : 0.0;
    }
  for (int sweep = 0; sweep < 12; ++sweep) {
    double off = 0.0;
    for (int p = 0; p < m; ++p)
      for (int q = p + 1; q < m; ++q) off = fmax(off, fabs(a[p][q]));
    if (!(off > 1e-17 * top)) break;
    for (int p = 0; p < m; ++p)
      for (int q = p + 1; q < m; ++q) {
        const double apq = a[p][q];
        if (apq == 0.0) continue;
        const double th = (a[q][q] - a[p][p]) / (2.0 * apq);
        const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(1.0 + th * th));
        const double c = rsqrt(1.0 + t * t), s = t * c;
        for (int k = 0; k < m; ++k) {
          const double x = a[k][p], y = a[k][q];
          a[k][p] = c * x - s * y;
          a[k][q] = s * x + c * y;
        }
        for (int k = 0; k < m; ++k) {
          const double x = a[p][k], y = a[q][k];
          a[p][k] = c * x - s * y;
          a[q][k] = s * x + c * y;
        }
        for (int k = 0; k < m; ++k) {
          const double x = v[k][p], y = v[k][q];
          v[k][p] = c * x - s * y;
          v[k][q] = s * x + c * y;
        }
      }
  }
  for (int j = 0; j < m; ++j) {  // ascending, by selection
    int b = -1;
    for (int k = 0; k < m; ++k)
      if (!isnan(a[k][k]) && (b < 0 || a[k][k] < a[b][b])) b = k;
    if (b < 0) {
      st->fail = 1;
      b = j;
    }
    for (int q = 0; q < m; ++q) J[(int64_t)q * n + i + j] = v[q][b];
    lam[i + j] = a[b][b];
    start[i + j] = i;
    size[i + j] = m;
    a[b][b] = __longlong_as_double(0x7ff8000000000000LL);  // taken
  }
}

// M = J (1 + E) - Rt J / 2.
__global__ void __launch_bounds__(256) k_refine_m(int n, const double *__restrict__ H,
                                                  const double *__restrict__ XX,
                                                  const double *__restrict__ J,
                                                  const double *__restrict__ lam,
                                                  const int *__restrict__ start,
                                                  const int *__restrict__ size,
                                                  const RefineStat *st, double *__restrict__ M) {
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= (int64_t)n * n || st->fail) return;
  const int i = (int)(e % n), j = (int)(e / n);
  const int si = start[i], mi = size[i], sj = start[j], mj = size[j];
  double v = 0.0;
  if (si == sj) {
    v = J[(int64_t)(i - sj) * n + j];
  } else {
    for (int a = 0; a < mi; ++a) {  // E_aj of the members of i's cluster
      double h = 0.0;
      for (int p = 0; p < mi; ++p)
        for (int q = 0; q < mj; ++q)
          h = fma(J[(int64_t)p * n + si + a] * H[(int64_t)(sj + q) * n + si + p],
                  J[(int64_t)q * n + j], h);
      v = fma(J[(int64_t)(i - si) * n + si + a], h / (lam[j] - lam[si + a]), v);
    }
  }
  for (int q = 0; q < mj; ++q) {
    const double rt = XX[(int64_t)(sj + q) * n + i] - (i == sj + q ? 1.0 : 0.0);
    v = fma(-0.5 * rt, J[(int64_t)q * n + j], v);
  }
  M[e] = v;
}

// M = (3 - X^T X) / 2, and the largest |X^T X - 1|.
__global__ void __launch_bounds__(256) k_refine_orth(int n, const double *__restrict__ XX,
                                                     RefineStat *st, double *__restrict__ M) {
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  unsigned long long r = 0;
  if (e < (int64_t)n * n) {
    const double one = e % n == e / n ? 1.0 : 0.0, rt = XX[e] - one;
    M[e] = fma(-0.5, rt, one);
    r = (unsigned long long)__double_as_longlong(rt) & 0x7fffffffffffffffULL;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r = max(r, __shfl_xor_sync(0xffffffffu, r, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&st->res, r);
}

int EighRefiner::reserve(Ctx *c, cusolverDnHandle_t sol, int n) {
  nmax = 0;
  if (n < 2 || n > kEighRefineMax) return BQC_OK;
  const size_t nn = (size_t)n * n;
  if (X.alloc(c, nn * 8) != BQC_OK || T.alloc(c, nn * 8) != BQC_OK || S.alloc(c, nn * 8) != BQC_OK ||
      XX.alloc(c, nn * 8) != BQC_OK || Af.alloc(c, nn * 4) != BQC_OK ||
      wf.alloc(c, (size_t)n * 4) != BQC_OK ||
      cusolverDnSsyevd_bufferSize(sol, CUSOLVER_EIG_MODE_VECTOR, CUBLAS_FILL_MODE_LOWER, n,
                                  Af.as<float>(), n, wf.as<float>(),
                                  &lwork) != CUSOLVER_STATUS_SUCCESS ||
      work.alloc(c, (size_t)std::max(lwork, 1) * 4) != BQC_OK ||
      J.alloc(c, (size_t)kClusterMax * n * 8) != BQC_OK || idx.alloc(c, (size_t)n * 8) != BQC_OK ||
      stat.alloc(c, 256) != BQC_OK)
    return BQC_OK;  // no room: the FP64 decomposition serves
  nmax = n;
  return BQC_OK;
}

int EighRefiner::run(cusolverDnHandle_t sol, const SmallGemm &mm, double *A, int n, double *evals,
                     bool *done, cudaStream_t s) {
  *done = false;
  if (n != nmax) return BQC_OK;
  const int64_t nn = (int64_t)n * n;
  const unsigned gb = (unsigned)((nn + 255) / 256);
  RefineStat *st = stat.as<RefineStat>();
  int *info = reinterpret_cast<int *>(stat.as<char>() + 128);
  double *x = X.as<double>(), *t = T.as<double>(), *sm = S.as<double>(), *xx = XX.as<double>();
  int *start = idx.as<int>(), *size = start + n;
  k_to_f32<<<gb, 256, 0, s>>>(nn, A, Af.as<float>());
  BQC_LAUNCH_CHECK();
  if (cusolverDnSsyevd(sol, CUSOLVER_EIG_MODE_VECTOR, CUBLAS_FILL_MODE_LOWER, n, Af.as<float>(), n,
                       wf.as<float>(), work.as<float>(), lwork, info) != CUSOLVER_STATUS_SUCCESS)
    return BQC_OK;
  k_to_f64<<<gb, 256, 0, s>>>(nn, Af.as<float>(), x);
  BQC_LAUNCH_CHECK();
  BQC_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(RefineStat), s));
  for (int round = 0; round < 5; ++round) {
    if (round) BQC_CUDA_TRY(cudaMemsetAsync(st, 0, 3 * sizeof(unsigned long long), s));
    BQC_TRY(mm.run(true, false, n, n, n, x, n, x, n, xx, n, s));
    BQC_TRY(mm.run(false, false, n, n, n, A, n, x, n, t, n, s));
    BQC_TRY(mm.run(true, false, n, n, n, x, n, t, n, sm, n, s));
    k_refine_h<<<gb, 256, 0, s>>>(n, sm, xx, t, st);
    BQC_LAUNCH_CHECK();
    k_refine_clusters<<<(unsigned)((n + 63) / 64), 64, 0, s>>>(n, t, st, J.as<double>(), evals,
                                                               start, size);
    BQC_LAUNCH_CHECK();
    k_refine_m<<<gb, 256, 0, s>>>(n, t, xx, J.as<double>(), evals, start, size, st, sm);
    BQC_LAUNCH_CHECK();
    BQC_TRY(mm.run(false, false, n, n, n, x, n, sm, n, t, n, s));
    std::swap(x, t);
    if (round < 2) continue;  // two rounds always; then look before another one
    BQC_TRY(mm.run(true, false, n, n, n, x, n, x, n, xx, n, s));
    k_refine_orth<<<gb, 256, 0, s>>>(n, xx, st, sm);
    BQC_LAUNCH_CHECK();
    BQC_TRY(mm.run(false, false, n, n, n, x, n, sm, n, t, n, s));
    std::swap(x, t);
    struct {
      RefineStat st;
      char pad[128 - sizeof(RefineStat)];
      int info;
    } h;
    BQC_CUDA_TRY(cudaMemcpyAsync(&h, stat.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    BQC_CUDA_TRY(cudaStreamSynchronize(s));
    double g, top, res;
    std::memcpy(&g, &h.st.g, 8);
    std::memcpy(&top, &h.st.top, 8);
    std::memcpy(&res, &h.st.res, 8);
    if (h.info || h.st.fail || !std::isfinite(g) || !std::isfinite(top) || !std::isfinite(res))
      return BQC_OK;
    if (g <= 1e-12 * top && res <= 1e-9) {
      BQC_CUDA_TRY(cudaMemcpyAsync(A, x, nn * 8, cudaMemcpyDeviceToDevice, s));
      *done = true;
      return BQC_OK;
    }
  }
  return BQC_OK;
}

}  // namespace bqc
