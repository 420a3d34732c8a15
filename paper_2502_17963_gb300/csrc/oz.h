// FP64 matrix products on the FP16 tensor cores by exact slicing (oz.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace bqc {

constexpr int kOzSlices = 7;  // base-256 digits of an operand element
constexpr int kOzKb = 32;     // contraction elements of a k-block

// Where operand element (row r, contraction index k) is read from.
enum OzSrcKind {
  kOzRows = 0,  // p[(k / k2) * s1 + r * ld + k % k2]
  kOzCols = 1,  // r = (z, i), i < n2:  p[z * sz + k * ld + i]
  kOzSym = 2,   // r = (z, m), m < n2:  packed symmetric p[z * sz + tri(max(m, k), min(m, k))]
};
struct OzSrc {
  int kind = kOzRows;
  const double *p = nullptr;
  int64_t rows = 0;
  int K = 0;
  int64_t ld = 0, s1 = 0, sz = 0;
  int k2 = 0;  // kOzRows: inner contraction length (0: K)
  int n2 = 0;  // kOzCols, kOzSym: inner row count (0: rows)
};

// A sliced operand in device memory: [k-block][slice][row][32] FP16 digits and
// one exponent per (contraction split, row).
struct OzOperand {
  const void *slices = nullptr;
  const int *exps = nullptr;
  int64_t rows = 0;
  int K = 0;
  int64_t stride = 0;  // rows of the whole sliced array when this is a row range of it (0: rows)
};

constexpr int oz_kblocks(int K) { return (K + kOzKb - 1) / kOzKb; }
inline size_t oz_align(size_t b) { return (b + 1023) & ~(size_t)1023; }
inline size_t oz_slice_bytes(int64_t rows, int K) {
  return oz_align((size_t)rows * oz_kblocks(K) * kOzSlices * kOzKb * 2);
}
inline size_t oz_exp_bytes(int64_t rows, int nsplit) {
  return oz_align((size_t)rows * nsplit * sizeof(int));
}
// k-blocks of one of at most nsplit equal contraction splits, and their count
inline int oz_split_kb(int K, int nsplit) {
  const int nkb = oz_kblocks(K);
  return (nkb + nsplit - 1) / nsplit;
}
inline int oz_splits(int K, int nsplit) {
  const int nkb = oz_kblocks(K), per = oz_split_kb(K, nsplit);
  return (nkb + per - 1) / per;
}

// Slices a source; exponents per row and split of split_kb k-blocks.
int oz_slice(const OzSrc &src, int split_kb, void *slices, int *exps, cudaStream_t s);

enum OzTri { kOzFull = 0, kOzLower = 1 };

// out[split][n * ldo + m] = beta out + alpha sum_k A(m, k) B(n, k), m < A.rows,
// n < B.rows, alpha = +-1, beta = 0 or 1; split covers split_kb k-blocks and
// its result goes to out + split * split_stride.  kOzLower (A.rows == B.rows):
// only tiles that hold an element with n <= m.
int oz_gemm(const OzOperand &A, const OzOperand &B, int split_kb, int alpha, int beta, double *out,
            int64_t ldo, int64_t split_stride, int tri, int *flag, cudaStream_t s);

// out (n x n, symmetric) = sum over splits of the lower parts of the partials
// (element (m, c), c <= m, at split * split_stride + c * ldp + m); both
// triangles are written.
int oz_sym_reduce(const double *part, int nsplit, int64_t split_stride, int n, int64_t ldp,
                  double *out, cudaStream_t s);

// 128 x 64 output tiles of a product (lower: of a symmetric one).
inline int64_t oz_tiles(int64_t M, int64_t N, bool lower) {
  const int64_t mt = (M + 127) / 128, nt = (N + 63) / 64;
  return lower ? mt * (mt - 1) + (nt < 2 * mt ? nt : 2 * mt) : mt * nt;
}

}  // namespace bqc
