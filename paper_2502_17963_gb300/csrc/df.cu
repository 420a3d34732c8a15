// Density-fitting tensor and the J/K build (Sec. 2.2).
//
// Stored mode (the three-index tensor depends only on basis and geometry, so
// it is computed once and kept):
//   V = (P|Q) -> L (Cholesky) -> raw (Q|mu nu) packed lower triangle in FP64
//   -> B = L^{-1} raw in place -> optional TF32-rounded full-square shadow.
// Each Fock build then makes two passes over B, as the paper notes for the
// Coulomb matrix: the X pass (X_P = B_P C_occ, with w_P = <X_P, C_occ>) and
// the J pass (J = sum_P w_P B_P); K = sum_P X_P X_P^T.
// Direct mode (regenerated per aux block at every build): see direct.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>

#include "bqc_internal.h"
#include "df_internal.h"
#include "gemm64.cuh"
#include "oz.h"

namespace bqc {

// w[P] = sum_{mu,i} X[P][mu][i] C[mu][i]  (one block of up to 1024 threads per
// P, FP64).  Bound by the load latency of the few blocks a chunk of P gives:
// four independent sums a thread keep four loads of each operand in flight.
__global__ void __launch_bounds__(1024) k_wdot(const double *X, const double *C, int64_t nc,
                                               double *w) {
  const int P = blockIdx.x;
  const double *x = X + (int64_t)P * nc;
  const int64_t st = blockDim.x;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int64_t i = threadIdx.x;
  for (; i + 3 * st < nc; i += 4 * st) {
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = fma(x[i + k * st], __ldg(C + i + k * st), s[k]);
  }
  for (; i < nc; i += st) s[0] = fma(x[i], __ldg(C + i), s[0]);
  __shared__ double red[1024];
  red[threadIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) w[P] = red[0];
}

// J pass over packed FP64 B: out[col] = sum_{P in [Pa, Pb)} w_P B[P][col] for
// the two adjacent columns c2, c2 + 1 a thread owns; P streams in increasing
// order (one read of B, coalesced), eight 16-byte loads in flight per thread,
// or, for an odd number of columns (every second row off a 16-byte boundary:
// half of all sizes), sixteen 8-byte ones.
__device__ __forceinline__ void jpass64_cols(const double *__restrict__ B,
                                             const double *__restrict__ w, int Pa, int Pb,
                                             int64_t npair, int64_t c2, double *__restrict__ out) {
  double a0 = 0.0, a1 = 0.0;
  const bool two = c2 + 1 < npair, even = npair % 2 == 0;
  const double *b = B + c2 + (int64_t)Pa * npair;
  const int o1 = two ? 1 : 0;
  auto load = [&](int64_t k) {
    const double *p = b + k * npair;
    return even ? __ldg(reinterpret_cast<const double2 *>(p))
                : make_double2(__ldg(p), __ldg(p + o1));
  };
  int P = Pa;
  for (; P + 8 <= Pb; P += 8, b += 8 * npair) {
    double2 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = load(k);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double wp = __ldg(w + P + k);
      a0 = fma(wp, v[k].x, a0);
      a1 = fma(wp, v[k].y, a1);
    }
  }
  for (; P < Pb; ++P, b += npair) {
    const double2 v = load(0);
    const double wp = __ldg(w + P);
    a0 = fma(wp, v.x, a0);
    a1 = fma(wp, v.y, a1);
  }
  out[c2] = a0;
  if (two) out[c2 + 1] = a1;
}

// Jp[y][col] = sum_{P in chunk y} w_P B[P][col]: gridDim.y aux chunks give
// small systems enough blocks; the chunk partials are summed in a fixed order
// by k_unpack_jsum.
__global__ void __launch_bounds__(256) k_jpass64(const double *__restrict__ B,
                                                 const double *__restrict__ w, int naux,
                                                 int64_t npair, double *__restrict__ Jp) {
  const int64_t c2 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 2;
  if (c2 >= npair) return;
  const int per = (naux + gridDim.y - 1) / gridDim.y;
  const int Pa = blockIdx.y * per, Pb = min(naux, Pa + per);
  jpass64_cols(B, w, Pa, Pb, npair, c2, Jp + (int64_t)blockIdx.y * npair);
}

// The same for aux functions [P0, P1), partials into the slices y0 .. y0 +
// gridDim.y - 1 (the pieces of the split-FP16 build's pipeline).
__global__ void __launch_bounds__(256) k_jpass64_range(const double *__restrict__ B,
                                                       const double *__restrict__ w, int P0,
                                                       int P1, int64_t npair, int y0,
                                                       double *__restrict__ Jp) {
  const int64_t c2 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 2;
  if (c2 >= npair) return;
  const int per = (P1 - P0 + gridDim.y - 1) / gridDim.y;
  const int Pa = P0 + blockIdx.y * per, Pb = min(P1, Pa + per);
  jpass64_cols(B, w, Pa, Pb, npair, c2, Jp + (int64_t)(y0 + blockIdx.y) * npair);
}

// (sh, sl) += (wh + wl) (bh + bl) in float-float arithmetic: the exact
// product wh*bh (its rounding error from one FMA), the two cross terms (wl*bl
// is below 2^-48 of the product), and a two-sum into the running pair.
__device__ __forceinline__ void ff_acc(float &sh, float &sl, float wh, float wl, float bh,
                                       float bl) {
  const float p = wh * bh;
  float e = fmaf(wh, bh, -p);
  e = fmaf(wh, bl, e);
  e = fmaf(wl, bh, e);
  const float t = sh + p;
  const float bp = t - sh;
  const float err = (sh - (t - bp)) + (p - bp);
  sh = t;
  sl += err + e;
}

// out[col] = sum_{P in [Pa, Pb)} w_P B[P][col] for the columns c2, c2 + 1 of
// a thread, from the float-pair B (one 16-byte load per P: hi0 lo0 hi1 lo1)
// and float-pair w, accumulated in float-float: the FP32 pipe does what the
// FP64 pipe (1/64 of its rate) would, at ~2^-46 relative per term, so the
// pass runs at the memory's speed.
__device__ __forceinline__ void jpass_ff_cols(const float4 *__restrict__ B2,
                                              const float2 *__restrict__ w2, int Pa, int Pb,
                                              int64_t npair, int64_t c2,
                                              double *__restrict__ out) {
  float h0 = 0.0f, l0 = 0.0f, h1 = 0.0f, l1 = 0.0f;
  const bool two = c2 + 1 < npair, even = npair % 2 == 0;
  const float2 *b = reinterpret_cast<const float2 *>(B2) + c2 + (int64_t)Pa * npair;
  const int o1 = two ? 1 : 0;
  auto load = [&](int64_t k) {  // as in jpass64_cols
    const float2 *p = b + k * npair;
    if (even) return __ldg(reinterpret_cast<const float4 *>(p));
    const float2 x = __ldg(p), y = __ldg(p + o1);
    return make_float4(x.x, x.y, y.x, y.y);
  };
  int P = Pa;
  for (; P + 8 <= Pb; P += 8, b += 8 * npair) {
    float4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = load(k);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float2 wp = __ldg(w2 + P + k);
      ff_acc(h0, l0, wp.x, wp.y, v[k].x, v[k].y);
      ff_acc(h1, l1, wp.x, wp.y, v[k].z, v[k].w);
    }
  }
  for (; P < Pb; ++P, b += npair) {
    const float4 v = load(0);
    const float2 wp = __ldg(w2 + P);
    ff_acc(h0, l0, wp.x, wp.y, v.x, v.y);
    ff_acc(h1, l1, wp.x, wp.y, v.z, v.w);
  }
  out[c2] = (double)h0 + (double)l0;
  if (two) out[c2 + 1] = (double)h1 + (double)l1;
}

__global__ void __launch_bounds__(256) k_jpass_ff_range(const float4 *__restrict__ B2,
                                                        const float2 *__restrict__ w2, int P0,
                                                        int P1, int64_t npair, int y0,
                                                        double *__restrict__ Jp) {
  const int64_t c2 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 2;
  if (c2 >= npair) return;
  const int per = (P1 - P0 + gridDim.y - 1) / gridDim.y;
  const int Pa = P0 + blockIdx.y * per, Pb = min(P1, Pa + per);
  jpass_ff_cols(B2, w2, Pa, Pb, npair, c2, Jp + (int64_t)(y0 + blockIdx.y) * npair);
}

// Grouped J pass of independent problems in one launch: problem k owns the
// blocks [off[k], off[k + 1]) as xb[k] column blocks times sp[k] aux chunks.
struct JGroup {
  const double *B[kMaxGroup];
  const double *w[kMaxGroup];
  const float4 *B2[kMaxGroup];  // float-pair B and w (ff variant)
  const float2 *w2[kMaxGroup];
  double *Jp[kMaxGroup];
  double *J[kMaxGroup];
  int64_t npair[kMaxGroup];
  int naux[kMaxGroup], sp[kMaxGroup], xb[kMaxGroup], n[kMaxGroup];
  int off[kMaxGroup + 1];
  int nprob;
};

template <bool FF>
__global__ void __launch_bounds__(256) k_jpass64_grp(const __grid_constant__ JGroup g) {
  const int bid = blockIdx.x;
  int k = 0;
  while (k + 1 < g.nprob && bid >= g.off[k + 1]) ++k;
  const int lb = bid - g.off[k], y = lb / g.xb[k], xb = lb % g.xb[k];
  const int64_t npair = g.npair[k];
  const int64_t c2 = ((int64_t)xb * blockDim.x + threadIdx.x) * 2;
  if (c2 >= npair) return;
  const int per = (g.naux[k] + g.sp[k] - 1) / g.sp[k];
  const int Pa = y * per, Pb = min(g.naux[k], Pa + per);
  if (FF)
    jpass_ff_cols(g.B2[k], g.w2[k], Pa, Pb, npair, c2, g.Jp[k] + (int64_t)y * npair);
  else
    jpass64_cols(g.B[k], g.w[k], Pa, Pb, npair, c2, g.Jp[k] + (int64_t)y * npair);
}

__device__ __forceinline__ void unpack_jsum_one(const double *Jp, int nsplit, int64_t npair, int n,
                                                double *J, int64_t i) {
  if (i >= (int64_t)n * n) return;
  const int64_t r = i / n, c = i % n;
  const int64_t hi = r > c ? r : c, lo = r > c ? c : r;
  const int64_t q = hi * (hi + 1) / 2 + lo;
  double s = Jp[q];
#pragma unroll 8
  for (int y = 1; y < nsplit; ++y) s += Jp[(int64_t)y * npair + q];
  J[i] = s;
}

__global__ void k_unpack_jsum(const double *Jp, int nsplit, int64_t npair, int n, double *J) {
  unpack_jsum_one(Jp, nsplit, npair, n, J, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void k_unpack_jsum_grp(const __grid_constant__ JGroup g) {
  const int k = blockIdx.y;
  unpack_jsum_one(g.Jp[k], g.sp[k], g.npair[k], g.n[k], g.J[k],
                  (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// aux chunks of the J pass: enough blocks for four per SM, at least min_aux P
// each.  64 for the passes of mixed builds (float-pair or FP64): their chunks are
// part of the mixed Fock matrix's last bits, which a staged SCF amplifies (see
// scf.cu; with 8 in the TF32x3 build its (H2O)_5 result moved by 1.3e-9).  8 for
// the J pass of FP64 builds, where 64 left a small system on a few blocks, each
// a serial stream.
int jpass_split(int64_t npair, int naux, int min_aux) {
  const int64_t blocks = (npair / 2 + 256) / 256;
  int sp = (int)std::min<int64_t>(min_aux >= kMixedJAux ? 16 : 64,
                                  (4 * (int64_t)sm_count() + blocks - 1) / blocks);
  sp = std::max(1, std::min(sp, naux / min_aux));
  return sp;
}

// Packed lower triangle -> full symmetric N x N.
__global__ void k_unpack_sym(const double *Jp, int n, double *J) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * n) return;
  const int64_t r = i / n, c = i % n;
  const int64_t hi = r > c ? r : c, lo = r > c ? c : r;
  J[i] = Jp[hi * (hi + 1) / 2 + lo];
}

int jpass_fp64(Df *df, double *J, cudaStream_t s, int min_aux) {
  const int n = df->basis->nbf, naux = df->naux_loc;
  const int64_t npair = df->npair;
  if (!df->B64.p) return BQC_E_INVALID;
  // as many chunks as there are slices for (AUTO mode may leave fewer)
  const int sp = (int)std::min<size_t>(jpass_split(npair, naux, min_aux),
                                       df->Jp.n / ((size_t)npair * 8));
  if (sp < jpass_split(npair, naux)) return BQC_E_INVALID;
  k_jpass64<<<dim3((unsigned)((npair / 2 + 256) / 256), (unsigned)sp), 256, 0, s>>>(
      df->B64.as<double>(), df->w.as<double>(), naux, npair, df->Jp.as<double>());
  BQC_LAUNCH_CHECK();
  k_unpack_jsum<<<(unsigned)(((int64_t)n * n + 255) / 256), 256, 0, s>>>(df->Jp.as<double>(), sp,
                                                                         npair, n, J);
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}


// Packed lower triangle of a symmetric N x N matrix with the off-diagonal
// doubled: D2[mu(mu+1)/2 + nu] = (2 - delta_mu nu) D[mu][nu] (so that
// B_P : D = sum over the packed entries of B_P D2).
__global__ void k_pack_sym2(const double *__restrict__ D, int n, double *__restrict__ D2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * (n + 1) / 2) return;
  int mu = (int)((sqrt(8.0 * (double)i + 1.0) - 1.0) * 0.5);
  while ((int64_t)(mu + 1) * (mu + 2) / 2 <= i) ++mu;
  while ((int64_t)mu * (mu + 1) / 2 > i) --mu;
  const int nu = (int)(i - (int64_t)mu * (mu + 1) / 2);
  D2[i] = (mu == nu ? 1.0 : 2.0) * D[(int64_t)mu * n + nu];
}

// w[P] = sum_c B[P][c] D2[c] over the packed FP64 B (one block per P; four
// loads of B in flight a thread).
__global__ void __launch_bounds__(256) k_bdot(const double *__restrict__ B, int64_t npair,
                                              const double *__restrict__ D2, double *w) {
  const double *b = B + (int64_t)blockIdx.x * npair;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int64_t c = threadIdx.x;
  for (; c + 3 * 256 < npair; c += 4 * 256) {
    double v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __ldg(b + c + 256 * k);
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = fma(v[k], __ldg(D2 + c + 256 * k), s[k]);
  }
  for (; c < npair; c += 256) s[0] = fma(__ldg(b + c), __ldg(D2 + c), s[0]);
  __shared__ double red[256];
  red[threadIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) w[blockIdx.x] = red[0];
}

// The packed, off-diagonal-doubled density as float pairs (hi, lo).
__global__ void k_pack_sym2_ff(const double *__restrict__ D, int n, float2 *__restrict__ D2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * (n + 1) / 2) return;
  int mu = (int)((sqrt(8.0 * (double)i + 1.0) - 1.0) * 0.5);
  while ((int64_t)(mu + 1) * (mu + 2) / 2 <= i) ++mu;
  while ((int64_t)mu * (mu + 1) / 2 > i) --mu;
  const int nu = (int)(i - (int64_t)mu * (mu + 1) / 2);
  const double v = (mu == nu ? 1.0 : 2.0) * D[(int64_t)mu * n + nu];
  const float h = (float)v;
  D2[i] = make_float2(h, (float)(v - (double)h));
}

// w[P] = sum_c B[P][c] D2[c] from the float pairs of B and D2 in float-float
// arithmetic (one block per P; the block's partial pairs summed in FP64);
// also w as float pairs for the J pass.  Bound by the read of B: four
// independent 16-byte loads of it in flight a thread (a row that starts off a
// 16-byte boundary is peeled by one element).
__global__ void __launch_bounds__(256) k_bdot_ff(const float2 *__restrict__ B2, int64_t npair,
                                                 const float2 *__restrict__ D2, double *w,
                                                 float2 *w2) {
  const int64_t at = (int64_t)blockIdx.x * npair;
  const int peel = (int)(at & 1);
  const float2 *b = B2 + at + peel, *d = D2 + peel;
  const int64_t n2 = (npair - peel) / 2;
  float h[4] = {0.0f, 0.0f, 0.0f, 0.0f}, l[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const float4 *b4 = reinterpret_cast<const float4 *>(b);
  int64_t c = threadIdx.x;
  for (; c + 3 * 256 < n2; c += 4 * 256) {
    float4 x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = __ldg(b4 + c + 256 * k);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 d0 = __ldg(d + 2 * (c + 256 * k)), d1 = __ldg(d + 2 * (c + 256 * k) + 1);
      ff_acc(h[k], l[k], d0.x, d0.y, x[k].x, x[k].y);
      ff_acc(h[k], l[k], d1.x, d1.y, x[k].z, x[k].w);
    }
  }
  for (; c < n2; c += 256) {
    const float4 x = __ldg(b4 + c);
    const float2 d0 = __ldg(d + 2 * c), d1 = __ldg(d + 2 * c + 1);
    ff_acc(h[0], l[0], d0.x, d0.y, x.x, x.y);
    ff_acc(h[0], l[0], d1.x, d1.y, x.z, x.w);
  }
  if (threadIdx.x == 0) {  // the peeled first and an odd last element
    const float2 *b0 = B2 + at;
    if (peel) ff_acc(h[1], l[1], D2[0].x, D2[0].y, b0[0].x, b0[0].y);
    const int64_t e = npair - 1;
    if ((npair - peel) & 1) ff_acc(h[2], l[2], D2[e].x, D2[e].y, b0[e].x, b0[e].y);
  }
  __shared__ double red[256];
  red[threadIdx.x] = (((double)h[0] + (double)l[0]) + ((double)h[1] + (double)l[1])) +
                     (((double)h[2] + (double)l[2]) + ((double)h[3] + (double)l[3]));
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double v = red[0];
    w[blockIdx.x] = v;
    const float fh = (float)v;
    w2[blockIdx.x] = make_float2(fh, (float)(v - (double)fh));
  }
}

int jff_of_density(Df *df, const double *D, double *D2, double *J, cudaStream_t s) {
  if (df->mode != BQC_DF_STORED || !df->B2f.p || !df->w2f.p) return BQC_E_INVALID;
  const int n = df->basis->nbf;
  float2 *d2 = reinterpret_cast<float2 *>(D2);  // npair doubles hold npair float pairs
  k_pack_sym2_ff<<<(unsigned)((df->npair + 255) / 256), 256, 0, s>>>(D, n, d2);
  BQC_LAUNCH_CHECK();
  k_bdot_ff<<<(unsigned)df->naux_loc, 256, 0, s>>>(df->B2f.as<float2>(), df->npair, d2,
                                                   df->w.as<double>(), df->w2f.as<float2>());
  BQC_LAUNCH_CHECK();
  const int sp = jpass_split(df->npair, df->naux_loc);
  BQC_TRY(jpass_ff_range(df, 0, df->naux_loc, 0, s));
  return jpass_unpack(df, sp, J, s);
}

int jfp64_of_density(Df *df, const double *D, double *D2, double *J, cudaStream_t s) {
  if (df->mode != BQC_DF_STORED || !df->B64.p) return BQC_E_INVALID;
  const int n = df->basis->nbf;
  k_pack_sym2<<<(unsigned)((df->npair + 255) / 256), 256, 0, s>>>(D, n, D2);
  BQC_LAUNCH_CHECK();
  k_bdot<<<(unsigned)df->naux_loc, 256, 0, s>>>(df->B64.as<double>(), df->npair, D2,
                                                df->w.as<double>());
  BQC_LAUNCH_CHECK();
  return jpass_fp64(df, J, s);
}

int jpass_fp64_range(Df *df, int P0, int P1, int y0, cudaStream_t s) {
  const int64_t npair = df->npair;
  const int sp = jpass_split(npair, P1 - P0);
  if (df->Jp.n < (size_t)(y0 + sp) * npair * 8) return BQC_E_INVALID;
  k_jpass64_range<<<dim3((unsigned)((npair / 2 + 256) / 256), (unsigned)sp), 256, 0, s>>>(
      df->B64.as<double>(), df->w.as<double>(), P0, P1, npair, y0, df->Jp.as<double>());
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

int jpass_ff_alloc(Df *df) {
  const int64_t count = (int64_t)df->naux_loc * df->npair;
  BQC_TRY(df->B2f.alloc(df->ctx, (size_t)count * 8));
  return df->w2f.alloc(df->ctx, (size_t)df->naux_loc * 8);
}

int jpass_ff_range(Df *df, int P0, int P1, int y0, cudaStream_t s) {
  const int64_t npair = df->npair;
  const int sp = jpass_split(npair, P1 - P0);
  if (!df->B2f.p || !df->w2f.p || df->Jp.n < (size_t)(y0 + sp) * npair * 8)
    return BQC_E_INVALID;
  k_jpass_ff_range<<<dim3((unsigned)((npair / 2 + 256) / 256), (unsigned)sp), 256, 0, s>>>(
      df->B2f.as<float4>(), df->w2f.as<float2>(), P0, P1, npair, y0, df->Jp.as<double>());
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

int jpass_unpack(Df *df, int nslice, double *J, cudaStream_t s) {
  const int n = df->basis->nbf;
  k_unpack_jsum<<<(unsigned)(((int64_t)n * n + 255) / 256), 256, 0, s>>>(df->Jp.as<double>(),
                                                                         nslice, df->npair, n, J);
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

int group_jpass(Df *const *dfs, double *const *J, int n, cudaStream_t s) {
  if (n <= 0 || n > kMaxGroup) return BQC_E_INVALID;
  JGroup g;
  std::memset(&g, 0, sizeof(g));
  int blocks = 0;
  bool ff = true;
  int64_t nn_max = 0;
  for (int k = 0; k < n; ++k) {
    Df *df = dfs[k];
    if (!df->B64.p) return BQC_E_INVALID;
    const int64_t npair = df->npair;
    const int naux = df->naux_loc, nb = df->basis->nbf;
    const int sp = jpass_split(npair, naux);
    if (df->Jp.n < (size_t)sp * npair * 8) return BQC_E_INVALID;
    g.B[k] = df->B64.as<double>();
    g.w[k] = df->w.as<double>();
    g.B2[k] = df->B2f.as<float4>();
    g.w2[k] = df->w2f.as<float2>();
    ff = ff && df->B2f.p && df->w2f.p;
    g.Jp[k] = df->Jp.as<double>();
    g.J[k] = J[k];
    g.npair[k] = npair;
    g.naux[k] = naux;
    g.sp[k] = sp;
    g.xb[k] = (int)((npair / 2 + 256) / 256);
    g.n[k] = nb;
    g.off[k] = blocks;
    blocks += g.xb[k] * sp;
    nn_max = std::max(nn_max, (int64_t)nb * nb);
  }
  g.off[n] = blocks;
  g.nprob = n;
  if (ff)
    k_jpass64_grp<true><<<(unsigned)blocks, 256, 0, s>>>(g);
  else
    k_jpass64_grp<false><<<(unsigned)blocks, 256, 0, s>>>(g);
  BQC_LAUNCH_CHECK();
  k_unpack_jsum_grp<<<dim3((unsigned)((nn_max + 255) / 256), (unsigned)n), 256, 0, s>>>(g);
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

// ------------------------------------------------ small molecules (FP64) --
// Up to kSmallN functions a Fock build is a few microseconds of DFMA work, and
// tiles of 64 or 128 would be mostly padding and too few to fill the chip.
// One block per aux function does everything that needs B_P while it is in
// shared memory: X_P = B_P C, w_P, and its contributions to K and J (packed
// lower triangles, one slice per block, accumulated by their owner threads
// over the block's aux functions); a second kernel sums the slices.
constexpr int kSmallN = 112;

__global__ void __launch_bounds__(256) k_jk64_small(const double *__restrict__ B,
                                                    const double *__restrict__ C, int n, int no,
                                                    int naux, double *__restrict__ w,
                                                    double *__restrict__ part) {
  extern __shared__ double sm[];
  const int npair = n * (n + 1) / 2, ldb = n | 1, ldx = no | 1, t = threadIdx.x;
  double *Bs = sm, *Cs = Bs + n * ldb, *Xs = Cs + n * no;
  __shared__ double red[8];
  double *pk = part + (int64_t)blockIdx.x * 2 * npair, *pj = pk + npair;
  for (int e = t; e < n * no; e += 256) Cs[e] = C[e];
  for (int P = blockIdx.x; P < naux; P += gridDim.x) {
    const double *b = B + (int64_t)P * npair;
    for (int q = t; q < npair; q += 256) {
      int mu = (int)((sqrtf(8.0f * q + 1.0f) - 1.0f) * 0.5f);
      while ((mu + 1) * (mu + 2) / 2 <= q) ++mu;
      while (mu * (mu + 1) / 2 > q) --mu;
      const int nu = q - mu * (mu + 1) / 2;
      const double v = b[q];
      Bs[mu * ldb + nu] = v;
      Bs[nu * ldb + mu] = v;
    }
    __syncthreads();
    double s = 0.0;
    for (int e = t; e < n * no; e += 256) {
      const int mu = e / no, i = e - mu * no;
      double x0 = 0.0, x1 = 0.0;
      int nu = 0;
      for (; nu + 1 < n; nu += 2) {
        x0 = fma(Bs[mu * ldb + nu], Cs[nu * no + i], x0);
        x1 = fma(Bs[mu * ldb + nu + 1], Cs[(nu + 1) * no + i], x1);
      }
      if (nu < n) x0 = fma(Bs[mu * ldb + nu], Cs[nu * no + i], x0);
      x0 += x1;
      Xs[mu * ldx + i] = x0;
      s = fma(x0, Cs[e], s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((t & 31) == 0) red[t >> 5] = s;
    __syncthreads();
    double wp = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) wp += red[k];
    if (t == 0) w[P] = wp;
    const bool first = P == blockIdx.x;
    for (int q = t; q < npair; q += 256) {
      int mu = (int)((sqrtf(8.0f * q + 1.0f) - 1.0f) * 0.5f);
      while ((mu + 1) * (mu + 2) / 2 <= q) ++mu;
      while (mu * (mu + 1) / 2 > q) --mu;
      const int nu = q - mu * (mu + 1) / 2;
      double k0 = first ? 0.0 : pk[q];
      for (int i = 0; i < no; ++i) k0 = fma(Xs[mu * ldx + i], Xs[nu * ldx + i], k0);
      pk[q] = k0;
      pj[q] = fma(wp, Bs[mu * ldb + nu], first ? 0.0 : pj[q]);
    }
    __syncthreads();
  }
}

// K and J (full, symmetric) from the slices: 32 elements and 8 slice classes
// per block, summed in a fixed order.
__global__ void __launch_bounds__(256) k_jk64_small_sum(const double *__restrict__ part, int nslice,
                                                        int n, double *__restrict__ K,
                                                        double *__restrict__ J) {
  __shared__ double t[8][33];
  const int npair = n * (n + 1) / 2, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int q = blockIdx.x * 32 + tx;  // over K's pairs, then J's
  double s = 0.0;
  if (q < 2 * npair)
    for (int k = ty; k < nslice; k += 8) s += part[(int64_t)k * 2 * npair + q];
  t[ty][tx] = s;
  __syncthreads();
  if (ty || q >= 2 * npair) return;
  s = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) s += t[k][tx];
  const int p = q < npair ? q : q - npair;
  int mu = (int)((sqrtf(8.0f * p + 1.0f) - 1.0f) * 0.5f);
  while ((mu + 1) * (mu + 2) / 2 <= p) ++mu;
  while (mu * (mu + 1) / 2 > p) --mu;
  const int nu = p - mu * (mu + 1) / 2;
  double *out = q < npair ? K : J;
  out[mu * n + nu] = s;
  out[nu * n + mu] = s;
}

static size_t jk64_small_smem(int n, int no) {
  return ((size_t)n * (n | 1) + (size_t)n * no + (size_t)n * (no | 1)) * 8;
}

// With nearly as many occupied orbitals as functions B_P, C and X_P may not fit
// beside one another in shared memory.
static bool jk64_small(int n, int no) {
  return n <= kSmallN && jk64_small_smem(n, no) <= (size_t)220 * 1024;
}

static int jk64_small_slices(int naux) { return std::min(naux, 2 * sm_count()); }

// Bytes of the FP64 X buffer: X, or the scratch of the small and the sliced
// builds where that is more (at most 32 MiB more).
static size_t x64_bytes(int n, int naux, int no);

static int jk_fp64_small(Df *df, const double *C, double *J, double *K, cudaStream_t s) {
  const int n = df->basis->nbf, naux = df->naux_loc, no = df->basis->nocc;
  const int npair = n * (n + 1) / 2, nsl = jk64_small_slices(naux);
  const size_t smem = jk64_small_smem(n, no);
  BQC_CUDA_TRY(cudaFuncSetAttribute(k_jk64_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem));
  df->mark(0, s);
  df->mark(1, s);
  k_jk64_small<<<(unsigned)nsl, 256, smem, s>>>(df->B64.as<double>(), C, n, no, naux,
                                                df->w.as<double>(), df->X64.as<double>());
  BQC_LAUNCH_CHECK();
  df->mark(2, s);
  df->mark(3, s);
  k_jk64_small_sum<<<(unsigned)((2 * npair + 31) / 32), 256, 0, s>>>(df->X64.as<double>(), nsl, n,
                                                                     K, J);
  BQC_LAUNCH_CHECK();
  df->mark(4, s);
  return BQC_OK;
}

// FP64 X pass and K on the tensor cores (oz.cu), over chunks of pc aux
// functions.  The handle's X buffer (Naux N nocc doubles) is the scratch: a
// chunk's sliced B, its X (FP64), its sliced X, and the K partials.
struct OzJkPlan {
  int pc = 0;               // aux functions per chunk (0: does not fit)
  int ns = 0;               // splits of the K contraction of a chunk
  size_t cs, ce, bs, be, x, xs, xe, kp, total;  // offsets, and the bytes used
};

static OzJkPlan oz_jk_layout(int n, int no, int pc, int ns) {
  OzJkPlan p;
  p.pc = pc;
  p.ns = oz_splits(pc * no, ns);
  size_t o = 0;
  auto take = [&o](size_t b) {
    const size_t at = o;
    o += oz_align(b);
    return at;
  };
  p.kp = take((size_t)p.ns * n * n * 8);
  p.cs = take(oz_slice_bytes(no, n));
  p.ce = take(oz_exp_bytes(no, 1));
  p.bs = take(oz_slice_bytes((int64_t)pc * n, n));
  p.be = take(oz_exp_bytes((int64_t)pc * n, 1));
  p.x = take((size_t)pc * n * no * 8);
  p.xs = take(oz_slice_bytes(n, pc * no));
  p.xe = take(oz_exp_bytes(n, p.ns));
  p.total = o;
  return p;
}

// Splits of a K contraction of length K: the count whose tiles fill whole waves
// best, splits of at least one accumulation chain (128).
static int oz_k_splits(int n, int K) {
  const int64_t tiles = oz_tiles(n, n, true);
  const int nsm = sm_count();
  int ns = 1;
  double eff = 0.0;
  for (int c = 1; c <= 2 * nsm && (c == 1 || c * 128 <= K); ++c) {
    const int64_t items = tiles * c;
    const double e = (double)items / ((double)((items + nsm - 1) / nsm) * nsm);
    if (e > eff + 1e-3) {
      eff = e;
      ns = c;
    }
    if (items >= 2 * nsm) break;
  }
  return ns;
}

static OzJkPlan oz_jk_plan(int n, int naux, int no, size_t bytes) {
  OzJkPlan best;
  for (int chunks = 1; chunks <= 64 && chunks <= naux; ++chunks) {
    const int pc = (naux + chunks - 1) / chunks;
    OzJkPlan p = oz_jk_layout(n, no, pc, oz_k_splits(n, pc * no));
    if (p.total <= bytes) return p;
  }
  return best;
}

static int oz_rows_of_b(const double *b, int64_t npair, int n, int np, void *slices, int *exps,
                        OzOperand *o, cudaStream_t s);
static int oz_rows_of_x(const double *X, int n, int no, int np, int ns, void *slices, int *exps,
                        OzOperand *o, cudaStream_t s);
static int oz_rows_of_c(const double *C, int n, int no, void *slices, int *exps, OzOperand *o,
                        cudaStream_t s);

static size_t x64_bytes(int n, int naux, int no) {
  const size_t x = (size_t)naux * n * no * 8;
  const size_t more = jk64_small(n, no) ? (size_t)jk64_small_slices(naux) * n * (n + 1) * 8
                                   : oz_jk_plan(n, naux, no, SIZE_MAX).total;
  return std::max(x, std::min<size_t>(more, (size_t)32 << 20));
}

static int jk_fp64_oz(Df *df, const OzJkPlan &p, const double *C, double *J, double *K,
                      cudaStream_t s) {
  const int n = df->basis->nbf, naux = df->naux_loc, no = df->basis->nocc;
  char *scr = df->X64.as<char>();
  double *X = reinterpret_cast<double *>(scr + p.x), *kp = reinterpret_cast<double *>(scr + p.kp);
  auto ints = [scr](size_t at) { return reinterpret_cast<int *>(scr + at); };
  df->mark(0, s);
  df->mark(1, s);
  OzOperand oc, ob, ox;
  BQC_TRY(oz_rows_of_c(C, n, no, scr + p.cs, ints(p.ce), &oc, s));
  const int ns = p.ns;
  for (int P0 = 0; P0 < naux; P0 += p.pc) {
    const int np = std::min(p.pc, naux - P0);
    BQC_TRY(oz_rows_of_b(df->B64.as<double>() + (int64_t)P0 * df->npair, df->npair, n, np,
                         scr + p.bs, ints(p.be), &ob, s));
    BQC_TRY(oz_gemm(oc, ob, oz_kblocks(n), 1, 0, X, no, 0, 0, df->ctx->flag, s));
    k_wdot<<<np, 1024, 0, s>>>(X, C, (int64_t)n * no, df->w.as<double>() + P0);
    BQC_LAUNCH_CHECK();
    // K partials; a short last chunk may have fewer splits than the others, and
    // adds to the first ones
    df->mark_k(s);
    BQC_TRY(oz_rows_of_x(X, n, no, np, ns, scr + p.xs, ints(p.xe), &ox, s));
    const int kb = oz_split_kb(ox.K, ns);
    BQC_TRY(oz_gemm(ox, ox, kb, 1, P0 > 0, kp, n, (int64_t)n * n, 1, df->ctx->flag, s));
    df->mark_k(s);
  }
  df->mark(2, s);
  BQC_TRY(jpass_fp64(df, J, s));
  df->mark(3, s);
  BQC_TRY(oz_sym_reduce(kp, ns, (int64_t)n * n, n, n, K, s));
  df->mark(4, s);
  return BQC_OK;
}

// Rows (P, mu) of np packed symmetric matrices as a sliced operand.
static int oz_rows_of_b(const double *b, int64_t npair, int n, int np, void *slices, int *exps,
                        OzOperand *o, cudaStream_t s) {
  OzSrc x;
  x.kind = kOzSym;
  x.p = b;
  x.rows = (int64_t)np * n;
  x.n2 = n;
  x.sz = npair;
  x.K = n;
  o->slices = slices;
  o->exps = exps;
  o->rows = x.rows;
  o->K = n;
  return oz_slice(x, oz_kblocks(n), slices, exps, s);
}

// Rows mu of np matrices X[P][mu][i], contraction (P, i), in at most ns splits.
static int oz_rows_of_x(const double *X, int n, int no, int np, int ns, void *slices, int *exps,
                        OzOperand *o, cudaStream_t s) {
  OzSrc x;
  x.kind = kOzRows;
  x.p = X;
  x.rows = n;
  x.K = np * no;
  x.k2 = no;
  x.s1 = (int64_t)n * no;
  x.ld = no;
  o->slices = slices;
  o->exps = exps;
  o->rows = n;
  o->K = x.K;
  return oz_slice(x, oz_split_kb(x.K, ns), slices, exps, s);
}

// C_occ^T: rows i, contraction nu.
static int oz_rows_of_c(const double *C, int n, int no, void *slices, int *exps, OzOperand *o,
                        cudaStream_t s) {
  OzSrc c;
  c.kind = kOzCols;
  c.p = C;
  c.rows = no;
  c.K = n;
  c.ld = no;
  o->slices = slices;
  o->exps = exps;
  o->rows = no;
  o->K = n;
  return oz_slice(c, oz_kblocks(n), slices, exps, s);
}

static size_t x_of_b_fixed(int n, int no) { return oz_slice_bytes(no, n) + oz_exp_bytes(no, 1); }

size_t x_of_b_bytes(int n, int no, int np) {
  return x_of_b_fixed(n, no) + oz_slice_bytes((int64_t)np * n, n) +
         oz_exp_bytes((int64_t)np * n, 1);
}

int x_of_b(Ctx *ctx, const double *b, int64_t npair, const double *C, int n, int no, int np,
           double *X, void *scratch, size_t bytes, cudaStream_t s) {
  int pc = std::min(np, 1 << 16);
  while (pc > 0 && x_of_b_bytes(n, no, pc) > bytes) pc = pc > 8 ? pc * 7 / 8 : 0;
  if (n > kSmallN && scratch && pc) {
    char *scr = static_cast<char *>(scratch);
    OzOperand oc, ob;
    BQC_TRY(oz_rows_of_c(C, n, no, scr, reinterpret_cast<int *>(scr + oz_slice_bytes(no, n)), &oc,
                         s));
    scr += x_of_b_fixed(n, no);
    int *be = reinterpret_cast<int *>(scr + oz_slice_bytes((int64_t)pc * n, n));
    for (int P0 = 0; P0 < np; P0 += pc) {
      BQC_TRY(oz_rows_of_b(b + (int64_t)P0 * npair, npair, n, std::min(pc, np - P0), scr, be, &ob,
                           s));
      BQC_TRY(oz_gemm(oc, ob, oz_kblocks(n), 1, 0, X + (int64_t)P0 * n * no, no, 0, 0, ctx->flag,
                      s));
    }
    return BQC_OK;
  }
  Gemm64Args g;  // batched over P
  g.M = n;
  g.N = no;
  g.K1 = 1;
  g.K2 = n;
  g.A = b;
  g.bsA = npair;
  g.B = C;
  g.ldb = no;
  g.C = X;
  g.ldc = no;
  g.bsC = (int64_t)n * no;
  g.batch = np;
  return launch_gemm64(kASym, false, g, s);
}

int k_of_x(Ctx *ctx, const double *X, int n, int no, int naux, void *scratch, size_t bytes,
           double *K, cudaStream_t s) {
  for (int pc = std::min(naux, (1 << 30) / std::max(1, no)); scratch && pc >= 1; pc /= 2) {
    const int ns = oz_splits(pc * no, oz_k_splits(n, pc * no));
    const size_t kp = oz_align((size_t)ns * n * n * 8), xs = oz_slice_bytes(n, pc * no);
    if (kp + xs + oz_exp_bytes(n, ns) > bytes) continue;
    char *scr = static_cast<char *>(scratch);
    double *part = reinterpret_cast<double *>(scr);
    for (int P0 = 0; P0 < naux; P0 += pc) {
      const int np = std::min(pc, naux - P0);
      OzOperand ox;
      BQC_TRY(oz_rows_of_x(X + (int64_t)P0 * n * no, n, no, np, ns, scr + kp,
                           reinterpret_cast<int *>(scr + kp + xs), &ox, s));
      BQC_TRY(oz_gemm(ox, ox, oz_split_kb(ox.K, ns), 1, P0 > 0, part, n, (int64_t)n * n, kOzLower,
                      ctx->flag, s));
    }
    return oz_sym_reduce(part, ns, (int64_t)n * n, n, n, K, s);
  }
  Gemm64Args k;  // one launch over (P, i)
  k.M = n;
  k.N = n;
  k.K1 = naux;
  k.K2 = no;
  k.A = X;
  k.lda = no;
  k.sA1 = (int64_t)n * no;
  k.B = X;
  k.ldb = no;
  k.sB1 = (int64_t)n * no;
  k.C = K;
  k.ldc = n;
  k.lower_only = 1;
  k.mirror = 1;
  return launch_gemm64(kAN, true, k, s);
}

int jk_fp64_stored(Df *df, const double *C, double *J, double *K, cudaStream_t s) {
  const Basis *b = df->basis;
  const int n = b->nbf, naux = df->naux_loc, no = b->nocc;
  const int64_t npair = df->npair;
  double *X = df->X64.as<double>();
  if (jk64_small(n, no) && df->X64.n >= x64_bytes(n, naux, no))
    return jk_fp64_small(df, C, J, K, s);
  if (n > 64) {
    const OzJkPlan p = oz_jk_plan(n, naux, no, df->X64.n);
    if (p.pc) return jk_fp64_oz(df, p, C, J, K, s);
  }
  df->mark(0, s);
  df->mark(1, s);
  BQC_TRY(x_of_b(df->ctx, df->B64.as<double>(), npair, C, n, no, naux, X, nullptr, 0, s));
  k_wdot<<<naux, 256, 0, s>>>(X, C, (int64_t)n * no, df->w.as<double>());
  BQC_LAUNCH_CHECK();
  df->mark(2, s);
  // J pass
  BQC_TRY(jpass_fp64(df, J, s));
  df->mark(3, s);
  BQC_TRY(k_of_x(df->ctx, X, n, no, naux, nullptr, 0, K, s));
  df->mark(4, s);
  return BQC_OK;
}

size_t df_stored_bytes(int n, int naux, int nocc, int shadow) {
  const size_t npair = (size_t)n * (n + 1) / 2;
  size_t b = (size_t)naux * naux * 8 + (size_t)naux * npair * 8;  // L, B64
  b += (size_t)naux * n * nocc * 8;                                // X64
  // (the X buffer's scratch, at most 32 MiB, and the J partials' further slices,
  // at most 3 MB, come on top: AUTO mode takes them from what its limit leaves,
  // serving from its allowance for small buffers)
  b += (size_t)jpass_split((int64_t)npair, naux) * npair * 8 + (size_t)naux * 8 * 2;
  if (shadow == BQC_SHADOW_TF32 || shadow == BQC_SHADOW_F16)
    b += mixed_workspace_bytes(n, naux, nocc, shadow);
  if (shadow == BQC_SHADOW_F16) {  // float-pair B and w of the J pass, the pieces' J partials
    b += (size_t)naux * npair * 8 + (size_t)naux * 8;
    const int np = std::min(kJPieces, std::max(naux, 1));
    for (int k = 0; k < np; ++k)
      b += (size_t)jpass_split((int64_t)npair, (int)((int64_t)naux * (k + 1) / np) -
                                                   (int)((int64_t)naux * k / np)) *
           npair * 8;
  }
  return b;
}

}  // namespace bqc

using namespace bqc;

extern "C" {

int bqc_df_coulomb(bqc_df *df, const double *D_dev, double *J_dev, int variant,
                   bqc_stream_t stream) {
  if (!df || !D_dev || !J_dev || (variant != BQC_COULOMB_FP64 && variant != BQC_COULOMB_FF))
    return BQC_E_INVALID;
  if (df->mode != BQC_DF_STORED || !df->B64.p) {
    set_error("bqc_df_coulomb needs a stored handle", __FILE__, __LINE__);
    return BQC_E_UNSUPPORTED;
  }
  if (variant == BQC_COULOMB_FF && !df->B2f.p) {
    set_error("the float-float Coulomb pass needs a handle built with BQC_SHADOW_F16",
              __FILE__, __LINE__);
    return BQC_E_UNSUPPORTED;
  }
  BQC_CUDA_TRY(cudaSetDevice(df->ctx->device));
  if (df->D2.n < (size_t)df->npair * 8) BQC_TRY(df->D2.alloc(df->ctx, (size_t)df->npair * 8));
  const int need = jpass_split(df->npair, df->naux_loc);
  if (df->Jp.n < (size_t)need * df->npair * 8)
    BQC_TRY(df->Jp.alloc(df->ctx, (size_t)need * df->npair * 8));
  cudaStream_t s = (cudaStream_t)stream;
  return variant == BQC_COULOMB_FF ? jff_of_density(df, D_dev, df->D2.as<double>(), J_dev, s)
                                   : jfp64_of_density(df, D_dev, df->D2.as<double>(), J_dev, s);
}

int bqc_df_build(bqc_ctx *ctx, const bqc_basis *basis, const bqc_df_opts *opts,
                 bqc_stream_t stream, bqc_df **out) {
  if (!ctx || !basis || !out) return BQC_E_INVALID;
  *out = nullptr;
  NvtxRange nv("bqc_df_build");
  BQC_CUDA_TRY(cudaSetDevice(ctx->device));
  bqc_df_opts o;
  o.mode = BQC_DF_STORED;
  o.schwarz = -1.0;
  o.aux_block = 1024;
  o.keep_fp32 = 1;
  o.hbm_limit = 0;
  o.aux_begin = 0;
  o.aux_end = 0;
  if (opts) o = *opts;
  cudaStream_t s = (cudaStream_t)stream;
  const int n = basis->nbf, naux = basis->naux, no = basis->nocc;
  const int64_t npair = (int64_t)n * (n + 1) / 2;
  int mode = o.mode;
  size_t room = SIZE_MAX;  // for scratch beyond df_stored_bytes
  if (mode == BQC_DF_AUTO) {
    size_t limit = o.hbm_limit;
    if (!limit) {
      size_t fr = 0, tot = 0;
      BQC_CUDA_TRY(cudaMemGetInfo(&fr, &tot));
      limit = (size_t)(fr * 0.9);
    }
    const size_t need = df_stored_bytes(n, naux, no, o.keep_fp32);
    mode = need <= limit ? BQC_DF_STORED : BQC_DF_DIRECT;
    room = need <= limit ? limit - need : 0;
  }
  if (mode != BQC_DF_STORED && mode != BQC_DF_DIRECT && mode != BQC_DF_NONE) return BQC_E_INVALID;
  if (o.keep_fp32 < BQC_SHADOW_NONE || o.keep_fp32 > BQC_SHADOW_F16) return BQC_E_INVALID;
  // aux shard [P0, P1) (stored mode): both 0 selects every aux function
  int P0 = o.aux_begin, P1 = o.aux_end;
  if (P0 == 0 && P1 == 0) P1 = naux;
  if (P0 < 0 || P1 > naux || P0 >= P1) {
    set_error("bqc_df_build: aux shard outside [0, Naux) or empty", __FILE__, __LINE__);
    return BQC_E_INVALID;
  }
  const bool shard = P0 != 0 || P1 != naux;
  if (shard && mode == BQC_DF_NONE) return BQC_E_INVALID;
  if (shard && mode != BQC_DF_STORED) {
    set_error("bqc_df_build: aux shards are a stored-mode feature", __FILE__, __LINE__);
    return BQC_E_UNSUPPORTED;
  }
  if (o.schwarz < 0.0) o.schwarz = (mode == BQC_DF_DIRECT) ? 1e-10 : 1e-12;
  if (o.aux_block <= 0) o.aux_block = 1024;
  bqc_df *df = new (std::nothrow) bqc_df();
  if (!df) return BQC_E_OOM;
  df->ctx = ctx;
  df->basis = basis;
  df->mode = mode;
  df->npair = npair;
  df->opts = o;
  df->p0 = P0;
  df->naux_loc = P1 - P0;
  auto fail = [&](int st) {
    cudaStreamSynchronize(s);
    delete df;
    return st;
  };
  int st;
  if (mode == BQC_DF_NONE) {  // conventional four-centre J/K: no auxiliary tensor
    if ((st = jk4c_setup(df, s)) != BQC_OK) return fail(st);
    if ((st = ctx->check_flag(s)) != BQC_OK) return fail(st);
    *out = df;
    return BQC_OK;
  }
  // metric and its Cholesky factor
  if ((st = df->L.alloc(ctx, (size_t)naux * naux * 8)) != BQC_OK) return fail(st);
  if ((st = launch_int2c(basis, df->L.as<double>(), s)) != BQC_OK) return fail(st);
  if ((st = df->Vdiag.alloc(ctx, (size_t)naux * naux * 8)) != BQC_OK) return fail(st);
  if (cudaMemcpyAsync(df->Vdiag.p, df->L.p, (size_t)naux * naux * 8, cudaMemcpyDeviceToDevice,
                      s) != cudaSuccess)
    return fail(BQC_E_CUDA);
  if ((st = cholesky_lower(ctx, df->L.as<double>(), naux, s)) != BQC_OK) return fail(st);
  if ((st = ctx->check_flag(s)) != BQC_OK) return fail(st);
  if ((st = eri3c_plan(basis, o.schwarz, df->Vdiag.as<double>(), s, &df->plan)) != BQC_OK)
    return fail(st);
  if ((st = df->w.alloc(ctx, (size_t)naux * 8)) != BQC_OK) return fail(st);
  if (mode == BQC_DF_STORED) {
    df->Vdiag.release();  // metric only needed for the screening plan
    // The sliced solve for handles without shadows only.  Its B is within 1e-12
    // of the substitution's and as near to 64 bits, but a split shadow keeps 22
    // bits: a few elements in a million of B then round the other way, which
    // moves the split-FP16 K of (H2O)_32 by 7e-10 of its norm and single elements
    // by 7e-8, and a staged SCF's mixed stage (see scf.cu) turns a change of B's
    // last bits into more than 1e-9 of its last Fock matrix ((H2O)_8: 4e-9,
    // (H2O)_12: 4e-9, against 1e-12).  What it costs: set-up of (H2O)_24 with FP16
    // shadows 570 ms, with the sliced solve 77.
    const bool sliced = o.keep_fp32 == BQC_SHADOW_NONE;
    // the FP64 X buffer, first the scratch of the sliced solve
    const int nl = df->naux_loc;
    const size_t x = (size_t)nl * n * no * 8;
    const size_t xs = x + std::min(room, x64_bytes(n, nl, no) - x);
    room -= xs - x;
    if (!shard) {
      if ((st = df->X64.alloc(ctx, xs)) != BQC_OK) return fail(st);
      if ((st = df->B64.alloc(ctx, (size_t)naux * npair * 8)) != BQC_OK) return fail(st);
      if (cudaMemsetAsync(df->B64.p, 0, (size_t)naux * npair * 8, s) != cudaSuccess)
        return fail(BQC_E_CUDA);
      if ((st = launch_eri3c(basis, &df->plan, 0, naux, df->B64.as<double>(), npair, s)) !=
          BQC_OK)
        return fail(st);
      if ((st = trsm_lower_left(ctx, df->L.as<double>(), naux, df->B64.as<double>(), npair,
                                npair, sliced ? df->X64.p : nullptr, sliced ? df->X64.n : 0,
                                s)) != BQC_OK)
        return fail(st);
    } else {
      // B_P for P in [P0, P1) depends on (Q|mu nu) for every Q <= P (the
      // triangular solve couples them): solve rows [0, P1) with the leading
      // P1 x P1 block of L and keep the shard's rows (raw is the largest array
      // of the build: the scratch beside it is given back before B is allocated)
      DBuf raw, Lb;
      if ((st = raw.alloc(ctx, (size_t)P1 * npair * 8)) != BQC_OK) return fail(st);
      if (cudaMemsetAsync(raw.p, 0, (size_t)P1 * npair * 8, s) != cudaSuccess)
        return fail(BQC_E_CUDA);
      if ((st = launch_eri3c(basis, &df->plan, 0, P1, raw.as<double>(), npair, s)) != BQC_OK)
        return fail(st);
      if ((st = Lb.alloc(ctx, (size_t)P1 * P1 * 8)) != BQC_OK) return fail(st);
      if (cudaMemcpy2DAsync(Lb.p, (size_t)P1 * 8, df->L.p, (size_t)naux * 8, (size_t)P1 * 8, P1,
                            cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return fail(BQC_E_CUDA);
      if (sliced && df->X64.alloc(ctx, xs) != BQC_OK) df->X64.release();
      if ((st = trsm_lower_left(ctx, Lb.as<double>(), P1, raw.as<double>(), npair, npair,
                                df->X64.p, df->X64.n, s)) != BQC_OK)
        return fail(st);
      if (cudaStreamSynchronize(s) != cudaSuccess) return fail(BQC_E_CUDA);
      df->X64.release();
      if ((st = df->B64.alloc(ctx, (size_t)(P1 - P0) * npair * 8)) != BQC_OK) return fail(st);
      if (cudaMemcpyAsync(df->B64.p, raw.as<double>() + (size_t)P0 * npair,
                          (size_t)(P1 - P0) * npair * 8, cudaMemcpyDeviceToDevice,
                          s) != cudaSuccess)
        return fail(BQC_E_CUDA);
      if (cudaStreamSynchronize(s) != cudaSuccess) return fail(BQC_E_CUDA);
    }
    if (!df->X64.p && (st = df->X64.alloc(ctx, xs)) != BQC_OK) return fail(st);
    const int jmin = jpass_split(npair, nl), jmax = jpass_split(npair, nl, kFp64JAux);
    const int js = jmin + (int)std::min<size_t>(jmax - jmin, room / ((size_t)npair * 8));
    if ((st = df->Jp.alloc(ctx, (size_t)js * npair * 8)) != BQC_OK) return fail(st);
    if (o.keep_fp32 != BQC_SHADOW_NONE)
      if ((st = mixed_setup(df, o.keep_fp32, s)) != BQC_OK) return fail(st);
  } else {
    if ((st = direct_setup(df, s)) != BQC_OK) return fail(st);
  }
  if ((st = ctx->check_flag(s)) != BQC_OK) return fail(st);
  *out = df;
  return BQC_OK;
}

int bqc_df_destroy(bqc_df *df) {
  if (!df) return BQC_E_INVALID;
  cudaSetDevice(df->ctx->device);
  cudaDeviceSynchronize();
  delete df;
  return BQC_OK;
}

int bqc_df_info(const bqc_df *df, int *mode, size_t *bytes) {
  if (!df) return BQC_E_INVALID;
  if (mode) *mode = df->mode;
  if (bytes) *bytes = df->device_bytes();
  return BQC_OK;
}

int bqc_df_shard(const bqc_df *df, int *aux_begin, int *aux_end) {
  if (!df) return BQC_E_INVALID;
  if (aux_begin) *aux_begin = df->p0;
  if (aux_end) *aux_end = df->p0 + df->naux_loc;
  return BQC_OK;
}

int bqc_df_screening(const bqc_df *df, int64_t *candidates, int64_t *survivors) {
  if (!df) return BQC_E_INVALID;
  if (candidates) *candidates = df->plan.candidates;
  if (survivors) *survivors = df->plan.survivors;
  return BQC_OK;
}

int bqc_df_copy(const bqc_df *df, int which, double *out, bqc_stream_t stream) {
  if (!df || !out) return BQC_E_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  const int naux = df->basis->naux;
  if (which == 0) {
    if (df->mode != BQC_DF_STORED) return BQC_E_INVALID;
    BQC_CUDA_TRY(cudaMemcpyAsync(out, df->B64.p, (size_t)df->naux_loc * df->npair * 8,
                                 cudaMemcpyDeviceToDevice, s));
  } else if (which == 1) {
    if (!df->L.p) return BQC_E_INVALID;
    BQC_CUDA_TRY(
        cudaMemcpyAsync(out, df->L.p, (size_t)naux * naux * 8, cudaMemcpyDeviceToDevice, s));
  } else {
    return BQC_E_INVALID;
  }
  return BQC_OK;
}

int bqc_int3c_screened(const bqc_df *df, int p0, int p1, int variant, double *out,
                       bqc_stream_t stream) {
  if (!df || !out || variant < 0 || variant > 2 || df->mode == BQC_DF_NONE)
    return BQC_E_INVALID;
  if (p0 < 0 || p1 > df->basis->naux || p0 >= p1) return BQC_E_INVALID;
  BQC_CUDA_TRY(cudaSetDevice(df->ctx->device));
  return launch_eri3c_variant(df->basis, &df->plan, p0, p1, out, df->npair, variant,
                              (cudaStream_t)stream);
}

int bqc_df_timing(bqc_df *df, int enable) {
  if (!df) return BQC_E_INVALID;
  if (enable) {
    for (auto &e : df->ev)
      if (!e) BQC_CUDA_TRY(cudaEventCreate(&e));
  }
  df->timing = enable != 0;
  return BQC_OK;
}

int bqc_df_phase_ms(bqc_df *df, float *ms, int n) {
  if (!df || !ms || n <= 0) return BQC_E_INVALID;
  if (!df->timed) return BQC_E_NOT_READY;
  BQC_CUDA_TRY(cudaEventSynchronize(df->ev[4]));
  float t[4] = {0, 0, 0, 0};
  BQC_CUDA_TRY(cudaEventElapsedTime(&t[0], df->ev[1], df->ev[2]));
  BQC_CUDA_TRY(cudaEventElapsedTime(&t[3], df->ev[0], df->ev[1]));
  if (df->mode == BQC_DF_STORED && df->side && df->last_mixed) {
    // mixed stored build: J (side stream, ev[j_from] -> ev5) runs beside the
    // tensor-core passes; K is the SYRK (ev2 -> ev3)
    BQC_CUDA_TRY(cudaEventElapsedTime(&t[1], df->ev[df->j_from], df->ev[5]));
    BQC_CUDA_TRY(cudaEventElapsedTime(&t[2], df->ev[2], df->ev[3]));
  } else {
    BQC_CUDA_TRY(cudaEventElapsedTime(&t[1], df->ev[2], df->ev[3]));
    BQC_CUDA_TRY(cudaEventElapsedTime(&t[2], df->ev[3], df->ev[4]));
    for (int k = 0; k + 1 < df->kev_used; k += 2) {
      float x = 0;
      BQC_CUDA_TRY(cudaEventElapsedTime(&x, df->kev[k], df->kev[k + 1]));
      t[0] -= x;
      t[2] += x;
    }
  }
  for (int i = 0; i < n && i < 4; ++i) ms[i] = t[i];
  return BQC_OK;
}

int bqc_jk(bqc_df *df, const double *C, int nocc, int prec, double *J, double *K,
           bqc_stream_t stream) {
  if (!df || !C || !J || !K) return BQC_E_INVALID;
  if (nocc != df->basis->nocc) return BQC_E_INVALID;
  NvtxRange nv(prec == BQC_PREC_FP64 ? "bqc_jk fp64" : "bqc_jk mixed");
  cudaStream_t s = (cudaStream_t)stream;
  if (df->timing) df->timed = true;
  df->kev_used = 0;
  df->last_mixed = prec != BQC_PREC_FP64;
  if (df->mode == BQC_DF_DIRECT) return jk_direct(df, C, prec, J, K, s);
  if (df->mode == BQC_DF_NONE) return jk_4c(df, C, prec, J, K, s);
  if (prec == BQC_PREC_FP64) return jk_fp64_stored(df, C, J, K, s);
  if (prec == BQC_PREC_MIXED_TF32 || prec == BQC_PREC_MIXED_TF32X3 ||
      prec == BQC_PREC_MIXED_F16X3) {
    if (!df->mixed) {
      set_error("mixed precision needs split shadows (bqc_df_opts.keep_fp32)", __FILE__, __LINE__);
      return BQC_E_INVALID;
    }
    return jk_mixed_stored(df, C, prec, J, K, s);
  }
  return BQC_E_INVALID;
}

int bqc_jk_host(bqc_df *df, const double *C, int nocc, int prec, double *J, double *K,
                bqc_stream_t stream) {
  if (!df || !C || !J || !K) return BQC_E_INVALID;
  if (nocc != df->basis->nocc) return BQC_E_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  const int n = df->basis->nbf;
  // a NaN or an infinity in the orbitals would poison every element of J
  // and K: refuse it on the host, before anything is copied or launched
  for (size_t i = 0, e = (size_t)n * nocc; i < e; ++i)
    if (!std::isfinite(C[i])) {
      char msg[96];
      std::snprintf(msg, sizeof(msg), "bqc_jk_host: C_occ[%zu] is not finite", i);
      set_error(msg, __FILE__, __LINE__);
      return BQC_E_INVALID;
    }
  if (!df->host_io.p) {
    BQC_TRY(df->host_io.alloc(df->ctx, ((size_t)n * nocc + 2 * (size_t)n * n) * 8));
  }
  double *dC = df->host_io.as<double>();
  double *dJ = dC + (size_t)n * nocc, *dK = dJ + (size_t)n * n;
  BQC_CUDA_TRY(cudaMemcpyAsync(dC, C, (size_t)n * nocc * 8, cudaMemcpyHostToDevice, s));
  BQC_TRY(bqc_jk(df, dC, nocc, prec, dJ, dK, stream));
  BQC_CUDA_TRY(cudaMemcpyAsync(J, dJ, (size_t)n * n * 8, cudaMemcpyDeviceToHost, s));
  BQC_CUDA_TRY(cudaMemcpyAsync(K, dK, (size_t)n * n * 8, cudaMemcpyDeviceToHost, s));
  BQC_CUDA_TRY(cudaStreamSynchronize(s));
  return df->ctx->check_flag(s);
}

}  // extern "C"
