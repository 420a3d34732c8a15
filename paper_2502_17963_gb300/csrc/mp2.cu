// DF-MP2 on the resident three-index tensor (Sec. 2.3).
//
// The paper's MP2 stage reuses the CD-ERIs of the mean field: in canonical
// SCF orbitals, B_P,ia = sum_{mu nu} C_mu i B_P,mu nu C_nu a, the
// integrals (ia|jb) = sum_P B_P,ia B_P,jb are formed block by block as
// matrix products, and the closed-shell second-order energy
//   E2 = sum_{ijab} (ia|jb) [2 (ia|jb) - (ib|ja)] / (e_i + e_j - e_a - e_b)
// (Szabo & Ostlund Eq. 6.74) is accumulated with the denominator applied in
// place, one block of occupied pairs at a time, so no four-index array is
// ever held.  FP64: sliced tensor-core products (oz.cu), (H2O)_10 in 6.7 ms
// against 96.8 on the DFMA GEMM of gemm64.cuh, which serves small systems;
// MIXED_F16X3: the pair blocks on the tensor cores (tc.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <memory>
#include <vector>

#include "bqc_internal.h"
#include "df_internal.h"
#include "gemm64.cuh"
#include "oz.h"

namespace bqc {

// 1 / x for x < 0 of normal size: FP32 seed of the mantissa and one step
// y (1 + e + e^2) with e = 1 - x y (the geometric series), error of the order
// of the seed's 2^-23 cubed; a third of the FP64 instructions of a division.
__device__ __forceinline__ double recip_neg(double x) {
  const int hi = __double2hiint(x);
  const int k = ((hi >> 20) & 0x7ff) - 1023;
  const double m = __hiloint2double(hi - (k << 20), __double2loint(x));  // -2 < m <= -1
  const double y = (double)(1.0f / (float)m);
  const double e = fma(-m, y, 1.0);
  const double r = fma(y * e, e + 1.0, y);
  return __hiloint2double(__double2hiint(r) - (k << 20), __double2loint(r));
}

// Energy of the occupied pairs (i, j), i >= j, of one block of
// V[(ii, a)][(jj, b)] = (i a | j b) with i = i0 + ii, j = j0 + jj: one CTA per
// pair, a fixed-order reduction, epair[i * nocc + j] = weight * sum_ab; the
// weight is 2 for i > j (the (j, i) term is equal) and 1 for i = j.
// Bound by the FP64 pipe: elements (a, b) and (b, a), which share their
// denominator, go together, v (2v - x) + x (2x - v) = 2 (v^2 - v x + x^2), from
// two 32 x 32 tiles read coalesced ((H2O)_10: 2.56 -> 0.7 ms in all).
__global__ void __launch_bounds__(256) k_mp2_pairs(const double *__restrict__ V, int64_t ldv,
                                                   int i0, int j0, int nvir,
                                                   const double *__restrict__ eps, int nocc,
                                                   double *__restrict__ epair) {
  const int ii = blockIdx.x, jj = blockIdx.y;
  const int i = i0 + ii, j = j0 + jj;
  if (j > i) return;  // uniform over the block
  __shared__ double tx[32][33];
  const double eij = eps[i] + eps[j];
  const double *ev = eps + nocc;
  const double *Vi = V + (int64_t)ii * nvir * ldv + (int64_t)jj * nvir;
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  double s = 0.0;
  const int nt = (nvir + 31) / 32;
  for (int ta = 0; ta < nt; ++ta)
    for (int tb = 0; tb <= ta; ++tb) {
      const int a0 = ta * 32, b0 = tb * 32;
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = ly + 8 * k;
        v[k] = (a0 + r < nvir && b0 + lx < nvir) ? Vi[(int64_t)(a0 + r) * ldv + b0 + lx] : 0.0;
        tx[r][lx] = (b0 + r < nvir && a0 + lx < nvir) ? Vi[(int64_t)(b0 + r) * ldv + a0 + lx] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int a = a0 + ly + 8 * k, b = b0 + lx;
        if (a < nvir && b <= a) {
          const double x = tx[lx][ly + 8 * k];
          const double q = fma(v[k], v[k], fma(x, x, -v[k] * x));  // v^2 when a == b
          const double den = eij - ev[a] - ev[b];
          const double r = den <= -2.2250738585072014e-308 && den >= -1.0e300 ? recip_neg(den)
                                                                           : 1.0 / den;
          s = fma(a == b ? q : 2.0 * q, r, s);
        }
      }
      __syncthreads();
    }
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) epair[(int64_t)i * nocc + j] = (i == j ? 1.0 : 2.0) * red[0];
}

// *out = sum of the lower triangle of epair (nocc x nocc), in a fixed order.
__global__ void __launch_bounds__(256) k_mp2_sum(const double *__restrict__ epair, int nocc,
                                                 double *out) {
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < (int64_t)nocc * nocc; e += blockDim.x) {
    const int i = (int)(e / nocc), j = (int)(e % nocc);
    if (j <= i) s += epair[e];
  }
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

// Occupied-index block size: (bi * nvir)^2 doubles of (ia|jb) at most ~1 GiB,
// and at most 16 occupied orbitals (small systems still run several blocks).
static int mp2_block(int nocc, int nvir) {
  const double cap = (double)(1 << 27);  // doubles
  int bi = std::max(1, (int)(std::sqrt(cap) / std::max(1, nvir)));
  return std::max(1, std::min({bi, 16, nocc}));
}

// X_P = B_P C_occ (into the handle's FP64 X buffer) and B_P,ia = sum_nu
// X_P[nu][i] C[nu][no + a] -> Bt[P][i][a] on the DFMA path.
static int mp2_transform_dfma(Df *df, const double *C, int nmo, double *Bt, cudaStream_t s) {
  const int n = df->basis->nbf, naux = df->basis->naux, no = df->basis->nocc, nv = nmo - no;
  Gemm64Args g;
  g.M = n;
  g.N = no;
  g.K1 = 1;
  g.K2 = n;
  g.A = df->B64.as<double>();
  g.bsA = df->npair;
  g.B = C;
  g.ldb = nmo;
  g.C = df->X64.as<double>();
  g.ldc = no;
  g.bsC = (int64_t)n * no;
  g.batch = naux;
  BQC_TRY(launch_gemm64(kASym, false, g, s));
  Gemm64Args t;
  t.M = no;
  t.N = nv;
  t.K1 = 1;
  t.K2 = n;
  t.A = df->X64.as<double>();
  t.lda = no;
  t.bsA = (int64_t)n * no;
  t.B = C + no;
  t.ldb = nmo;
  t.C = Bt;
  t.ldc = nv;
  t.bsC = (int64_t)no * nv;
  t.batch = naux;
  return launch_gemm64(kAT, false, t, s);
}

// The same as sliced tensor-core products (oz.cu), chunks of pc aux functions.
// Scratch: the sliced C_occ^T and C_vir^T, then a chunk's sliced B (rows
// (P, mu)) or X (rows (P, i)).
static int mp2_transform_pc(int n, int naux, int no, int nv, size_t bytes) {
  const size_t fixed = oz_slice_bytes(no, n) + oz_exp_bytes(no, 1) + oz_slice_bytes(nv, n) +
                       oz_exp_bytes(nv, 1) + 4096;
  const size_t row = (size_t)oz_kblocks(n) * kOzSlices * kOzKb * 2 + sizeof(int);
  if (bytes <= fixed) return 0;
  return (int)std::min<size_t>((bytes - fixed) / (row * n), (size_t)naux);
}

static int mp2_transform_oz(Df *df, const double *C, int nmo, double *Bt, char *scr, int pc,
                            cudaStream_t s) {
  const int n = df->basis->nbf, naux = df->basis->naux, no = df->basis->nocc, nv = nmo - no;
  const int kb = oz_kblocks(n);
  int *flag = df->ctx->flag;
  double *X = df->X64.as<double>();
  OzOperand oc[2];
  for (int k = 0; k < 2; ++k) {
    OzSrc c;
    c.kind = kOzCols;
    c.p = C + (k ? no : 0);
    c.rows = k ? nv : no;
    c.K = n;
    c.ld = nmo;
    oc[k].slices = scr;
    int *e = reinterpret_cast<int *>(scr + oz_slice_bytes(c.rows, n));
    oc[k].exps = e;
    oc[k].rows = c.rows;
    oc[k].K = n;
    BQC_TRY(oz_slice(c, kb, scr, e, s));
    scr += oz_slice_bytes(c.rows, n) + oz_exp_bytes(c.rows, 1);
  }
  for (int P0 = 0; P0 < naux; P0 += pc) {
    const int np = std::min(pc, naux - P0);
    for (int k = 0; k < 2; ++k) {
      OzSrc b;
      b.K = n;
      if (k == 0) {
        b.kind = kOzSym;
        b.p = df->B64.as<double>() + (int64_t)P0 * df->npair;
        b.n2 = n;
        b.sz = df->npair;
      } else {
        b.kind = kOzCols;
        b.p = X + (int64_t)P0 * n * no;
        b.n2 = no;
        b.sz = (int64_t)n * no;
        b.ld = no;
      }
      b.rows = (int64_t)np * b.n2;
      OzOperand ob;
      ob.slices = scr;
      int *e = reinterpret_cast<int *>(scr + oz_slice_bytes(b.rows, n));
      ob.exps = e;
      ob.rows = b.rows;
      ob.K = n;
      BQC_TRY(oz_slice(b, kb, scr, e, s));
      BQC_TRY(oz_gemm(oc[k], ob, kb, 1, 0,
                      k == 0 ? X + (int64_t)P0 * n * no : Bt + (int64_t)P0 * no * nv,
                      k == 0 ? no : nv, 0, 0, flag, s));
    }
  }
  return BQC_OK;
}

// prec FP64: the transform and the pair blocks V = B_ia^T B_jb as sliced
// FP64-accurate tensor-core products; MIXED_F16X3: the pair blocks as
// split-FP16 tensor-core GEMMs (FP32 accumulation in short chains, float-float
// drains, FP64 blocks); the energy in FP64.  Without memory for the slices the
// DFMA GEMM, and for few functions, where a tile is mostly padding: in FP64 up
// to 64 (whole energy, N = 75: 614 us sliced, 1000 DFMA; 100: 820 and 2634), in
// MIXED_F16X3, where only the transform is at stake, up to 80 (75: 672 us with the
// sliced transform, 585 without; 100: 838 and 1227).
constexpr int kMp2DfmaMax = 64, kMp2DfmaMaxF16 = 80;
static int mp2_run(Df *df, const double *C, const double *eps, int nmo, int prec, double *e2,
                   cudaStream_t s) {
  const Basis *b = df->basis;
  const int n = b->nbf, naux = b->naux, no = b->nocc, nv = nmo - no;
  Ctx *ctx = df->ctx;
  DBuf Bt, V, ep, out, Ts;
  std::unique_ptr<Mp2Tc, Mp2TcDeleter> tcs;
  BQC_TRY(ep.alloc(ctx, (size_t)no * no * 8));
  BQC_TRY(out.alloc(ctx, 8));
  StreamGuard guard{s};
  BQC_CUDA_TRY(cudaMemsetAsync(ep.p, 0, ep.n, s));
  if (nv > 0) {
    const int64_t Q = (int64_t)no * nv;
    BQC_TRY(Bt.alloc(ctx, (size_t)naux * Q * 8));
    const int bi = mp2_block(no, nv);
    int pc = 0;
    if (n > (prec == BQC_PREC_FP64 ? kMp2DfmaMax : kMp2DfmaMaxF16) &&
        Ts.alloc(ctx, oz_slice_bytes(Q, naux) + oz_exp_bytes(Q, 1)) == BQC_OK)
      pc = mp2_transform_pc(n, naux, no, nv, Ts.n);
    bool oz = prec == BQC_PREC_FP64 && Ts.p;
    if (pc)
      BQC_TRY(mp2_transform_oz(df, C, nmo, Bt.as<double>(), Ts.as<char>(), pc, s));
    else
      BQC_TRY(mp2_transform_dfma(df, C, nmo, Bt.as<double>(), s));
    if (prec == BQC_PREC_MIXED_F16X3) {
      if (Ts.p) {
        BQC_CUDA_TRY(cudaStreamSynchronize(s));
        Ts.release();
      }
      BQC_TRY(mp2_tc_setup(ctx, Bt.as<double>(), naux, no, nv, ctx->flag, tcs, s));
      BQC_CUDA_TRY(cudaStreamSynchronize(s));
      Bt.release();  // the split operand replaces it
    }
    int *te = oz ? reinterpret_cast<int *>(Ts.as<char>() + oz_slice_bytes(Q, naux)) : nullptr;
    if (oz) {  // rows (i, a), contraction P
      OzSrc q;
      q.kind = kOzCols;
      q.p = Bt.as<double>();
      q.rows = Q;
      q.K = naux;
      q.ld = Q;
      BQC_TRY(oz_slice(q, oz_kblocks(naux), Ts.p, te, s));
    }
    if (V.alloc(ctx, (size_t)bi * nv * bi * nv * 8) != BQC_OK) {
      if (!oz) return BQC_E_OOM;
      // the slices' memory is what the pair block lacks: do without them
      BQC_CUDA_TRY(cudaStreamSynchronize(s));
      Ts.release();
      oz = false;
      BQC_TRY(V.alloc(ctx, (size_t)bi * nv * bi * nv * 8));
    }
    for (int i0 = 0; i0 < no; i0 += bi) {
      const int ni = std::min(bi, no - i0);
      for (int j0 = 0; j0 <= i0; j0 += bi) {
        const int nj = std::min(bi, no - j0);
        // V[(ii,a)][(jj,b)] = sum_P Bt[P][i0+ii][a] Bt[P][j0+jj][b]
        if (tcs) {
          BQC_TRY(mp2_tc_block(tcs.get(), nv, i0, ni, j0, nj, V.as<double>(), (int64_t)nj * nv,
                               ctx->flag, s));
        } else if (oz) {
          auto rows = [&](int o0, int cnt) {
            OzOperand r;
            r.slices = Ts.as<char>() + (int64_t)o0 * nv * kOzKb * 2;
            r.exps = te + (int64_t)o0 * nv;
            r.rows = (int64_t)cnt * nv;
            r.K = naux;
            r.stride = Q;
            return r;
          };
          BQC_TRY(oz_gemm(rows(j0, nj), rows(i0, ni), oz_kblocks(naux), 1, 0, V.as<double>(),
                          (int64_t)nj * nv, 0, 0, ctx->flag, s));
        } else {
          Gemm64Args v;
          v.M = ni * nv;
          v.N = nj * nv;
          v.K1 = 1;
          v.K2 = naux;
          v.A = Bt.as<double>() + (int64_t)i0 * nv;
          v.lda = Q;
          v.B = Bt.as<double>() + (int64_t)j0 * nv;
          v.ldb = Q;
          v.C = V.as<double>();
          v.ldc = (int64_t)nj * nv;
          BQC_TRY(launch_gemm64(kAT, false, v, s));
        }
        k_mp2_pairs<<<dim3((unsigned)ni, (unsigned)nj), 256, 0, s>>>(
            V.as<double>(), (int64_t)nj * nv, i0, j0, nv, eps, no, ep.as<double>());
        BQC_LAUNCH_CHECK();
      }
    }
  }
  k_mp2_sum<<<1, 256, 0, s>>>(ep.as<double>(), no, out.as<double>());
  BQC_LAUNCH_CHECK();
  BQC_CUDA_TRY(cudaMemcpyAsync(e2, out.p, 8, cudaMemcpyDeviceToHost, s));
  BQC_CUDA_TRY(cudaStreamSynchronize(s));
  return ctx->check_flag(s);
}

}  // namespace bqc

using namespace bqc;

extern "C" int bqc_mp2(bqc_df *df, const double *C_dev, const double *eps_dev, int nmo, int prec,
                       double *e2, bqc_stream_t stream) {
  if (!df || !C_dev || !eps_dev || !e2) return BQC_E_INVALID;
  NvtxRange nv("bqc_mp2");
  if (df->mode != BQC_DF_STORED || !df->B64.p || !df->X64.p || df->is_shard()) {
    set_error("bqc_mp2 needs a stored-mode DF handle holding the whole tensor", __FILE__, __LINE__);
    return BQC_E_INVALID;
  }
  if (nmo < df->basis->nocc || nmo > df->basis->nbf) return BQC_E_INVALID;
  BQC_CUDA_TRY(cudaSetDevice(df->ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  if (prec == BQC_PREC_FP64 || prec == BQC_PREC_MIXED_F16X3)
    return mp2_run(df, C_dev, eps_dev, nmo, prec, e2, s);
  set_error("bqc_mp2: precision not available", __FILE__, __LINE__);
  return BQC_E_UNSUPPORTED;
}
