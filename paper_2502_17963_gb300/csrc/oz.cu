// FP64 matrix products on the 5th-generation tensor cores (tcgen05 kind::f16)
// by exact slicing (Ozaki, Ogita, Oishi, Rump 2012; on FP16 tensor cores:
// Mukunoki, Ozaki, Ogita, Imamura 2020).
//
// FP64 runs at 1/64 of FP32 here (1.2 TFLOP/s measured), FP16 MMAs at 1.9
// PFLOP/s, so an FP64 product assembled from 34 FP16 products of slices is
// still more than an order of magnitude faster than DFMA.
//
//  * Slices.  With 2^e an upper bound of the row's elements, an element is
//    held as the integer round(a 2^(55 - e)), |.| <= 2^55, in seven balanced
//    base-256 digits (the first in [-128, 128], the others in [-128, 127]),
//    each exact in FP16.  The row's largest elements keep all their 53 bits;
//    smaller ones are rounded at 2^(e - 56).
//  * Products.  Digit products are integers of at most 2^14.  Products of
//    slices i and j carry the weight 2^(-8 (i + j)); those of one level
//    d = i + j <= 7 (at most seven) add into one TMEM accumulator over 128
//    contraction elements: at most 7 * 128 * 2^14 < 2^24, so every FP32
//    partial sum is an exact integer and the tensor core's truncation has
//    nothing to truncate.  Levels 8 and up (below 2^-64 of the row bounds'
//    product times about 5 K) are left out.  For rows of even size the result is
//    closer to the exact one than a DFMA chain's; the bound is one of the rows,
//    not of the terms (rows spread log-normally over e^(+-3): 5.6e-15 of the
//    norm, DFMA 7.4e-16).
//  * Chains are drained into two 64-bit integers per element (levels 0-3 and
//    4-7, one IMAD.WIDE per level), exact for up to 2^15 chains, and turned
//    into FP64 once per tile with integer arithmetic (the FP64 pipe would
//    take longer than the MMAs of a short contraction).
// A row with an infinity or a NaN makes every result it enters a NaN.
//
// Tile 128 x 64 (eight levels x 64 columns fill the 512 TMEM columns), k-block
// 32: 14 slices of a k-block (84 KB) arrive as two TMA boxes and feed 34 x 2
// MMAs, so shared-memory reads (6 KB an MMA, 48 clocks where the arithmetic takes
// 32; measured) and not the load path bound the main loop: multicasting an
// operand tile to CTA pairs changed nothing.  30000 x 900 x 900: 30 to 31.6
// TFLOP/s of FP64 product (1031 to 1075 of FP16 issued, 0.53 to 0.55 of the
// measured 1942; DFMA 1.2), error of normal deviates 5.9e-17 of the result's norm
// against DFMA's 9.2e-16; 60000 x 64 x 64, where the drain and the conversion of a
// tile take as long as its MMAs, about 8.  The accumulators are single-buffered: a
// level is handed over as soon as its last MMA of the chain is issued, the MMAs of
// a k-block run level by level, and so the eight epilogue warps drain level d while
// levels d + 1 ... and the next chain's first levels are computed.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "bqc_internal.h"
#include "df_internal.h"
#include "oz.h"
#include "tc_util.cuh"

namespace bqc {

using namespace tc;

int make_tmap_f16_sw64(CUtensorMap *map, const void *base, int rank, const uint64_t *dims,
                       const uint64_t *strides_bytes, const uint32_t *box);  // tc.cu

// ----------------------------------------------------------------- slicing --

constexpr int kOzBadExp = 1 << 28;  // exponent of a row with a non-finite element

template <int KIND>
__device__ __forceinline__ double oz_load(const OzSrc &a, int64_t z, int64_t i, int64_t r, int k) {
  if (KIND == kOzRows) {
    const int k1 = k / a.k2;
    return __ldg(a.p + (int64_t)k1 * a.s1 + r * a.ld + (k - k1 * a.k2));
  }
  if (KIND == kOzCols) return __ldg(a.p + z * a.sz + (int64_t)k * a.ld + i);
  const int64_t hi = i > k ? i : k, lo = i > k ? k : i;
  return __ldg(a.p + z * a.sz + hi * (hi + 1) / 2 + lo);
}

// a as the integer round(a 2^(55 - e)) plus 0x80 in each of its seven bytes,
// so that byte s from the top is digit s + 128.  emax = e + 1022 is the
// largest exponent field of the row.
__device__ __forceinline__ unsigned long long oz_fixed(double a, int emax) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(a);
  const int ef = (int)(bits >> 52) & 0x7ff;
  unsigned long long m = bits & 0xfffffffffffffULL;
  if (ef) m |= 1ULL << 52;
  const int sh = max(ef, 1) - emax + 2;  // <= 2
  if (sh >= 0)
    m <<= sh;
  else
    m = sh > -55 ? (m + (1ULL << (-sh - 1))) >> (-sh) : 0ULL;
  const long long v = (long long)bits < 0 ? -(long long)m : (long long)m;
  return (unsigned long long)(v + 0x0080808080808080LL);
}

// One block: 8 rows, one contraction split.  A lane owns a row and 8
// consecutive contraction elements, so a warp writes the 512 contiguous bytes
// of (k-block, slice, 8 rows) per slice, and reads whole 64-byte segments for
// either source order.  The first sweep finds the rows' exponents, the second
// reads again (from L1 / L2) and writes; with one k-block per warp the
// elements stay in registers.  Bound by the writes: 14 bytes per element.
template <int KIND>
__global__ void __launch_bounds__(256) k_oz_slice(OzSrc a, int split_kb, __half *out, int *exps) {
  __shared__ int emax_s[8][8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rl = lane >> 2, kg = lane & 3;
  const int64_t r = (int64_t)blockIdx.x * 8 + rl;
  const bool rok = r < a.rows;
  const int nkb = oz_kblocks(a.K), kb0 = blockIdx.y * split_kb, kb1 = min(nkb, kb0 + split_kb);
  int64_t z = 0, i = r;
  if (KIND != kOzRows && a.n2 < a.rows) {
    z = r / a.n2;
    i = r - z * a.n2;
  }
  const bool once = kb1 - kb0 <= 8;
  double v[8];
  int em = 1;
  for (int kb = kb0 + warp; kb < kb1; kb += 8) {
    const int k = kb * kOzKb + kg * 8;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      v[t] = (rok && k + t < a.K) ? oz_load<KIND>(a, z, i, r, k + t) : 0.0;
      em = max(em, (__double2hiint(v[t]) >> 20) & 0x7ff);
    }
  }
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 1));
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 2));
  if (kg == 0) emax_s[warp][rl] = em;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) em = max(em, emax_s[w][rl]);
  const bool bad = em == 0x7ff;
  if (warp == 0 && kg == 0 && rok)
    exps[(int64_t)blockIdx.y * a.rows + r] = bad ? kOzBadExp : em - 1022;
  if (!rok) return;
  const __half2 off = __half2half2(__ushort_as_half(0x6480));  // 1024 + 128
  for (int kb = kb0 + warp; kb < kb1; kb += 8) {
    const int k = kb * kOzKb + kg * 8;
    unsigned long long u[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (!once) v[t] = k + t < a.K ? oz_load<KIND>(a, z, i, r, k + t) : 0.0;
      u[t] = bad ? 0x0080808080808080ULL : oz_fixed(v[t], em);
    }
#pragma unroll
    for (int sl = 0; sl < kOzSlices; ++sl) {
      uint4 w;
      uint32_t *wp = &w.x;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int sh = 8 * (kOzSlices - 1 - sl);
        uint32_t lo = (uint32_t)(u[2 * t] >> sh), hi = (uint32_t)(u[2 * t + 1] >> sh);
        if (sl > 0) {
          lo &= 0xff;
          hi &= 0xff;
        }
        const uint32_t h = (lo | (hi << 16)) + 0x64006400u;  // 1024 + digit + 128, exact in FP16
        const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&h), off);
        wp[t] = *reinterpret_cast<const uint32_t *>(&d);
      }
      __half *dst = out + (((int64_t)kb * kOzSlices + sl) * a.rows + r) * kOzKb + kg * 8;
      *reinterpret_cast<uint4 *>(dst) = w;
    }
  }
}

int oz_slice(const OzSrc &src, int split_kb, void *slices, int *exps, cudaStream_t s) {
  if (src.rows <= 0 || src.K <= 0 || split_kb <= 0) return BQC_E_INVALID;
  OzSrc a = src;
  if (!a.k2) a.k2 = a.K;
  if (!a.n2) a.n2 = (int)std::min<int64_t>(a.rows, 0x7fffffff);
  const int ns = (oz_kblocks(a.K) + split_kb - 1) / split_kb;
  const dim3 grid((unsigned)((a.rows + 7) / 8), (unsigned)ns);
  if (ns > 65535 || (a.rows + 7) / 8 > 0x7fffffff) return BQC_E_INVALID;
  __half *o = static_cast<__half *>(slices);
  if (a.kind == kOzRows) k_oz_slice<kOzRows><<<grid, 256, 0, s>>>(a, split_kb, o, exps);
  else if (a.kind == kOzCols) k_oz_slice<kOzCols><<<grid, 256, 0, s>>>(a, split_kb, o, exps);
  else k_oz_slice<kOzSym><<<grid, 256, 0, s>>>(a, split_kb, o, exps);
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

// ----------------------------------------------------------------- product --

constexpr int kOzM = 128, kOzN = 64, kOzLevels = 8, kOzStages = 2;
constexpr int kOzChain = 4;  // k-blocks per accumulation chain (128 elements)
constexpr int kOzEpiWarps = 8;
constexpr int kOzThreads = 64 + 32 * kOzEpiWarps;
constexpr uint32_t kOzASlice = kOzM * 64, kOzBSlice = kOzN * 64;
constexpr uint32_t kOzStage = kOzSlices * (kOzASlice + kOzBSlice);
constexpr size_t kOzSmem = 1024 + (size_t)kOzStages * kOzStage + 256;

// K-major operand tile with 64-byte rows in the 64-byte swizzle (8-row groups
// 512 bytes apart).
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;           // LBO (ignored for swizzled K-major)
  d |= (uint64_t)(512 >> 4) << 32;  // SBO
  d |= (uint64_t)1 << 46;           // descriptor version
  d |= (uint64_t)4 << 61;           // SWIZZLE_64B
  return d;
}

struct OzParams {
  int64_t M;
  int N, nt;
  int nkb, split_kb, ns;
  int tiles;  // tiles of one split
  int tri;
  const int *eA, *eB;
  double *out;
  int64_t ldo, split_stride;
  int alpha, beta;
  int *flag;
};

struct OzItem {
  int split, tm, tn, kb0, kb1;
};

__device__ __forceinline__ OzItem oz_item(const OzParams &p, int64_t it) {
  OzItem x;
  x.split = (int)(it / p.tiles);
  const int t = (int)(it - (int64_t)x.split * p.tiles);
  if (p.tri) {  // row tile tm has column tiles 0 .. 2 tm + 1
    int tm = (int)((sqrtf(4.0f * t + 1.0f) - 1.0f) * 0.5f);
    while ((tm + 1) * (tm + 2) <= t) ++tm;
    while (tm * (tm + 1) > t) --tm;
    x.tm = tm;
    x.tn = t - tm * (tm + 1);
  } else {
    x.tm = t / p.nt;
    x.tn = t - x.tm * p.nt;
  }
  x.kb0 = x.split * p.split_kb;
  x.kb1 = min(p.nkb, x.kb0 + p.split_kb);
  return x;
}

// (hi 2^32 + lo) 2^e as a double, rounded once; integer arithmetic only.
__device__ __forceinline__ double oz_value(long long hi, long long lo, int e) {
  long long h = hi + (lo >> 32);
  uint32_t l = (uint32_t)lo;
  const bool neg = h < 0;
  if (neg) {
    h = ~h + (l == 0);
    l = 0u - l;
  }
  unsigned long long m;
  int n;
  if (h) {
    n = __clzll(h);  // 1 .. 63
    m = ((unsigned long long)h << n) |
        (n <= 32 ? (unsigned long long)(l >> (32 - n)) : (unsigned long long)l << (n - 32));
  } else {
    if (!l) return 0.0;
    n = __clz(l);
    m = (unsigned long long)l << (32 + n);
    n += 64;
  }
  const int be = 63 + 32 - n + e + 1023;  // biased exponent of the leading bit
  if (be <= 0) return 0.0;
  unsigned long long r = ((m >> 10) + 1) >> 1;
  r += (unsigned long long)(be - 1) << 52;  // the leading bit adds one
  if ((r >> 52) >= 0x7ff) r = 0x7ffULL << 52;
  if (neg) r |= 1ULL << 63;
  return __longlong_as_double((long long)r);
}

__global__ void __launch_bounds__(kOzThreads, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
              const OzParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t *smem = smem_raw + ((1024 - (raw & 1023)) & 1023);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + (size_t)kOzStages * kOzStage);
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * kOzStages + 2 * kOzLevels);
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kOzStages;
  const uint32_t tfull0 = empty0 + 8 * kOzStages, tempty0 = tfull0 + 8 * kOzLevels;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t items = (int64_t)p.tiles * p.ns;
  if (threadIdx.x == 0) {
    prefetch_tmap(&mapA);
    prefetch_tmap(&mapB);
    for (int st = 0; st < kOzStages; ++st) {
      mbar_init(full0 + 8 * st, 1);
      mbar_init(empty0 + 8 * st, 1);
    }
    for (int d = 0; d < kOzLevels; ++d) {
      mbar_init(tfull0 + 8 * d, 1);
      mbar_init(tempty0 + 8 * d, kOzEpiWarps);
    }
    fence_barrier_init();
  }
  if (warp == 0) tmem_alloc(smem_u32(tslot), 512);
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tslot;
  const uint32_t sbase = smem_u32(smem);
  bool ok = true;
  if (warp == 0) {
    if (lane == 0) {
      int64_t kg = 0;
      for (int64_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
        const OzItem x = oz_item(p, it);
        for (int kb = x.kb0; kb < x.kb1; ++kb, ++kg) {
          const int st = (int)(kg % kOzStages);
          if (kg >= kOzStages)
            ok = mbar_wait(empty0 + 8 * st, (uint32_t)(((kg / kOzStages) - 1) & 1), p.flag, 61);
          if (!ok) break;
          const uint32_t a = sbase + st * kOzStage, bar = full0 + 8 * st;
          mbar_arrive_expect_tx(bar, kOzStage);
          tma_load_3d(a, &mapA, bar, 0, x.tm * kOzM, kb * kOzSlices);
          tma_load_3d(a + kOzSlices * kOzASlice, &mapB, bar, 0, x.tn * kOzN, kb * kOzSlices);
        }
      }
    }
  } else if (warp == 1) {
    constexpr uint32_t idesc = idesc_f16(kOzM, kOzN);
    int64_t kg = 0, g = 0;
    for (int64_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
      const OzItem x = oz_item(p, it);
      for (int c0 = x.kb0; c0 < x.kb1 && ok; c0 += kOzChain, ++g) {
        const int c1 = min(x.kb1, c0 + kOzChain);
        for (int kb = c0; kb < c1 && ok; ++kb, ++kg) {
          const int st = (int)(kg % kOzStages);
          ok = mbar_wait_warp(full0 + 8 * st, (uint32_t)((kg / kOzStages) & 1), p.flag, 62);
          if (!ok) break;
          tc_fence_after();
          const uint64_t a = sdesc_sw64(sbase + st * kOzStage);
          const uint64_t b = a + ((kOzSlices * kOzASlice) >> 4);
#pragma unroll
          for (int d = 0; d < kOzLevels; ++d) {
            if (kb == c0 && g > 0) {
              ok = mbar_wait_warp(tempty0 + 8 * d, (uint32_t)((g - 1) & 1), p.flag, 63);
              if (!ok) break;
              tc_fence_after();
            }
            uint32_t acc = kb != c0;
#pragma unroll
            for (int i = 0; i < kOzSlices; ++i) {
              const int j = d - i;
              if (j < 0 || j >= kOzSlices) continue;
#pragma unroll
              for (int k2 = 0; k2 < 2; ++k2) {
                mma_f16(tbase + d * kOzN, a + ((i * kOzASlice + k2 * 32) >> 4),
                        b + ((j * kOzBSlice + k2 * 32) >> 4), idesc, acc);
                acc = 1;
              }
            }
            if (kb == c1 - 1) mma_commit(tfull0 + 8 * d);
          }
          if (ok) mma_commit(empty0 + 8 * st);
        }
      }
    }
  } else {
    const int q = warp & 3, h = (warp - 2) >> 2;
    const uint32_t tl = tbase + ((uint32_t)(q * 32) << 16) + h * 32;
    int64_t g = 0;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
      const OzItem x = oz_item(p, it);
      long long hi[32], lo[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
      for (int c0 = x.kb0; c0 < x.kb1; c0 += kOzChain, ++g) {
#pragma unroll
        for (int d = 0; d < kOzLevels; ++d) {
          if (ok) ok = mbar_wait(tfull0 + 8 * d, (uint32_t)(g & 1), p.flag, 64);
          __syncwarp();
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < 32; c += 16) {
            float v[16];
            tmem_ld16(tl + d * kOzN + c, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int iv = __float2int_rn(v[i]);
              if (d < 4)
                hi[c + i] += (long long)iv * (1 << (8 * (3 - d)));
              else
                lo[c + i] += (long long)iv * (1 << (8 * (7 - d)));
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty0 + 8 * d);
        }
      }
      const int64_t m = (int64_t)x.tm * kOzM + q * 32 + lane;
      const int n0 = x.tn * kOzN + h * 32;
      if (ok && m < p.M) {
        const int ea = p.eA[(int64_t)x.split * p.M + m];
        double *o = p.out + (int64_t)x.split * p.split_stride + m;
#pragma unroll
        for (int c = 0; c < 32; c += 8) {
          // the old values of eight columns together: loads between stores to
          // the same array are not reordered, and 32 of them in a chain took
          // longer than a short contraction
          double old[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            old[k] = p.beta && n0 + c + k < p.N ? o[(int64_t)(n0 + c + k) * p.ldo] : 0.0;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (n0 + c + k < p.N) {
              const int eb = __ldg(p.eB + (int64_t)x.split * p.N + n0 + c + k);
              double v = (ea == kOzBadExp || eb == kOzBadExp)
                             ? __longlong_as_double(0x7ff8000000000000LL)
                             : oz_value(hi[c + k], lo[c + k], ea + eb - 70);
              if (p.alpha < 0) v = -v;
              o[(int64_t)(n0 + c + k) * p.ldo] = p.beta ? old[k] + v : v;
            }
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tbase, 512);
}

static int oz_map(CUtensorMap *map, const OzOperand &o, int box_rows) {
  const uint64_t dims[3] = {(uint64_t)kOzKb, (uint64_t)o.rows,
                            (uint64_t)oz_kblocks(o.K) * kOzSlices};
  const uint64_t str[2] = {(uint64_t)kOzKb * 2, (uint64_t)(o.stride ? o.stride : o.rows) * kOzKb * 2};
  const uint32_t box[3] = {(uint32_t)kOzKb, (uint32_t)box_rows, (uint32_t)kOzSlices};
  return make_tmap_f16_sw64(map, o.slices, 3, dims, str, box);
}

int oz_gemm(const OzOperand &A, const OzOperand &B, int split_kb, int alpha, int beta, double *out,
            int64_t ldo, int64_t split_stride, int tri, int *flag, cudaStream_t s) {
  if (A.rows <= 0 || B.rows <= 0 || A.K <= 0 || A.K != B.K || split_kb <= 0 ||
      A.rows > 0x7fffff00 || B.rows > 0x7fffff00 || (tri && A.rows != B.rows))
    return BQC_E_INVALID;
  CUtensorMap ma, mb;
  BQC_TRY(oz_map(&ma, A, kOzM));
  BQC_TRY(oz_map(&mb, B, kOzN));
  OzParams p;
  p.M = A.rows;
  p.N = (int)B.rows;
  p.nt = (int)((B.rows + kOzN - 1) / kOzN);
  p.nkb = oz_kblocks(A.K);
  p.split_kb = split_kb;
  p.ns = (p.nkb + split_kb - 1) / split_kb;
  p.tri = tri;
  const int64_t tiles = oz_tiles(A.rows, B.rows, tri == kOzLower);
  if (tiles > (1 << 30)) return BQC_E_INVALID;
  p.tiles = (int)tiles;
  p.eA = A.exps;
  p.eB = B.exps;
  p.out = out;
  p.ldo = ldo;
  p.split_stride = split_stride;
  p.alpha = alpha;
  p.beta = beta;
  p.flag = flag;
  BQC_CUDA_TRY(cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kOzSmem));
  const int64_t grid = std::min<int64_t>(tiles * p.ns, sm_count());
  k_oz_gemm<<<(unsigned)grid, kOzThreads, kOzSmem, s>>>(ma, mb, p);
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

// One thread per element of a 32 x 32 tile of the lower triangle: sums the
// partials in a fixed order, writes both triangles coalesced.
__global__ void __launch_bounds__(256) k_oz_sym_reduce(const double *part, int nsplit,
                                                       int64_t stride, int n, int64_t ldp,
                                                       double *out) {
  if (blockIdx.y > blockIdx.x) return;  // x: row tile m, y: column tile n <= m
  __shared__ double t[32][33];
  const int m0 = blockIdx.x * 32, n0 = blockIdx.y * 32, tx = threadIdx.x & 31;
  for (int ty = threadIdx.x >> 5; ty < 32; ty += 8) {
    const int m = m0 + tx, c = n0 + ty;
    double s = 0.0;
    if (m < n && c <= m)
      for (int k = 0; k < nsplit; ++k) s += part[k * stride + (int64_t)c * ldp + m];
    t[ty][tx] = s;
    if (m < n && c <= m) out[(int64_t)c * n + m] = s;
  }
  __syncthreads();
  for (int ty = threadIdx.x >> 5; ty < 32; ty += 8) {
    const int m = m0 + ty, c = n0 + tx;
    if (m < n && c < m) out[(int64_t)m * n + c] = t[tx][ty];
  }
}

int oz_sym_reduce(const double *part, int nsplit, int64_t split_stride, int n, int64_t ldp,
                  double *out, cudaStream_t s) {
  const unsigned t = (unsigned)((n + 31) / 32);
  k_oz_sym_reduce<<<dim3(t, t), 256, 0, s>>>(part, nsplit, split_stride, n, ldp, out);
  BQC_LAUNCH_CHECK();
  return BQC_OK;
}

}  // namespace bqc

using namespace bqc;

extern "C" int bqc_gemm_sliced(bqc_ctx *ctx, int m, int n, int k, const double *A_dev,
                               const double *B_dev, int splits, int lower, double *C_dev,
                               bqc_stream_t stream) {
  if (!ctx || m < 1 || n < 1 || k < 1 || !A_dev || !B_dev || !C_dev || splits < 1 ||
      splits > 65535 || (lower && m != n))
    return BQC_E_INVALID;
  BQC_CUDA_TRY(cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  const int ns = oz_splits(k, splits), kb = oz_split_kb(k, splits);
  DBuf buf[2];
  OzOperand o[2];
  StreamGuard guard{s};
  BQC_CUDA_TRY(cudaMemsetAsync(C_dev, 0, (size_t)splits * m * n * 8, s));
  for (int q = 0; q < 2; ++q) {
    OzSrc x;
    x.p = q ? B_dev : A_dev;
    x.rows = q ? n : m;
    x.K = k;
    x.ld = k;
    BQC_TRY(buf[q].alloc(ctx, oz_slice_bytes(x.rows, k) + oz_exp_bytes(x.rows, ns)));
    o[q].slices = buf[q].p;
    int *e = reinterpret_cast<int *>(buf[q].as<char>() + oz_slice_bytes(x.rows, k));
    o[q].exps = e;
    o[q].rows = x.rows;
    o[q].K = k;
    BQC_TRY(oz_slice(x, kb, buf[q].p, e, s));
  }
  BQC_TRY(oz_gemm(o[0], o[1], kb, 1, 0, C_dev, m, (int64_t)m * n, lower ? kOzLower : kOzFull,
                  ctx->flag, s));
  return ctx->check_flag(s);
}
