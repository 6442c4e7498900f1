// FP64 GEMM on the FP16 tensor cores, by exact integer products (the scheme of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 95 (2012), with the
// error-free slices held as fixed-point digits).
//
// Why: GB300 retires 2 FP64 FMAs per SM and clock, and 1 018 FP16 ones on
// mma.sync (both measured).  Over a K range every row of op(A) and every column
// of B is scaled by the power of two above its largest magnitude and held as a
// 63-bit fixed-point number, written in eight balanced base-256 digits
// d_0 .. d_7 in [-128, 127]: a = 2^e sum_s d_s 2^{-8s}.  FP16 holds the digits
// exactly, a product of two is at most 2^14, and the 36 digit products with
// s + t <= 7 go to eight accumulators, one per weight 2^{-8(s+t)}.
//
// Exactness: an accumulator starts at 1.5 * 2^23 and takes 32 k-values of at
// most 8 digit pairs, |sum| <= 32 * 8 * 2^14 = 2^22, so it stays in
// [2^23, 2^24] where FP32 is spaced by 1: every addition is exact, and the
// float's bit pattern minus that of 1.5 * 2^23 IS the integer sum.  The sums
// are added to two 64-bit integers per output (weights 2^-24 and 2^-56), so
// the only errors are the fixed-point truncation of the operands (2^-61 of the
// row's / column's largest value A / B), the dropped products (s + t >= 8,
// together below 2^-57.1 A B per k-value) and the final rounding to FP64: in
// all below K 2^-56.8 A B over a range of K values, where a chain of FP64 FMAs
// is held to K 2^-53 sum_k |a_k b_k|.
//
// That is a bound by the row and the column as wholes.  Where large entries of
// the one only meet small ones of the other, sum_k |a_k b_k| is far below A B and
// the FMAs are the more accurate: a = (1, 2^-70) times b = (2^-70, 1) is 0 here,
// 2^-69 there.  The library's own products (projections, Rayleigh-Ritz, Lanczos)
// are of vectors whose components carry rounding errors of 2^-53 of the largest
// one, from H x, so that nothing is lost.  A product of the caller's own numbers
// sets 'graded': |d_0| |d_0'| is summed beside the products (one more of 36, the
// signs masked off), and an output where it stays below 128 -- between 1/8 and
// 1/32 of A B, whose leading digits are 32 to 64 -- is computed again with FP64
// FMAs, a warp per output.  Screening of 7 vectors with 128 on 48^3: 103.7 -> 106.6
// us, of 100 with 200: 265 -> 272 us.
//
// 36 FP16 products per FP64 one leave 28 FP64-accurate FMAs per SM and clock,
// 14 times the FP64 pipe.  A 32 x 32 tile per CTA of four warps (three CTAs per
// SM) pads small products little and splits K finely; what bounds it is the
// issue of the digit conversion (about 27 instructions per operand element)
// beside the products.  Against the FP64 FMA kernel it replaced: 80 x 256 x 6859
// and 6859 x 256 x 80 together 0.53 -> 0.13 ms, 128 x 7 x 6858 with its
// transpose 0.48 -> 0.08 ms, 80 x 8192 x 6859 (then in double-float) 2.9 -> 2.1
// ms; relative error against long double, 128 x 3 x 6858 and back, 7.1e-16 ->
// 2.6e-16 (flat), 7.8e-16 -> 1.2e-16 (falling by 26 orders of magnitude).
#include <algorithm>
#include <cstdint>

#include "fx.cuh"
#include "linalg.cuh"
#include "profile.cuh"

namespace pdep {
namespace {

constexpr int FX_BM = 32, FX_BN = 32;         // CTA tile, four warps of 16 x 16
constexpr int FX_KS = 32;                     // k-values per stage (and per exact accumulation)
constexpr int FX_THREADS = 128;
constexpr int FX_ROWS = FX_BM + FX_BN;
// digit rows of a stage: 32 halves padded to 40 (80 bytes): the eight 16-byte
// rows of an ldmatrix tile fall on distinct banks
constexpr int FX_LD = 40;
constexpr int FX_SMEM = FX_S * FX_ROWS * FX_LD * 2;
// K range of one CTA: the high sum stays below 2^51 (2^38 per k-value)
constexpr int FX_KMAX = 4096;

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
// (hi 2^-24 + lo 2^-56) 2^q2 rounded to FP64 (integer arithmetic: the FP64
// pipe would take as long for this as the tensor cores for the products)
__device__ __forceinline__ double fx_result(long long hi, long long lo, int q2) {
  hi += lo >> 32;
  uint32_t l = (uint32_t)lo;
  const bool neg = hi < 0;
  if (neg) {
    hi = ~hi;
    l = 0u - l;
    if (l == 0) ++hi;
  }
  unsigned long long top;
  int z;
  if (hi != 0) {
    z = __clzll(hi);
    top = ((unsigned long long)hi << z) | (((unsigned long long)l << 32) >> (64 - z));  // z >= 1
  } else {
    if (l == 0) return 0.0;
    const int c = __clz(l);
    z = 64 + c;
    top = (unsigned long long)l << (32 + c);
  }
  // top 2^(-z) units of 2^(q2 - 24), top in [2^63, 2^64)
  const unsigned long long mant = (top >> 11) + ((top >> 10) & 1ull);
  const int q = q2 - 24 - z + 11;
  const int be = q + 52 + 1023;
  double r;
  if (be > 0 && be < 2046)
    r = __longlong_as_double((long long)(((unsigned long long)(be - 1) << 52) + mant));
  else
    r = scalbn((double)mant, q);
  return neg ? -r : r;
}

// C (m x n) = alpha op(A) B + beta C over the K range of blockIdx.z; with
// atomic set, alpha op(A) B is added to C (scaled beforehand).
template <bool TA, bool GRADED>
__global__ void __launch_bounds__(FX_THREADS, 3)
    k_gemm_fx(int m, int n, int k, double alpha, const double* __restrict__ A, long long lda,
              const double* __restrict__ B, long long ldb, double beta, double* __restrict__ C,
              long long ldc, int kchunk, int atomic, const int* __restrict__ bmap,
              const int* __restrict__ cmap, const int* __restrict__ ndev, int has_beta) {
  extern __shared__ __align__(16) unsigned char fx_sh[];
  __shared__ int rexp[FX_ROWS];
  __shared__ int n_again;
  if (ndev) n = min(n, *ndev);
  const int row0 = blockIdx.x * FX_BM, col0 = blockIdx.y * FX_BN;
  if (col0 >= n) return;
  const int kbeg = blockIdx.z * kchunk, kend = min(k, kbeg + kchunk);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // element (row r of the stage, k): r < 32 rows of op(A), then columns of B
  auto value = [&](int r, int kk) -> double {
    if (kk >= kend) return 0.0;
    if (r < FX_BM) {
      const int gi = row0 + r;
      if (gi >= m) return 0.0;
      return TA ? A[kk + (long long)gi * lda] : A[gi + (long long)kk * lda];
    }
    const int gj = col0 + r - FX_BM;
    if (gj >= n) return 0.0;
    return B[kk + (long long)(bmap ? bmap[gj] : gj) * ldb];
  };
  // A thread's elements of a stage: eight pairs (k, k + 1), pair q in row
  // pr(q) at k-offset pk(q).  Rows contiguous in k (B, and A when TA): half a
  // warp reads 32 consecutive k; A contiguous in its rows: a quarter warp
  // reads 8 consecutive rows.
  auto pr = [&](int q) { return (q < 4 && !TA) ? (lane & 7) + 8 * warp : warp * 2 + (lane >> 4) + 8 * q; };
  auto pk = [&](int q) { return (q < 4 && !TA) ? 2 * ((lane >> 3) + 4 * q) : 2 * (lane & 15); };

  // largest exponent of every row over the K range
  for (int r = tid; r < FX_ROWS; r += FX_THREADS) rexp[r] = 1;
  __syncthreads();
  {
    int ex[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) ex[q] = 1;
    for (int k0 = kbeg; k0 < kend; k0 += FX_KS) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int r = pr(q), kk = k0 + pk(q);
        ex[q] = max(ex[q], max(exp_of(value(r, kk)), exp_of(value(r, kk + 1))));
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) atomicMax(&rexp[pr(q)], ex[q]);
  }
  __syncthreads();
  int top = 0;
  if (tid < FX_ROWS) top = rexp[tid];
  if (__syncthreads_or(top == 0x7ff)) {
    // an infinity or NaN in the tile: plain FP64 arithmetic propagates it
    for (int e = tid; e < FX_BM * FX_BN; e += FX_THREADS) {
      const int gi = row0 + e % FX_BM, gj = col0 + e / FX_BM;
      if (gi >= m || gj >= n) continue;
      double s = 0.0;
      for (int kk = kbeg; kk < kend; ++kk) s += value(e % FX_BM, kk) * value(FX_BM + e / FX_BM, kk);
      double* c = C + gi + (long long)(cmap ? cmap[gj] : gj) * ldc;
      if (atomic)
        atomicAdd(c, alpha * s);
      else
        *c = has_beta ? alpha * s + beta * *c : alpha * s;
    }
    return;
  }

  int er[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) er[q] = rexp[pr(q)];
  const int wm = warp >> 1, wn = warp & 1;
  const uint32_t sh0 = (uint32_t)__cvta_generic_to_shared(fx_sh);
  constexpr uint32_t SLICE = FX_ROWS * FX_LD * 2;
  // ldmatrix rows: A 16 x 16 (rows 0-7 | 8-15 at k 0, then at k 8); B two
  // 8-column tiles (columns 0-7 at k 0, k 8, then columns 8-15)
  const uint32_t a_addr = sh0 + 2 * ((wm * 16 + (lane & 15)) * FX_LD + (lane >> 4) * 8);
  const uint32_t b_addr = sh0 + 2 * ((FX_BM + wn * 16 + (lane & 7) + ((lane >> 4) << 3)) * FX_LD +
                                     ((lane >> 3) & 1) * 8);
  long long hi[2][4], lo[2][4];
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int e = 0; e < 4; ++e) hi[b][e] = lo[b][e] = 0;
  float lead[2][4] = {};  // GRADED: sum of |d_0| |d_0'|

  double x[8][2];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    x[q][0] = value(pr(q), kbeg + pk(q));
    x[q][1] = value(pr(q), kbeg + pk(q) + 1);
  }
  int stages = 0;
  for (int k0 = kbeg; k0 < kend; k0 += FX_KS) {
    if (stages) __syncthreads();  // the last stage's digits have been read
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint2 u0 = biased(fx_of(x[q][0], er[q])), u1 = biased(fx_of(x[q][1], er[q]));
      uint32_t* d = (uint32_t*)(fx_sh + 2 * (pr(q) * FX_LD + pk(q)));
#pragma unroll
      for (int s = 0; s < FX_S; ++s) d[s * (SLICE / 4)] = digit_pair(u0, u1, s);
    }
    __syncthreads();
    if (k0 + FX_KS < kend) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        x[q][0] = value(pr(q), k0 + FX_KS + pk(q));
        x[q][1] = value(pr(q), k0 + FX_KS + pk(q) + 1);
      }
    }
    float acc[FX_S][2][4];
#pragma unroll
    for (int s = 0; s < FX_S; ++s)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[s][b][e] = __uint_as_float(FX_MAGIC);
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      uint32_t bf[FX_S][4];
#pragma unroll
      for (int s = 0; s < FX_S; ++s) ldsm4(bf[s], b_addr + s * SLICE + kk * 32);
#pragma unroll
      for (int s = 0; s < FX_S; ++s) {
        uint32_t af[4];
        ldsm4(af, a_addr + s * SLICE + kk * 32);
        if constexpr (GRADED) {
          if (s == 0) {
            constexpr uint32_t M = 0x7fff7fffu;
            const uint32_t aa[4] = {af[0] & M, af[1] & M, af[2] & M, af[3] & M};
            mma_f16(lead[0], aa, bf[0][0] & M, bf[0][1] & M);
            mma_f16(lead[1], aa, bf[0][2] & M, bf[0][3] & M);
          }
        }
#pragma unroll
        for (int t = 0; t + s < FX_S; ++t) {
          mma_f16(acc[s + t][0], af, bf[t][0], bf[t][1]);
          mma_f16(acc[s + t][1], af, bf[t][2], bf[t][3]);
        }
      }
    }
    // exact integer sums into the 64-bit accumulators (the magic numbers'
    // bits are taken off after the loop)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          hi[b][e] += (long long)__float_as_int(acc[s][b][e]) * (1 << (24 - 8 * s));
          lo[b][e] += (long long)__float_as_int(acc[s + 4][b][e]) * (1 << (24 - 8 * s));
        }
      }
    ++stages;
  }
  const long long bias = (long long)stages * ((long long)FX_MAGIC * 0x1010101ll);
  const int g = lane >> 2, t = lane & 3;
  unsigned short* again = reinterpret_cast<unsigned short*>(fx_sh);  // over the digits
  if constexpr (GRADED) {
    if (tid == 0) n_again = 0;
    __syncthreads();
  }
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = wm * 16 + g + (e >= 2 ? 8 : 0), cl = wn * 16 + b * 8 + 2 * t + (e & 1);
      const int gi = row0 + r, gj = col0 + cl;
      if (gi >= m || gj >= n) continue;
      if constexpr (GRADED) {
        // (rows of zeros, exponent field 1 as of subnormals, are exact)
        if (lead[b][e] < 128.0f && rexp[r] > 1 && rexp[FX_BM + cl] > 1) {
          again[atomicAdd(&n_again, 1)] = (unsigned short)(r * FX_BN + cl);
          continue;
        }
      }
      // operand scales 2^(er - 1084 + 56) each
      double v = fx_result(hi[b][e] - bias, lo[b][e] - bias, rexp[r] + rexp[FX_BM + cl] - 2056);
      v = alpha == 1.0 ? v : alpha == -1.0 ? -v : alpha * v;
      double* c = C + gi + (long long)(cmap ? cmap[gj] : gj) * ldc;
      if (atomic)
        atomicAdd(c, v);
      else
        *c = has_beta ? v + beta * *c : v;
    }
  if constexpr (GRADED) {
    __syncthreads();
    for (int q = warp; q < n_again; q += FX_THREADS / 32) {
      const int r = again[q] / FX_BN, cl = again[q] % FX_BN;
      double s = 0.0;
      for (int kk = kbeg + lane; kk < kend; kk += 32)
        s = fma(value(r, kk), value(FX_BM + cl, kk), s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        const int gj = col0 + cl;
        double* c = C + row0 + r + (long long)(cmap ? cmap[gj] : gj) * ldc;
        if (atomic)
          atomicAdd(c, alpha * s);
        else
          *c = has_beta ? alpha * s + beta * *c : alpha * s;
      }
    }
  }
}

__global__ void k_scale_fx(double* C, long long ldc, int m, int n, double beta, const int* cmap,
                           const int* ndev) {
  if (ndev) n = min(n, *ndev);
  const long long tot = (long long)m * n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e % m), j = (int)(e / m);
    double* c = C + i + (long long)(cmap ? cmap[j] : j) * ldc;
    *c = beta == 0.0 ? 0.0 : beta * *c;
  }
}

}  // namespace

cudaError_t gemm_fx(bool transA, int m, int n, int k, double alpha, const double* A, long long lda,
                    const double* B, long long ldb, double beta, double* C, long long ldc, int sms,
                    cudaStream_t st, const int* bmap, const int* cmap, const int* ndev,
                    int split_x8, bool mixed, bool graded) {
  const int tm = (m + FX_BM - 1) / FX_BM, tn = (n + FX_BN - 1) / FX_BN;
  const long long tiles = (long long)tm * tn;
  // about three resident CTAs per SM, at least four stages each
  int splits = (int)std::max<long long>(1, (3LL * sms + tiles - 1) / tiles);
  if (split_x8 > 0) splits = std::max(1, (splits * split_x8 + 7) / 8);
  splits = std::min(splits, std::max(1, k / (4 * FX_KS)));
  splits = std::max(splits, (k + FX_KMAX - 1) / FX_KMAX);
  int kchunk = (std::max(k, 1) + splits - 1) / splits;
  kchunk = ((kchunk + FX_KS - 1) / FX_KS) * FX_KS;
  splits = std::max(1, (k + kchunk - 1) / kchunk);
  int atomic = 0;
  if (splits > 1 || k <= 0) {
    const long long tot = (long long)m * n;
    const int blocks = (int)std::min<long long>((tot + 255) / 256, 4096);
    if (beta != 1.0 || k <= 0) {
      count_launch();
      k_scale_fx<<<blocks, 256, 0, st>>>(C, ldc, m, n, beta, cmap, ndev);
    }
    if (k <= 0) return cudaGetLastError();
    atomic = 1;
  }
  dim3 grid(tm, tn, splits);
  if (tn > 65535 || splits > 65535) return cudaErrorInvalidValue;
  ProfScope ps(mixed ? PC_GEMM_DF : PC_GEMM_F64, st, 2.0 * m * n * (double)k,
               ((double)m * k + (double)k * n + (beta != 0.0 ? 2.0 : 1.0) * m * n) * sizeof(double),
               ndev, n);
  count_launch();
  const int hb = beta != 0.0 ? 1 : 0;
  auto kern = transA ? (graded ? k_gemm_fx<true, true> : k_gemm_fx<true, false>)
                     : (graded ? k_gemm_fx<false, true> : k_gemm_fx<false, false>);
  kern<<<grid, FX_THREADS, FX_SMEM, st>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, kchunk,
                                          atomic, bmap, cmap, ndev, hb);
  return cudaGetLastError();
}

}  // namespace pdep
