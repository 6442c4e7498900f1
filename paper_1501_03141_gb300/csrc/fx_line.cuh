// FP64-accurate line transforms on the FP16 tensor cores (the passes of
// transforms.cuh for FP64 data; transforms_fx.cu, transforms_fx_cols.cu).
//
// Why: FP64 line FFTs are bound by the FP64 pipe (2 FMAs per SM and clock), and
// double-float ones by ten FP32 instructions per flop.  A line DFT is also a
// small matrix product, and fx.cuh's exact digit products give 28
// FP64-accurate FMAs per SM and clock.
//
// The DFT of a line of N points whose frequencies satisfy |n| < N/4 is folded
// twice before it becomes a product.  With E_n = z_n + z_-n and O_n = z_n - z_-n,
// X(j) = sum_n E_n cos(2 pi n j / N) + i sum_n O_n sin(2 pi n j / N); split
// into even and odd n, the four real sums Ce, Co, Se, So over N/8 frequencies
// each, taken at j = 0 .. N/4 only, give
//   X(j), X(-j)             = (Ce + Co) +- i (Se + So)
//   X(N/2 - j), X(N/2 + j)  = (Ce - Co) +- i (So - Se).
// The way back is the transpose: the four values of a quadruple are folded the
// same way and multiplied by the transposed tables (weights 1/2 at j = 0 and
// N/4, whose quadruples hold each position twice).  That leaves 1/8 of the
// dense product: 6 x 13 instead of 23 x 48 entries for N = 48, four times.
//
// Layout: the lines are the rows of the tensor-core tiles (M), real part of
// line g in row g and imaginary part in row g + 8, so one thread holds both;
// frequencies are K on the way in and N on the way out.  The accumulator
// fragment of the inverse transform has the layout of the A fragment of the
// forward one, so a z-line goes sphere -> grid -> (density, potential) ->
// sphere in registers.
//
// Numbers are 64-bit integers with one power-of-two scale per plane and pass,
// chosen from the largest value after every pass (a block maximum), so the
// rounding of a pass is 2^-58 of the plane's largest value or less.
#pragma once

#include <type_traits>

#include "fx.cuh"
#include "transforms.cuh"

namespace pdep {

template <int N>
struct FxLine {
  static constexpr int KI = N / 8;             // frequencies per parity
  static constexpr int KS = (KI + 7) / 8;      // k-steps of 8, sphere -> grid
  static constexpr int NTJ = (N / 4 + 8) / 8;  // tiles of 8 positions j <= N/4
  static constexpr int NTN = (KI + 7) / 8;     // tiles of 8 frequencies per parity
  static constexpr int NC = (NTJ + 1) / 2;     // chunks of two position tiles
  // table words: B fragments, sixteen words per lane (see paired_products)
  static constexpr int INV = KS * NTJ * 4 * 32 * 16;
  static constexpr int FWD = NC * NTN * 4 * 32 * 16;
};

// Scales.  A pass multiplies integers v of scale 2^e by table entries of scale
// 2^-62 and returns sums in units 2^SH of the leading digit product, that is of
// scale 2^(e + 50 - SH).  With C = 31 sqrt(2) < 2^5.5 lines' coefficients (95
// sqrt(2) < 2^7.1 for N = 192) and 64 sqrt(2) < 2^6.5 (2^8.1) positions:
//   columns in         |v| < 2^61
//   y inverse, SH 44:  |X| < 2^(61 + 5.5 - 6)       < 2^61, shifted left to < 2^61
//   z inverse, SH 45:  |X| < 2^(61 + 5.5 - 5)       < 2^62  (N = 192: SH 43)
//   times V:           X shifted left to < 2^62, the high word of X V < 2^60
//   z forward, SH 46:  |F| < 2^(60 + 6.5 - 4)       < 2^63  (N = 192: SH 44)
//   y forward, SH 46:  F shifted to < 2^60          |.| < 2^62.5
// Sums of two (inverse) or four (forward) of them are what becomes digits, below
// 2^62 in magnitude.
constexpr int SH_Y = 44, SH_YB = 46;
template <int N3>
constexpr int SH_Z = N3 <= 64 ? 45 : 43;
template <int N3>
constexpr int SH_ZB = N3 <= 64 ? 46 : 44;

struct cl {
  long long x, y;
};
// |v| < 2^(bit_length) for every v whose folded high word is at most m
__device__ __forceinline__ unsigned high_mag(long long v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ int bit_length(unsigned m) { return 64 - __clz(m); }

// v 2^-62 rounded to FP64 (integer arithmetic: a conversion on the FP64 pipe
// takes 32 clocks per warp), and 2^(q + 62), so that their product is v 2^q
__device__ __forceinline__ double fx_frac(long long v) {
  unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll(m);
  m <<= z & 63;
  const unsigned long long b =
      ((unsigned long long)(unsigned)(1023 - z) << 52) + (m >> 11) + ((m >> 10) & 1ull);
  const double r = m ? __longlong_as_double((long long)b) : 0.0;
  return v < 0 ? -r : r;
}
__device__ __forceinline__ double fx_unit(int q) { return scalbn(1.0, q + 62); }
// the S exact accumulators as one integer, units 2^SH of the leading one
template <int S, int SH>
__device__ __forceinline__ long long combine(const float (&acc)[S][4], int e) {
  constexpr unsigned long long M = FX_MAGIC;
  constexpr unsigned long long bias = (M << SH) + (M << (SH - 8)) + (M << (SH - 16)) +
                                      (M << (SH - 24)) + (M << (SH - 32)) + (M << (SH - 40));
  long long r = (long long)(0ull - bias);
  uint32_t top = 0;
#pragma unroll
  for (int d = 5; d >= 0; --d) {
    const int b = __float_as_int(acc[d][e]), sh = SH - 8 * d;
    if (sh >= 32)
      top += (uint32_t)b << (sh >= 32 ? sh - 32 : 0);
    else
      r += (long long)b * (1 << (sh < 31 ? sh : 0));
  }
  // the last sums lie below the unit: rounded
  uint32_t t = (uint32_t)__float_as_int(acc[6][e]) << 8;
  if constexpr (S == 8) t += (uint32_t)__float_as_int(acc[7][e]);
  constexpr int sr = 56 - SH;
  constexpr uint32_t c0 = (1u << (sr - 1)) - FX_MAGIC * (S == 8 ? 257u : 256u);
  r += (int)(t + c0) >> sr;
  return (long long)((unsigned long long)r + ((unsigned long long)top << 32));
}

template <int S>
__device__ __forceinline__ void digits(long long v0, long long v1, uint32_t (&d)[S]) {
  const uint2 u0 = biased(v0), u1 = biased(v1);
#pragma unroll
  for (int s = 0; s < S; ++s) d[s] = digit_pair(u0, u1, s);
}
__device__ __forceinline__ void load8(const uint4* p, uint32_t* b) {
  const uint4 q0 = __ldg(p), q1 = __ldg(p + 1);
  b[0] = q0.x;
  b[1] = q0.y;
  b[2] = q0.z;
  b[3] = q0.w;
  b[4] = q1.x;
  b[5] = q1.y;
  b[6] = q1.z;
  b[7] = q1.w;
}
__device__ __forceinline__ void magic4(float (&m)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) m[e] = __uint_as_float(FX_MAGIC);
}

// All digit products s + u <= S - 1 of operands with eight k-values.  The
// m16n8k8 and m16n8k16 shapes take the same time here, so two products of one
// accumulator, (s, u) and (s + 1, u - 1), share an m16n8k16: digit s fills its
// first eight k-values, digit s + 1 the other eight (20 instructions instead
// of 36).  Table words b: digits (1,0)(3,2)(5,4)(7,6), then (0,-)(2,1)(4,3)(6,5).
template <int S>
__device__ __forceinline__ void paired_products(float (&acc)[S][4], const uint32_t (&a0)[S],
                                                const uint32_t (&a1)[S], const uint32_t (&b)[16],
                                                bool first) {
  float m[4];
  magic4(m);
#pragma unroll
  for (int d = 0; d < S; ++d)
#pragma unroll
    for (int s = 0; s <= d; s += 2) {
      const int u = d - s;
      if (s + 1 <= d) {
        const uint32_t as[4] = {a0[s], a1[s], a0[s + 1], a1[s + 1]};
        // digit u: u odd in the first half at (u - 1), u even in the second at u
        const uint32_t bu = u & 1 ? b[u - 1] : b[8 + u], bl = u & 1 ? b[u] : b[8 + u + 1];
        if (first && s == 0)
          mma_f16_from(acc[d], m, as, bu, bl);
        else
          mma_f16(acc[d], as, bu, bl);
      } else if (first && s == 0) {
        mma_f16_k8_from(acc[d], m, a0[s], a1[s], b[8]);
      } else {
        mma_f16_k8(acc[d], a0[s], a1[s], b[8]);
      }
    }
}

// The sums over even and odd n of the cosine and sine parts of eight lines at
// the NT2 position tiles from nt0: q[0], q[2] = Ce + Co, Ce - Co and q[1], q[3] =
// Se + So, So - Se; ld(n): coefficient n of this thread's line, scaled by 2^sh
// here.
template <int N, int S, int SH, int NT2, typename LD>
__device__ __forceinline__ void inv_sums(const uint32_t* __restrict__ tab, int nt0, const LD& ld,
                                         int sh, long long (&q)[4][NT2][4]) {
  using L = FxLine<N>;
  const int lane = threadIdx.x & 31, t = lane & 3;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int i = 0; i < NT2; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) q[k][i][e] = 0;
  // one copy of the code for both parities: the kernel is long enough for the
  // instruction cache to matter
#pragma unroll 1
  for (int par = 0; par < 2; ++par) {
    cl p0[L::KS], p1[L::KS], m0[L::KS], m1[L::KS];
#pragma unroll
    for (int ks = 0; ks < L::KS; ++ks) {
      const int n0 = 2 * (8 * ks + 2 * t) + par;
      p0[ks] = ld(n0);
      p1[ks] = ld(n0 + 2);
      m1[ks] = ld(-n0 - 2);
      m0[ks] = n0 == 0 ? cl{0, 0} : ld(-n0);
    }
#pragma unroll
    for (int sine = 0; sine < 2; ++sine) {
      float acc[NT2][S][4];
#pragma unroll
      for (int ks = 0; ks < L::KS; ++ks) {
        uint32_t a0[S], a1[S];
        if (!sine) {
          digits<S>((p0[ks].x + m0[ks].x) << sh, (p1[ks].x + m1[ks].x) << sh, a0);
          digits<S>((p0[ks].y + m0[ks].y) << sh, (p1[ks].y + m1[ks].y) << sh, a1);
        } else {
          digits<S>((m0[ks].y - p0[ks].y) << sh, (m1[ks].y - p1[ks].y) << sh, a0);
          digits<S>((p0[ks].x - m0[ks].x) << sh, (p1[ks].x - m1[ks].x) << sh, a1);
        }
#pragma unroll
        for (int i = 0; i < NT2; ++i) {
          uint32_t b[16];
          const uint4* tb =
              (const uint4*)tab + (((ks * L::NTJ + nt0 + i) * 4 + 2 * sine + par) * 32 + lane) * 4;
          load8(tb, b);
          load8(tb + 2, b + 8);
          paired_products<S>(acc[i], a0, a1, b, ks == 0);
        }
      }
#pragma unroll
      for (int i = 0; i < NT2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const long long v = combine<S, SH>(acc[i], e);
          q[sine][i][e] += v;
          if (par == sine)
            q[2 + sine][i][e] += v;
          else
            q[2 + sine][i][e] -= v;
        }
    }
  }
}

// quadruples q[0..3] = X(j), X(-j), X(N/2 - j), X(N/2 + j), j = 8 (nt0 + i) +
// 2 t + (e & 1); e < 2 the real part, e >= 2 the imaginary part of line g
template <int N, int S, int SH, int NT2, typename LD>
__device__ __forceinline__ void line_inverse(const uint32_t* __restrict__ tab, int nt0,
                                             const LD& ld, int sh, long long (&q)[4][NT2][4]) {
  inv_sums<N, S, SH, NT2>(tab, nt0, ld, sh, q);
#pragma unroll
  for (int i = 0; i < NT2; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const long long cp = q[0][i][e], cm = q[2][i][e], sp = q[1][i][e], sm = q[3][i][e];
      q[0][i][e] = cp + sp;
      q[1][i][e] = cp - sp;
      q[2][i][e] = cm + sm;
      q[3][i][e] = cm - sm;
    }
}
// grid position of member k of the quadruple of j
template <int N>
__device__ __forceinline__ int quad_pos(int k, int j) {
  return k == 0 ? j : k == 1 ? (j ? N - j : 0) : k == 2 ? N / 2 - j : N / 2 + j;
}
// members 1 and 3 repeat 0 and 2 at j = 0, members 2 and 3 repeat 0 and 1 at N/4
template <int N>
__device__ __forceinline__ bool quad_new(int k, int j) {
  return j <= N / 4 && !(j == 0 && (k & 1)) && !(j == N / 4 && k >= 2);
}

// One group's product (grp: cosine even, cosine odd, sine even, sine odd n)
// over the NT2 position tiles of chunk c from the folded quadruples f:
// frequencies 2 kk + (grp & 1), kk = 8 nt + 2 t + (e & 1).
template <int N, int S, int SH, int NT2, int SINE>
__device__ __forceinline__ void fwd_group(const uint32_t* __restrict__ tab, int c, int nt, int par,
                                          const long long (&f)[NT2][4], long long (&out)[4]) {
  using L = FxLine<N>;
  const int lane = threadIdx.x & 31;
  float acc[S][4];
  uint32_t a[2 * NT2][S];
#pragma unroll
  for (int i = 0; i < NT2; ++i) {
    if (!SINE) {
      digits<S>(f[i][0], f[i][1], a[2 * i]);
      digits<S>(f[i][2], f[i][3], a[2 * i + 1]);
    } else {
      // -i Q: the real row takes the imaginary part, the imaginary row minus
      // the real part
      digits<S>(f[i][2], f[i][3], a[2 * i]);
      digits<S>(-f[i][0], -f[i][1], a[2 * i + 1]);
    }
  }
  const uint4* tb =
      (const uint4*)tab + (((c * L::NTN + nt) * 4 + 2 * SINE + par) * 32 + lane) * 4;
  uint32_t b[16];
  load8(tb, b);
  load8(tb + 2, b + 8);
  if constexpr (NT2 == 2) {
    // sixteen k-values: digit u is b[2 u], b[2 u + 1]
    float m[4];
    magic4(m);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const uint32_t as[4] = {a[0][s], a[1][s], a[2][s], a[3][s]};
#pragma unroll
      for (int u = 0; u + s < S; ++u) {
        if (s == 0)
          mma_f16_from(acc[u], m, as, b[2 * u], b[2 * u + 1]);
        else
          mma_f16(acc[s + u], as, b[2 * u], b[2 * u + 1]);
      }
    }
  } else {
    paired_products<S>(acc, a[0], a[1], b, true);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) out[e] = combine<S, SH>(acc, e);
}
// first fold of the quadruples: u from X(j), X(-j), w from X(N/2 -+ j); the
// even (odd) frequencies take u + w (u - w) in the cosine part and u - w
// (u + w) in the sine part
template <int NT2, int SINE>
__device__ __forceinline__ void fold(const long long (&q)[4][NT2][4], long long (&u)[NT2][4],
                                     long long (&w)[NT2][4]) {
#pragma unroll
  for (int i = 0; i < NT2; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      u[i][e] = SINE ? q[0][i][e] - q[1][i][e] : q[0][i][e] + q[1][i][e];
      w[i][e] = SINE ? q[2][i][e] - q[3][i][e] : q[2][i][e] + q[3][i][e];
    }
}
template <int NT2, int SINE>
__device__ __forceinline__ void fold2(const long long (&u)[NT2][4], const long long (&w)[NT2][4],
                                      int par, long long (&f)[NT2][4]) {
#pragma unroll
  for (int i = 0; i < NT2; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) f[i][e] = par == SINE ? u[i][e] + w[i][e] : u[i][e] - w[i][e];
}

}  // namespace pdep
