// The FP64 column passes on the tensor cores (fx_line.cuh): x-lines between the
// sphere and the column scratch.
#include <algorithm>
#include <cmath>
#include <vector>

#include "fx_line.cuh"
#include "profile.cuh"

namespace pdep {
namespace {

// Two warps per eight upper columns: the eight lines and their mirror lines are
// two tiles of rows made from the same sphere members.  A column group scales by
// its own largest member, and the scratch holds FP64 numbers.
//
// Bound by the latency of a warp's chain (conversion, digits, products, sums):
// a tile per warp, with the members (in) or the coefficients (out) exchanged
// through shared memory, halves it against one warp for both tiles.  A pass over
// 128 items on 24^3 19.3 -> 14.2 us, on 48^3 53.6 -> 50.1 us (82 us as FP64
// FFTs).
constexpr int COLS_PAIRS = 2;  // column groups per block
constexpr int COLS_THREADS = 64 * COLS_PAIRS;

struct Member {
  double ax, ay, bx, by;
};

// Frequencies |n| <= 15: the digit tables' entries of |n| >= N1 / 4 are zero.
template <int N1, int S, bool COUL>
__global__ void __launch_bounds__(COLS_THREADS, 3)
    k_cols_fx_fwd(SphereDev<double> s, const double* __restrict__ x, long long ldx, ItemMap map,
                  int n_items, cpx<double>* __restrict__ b1) {
  using L = FxLine<N1>;
  __shared__ __align__(16) long long mem[COLS_PAIRS][32 * 8][4];
  __shared__ int exps[2 * COLS_PAIRS];
  const int nl = listed_count(map);
  const int units = (s.n_ucol + 7) / 8, warp = threadIdx.x >> 5, pair = warp >> 1, mirror = warp & 1;
  const long long unit = (long long)blockIdx.x * COLS_PAIRS + pair;
  int item = (int)(unit / units);
  if ((long long)blockIdx.x * COLS_PAIRS / units >= items_of(map, n_items, nl)) return;
  const bool any = item < items_of(map, n_items, nl);
  if (!any) item = 0;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int uc = any ? (int)(unit - (long long)item * units) * 8 + g : s.n_ucol;
  const UCol c = s.ucol[min(uc, s.n_ucol - 1)];
  const bool live = uc < s.n_ucol && ucol_in_range(s, c), self = c.col == c.mcol;
  const int R1 = live ? c.R1 : -1;
  const int ia = map.vec(item, 0, nl), ib = map.vec(item, 1, nl);
  const double* xa = ia >= 0 ? x + (long long)ia * ldx : nullptr;
  const double* xb = ib >= 0 ? x + (long long)ib * ldx : nullptr;

  // member n1 of this thread's column (|n| for the self-mirrored one, whose
  // n = 0 holds c(0), sqrt 2 below the others' scale)
  auto member = [&](int n) {
    Member m{0.0, 0.0, 0.0, 0.0};
    if (n > R1 || n < -R1) return m;
    if (self && n == 0) {
      if (!COUL) {
        const int k0 = 2 * s.n_half;
        m.ax = xa ? xa[k0] * 1.4142135623730951 : 0.0;
        m.bx = xb ? xb[k0] * 1.4142135623730951 : 0.0;
      }
      return m;
    }
    const int k = self ? c.h0 + abs(n) - 1 : c.h0 + n + c.R1;
    if (xa) {
      m.ax = xa[2 * k];
      m.ay = xa[2 * k + 1];
    }
    if (xb) {
      m.bx = xb[2 * k];
      m.by = xb[2 * k + 1];
    }
    if constexpr (COUL) {
      const double w = sqrt(12.566370614359172953850573533118 / s.g2[k]);
      m.ax *= w;
      m.ay *= w;
      m.bx *= w;
      m.by *= w;
    }
    return m;
  };
  // the group's members as integers below 2^60 (their packed sums stay below
  // 2^61), each read once: n >= 0 by the first warp, n < 0 by the second
  long long(*mine)[4] = mem[pair] + g * 32;
  Member m[4];
  int ex = 1;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int n = 4 * t + q;
    m[q] = member(mirror ? -n : n);
    ex = max(ex, max(max(exp_of(m[q].ax), exp_of(m[q].ay)), max(exp_of(m[q].bx), exp_of(m[q].by))));
  }
  ex = __reduce_max_sync(0xffffffffu, ex);
  if (lane == 0) exps[warp] = ex;
  __syncthreads();
  const int er = max(exps[2 * pair], exps[2 * pair + 1]);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int n = 4 * t + q;
    if (mirror && n == 0) continue;
    longlong2* d = reinterpret_cast<longlong2*>(mine[mirror ? 16 - n : 16 + n]);
    d[0] = make_longlong2(fx_of(m[q].ax, er) >> 2, fx_of(m[q].ay, er) >> 2);
    d[1] = make_longlong2(fx_of(m[q].bx, er) >> 2, fx_of(m[q].by, er) >> 2);
  }
  __syncthreads();
  const double scale = er == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                   : fx_unit(er - 1082 + 50 - SH_Y) * 0.70710678118654752440;
  // (a + i b)(n) on the column, its mirror's conj(a + i b)(-n) on the mirror
  auto ld = [&](int n) {
    const bool flip = mirror != (self && n < 0);
    const longlong2* d = reinterpret_cast<const longlong2*>(mine[16 + (mirror ? -n : n)]);
    const longlong2 a = d[0], b = d[1];
    return flip ? cl{a.x + b.y, b.x - a.y} : cl{a.x - b.y, b.x + a.y};
  };
  const int col = mirror ? c.mcol : c.col;
  cpx<double>* base = b1 + (long long)item * N1 * s.n_col + col;
  auto chunk = [&](auto nt2, int nt0) {
    constexpr int NT2 = decltype(nt2)::value;
    long long q[4][NT2][4];
    line_inverse<N1, S, SH_Y, NT2>(s.fx1, nt0, ld, 0, q);
    if (!live || (mirror && self)) return;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < NT2; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = 8 * (nt0 + i) + 2 * t + e;
          if (!quad_new<N1>(k, j)) continue;
          base[(long long)quad_pos<N1>(k, j) * s.n_col] =
              mk(fx_frac(q[k][i][e]) * scale, fx_frac(q[k][i][e + 2]) * scale);
        }
  };
  if constexpr (L::NTJ >= 2) chunk(std::integral_constant<int, 2>{}, 0);
  if constexpr (L::NTJ % 2) chunk(std::integral_constant<int, 1>{}, L::NTJ - 1);
}

template <int N1, int S>
__global__ void __launch_bounds__(COLS_THREADS, 3)
    k_cols_fx_bwd(SphereDev<double> s, const cpx<double>* __restrict__ b1, ItemMap map, int n_items,
                  Epilogue<double> ep) {
  using L = FxLine<N1>;
  // coefficients of the warps' lines at n and -n (element 2 (2 par + e) and the
  // next) in units of their own scale
  __shared__ __align__(16) cl coef[2 * COLS_PAIRS][8][32];
  __shared__ int exps[2 * COLS_PAIRS];
  const int nl = listed_count(map);
  const int units = (s.n_ucol + 7) / 8, warp = threadIdx.x >> 5, pair = warp >> 1, mirror = warp & 1;
  const long long unit = (long long)blockIdx.x * COLS_PAIRS + pair;
  int item = (int)(unit / units);
  if ((long long)blockIdx.x * COLS_PAIRS / units >= items_of(map, n_items, nl)) return;
  const bool any = item < items_of(map, n_items, nl);
  if (!any) item = 0;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int uc = any ? (int)(unit - (long long)item * units) * 8 + g : s.n_ucol;
  const UCol c = s.ucol[min(uc, s.n_ucol - 1)];
  const bool live = uc < s.n_ucol && ucol_in_range(s, c), self = c.col == c.mcol;
  {
    const bool use = live && !(mirror && self);
    const cpx<double>* column =
        b1 + (long long)item * N1 * s.n_col + (mirror ? c.mcol : c.col);
    long long co[2][4], so[2][4];
#pragma unroll
    for (int par = 0; par < 2; ++par)
#pragma unroll
      for (int e = 0; e < 4; ++e) co[par][e] = so[par][e] = 0;
    // the largest exponent of the warp's lines: up to 48 points they stay in
    // registers meanwhile, the 64-point ones are read twice
    int er = 1;
    if constexpr (L::NTJ > 2) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < 2 * L::NTJ; ++i) {
          const int j = 8 * (i >> 1) + 2 * t + (i & 1);
          if (!use || j > N1 / 4) continue;
          const cpx<double> z = column[(long long)quad_pos<N1>(k, j) * s.n_col];
          er = max(er, max(exp_of(z.x), exp_of(z.y)));
        }
      er = __reduce_max_sync(0xffffffffu, er);
    }
    auto chunk = [&](auto nt2, int ch) {
      constexpr int NT2 = decltype(nt2)::value;
      double z[4][NT2][4];
      long long q[4][NT2][4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < NT2; ++i)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = 8 * (2 * ch + i) + 2 * t + e;
            cpx<double> v = mk(0.0, 0.0);
            if (use && j <= N1 / 4) v = column[(long long)quad_pos<N1>(k, j) * s.n_col];
            z[k][i][e] = v.x;
            z[k][i][e + 2] = v.y;
            if constexpr (L::NTJ <= 2) er = max(er, max(exp_of(v.x), exp_of(v.y)));
          }
      if constexpr (L::NTJ <= 2) er = __reduce_max_sync(0xffffffffu, er);
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < NT2; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) q[k][i][e] = fx_of(z[k][i][e], er) >> 2;
      long long cu[NT2][4], cw[NT2][4], su[NT2][4], sw[NT2][4];
      fold<NT2, 0>(q, cu, cw);
      fold<NT2, 1>(q, su, sw);
#pragma unroll 1
      for (int par = 0; par < 2; ++par) {
        long long y[NT2][4], v[4], w[4];
        fold2<NT2, 0>(cu, cw, par, y);
        fwd_group<N1, S, SH_YB, NT2, 0>(s.fx1 + L::INV, ch, 0, par, y, v);
        fold2<NT2, 1>(su, sw, par, y);
        fwd_group<N1, S, SH_YB, NT2, 1>(s.fx1 + L::INV, ch, 0, par, y, w);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (par == 0) {
            co[0][e] += v[e];
            so[0][e] += w[e];
          } else {
            co[1][e] += v[e];
            so[1][e] += w[e];
          }
        }
      }
    };
    if constexpr (L::NTJ >= 2) chunk(std::integral_constant<int, 2>{}, 0);
    if constexpr (L::NTJ % 2) chunk(std::integral_constant<int, 1>{}, L::NTJ / 2);
    // one bit of headroom for the sum with the mirror line
#pragma unroll
    for (int par = 0; par < 2; ++par)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        coef[warp][2 * (2 * par + e)][lane] =
            cl{(co[par][e] + so[par][e]) >> 1, (co[par][e + 2] + so[par][e + 2]) >> 1};
        coef[warp][2 * (2 * par + e) + 1][lane] =
            cl{(co[par][e] - so[par][e]) >> 1, (co[par][e + 2] - so[par][e + 2]) >> 1};
      }
    if (lane == 0) exps[warp] = er;
  }
  __syncthreads();
  if (!live) return;
  // Hermitian unpacking of the two real fields, both lines in the larger unit,
  // and the epilogue: the first warp writes the members at n, the second those
  // at -n
  const int e0 = exps[2 * pair], e1 = exps[2 * pair + 1], em = max(e0, e1);
  const int r0 = min(em - e0, 63), r1 = min(em - e1, 63);
  const double fu = em == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                : fx_unit(em - 1082 + 50 - SH_YB + 1) * ep.scale;
  const int ia = map.vec(item, 0, nl), ib = map.vec(item, 1, nl);
  double* ya = ia >= 0 ? ep.y + (long long)ia * ep.ldy : nullptr;
  double* yb = ib >= 0 ? ep.y + (long long)ib * ep.ldy : nullptr;
  const double* xa = ep.x_in && ia >= 0 ? ep.x_in + (long long)ia * ep.ldx : nullptr;
  const double* xb = ep.x_in && ib >= 0 ? ep.x_in + (long long)ib * ep.ldx : nullptr;
  const double sa = xa && ep.shift ? ep.shift[ia % ep.shift_period] : 0.0;
  const double sb = xb && ep.shift ? ep.shift[ib % ep.shift_period] : 0.0;
  auto write = [&](double* y, const double* x, int j, long long v, double cf, double diag) {
    if (!y) return;
    double r = cf * fx_frac(v);
    if (x) r += diag * x[j];
    if (ep.beta != 0) r += ep.beta * y[j];
    y[j] = r;
  };
  const int w0 = 2 * pair;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int n = 2 * (2 * t + (q & 1)) + (q >> 1);
    if (n > c.R1 || (mirror && (n == 0 || self))) continue;
    cl d = coef[w0][2 * q + mirror][lane];
    d.x >>= r0;
    d.y >>= r0;
    if (self && n == 0) {
      const double cf = ep.coef == COEF_ONE ? fu : 0.0;
      write(ya, xa, 2 * s.n_half, d.x, cf, sa);
      write(yb, xb, 2 * s.n_half, d.y, cf, sb);
      continue;
    }
    // the mirror line at -n (the self-mirrored column's own)
    cl dm = self ? coef[w0][2 * q + 1][lane] : coef[w0 + 1][2 * q + 1 - mirror][lane];
    const int rm = self ? r0 : r1;
    dm.x >>= rm;
    dm.y >>= rm;
    const int k = self ? c.h0 + n - 1 : c.h0 + (mirror ? -n : n) + c.R1;
    double cf = fu * 0.70710678118654752440084436210485;
    if (ep.coef == COEF_SQRT_COULOMB) cf *= sqrt(12.566370614359172953850573533118 / s.g2[k]);
    const double dg = ep.kin != 0 ? s.kin[k] : 0.0;
    write(ya, xa, 2 * k, d.x + dm.x, cf, dg + sa);
    write(ya, xa, 2 * k + 1, d.y - dm.y, cf, dg + sa);
    write(yb, xb, 2 * k, d.y + dm.y, cf, dg + sb);
    write(yb, xb, 2 * k + 1, dm.x - d.x, cf, dg + sb);
  }
}

template <int N1>
cudaError_t cols_fwd_fx_impl(const SphereDev<double>& s, const double* x, long long ldx,
                             const ItemMap& map, int n_items, int coef, cpx<double>* b1,
                             int digits, cudaStream_t st) {
  const long long units = (long long)n_items * ((s.n_ucol + 7) / 8);
  const unsigned blocks = (unsigned)((units + COLS_PAIRS - 1) / COLS_PAIRS);
  const double lines = (double)n_items * s.n_col;
  ProfScope ps(digits < FX_S ? PC_COLS_DF : PC_COLS_F64, st, lines * 5.0 * N1 * std::log2((double)N1),
               (double)n_items * 2.0 * s.n_pw * sizeof(double) + lines * N1 * 2.0 * sizeof(double),
               map.list ? map.n_dev : nullptr, map.n_list);
  count_launch();
  auto kern = coef == COEF_SQRT_COULOMB ? k_cols_fx_fwd<N1, 8, true>
              : digits < FX_S           ? k_cols_fx_fwd<N1, 7, false>
                                        : k_cols_fx_fwd<N1, 8, false>;
  kern<<<blocks, COLS_THREADS, 0, st>>>(s, x, ldx, map, n_items, b1);
  return cudaGetLastError();
}
template <int N1>
cudaError_t cols_bwd_fx_impl(const SphereDev<double>& s, const cpx<double>* b1, const ItemMap& map,
                             int n_items, const Epilogue<double>& ep, int digits, cudaStream_t st) {
  const long long units = (long long)n_items * ((s.n_ucol + 7) / 8);
  const unsigned blocks = (unsigned)((units + COLS_PAIRS - 1) / COLS_PAIRS);
  const double lines = (double)n_items * s.n_col;
  const double vecs = (double)n_items * 2.0 * s.n_pw * sizeof(double);
  ProfScope ps(digits < FX_S ? PC_COLS_DF : PC_COLS_F64, st, lines * 5.0 * N1 * std::log2((double)N1),
               lines * N1 * 2.0 * sizeof(double) +
                   vecs * (1.0 + (ep.x_in ? 1.0 : 0.0) + (ep.beta != 0 ? 1.0 : 0.0)),
               map.list ? map.n_dev : nullptr, map.n_list);
  count_launch();
  auto kern = digits < FX_S ? k_cols_fx_bwd<N1, 7> : k_cols_fx_bwd<N1, 8>;
  kern<<<blocks, COLS_THREADS, 0, st>>>(s, b1, map, n_items, ep);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cols_fwd(const SphereDev<double>& s, const double* x, long long ldx, ItemMap map,
                            int n_items, int coef, cpx<double>* b1, cudaStream_t st, int digits) {
  if (n_items <= 0) return cudaSuccess;
  switch (s.N1) {
    case 24: return cols_fwd_fx_impl<24>(s, x, ldx, map, n_items, coef, b1, digits, st);
    case 32: return cols_fwd_fx_impl<32>(s, x, ldx, map, n_items, coef, b1, digits, st);
    case 40: return cols_fwd_fx_impl<40>(s, x, ldx, map, n_items, coef, b1, digits, st);
    case 48: return cols_fwd_fx_impl<48>(s, x, ldx, map, n_items, coef, b1, digits, st);
    case 64: return cols_fwd_fx_impl<64>(s, x, ldx, map, n_items, coef, b1, digits, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_cols_bwd(const SphereDev<double>& s, const cpx<double>* b1, ItemMap map,
                            int n_items, const Epilogue<double>& ep, cudaStream_t st, int digits) {
  if (n_items <= 0) return cudaSuccess;
  switch (s.N1) {
    case 24: return cols_bwd_fx_impl<24>(s, b1, map, n_items, ep, digits, st);
    case 32: return cols_bwd_fx_impl<32>(s, b1, map, n_items, ep, digits, st);
    case 40: return cols_bwd_fx_impl<40>(s, b1, map, n_items, ep, digits, st);
    case 48: return cols_bwd_fx_impl<48>(s, b1, map, n_items, ep, digits, st);
    case 64: return cols_bwd_fx_impl<64>(s, b1, map, n_items, ep, digits, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pdep
