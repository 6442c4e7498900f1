// The FP64 column passes on the tensor cores (fx_line.cuh): x-lines between the
// sphere and the column scratch.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

#include "fx_line.cuh"
#include "profile.cuh"

namespace pdep {
namespace {

// One warp per eight upper columns: the eight lines and their mirror lines are
// two tiles of rows made from the same sphere members.  Each warp scales by
// its own largest member, and the scratch holds FP64 numbers.
constexpr int COLS_WARPS = 4;

// Frequencies |n| <= 15: the digit tables' entries of |n| >= N1 / 4 are zero.
struct Member {
  double ax, ay, bx, by;
};

template <int N1, int S, bool COUL>
__global__ void __launch_bounds__(32 * COLS_WARPS, 3)
    k_cols_fx_fwd(SphereDev<double> s, const double* __restrict__ x, long long ldx, ItemMap map,
                  int n_items, cpx<double>* __restrict__ b1) {
  using L = FxLine<N1>;
  const int nl = listed_count(map);
  const int units = (s.n_ucol + 7) / 8;
  const long long unit = (long long)blockIdx.x * COLS_WARPS + (threadIdx.x >> 5);
  const int item = (int)(unit / units);
  if (item >= items_of(map, n_items, nl)) return;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int uc = (int)(unit - (long long)item * units) * 8 + g;
  const UCol c = s.ucol[min(uc, s.n_ucol - 1)];
  const bool live = uc < s.n_ucol && ucol_in_range(s, c), self = c.col == c.mcol;
  const int R1 = live ? c.R1 : -1;
  const int ia = map.vec(item, 0, nl), ib = map.vec(item, 1, nl);
  const double* xa = ia >= 0 ? x + (long long)ia * ldx : nullptr;
  const double* xb = ib >= 0 ? x + (long long)ib * ldx : nullptr;
  cpx<double>* base = b1 + (long long)item * N1 * s.n_col;

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
  // the warp's members as integers below 2^60 in shared memory (their packed
  // sums stay below 2^61), each read once from the sphere
  __shared__ __align__(16) long long mem[COLS_WARPS][32 * 8][4];
  long long(*mine)[4] = mem[threadIdx.x >> 5] + g * 32;
  Member m[8];
  int ex = 1;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int n = 4 * t + (q & 3);
    m[q] = member(q < 4 ? n : -n);
    ex = max(ex, max(max(exp_of(m[q].ax), exp_of(m[q].ay)), max(exp_of(m[q].bx), exp_of(m[q].by))));
  }
  const int er = __reduce_max_sync(0xffffffffu, ex);
  const double scale = er == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                   : fx_unit(er - 1082 + 50 - SH_Y) * 0.70710678118654752440;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int n = 4 * t + (q & 3);
    longlong2* d = reinterpret_cast<longlong2*>(mine[q < 4 ? 16 + n : 16 - n]);
    if (q >= 4 && n == 0) continue;
    d[0] = make_longlong2(fx_of(m[q].ax, er) >> 2, fx_of(m[q].ay, er) >> 2);
    d[1] = make_longlong2(fx_of(m[q].bx, er) >> 2, fx_of(m[q].by, er) >> 2);
  }
  __syncwarp();
#pragma unroll 1
  for (int mirror = 0; mirror < 2; ++mirror) {
    // (a + i b)(n) on the column, its mirror's conj(a + i b)(-n) on the mirror
    auto ld = [&](int n) {
      const bool flip = mirror != (self && n < 0);
      const longlong2* d = reinterpret_cast<const longlong2*>(mine[16 + (mirror ? -n : n)]);
      const longlong2 a = d[0], b = d[1];
      return flip ? cl{a.x + b.y, b.x - a.y} : cl{a.x - b.y, b.x + a.y};
    };
    auto chunk = [&](auto nt2, int nt0) {
      constexpr int NT2 = decltype(nt2)::value;
      long long q[4][NT2][4];
      line_inverse<N1, S, SH_Y, NT2>(s.fx1, nt0, ld, 0, q);
      if (!live || (mirror && self)) return;
      const int col = mirror ? c.mcol : c.col;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < NT2; ++i)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = 8 * (nt0 + i) + 2 * t + e;
            if (!quad_new<N1>(k, j)) continue;
            base[(long long)quad_pos<N1>(k, j) * s.n_col + col] =
                mk(fx_frac(q[k][i][e]) * scale, fx_frac(q[k][i][e + 2]) * scale);
          }
    };
    if constexpr (L::NTJ >= 2) chunk(std::integral_constant<int, 2>{}, 0);
    if constexpr (L::NTJ % 2) chunk(std::integral_constant<int, 1>{}, L::NTJ - 1);
  }
}

template <int N1, int S>
__global__ void __launch_bounds__(32 * COLS_WARPS, 3)
    k_cols_fx_bwd(SphereDev<double> s, const cpx<double>* __restrict__ b1, ItemMap map, int n_items,
                  Epilogue<double> ep) {
  using L = FxLine<N1>;
  const int nl = listed_count(map);
  const int units = (s.n_ucol + 7) / 8;
  const long long unit = (long long)blockIdx.x * COLS_WARPS + (threadIdx.x >> 5);
  const int item = (int)(unit / units);
  if (item >= items_of(map, n_items, nl)) return;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int uc = (int)(unit - (long long)item * units) * 8 + g;
  const UCol c = s.ucol[min(uc, s.n_ucol - 1)];
  const bool live = uc < s.n_ucol && ucol_in_range(s, c), self = c.col == c.mcol;
  const cpx<double>* base = b1 + (long long)item * N1 * s.n_col;

  // F[par][e][0 / 1]: the line's coefficients at +-n, n = 2 (2 t + e) + par
  cpx<double> f[2][2][2][2];
#pragma unroll
  for (int mirror = 0; mirror < 2; ++mirror) {
    const bool use = live && !(mirror && self);
    const cpx<double>* column = base + (mirror ? c.mcol : c.col);
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
    const double scale = er == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                     : fx_unit(er - 1082 + 50 - SH_YB);
#pragma unroll
    for (int par = 0; par < 2; ++par)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        f[mirror][par][e][0] = mk(fx_frac(co[par][e] + so[par][e]) * scale,
                                  fx_frac(co[par][e + 2] + so[par][e + 2]) * scale);
        f[mirror][par][e][1] = mk(fx_frac(co[par][e] - so[par][e]) * scale,
                                  fx_frac(co[par][e + 2] - so[par][e + 2]) * scale);
      }
  }
  if (!live) return;
  // Hermitian unpacking of the two real fields and the epilogue
  const int ia = map.vec(item, 0, nl), ib = map.vec(item, 1, nl);
  const double rs2 = 0.70710678118654752440084436210485 * ep.scale;
  auto write = [&](int vec, int j, double val, double diag) {
    if (vec < 0) return;
    double* y = ep.y + (long long)vec * ep.ldy;
    double r = val;
    if (ep.x_in) {
      const double sh = ep.shift ? ep.shift[vec % ep.shift_period] : 0.0;
      r += (diag + sh) * ep.x_in[(long long)vec * ep.ldx + j];
    }
    if (ep.beta != 0) r += ep.beta * y[j];
    y[j] = r;
  };
#pragma unroll
  for (int par = 0; par < 2; ++par)
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int neg = 0; neg < 2; ++neg) {
        const int n = 2 * (2 * t + e) + par;
        if (n > c.R1 || (neg && (n == 0 || self))) continue;
        const cpx<double> d = f[0][par][e][neg];
        if (self && n == 0) {
          const double cf = ep.coef == COEF_ONE ? ep.scale : 0.0;
          write(ia, 2 * s.n_half, cf * d.x, 0.0);
          write(ib, 2 * s.n_half, cf * d.y, 0.0);
          continue;
        }
        // the mirror line at -n (the self-mirrored column's own)
        const cpx<double> dm = self ? f[0][par][e][1] : f[1][par][e][1 - neg];
        const int k = self ? c.h0 + n - 1 : c.h0 + (neg ? -n : n) + c.R1;
        const double cf =
            ep.coef == COEF_SQRT_COULOMB ? rs2 * sqrt(12.566370614359172953850573533118 / s.g2[k]) : rs2;
        const double dg = ep.kin * s.kin[k];
        write(ia, 2 * k, cf * (d.x + dm.x), dg);
        write(ia, 2 * k + 1, cf * (d.y - dm.y), dg);
        write(ib, 2 * k, cf * (d.y + dm.y), dg);
        write(ib, 2 * k + 1, -(cf * (d.x - dm.x)), dg);
      }
}

template <int N1>
cudaError_t cols_fwd_fx_impl(const SphereDev<double>& s, const double* x, long long ldx,
                             const ItemMap& map, int n_items, int coef, cpx<double>* b1,
                             int digits, cudaStream_t st) {
  const long long units = (long long)n_items * ((s.n_ucol + 7) / 8);
  const unsigned blocks = (unsigned)((units + COLS_WARPS - 1) / COLS_WARPS);
  const double lines = (double)n_items * s.n_col;
  ProfScope ps(digits < FX_S ? PC_COLS_DF : PC_COLS_F64, st, lines * 5.0 * N1 * std::log2((double)N1),
               (double)n_items * 2.0 * s.n_pw * sizeof(double) + lines * N1 * 2.0 * sizeof(double),
               map.list ? map.n_dev : nullptr, map.n_list);
  count_launch();
  auto kern = coef == COEF_SQRT_COULOMB ? k_cols_fx_fwd<N1, 8, true>
              : digits < FX_S           ? k_cols_fx_fwd<N1, 7, false>
                                        : k_cols_fx_fwd<N1, 8, false>;
  kern<<<blocks, 32 * COLS_WARPS, 0, st>>>(s, x, ldx, map, n_items, b1);
  return cudaGetLastError();
}
template <int N1>
cudaError_t cols_bwd_fx_impl(const SphereDev<double>& s, const cpx<double>* b1, const ItemMap& map,
                             int n_items, const Epilogue<double>& ep, int digits, cudaStream_t st) {
  const long long units = (long long)n_items * ((s.n_ucol + 7) / 8);
  const unsigned blocks = (unsigned)((units + COLS_WARPS - 1) / COLS_WARPS);
  const double lines = (double)n_items * s.n_col;
  const double vecs = (double)n_items * 2.0 * s.n_pw * sizeof(double);
  ProfScope ps(digits < FX_S ? PC_COLS_DF : PC_COLS_F64, st, lines * 5.0 * N1 * std::log2((double)N1),
               lines * N1 * 2.0 * sizeof(double) +
                   vecs * (1.0 + (ep.x_in ? 1.0 : 0.0) + (ep.beta != 0 ? 1.0 : 0.0)),
               map.list ? map.n_dev : nullptr, map.n_list);
  count_launch();
  auto kern = digits < FX_S ? k_cols_fx_bwd<N1, 7> : k_cols_fx_bwd<N1, 8>;
  kern<<<blocks, 32 * COLS_WARPS, 0, st>>>(s, b1, map, n_items, ep);
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
