// The FP64 slab pass on the tensor cores (fx_line.cuh): y- and z-lines of one
// x-plane of one item per block.
//
// Bound by the issue of the digit conversions and the integer sums and their
// latency (seven digits with the density on 48^3: 43% of the issue slots, ALU 49%,
// FP64 pipe 39%, tensor pipe 17%, two blocks of six warps per SM), no longer by the
// FP64 pipe.  128 items on 48^3: 0.88 -> 0.27 ms; the mixed
// refinement's passes (seven digits, before in double-float) over 4096 items,
// there and back with the density and from the grid, 35.9 -> 25.3 ms.
#pragma once

#include "fx_line.cuh"
#include "profile.cuh"

namespace pdep {
namespace {

// Element (n3 slot, i2) of the shared plane: rows of N2 complex integers,
// columns swizzled inside blocks of eight so that the four rows (4 apart) of a
// z-line access and the two rows of a y-line access fall on distinct banks.
template <int N2>
__device__ __forceinline__ int t2_fx(int row, int col) {
  return row * N2 + (col ^ ((((row >> 2) & 3) << 1) | (row & 1)));
}

constexpr int FX_MX = 8;  // block maxima: 0 plane in, 1 after y, 2 .. z chunks, 7 after z

__device__ __forceinline__ void block_max(unsigned* slot, unsigned m) {
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(slot, m);
}

// z-lines of one warp (eight lines): the NT2 position tiles of chunk c.
// Adds the chunk's forward sums to fo (units 2^fe).
template <int S, int N2, int N3, int NT2, int SINE>
__device__ __forceinline__ void z_back(const SphereDev<double>& s, int c, int rs,
                                       const long long (&q)[4][NT2][4],
                                       long long (&fo)[4][FxLine<N3>::NTN][4]) {
  using L = FxLine<N3>;
  long long u[NT2][4], w[NT2][4];
  fold<NT2, SINE>(q, u, w);
#pragma unroll 1
  for (int par = 0; par < 2; ++par) {
    long long f[NT2][4];
    fold2<NT2, SINE>(u, w, par, f);
#pragma unroll
    for (int i = 0; i < L::NTN; ++i) {
      long long v[4];
      fwd_group<N3, S, SH_ZB<N3>, NT2, SINE>(s.fx3 + L::INV, c, i, par, f, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const long long x = v[e] >> min(rs, 63);
        if (par == 0)
          fo[2 * SINE][i][e] = (c > 0 ? fo[2 * SINE][i][e] : 0) + x;
        else
          fo[2 * SINE + 1][i][e] = (c > 0 ? fo[2 * SINE + 1][i][e] : 0) + x;
      }
    }
  }
}

// AT (HPSI): with the density response, its array from a.dn_at
template <int MODE, bool AT, int S, int N2, int N3, int NT2>
__device__ __forceinline__ void z_chunk(const SphereDev<double>& s, const SlabArgs<double>& a, int nl,
                                        int item, long long plane, const cl* T2, unsigned* mx,
                                        int c, int e2, int sh2,
                                        long long (&fo)[4][FxLine<N3>::NTN][4], int& fe) {
  using L = FxLine<N3>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int i2 = warp * 8 + g;
  const int R3 = s.R3;
  const long long line = plane + (long long)i2 * N3;
  long long q[4][NT2][4];
  int e4;
  if constexpr (MODE == SLAB_FROM_GRID) {
    const int grp = item / a.map.items_per_group;
    const int w = item - grp * a.map.items_per_group;
    const double* f = a.src.f ? a.src.f + (long long)grp * a.src.f_stride + line : nullptr;
    const double* ga = a.src.g + (long long)(2 * w) * a.src.g_stride + line;
    const double* gb = 2 * w + 1 < a.map.vecs_per_group ? ga + a.src.g_stride : nullptr;
    int ex = 1;
    double p[4][NT2][4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < NT2; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = 8 * (2 * c + i) + 2 * t + e;
          const int pos = quad_pos<N3>(k, min(j, N3 / 4));
          const double fv = f ? f[pos] : 1.0;
          const double va = j <= N3 / 4 ? fv * ga[pos] : 0.0;
          const double vb = j <= N3 / 4 && gb ? fv * gb[pos] : 0.0;
          p[k][i][e] = va;
          p[k][i][e + 2] = vb;
          ex = max(ex, max(exp_of(va), exp_of(vb)));
        }
    block_max(&mx[2 + c], (unsigned)ex);
    __syncthreads();
    const int er = (int)mx[2 + c];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < NT2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) q[k][i][e] = fx_of(p[k][i][e], er == 0x7ff ? 0x7fe : er) >> 2;
    e4 = er - 1082;
  } else {
    auto ld = [&](int n) {
      cl v{0, 0};
      if (n <= R3 && n >= -R3) v = T2[t2_fx<N2>(n + R3, i2)];
      return v;
    };
    line_inverse<N3, S, SH_Z<N3>, NT2>(s.fx3, 2 * c, ld, sh2, q);
    const int e3 = e2 - sh2 + 50 - SH_Z<N3>;
    if constexpr (MODE == SLAB_TO_GRID) {
      const int ia = a.map.vec(item, 0, nl), ib = a.map.vec(item, 1, nl);
      double* oa = ia >= 0 ? a.out + (long long)ia * a.out_stride + line : nullptr;
      double* ob = ib >= 0 ? a.out + (long long)ib * a.out_stride + line : nullptr;
      const double unit = fx_unit(e3) * a.out_scale;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < NT2; ++i)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = 8 * (2 * c + i) + 2 * t + e;
            if (!quad_new<N3>(k, j)) continue;
            const int pos = quad_pos<N3>(k, j);
            if (oa) oa[pos] = fx_frac(q[k][i][e]) * unit;
            if (ob) ob[pos] = fx_frac(q[k][i][e + 2]) * unit;
          }
      return;
    }
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < NT2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) m = max(m, high_mag(q[k][i][e]));
    block_max(&mx[2 + c], m);
    __syncthreads();
    // potential values below 2^62, X below 2^62: products below 2^60
    const int shx = 62 - bit_length(mx[2 + c]);
    if (AT || a.dn) {
      // density response of the two vectors of the item (Eq. deltani),
      // accumulated over the occupied states v
      const int ia = a.map.vec(item, 0, nl), ib = a.map.vec(item, 1, nl);
      const int ja = ia / a.dn_nocc, jb = ib >= 0 ? ib / a.dn_nocc : -1;
      const double* ua = a.u + (long long)(ia - ja * a.dn_nocc) * a.dn_stride + line;
      const double* ub = ib >= 0 ? a.u + (long long)(ib - jb * a.dn_nocc) * a.dn_stride + line : ua;
      double* const dn = AT ? *a.dn_at : a.dn;
      double* da = dn + (long long)ja * a.dn_stride + line;
      double* db = ib >= 0 ? dn + (long long)jb * a.dn_stride + line : da;
      const double sc = a.dn_scale * fx_unit(e3);
      const bool same = jb == ja;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < NT2; ++i)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = 8 * (2 * c + i) + 2 * t + e;
            if (!quad_new<N3>(k, j)) continue;
            const int pos = quad_pos<N3>(k, j);
            // without a second vector its values are zero
            double ca = fx_frac(q[k][i][e]) * ua[pos];
            const double cb = fx_frac(q[k][i][e + 2]) * ub[pos];
            ca += same ? cb : 0.0;
            atomicAdd(da + pos, sc * ca);
            if (!same) atomicAdd(db + pos, sc * cb);
          }
    }
    const long long* vx = s.vfx + line;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < NT2; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = 8 * (2 * c + i) + 2 * t + e;
          const long long v = __ldg(vx + quad_pos<N3>(k, min(j, N3 / 4)));
          q[k][i][e] = __mul64hi(q[k][i][e] << shx, v);
          q[k][i][e + 2] = __mul64hi(q[k][i][e + 2] << shx, v);
        }
    e4 = e3 - shx + s.v_exp + 64;
  }
  // back to the sphere's n3 frequencies
  const int ec = e4 + 50 - SH_ZB<N3>;
  int rs = 0;  // right shift of this chunk's sums
  if (c > 0) {
    const int m = max(fe, ec), r0 = m - fe;
    rs = m - ec;
    if (r0) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < L::NTN; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) fo[k][i][e] >>= min(r0, 63);
    }
    fe = m;
  } else {
    fe = ec;
  }
  z_back<S, N2, N3, NT2, 0>(s, c, rs, q, fo);
  z_back<S, N2, N3, NT2, 1>(s, c, rs, q, fo);
}

// Every value of the plane is NaN: an infinity or NaN came in
template <bool AT, int N2, int N3>
__device__ void slab_nan(const SphereDev<double>& s, const SlabArgs<double>& a, int nl, int item,
                         long long plane, cpx<double>* row) {
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  const int ia = a.map.vec(item, 0, nl), ib = a.map.vec(item, 1, nl);
  for (int p = threadIdx.x; p < N2 * N3; p += blockDim.x) {
    if (a.mode == SLAB_TO_GRID) {
      if (ia >= 0) a.out[(long long)ia * a.out_stride + plane + p] = nan;
      if (ib >= 0) a.out[(long long)ib * a.out_stride + plane + p] = nan;
    } else if (a.mode == SLAB_HPSI && (AT || a.dn)) {
      double* const dn = AT ? *a.dn_at : a.dn;
      atomicAdd(dn + (long long)(ia / a.dn_nocc) * a.dn_stride + plane + p, nan);
      if (ib >= 0) atomicAdd(dn + (long long)(ib / a.dn_nocc) * a.dn_stride + plane + p, nan);
    }
  }
  if (a.mode == SLAB_TO_GRID) return;
  for (int j = threadIdx.x; j < s.n_col; j += blockDim.x) row[j] = mk(nan, nan);
}

template <int N2>
struct FxBlocks {  // resident blocks per SM the registers are held to
  static constexpr int v = N2 <= 24 ? 4 : N2 <= 32 ? 3 : N2 <= 48 ? 2 : 1;
};

template <int MODE, bool AT, int S, int N2, int N3>
__global__ void __launch_bounds__(N2 * 4, FxBlocks<N2>::v)
    k_slab_fx(SphereDev<double> s, SlabArgs<double> a) {
  using L2 = FxLine<N2>;
  using L3 = FxLine<N3>;
  constexpr int W = N2 / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned mx[FX_MX];
  cl* S1 = reinterpret_cast<cl*>(smem_raw);
  cl* T2 = S1 + s.n_col;
  const int nl = listed_count(a.map);
  const int item = blockIdx.x, i1 = blockIdx.y;
  if (item >= items_of(a.map, a.n_items, nl)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const long long plane = (long long)i1 * N2 * N3;
  cpx<double>* row = a.b1 + ((long long)item * s.N1 + i1) * s.n_col;
  const int nslot = 2 * s.R3 + 1, mt2 = (nslot + 7) / 8;
  if (tid < FX_MX) mx[tid] = 0;
  __syncthreads();

  int e2 = 0, sh2 = 0;  // the shared plane's scale, and the shift it is read with
  if constexpr (MODE != SLAB_FROM_GRID) {
    // the plane's columns as integers below 2^61
    int ex = 1;
    for (int j = tid; j < s.n_col; j += blockDim.x) {
      const cpx<double> z = row[j];
      ex = max(ex, max(exp_of(z.x), exp_of(z.y)));
    }
    block_max(&mx[0], (unsigned)ex);
    __syncthreads();
    const int er = (int)mx[0];
    if (er == 0x7ff) {
      slab_nan<AT, N2, N3>(s, a, nl, item, plane, row);
      return;
    }
    for (int j = tid; j < s.n_col; j += blockDim.x) {
      const cpx<double> z = row[j];
      S1[j] = cl{fx_of(z.x, er) >> 1, fx_of(z.y, er) >> 1};
    }
    __syncthreads();
    // y-lines: eight n3 slots and one tile of positions per unit
    unsigned m = 0;
    for (int u = warp; u < mt2 * L2::NTJ; u += W) {
      const int nt = u / mt2, sl = 8 * (u - nt * mt2) + g;
      int2 info = sl < nslot ? s.slot[sl] : make_int2(-1, 0);
      if (sl < nslot && !slot_in_range(s, info)) info.x = -1;
      auto ld = [&](int n) {
        return n <= info.x && n >= -info.x ? S1[info.y + n + info.x] : cl{0, 0};
      };
      long long q[4][1][4];
      line_inverse<N2, S, SH_Y, 1>(s.fx2, nt, ld, 0, q);
      if (sl < nslot) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = 8 * nt + 2 * t + e;
            if (!quad_new<N2>(k, j)) continue;
            const cl v{q[k][0][e], q[k][0][e + 2]};
            m = max(m, max(high_mag(v.x), high_mag(v.y)));
            T2[t2_fx<N2>(sl, quad_pos<N2>(k, j))] = v;
          }
      }
    }
    block_max(&mx[1], m);
    __syncthreads();
    sh2 = 61 - bit_length(mx[1]);
    e2 = er - 1083 + 50 - SH_Y;
  }

  // z-lines: eight per warp, in registers from n3 back to n3
  long long fo[4][L3::NTN][4];
  int fe = 0;
  constexpr int full = L3::NTJ / 2;
  if constexpr (full > 0) {
    if constexpr (full == 1) {
      z_chunk<MODE, AT, S, N2, N3, 2>(s, a, nl, item, plane, T2, mx, 0, e2, sh2, fo, fe);
    } else {
#pragma unroll 1
      for (int c = 0; c < full; ++c)
        z_chunk<MODE, AT, S, N2, N3, 2>(s, a, nl, item, plane, T2, mx, c, e2, sh2, fo, fe);
    }
  }
  if constexpr (L3::NTJ % 2)
    z_chunk<MODE, AT, S, N2, N3, 1>(s, a, nl, item, plane, T2, mx, full, e2, sh2, fo, fe);
  if constexpr (MODE == SLAB_TO_GRID) {
    return;
  } else {
  if constexpr (MODE == SLAB_FROM_GRID) {
    bool bad = false;
#pragma unroll
    for (int c = 0; c < L3::NC; ++c) bad |= mx[2 + c] == 0x7ff;
    if (bad) {  // uniform: every chunk's maximum was written before a barrier
      slab_nan<AT, N2, N3>(s, a, nl, item, plane, row);
      return;
    }
  }
  {
    __syncwarp();  // the warp's own columns have been read
    const int i2 = warp * 8 + g;
    unsigned m = 0;
#pragma unroll
    for (int par = 0; par < 2; ++par)
#pragma unroll
      for (int i = 0; i < L3::NTN; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int n = 2 * (8 * i + 2 * t + e) + par;
          if (n > s.R3) continue;
          const cl p{fo[par][i][e] + fo[2 + par][i][e], fo[par][i][e + 2] + fo[2 + par][i][e + 2]};
          const cl q{fo[par][i][e] - fo[2 + par][i][e], fo[par][i][e + 2] - fo[2 + par][i][e + 2]};
          m = max(m, max(high_mag(p.x), high_mag(p.y)));
          T2[t2_fx<N2>(s.R3 + n, i2)] = p;
          if (n > 0) {
            m = max(m, max(high_mag(q.x), high_mag(q.y)));
            T2[t2_fx<N2>(s.R3 - n, i2)] = q;
          }
        }
    block_max(&mx[FX_MX - 1], m);
  }
  __syncthreads();
  const int sh5 = 60 - bit_length(mx[FX_MX - 1]);
  const double unit = fx_unit(fe - sh5 + 50 - SH_YB);
  // y-lines back: eight n3 slots and one parity of n2 per unit
  for (int u = warp; u < mt2 * 2; u += W) {
    const int par = u / mt2, sl = 8 * (u - par * mt2) + g;
    int2 info = sl < nslot ? s.slot[sl] : make_int2(-1, 0);
    if (sl < nslot && !slot_in_range(s, info)) info.x = -1;
    long long co[4] = {0, 0, 0, 0}, so[4] = {0, 0, 0, 0};
    auto chunk = [&](auto nt2, int c) {
      constexpr int NT2 = decltype(nt2)::value;
      long long q[4][NT2][4], x[NT2][4], w[NT2][4], f[NT2][4], v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < NT2; ++i)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = 8 * (2 * c + i) + 2 * t + e;
            cl z{0, 0};
            if (sl < nslot && j <= N2 / 4) z = T2[t2_fx<N2>(sl, quad_pos<N2>(k, j))];
            q[k][i][e] = z.x;
            q[k][i][e + 2] = z.y;
          }
      if (sh5 >= 0) {
#pragma unroll
        for (int k = 0; k < 16 * NT2; ++k) q[k / (4 * NT2)][k / 4 % NT2][k % 4] <<= sh5;
      } else {
#pragma unroll
        for (int k = 0; k < 16 * NT2; ++k) q[k / (4 * NT2)][k / 4 % NT2][k % 4] >>= -sh5;
      }
      fold<NT2, 0>(q, x, w);
      fold2<NT2, 0>(x, w, par, f);
      fwd_group<N2, S, SH_YB, NT2, 0>(s.fx2 + L2::INV, c, 0, par, f, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) co[e] += v[e];
      fold<NT2, 1>(q, x, w);
      fold2<NT2, 1>(x, w, par, f);
      fwd_group<N2, S, SH_YB, NT2, 1>(s.fx2 + L2::INV, c, 0, par, f, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) so[e] += v[e];
    };
#pragma unroll
    for (int c = 0; c < L2::NTJ / 2; ++c) chunk(std::integral_constant<int, 2>{}, c);
    if constexpr (L2::NTJ % 2) chunk(std::integral_constant<int, 1>{}, L2::NTJ / 2);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int n = 2 * (2 * t + e) + par;
      if (n > info.x) continue;
      row[info.y + info.x + n] = mk(fx_frac(co[e] + so[e]) * unit, fx_frac(co[e + 2] + so[e + 2]) * unit);
      if (n > 0)
        row[info.y + info.x - n] =
            mk(fx_frac(co[e] - so[e]) * unit, fx_frac(co[e + 2] - so[e + 2]) * unit);
    }
  }
  }
}

template <int MODE, bool AT, int S, int N2, int N3>
cudaError_t slab_fx_mode(const SphereDev<double>& s, const SlabArgs<double>& a, cudaStream_t st) {
  if (a.n_items <= 0) return cudaSuccess;
  const size_t smem = slab_smem_bytes(s.n_col, s.R3, N2, 8);
  auto kern = k_slab_fx<MODE, AT, S, N2, N3>;
  static OncePerDevice limit;  // per instantiation
  if (const cudaError_t e = raise_smem_limit(limit, kern, 200 * 1024)) return e;
  double fl = 0, by = 0;
  slab_work(s, a, fl, by);
  ProfScope ps(S < FX_S ? PC_SLAB_DF : PC_SLAB_F64, st, fl, by,
               a.map.list ? a.map.n_dev : nullptr, a.map.n_list);
  count_launch();
  kern<<<dim3(a.n_items, s.N1), N2 * 4, smem, st>>>(s, a);
  return cudaGetLastError();
}

}  // namespace
}  // namespace pdep
