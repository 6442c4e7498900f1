// The FP64 slab pass (fx_slab.cuh): its launches, the digit tables of the lines
// and the potential as integers.
#include <algorithm>
#include <cmath>
#include <vector>

#include "fx_slab.cuh"

namespace pdep {
namespace {

uint16_t half_of_int(int v) {
  if (v == 0) return 0;
  const uint16_t s = v < 0 ? 0x8000 : 0;
  int a = v < 0 ? -v : v, e = 0;
  while ((1 << (e + 1)) <= a) ++e;
  return (uint16_t)(s | ((e + 15) << 10) | ((a << (10 - e)) & 0x3ff));
}
// digit s of w 2^62
int host_digit(long double w, int s) {
  const long long v = llroundl(w * 4611686018427387904.0L);
  const unsigned long long u = (unsigned long long)v + 0x8080808080808080ull;
  return (int)((u >> (8 * (7 - s))) & 0xff) - 128;
}

template <int N>
std::vector<uint32_t> build_table() {
  using L = FxLine<N>;
  std::vector<uint32_t> tab(L::INV + L::FWD, 0u);
  const long double two_pi = 6.283185307179586476925286766559005768L;
  // table entry of frequency index kk of a parity and position j
  auto entry = [&](int grp, int kk, int j, bool fwd) -> long double {
    if (kk >= L::KI || j > N / 4) return 0.0L;
    const int n = 2 * kk + (grp & 1);
    const int r = (int)(((long long)n * j) % N);
    // reduced to the first octant so that symmetric entries are exact
    const long double x = two_pi * r / N;
    long double v = grp < 2 ? cosl(x) : sinl(x);
    if (grp < 2 ? (4 * r == N || 4 * r == 3 * N) : (2 * r == N || r == 0)) v = 0.0L;
    return fwd && (j == 0 || j == N / 4) ? 0.5L * v : v;
  };
  // digit order of the paired layout: (1,0)(3,2)(5,4)(7,6)(0,-)(2,1)(4,3)(6,5)
  const int order[16] = {1, 0, 3, 2, 5, 4, 7, 6, 0, -1, 2, 1, 4, 3, 6, 5};
  auto word = [&](int grp, int k0, int k1, int j0, int j1, int d, bool fwd) -> uint32_t {
    if (d < 0) return 0u;
    const uint32_t lo = half_of_int(host_digit(entry(grp, k0, j0, fwd), d));
    const uint32_t hi = half_of_int(host_digit(entry(grp, k1, j1, fwd), d));
    return lo | hi << 16;
  };
  for (int ks = 0; ks < L::KS; ++ks)
    for (int nt = 0; nt < L::NTJ; ++nt)
      for (int grp = 0; grp < 4; ++grp)
        for (int lane = 0; lane < 32; ++lane)
          for (int w = 0; w < 16; ++w) {
            const int kk = 8 * ks + 2 * (lane & 3), j = 8 * nt + (lane >> 2);
            tab[((((size_t)ks * L::NTJ + nt) * 4 + grp) * 32 + lane) * 16 + w] =
                word(grp, kk, kk + 1, j, j, order[w], false);
          }
  for (int c = 0; c < L::NC; ++c) {
    const bool two = 2 * c + 1 < L::NTJ;  // a chunk of two position tiles: digit u at 2 u, 2 u + 1
    for (int nt = 0; nt < L::NTN; ++nt)
      for (int grp = 0; grp < 4; ++grp)
        for (int lane = 0; lane < 32; ++lane)
          for (int w = 0; w < 16; ++w) {
            const int kk = 8 * nt + (lane >> 2), j = 16 * c + (two ? 8 * (w & 1) : 0) + 2 * (lane & 3);
            tab[L::INV + ((((size_t)c * L::NTN + nt) * 4 + grp) * 32 + lane) * 16 + w] =
                word(grp, kk, kk, j, j + 1, two ? w >> 1 : order[w], true);
          }
  }
  return tab;
}

template <int N2, int N3>
cudaError_t slab_fx_impl(const SphereDev<double>& s, const SlabArgs<double>& a, cudaStream_t st) {
  const bool few = a.digits < FX_S;
  switch (a.mode) {
    case SLAB_HPSI:
      return few ? slab_fx_mode<SLAB_HPSI, false, 7, N2, N3>(s, a, st)
                 : slab_fx_mode<SLAB_HPSI, false, 8, N2, N3>(s, a, st);
    case SLAB_FROM_GRID:
      return few ? slab_fx_mode<SLAB_FROM_GRID, false, 7, N2, N3>(s, a, st)
                 : slab_fx_mode<SLAB_FROM_GRID, false, 8, N2, N3>(s, a, st);
    case SLAB_TO_GRID: return slab_fx_mode<SLAB_TO_GRID, false, 8, N2, N3>(s, a, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

std::vector<uint32_t> fx_line_table(int N) {
  switch (N) {
    case 24: return build_table<24>();
    case 32: return build_table<32>();
    case 40: return build_table<40>();
    case 48: return build_table<48>();
    case 64: return build_table<64>();
    case 192: return build_table<192>();
  }
  return {};
}

__global__ void k_fixed_potential(const double* __restrict__ v, int n, int er, long long* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = fx_of(v[i], er);
}
cudaError_t fixed_potential(const double* v, int n, int er, long long* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  count_launch();
  k_fixed_potential<<<std::min((n + 255) / 256, 4096), 256, 0, st>>>(v, n, er, out);
  return cudaGetLastError();
}

cudaError_t launch_slab(const SphereDev<double>& s, const SlabArgs<double>& a, cudaStream_t st) {
  if (a.dn_at && !a.dn) return launch_slab_rounds(s, a, st);
  if (s.N2 == s.N3) {
    switch (s.N2) {
      case 24: return slab_fx_impl<24, 24>(s, a, st);
      case 32: return slab_fx_impl<32, 32>(s, a, st);
      case 40: return slab_fx_impl<40, 40>(s, a, st);
      case 48: return slab_fx_impl<48, 48>(s, a, st);
      case 64: return slab_fx_impl<64, 64>(s, a, st);
    }
  } else if (s.N2 == 64 && s.N3 == 192) {
    return slab_fx_impl<64, 192>(s, a, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pdep
