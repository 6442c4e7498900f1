// Plane-wave sphere <-> grid transforms (see transforms.cuh for the scheme).
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "fft.cuh"
#include "transforms.cuh"
#include "profile.cuh"

namespace pdep {


cudaError_t upload_local_twiddles() {
  static const int sizes[] = {6, 8, 10, 12, 16, 20, 24, 32, 40, 48, 64};
  float2 hf[LOCAL_TW_SIZE];
  const double two_pi = 6.283185307179586476925286766559;
  for (int M : sizes) {
    int off = local_tw_offset(M);
    for (int j = 0; j < M; ++j) {
      double a = two_pi * (double)j / (double)M;
      hf[off + j] = make_float2((float)cos(a), (float)sin(a));
    }
  }
  return cudaMemcpyToSymbol(c_local_tw_f, hf, sizeof(hf));
}

// Lanes per line for each supported length (N / TPL registers per lane).
// Four lanes per line up to N = 64 measured faster than two for FP32 too:
// the extra shuffle stage costs less than the occupancy two-lane lines lose.
template <typename R, int N>
struct Tpl;
template <typename R> struct Tpl<R, 24> { static constexpr int v = 2; };
template <typename R> struct Tpl<R, 32> { static constexpr int v = 4; };
template <typename R> struct Tpl<R, 40> { static constexpr int v = 4; };
// 48-point FP32 lines: 4 lanes measured fastest per PDEP solve once the
// line FFTs skip the registers outside every sphere — half of each lane's
// 12 here — 2.4% ahead of 8 lanes and 26% ahead of 2
template <typename R> struct Tpl<R, 48> { static constexpr int v = 4; };
template <typename R> struct Tpl<R, 64> { static constexpr int v = 4; };
template <typename R> struct Tpl<R, 192> { static constexpr int v = 8; };

bool grid_supported(int N1, int N2, int N3) {
  bool n1 = (N1 == 24 || N1 == 32 || N1 == 40 || N1 == 48 || N1 == 64);
  bool cube = (N2 == N3) && (N2 == 24 || N2 == 32 || N2 == 40 || N2 == 48 || N2 == 64);
  bool slab = (N2 == 64 && N3 == 192);
  return n1 && (cube || slab);
}

static __device__ __forceinline__ int iabs(int a) { return a < 0 ? -a : a; }

template <typename R>
__device__ __forceinline__ cpx<R> zero() { return mk(R(0), R(0)); }

template <typename R>
__device__ __forceinline__ R coef_of(int kind, const double* __restrict__ g2, int k) {
  if (kind == COEF_SQRT_COULOMB) return R(sqrt(12.566370614359172953850573533118 / g2[k]));
  return R(1);
}

// ---------------------------------------------------------------------------
// column pass: sphere -> x-lines (inverse transform, S = +1)
// ---------------------------------------------------------------------------
template <typename R, int N1>
__device__ __forceinline__ void cols_fwd_line(const SphereDev<R>& s,
                                              const R* __restrict__ x,
                                              long long ldx, const ItemMap& map, int nl,
                                              int coef, cpx<R>* __restrict__ b1, long long g,
                                              long long total);
template <typename R, int N1, typename TW>
__device__ __forceinline__ void xline_inverse(const SphereDev<R>& s,
                                              const R* __restrict__ x,
                                              long long ldx, const ItemMap& map, int nl, int coef,
                                              int item, int uc, bool live, cpx<R>* base,
                                              const TW& tws);

template <typename R, int N1>
__global__ void __launch_bounds__(128) k_cols_fwd(SphereDev<R> s,
                                                  const R* __restrict__ x,
                                                  long long ldx, ItemMap map, int n_items,
                                                  int coef, cpx<R>* __restrict__ b1) {
  const int nl = listed_count(map);
  const long long total = (long long)items_of(map, n_items, nl) * s.n_ucol;
  const int per = blockDim.x / Tpl<R, N1>::v;
  // the launch covers the largest count; blocks past the device count exit
  // (a grid-stride loop here costs 40-70% more registers)
  const long long g0 = (long long)blockIdx.x * per;
  if (g0 < total)
    cols_fwd_line<R, N1>(s, x, ldx, map, nl, coef, b1, g0 + threadIdx.x / Tpl<R, N1>::v, total);
}

template <typename R, int N1>
__device__ __forceinline__ void cols_fwd_line(const SphereDev<R>& s,
                                              const R* __restrict__ x,
                                              long long ldx, const ItemMap& map, int nl,
                                              int coef, cpx<R>* __restrict__ b1, long long g,
                                              long long total) {
  const bool live = g < total;
  const int item = live ? (int)(g / s.n_ucol) : 0;
  const int uc = live ? (int)(g - (long long)item * s.n_ucol) : 0;
  xline_inverse<R, N1>(s, x, ldx, map, nl, coef, item, uc, live,
                       b1 + (long long)item * N1 * s.n_col, TableTw<R>{s.tw1});
}

// x-line uc of item (both members of its mirror pair) from the sphere into
// the item's column scratch 'base' ([N1][n_col], global or shared memory);
// every lane of the warp must call it (the FFT shuffles), live or not.
template <typename R, int N1, typename TW>
__device__ __forceinline__ void xline_inverse(const SphereDev<R>& s,
                                              const R* __restrict__ x,
                                              long long ldx, const ItemMap& map, int nl, int coef,
                                              int item, int uc, bool live, cpx<R>* base,
                                              const TW& tws) {
  constexpr int TPL = Tpl<R, N1>::v;
  constexpr int M = N1 / TPL;
  const int t = threadIdx.x & (TPL - 1);
  const UCol c = s.ucol[live ? uc : 0];
  const bool active = live && ucol_in_range(s, c);
  const bool self = (c.col == c.mcol);
  const int ia = map.vec(item, 0, nl), ib = map.vec(item, 1, nl);
  const R* xa = (active && ia >= 0) ? x + (long long)ia * ldx : nullptr;
  const R* xb = (active && ib >= 0) ? x + (long long)ib * ldx : nullptr;
  const R rs2 = R(0.70710678118654752440084436210485);

  cpx<R> v0[M], v1[M];
#pragma unroll
  for (int i = 0; i < M; ++i) {
    v0[i] = zero<R>();
    v1[i] = zero<R>();
    if (a_outside(N1, TPL, i)) continue;
    const int n1 = freq_of(pos_a<N1, TPL>(t, i), N1);
    if (!active) continue;
    if (!self) {
      if (iabs(n1) <= c.R1) {
        // line c at n1: member k;  mirror line at n1: conj of member k'
        const int k = c.h0 + n1 + c.R1;
        const int k2 = c.h0 - n1 + c.R1;
        const R w = coef_of<R>(coef, s.g2, k) * rs2;
        const R w2 = coef_of<R>(coef, s.g2, k2) * rs2;
        cpx<R> A = xa ? mk(*(xa + 2 * k) * w, *(xa + 2 * k + 1) * w) : zero<R>();
        cpx<R> B = xb ? mk(*(xb + 2 * k) * w, *(xb + 2 * k + 1) * w) : zero<R>();
        v0[i] = mk(A.x - B.y, A.y + B.x);
        cpx<R> A2 = xa ? mk(*(xa + 2 * k2) * w2, *(xa + 2 * k2 + 1) * w2) : zero<R>();
        cpx<R> B2 = xb ? mk(*(xb + 2 * k2) * w2, *(xb + 2 * k2 + 1) * w2) : zero<R>();
        v1[i] = mk(A2.x + B2.y, B2.x - A2.y);
      }
    } else {
      if (n1 == 0) {
        const R w = (coef == COEF_ONE) ? R(1) : R(0);
        const int k0 = 2 * s.n_half;
        v0[i] = mk(xa ? *(xa + k0) * w : R(0), xb ? *(xb + k0) * w : R(0));
      } else if (iabs(n1) <= c.R1) {
        const int k = c.h0 + iabs(n1) - 1;
        const R w = coef_of<R>(coef, s.g2, k) * rs2;
        cpx<R> A = xa ? mk(*(xa + 2 * k) * w, *(xa + 2 * k + 1) * w) : zero<R>();
        cpx<R> B = xb ? mk(*(xb + 2 * k) * w, *(xb + 2 * k + 1) * w) : zero<R>();
        v0[i] = n1 > 0 ? mk(A.x - B.y, A.y + B.x) : mk(A.x + B.y, B.x - A.y);
      }
    }
  }
  fft_a2b<R, N1, TPL, +1>(v0, t, tws);
  fft_a2b<R, N1, TPL, +1>(v1, t, tws);
  if (!active) return;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const int i1 = pos_b<N1, TPL>(t, i);
    base[(long long)i1 * s.n_col + c.col] = v0[i];
    if (!self) base[(long long)i1 * s.n_col + c.mcol] = v1[i];
  }
}

// ---------------------------------------------------------------------------
// column pass back: x-lines -> sphere (forward transform, S = -1), Hermitian
// unpacking of the two real fields and the epilogue
// ---------------------------------------------------------------------------
// One output vector's epilogue state: its output and input rows and its shift,
// set up once per line.
template <typename R>
struct OutRow {
  R* y_;
  const R* x_;  // null: no diagonal term
  R sh_;
  __device__ __forceinline__ OutRow(const Epilogue<R>& ep, int vec) {
    y_ = ep.y + (long long)(vec >= 0 ? vec : 0) * ep.ldy;
    x_ = ep.x_in ? ep.x_in + (long long)(vec >= 0 ? vec : 0) * ep.ldx : nullptr;
    sh_ = (ep.x_in && ep.shift && vec >= 0) ? ep.shift[vec % ep.shift_period] : R(0);
  }
};
template <typename R>
__device__ __forceinline__ void write_out(const Epilogue<R>& ep, const OutRow<R>& o, int j, R val,
                                          R coefv, R diag) {
  R r = ep.scale * coefv * val;
  if (o.x_) r += (diag + o.sh_) * o.x_[j];
  if (ep.beta != 0) r += ep.beta * o.y_[j];
  o.y_[j] = r;
}

template <typename R, int N1>
__device__ __forceinline__ void cols_bwd_line(const SphereDev<R>& s,
                                              const cpx<R>* __restrict__ b1, const ItemMap& map,
                                              int nl, const Epilogue<R>& ep, long long g,
                                              long long total);
template <typename R, int N1, typename TW>
__device__ __forceinline__ void xline_forward(const SphereDev<R>& s, const cpx<R>* base,
                                              const ItemMap& map, int nl, const Epilogue<R>& ep,
                                              int item, int uc, bool live, const TW& tws);

template <typename R, int N1>
__global__ void __launch_bounds__(128) k_cols_bwd(SphereDev<R> s, const cpx<R>* __restrict__ b1,
                                                  ItemMap map, int n_items, Epilogue<R> ep) {
  const int nl = listed_count(map);
  const long long total = (long long)items_of(map, n_items, nl) * s.n_ucol;
  const int per = blockDim.x / Tpl<R, N1>::v;
  const long long g0 = (long long)blockIdx.x * per;
  if (g0 < total)
    cols_bwd_line<R, N1>(s, b1, map, nl, ep, g0 + threadIdx.x / Tpl<R, N1>::v, total);
}

template <typename R, int N1>
__device__ __forceinline__ void cols_bwd_line(const SphereDev<R>& s,
                                              const cpx<R>* __restrict__ b1, const ItemMap& map,
                                              int nl, const Epilogue<R>& ep, long long g,
                                              long long total) {
  const bool live = g < total;
  const int item = live ? (int)(g / s.n_ucol) : 0;
  const int uc = live ? (int)(g - (long long)item * s.n_ucol) : 0;
  xline_forward<R, N1>(s, b1 + (long long)item * N1 * s.n_col, map, nl, ep, item, uc, live,
                       TableTw<R>{s.tw1});
}

// x-line uc of item from its column scratch 'base' back to the sphere, the
// two real fields unpacked, through the epilogue; every lane of the warp
// must call it.
template <typename R, int N1, typename TW>
__device__ __forceinline__ void xline_forward(const SphereDev<R>& s, const cpx<R>* base,
                                              const ItemMap& map, int nl, const Epilogue<R>& ep,
                                              int item, int uc, bool live, const TW& tws) {
  constexpr int TPL = Tpl<R, N1>::v;
  constexpr int M = N1 / TPL;
  const int lane = threadIdx.x & 31;
  const int t = threadIdx.x & (TPL - 1);
  const UCol c = s.ucol[live ? uc : 0];
  const bool active = live && ucol_in_range(s, c);
  const bool self = (c.col == c.mcol);

  cpx<R> v0[M], v1[M];
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const int i1 = pos_b<N1, TPL>(t, i);
    v0[i] = active ? base[(long long)i1 * s.n_col + c.col] : zero<R>();
    v1[i] = (active && !self) ? base[(long long)i1 * s.n_col + c.mcol] : zero<R>();
  }
  fft_b2a<R, N1, TPL, -1>(v0, t, tws);
  fft_b2a<R, N1, TPL, -1>(v1, t, tws);

  const int src = (lane & ~(TPL - 1)) | ((TPL - t) & (TPL - 1));
  const int ia = map.vec(item, 0, nl), ib = map.vec(item, 1, nl);
  const OutRow<R> oa(ep, ia), ob(ep, ib);
  const R rs2 = R(0.70710678118654752440084436210485);
#pragma unroll
  for (int i = 0; i < M; ++i) {
    if (a_outside(N1, TPL, i)) continue;  // the same i in every lane
    // value of the mirror line at position (N1 - p) mod N1
    cpx<R> send = self ? v0[M - 1 - i] : v1[M - 1 - i];
    cpx<R> dm = shfl_idx(send, src);
    if (t == 0) dm = self ? v0[(M - i) % M] : v1[(M - i) % M];
    if (!active) continue;
    const int n1 = freq_of(pos_a<N1, TPL>(t, i), N1);
    int k = -1;
    if (!self) {
      if (iabs(n1) <= c.R1) k = c.h0 + n1 + c.R1;
    } else if (n1 > 0 && n1 <= c.R1) {
      k = c.h0 + n1 - 1;
    }
    const cpx<R> d = v0[i];
    if (k >= 0) {
      const cpx<R> sa = d + conj(dm);   // 2 Va
      const cpx<R> sb = d - conj(dm);   // 2 i Vb
      const R cf = coef_of<R>(ep.coef, s.g2, k);
      const R dg = ep.kin * s.kin[k];
      if (ia >= 0) {
        write_out(ep, oa, 2 * k, rs2 * sa.x, cf, dg);
        write_out(ep, oa, 2 * k + 1, rs2 * sa.y, cf, dg);
      }
      if (ib >= 0) {
        write_out(ep, ob, 2 * k, rs2 * sb.y, cf, dg);
        write_out(ep, ob, 2 * k + 1, -rs2 * sb.x, cf, dg);
      }
    } else if (self && n1 == 0) {
      const R cf = (ep.coef == COEF_ONE) ? R(1) : R(0);
      const int j0 = 2 * s.n_half;
      if (ia >= 0) write_out(ep, oa, j0, d.x, cf, R(0));
      if (ib >= 0) write_out(ep, ob, j0, d.y, cf, R(0));
    }
  }
}

// ---------------------------------------------------------------------------
// slab pass, FP32: one x-plane i1 of one item (FP64 data take
// transforms_fx.cu)
// ---------------------------------------------------------------------------
// largest block a slab of this shape launches with: every z-line (N2 lines)
// or every y-line (at most N3/2 + 1 planes) in one round
template <int N2, int N3>
struct SlabThreads {
  static constexpr int z = N2 * Tpl<float, N3>::v;
  static constexpr int y = (N3 / 2 + 1) * Tpl<float, N2>::v;
  static constexpr int v = (((z > y ? z : y) + 31) / 32) * 32;
};
// three blocks of up to 256 threads per SM stay resident (register budget
// ~85-110)
template <int N2, int N3>
struct SlabMinBlocks {
  static constexpr int t = SlabThreads<N2, N3>::v;
  static constexpr int v = t <= 128 ? 384 / t : t <= 256 ? 3 : t <= 384 ? 2 : 1;
};
// Row stride of the (n3, i2) shared-memory plane (rows padded by 8 complex)
// and a column swizzle: element (row, col) sits at row * TS + (col ^ (row &
// 7)).  The swizzle stays inside each aligned block of 8 columns (N2 is a
// multiple of 8) and spreads the eight y-line slots a warp touches, whose four
// lanes' positions are 12 complex apart, over all banks (a third of the
// shared-memory wavefronts of the LSU-bound slab); the four n3 rows of a
// z-line access keep their distinct halves.
template <int N2>
struct T2Stride {
  static constexpr int v = N2 + 8;
};
__device__ __forceinline__ int t2_at(int row, int col, int ts) {
  return row * ts + (col ^ (row & 7));
}

// tid / nthreads: the thread's index in, and the size of, the (warp-aligned)
// group of threads that transforms this plane
template <int N2, typename TW>
__device__ __forceinline__ void y_inverse(const SphereDev<float>& s, const cpx<float>* S1, cpx<float>* T2,
                                          int tid, int nthreads, const TW& tws) {
  constexpr int TL = Tpl<float, N2>::v;
  constexpr int TS = T2Stride<N2>::v;
  constexpr int M = N2 / TL;
  const int nslot = 2 * s.R3 + 1;
  const int per = nthreads / TL;
  const int t = tid & (TL - 1);
  // first slot of this warp in a round: warps whose slots all lie past the
  // last (n3) row skip the line FFTs instead of transforming zeros
  const int wslot0 = (tid & ~31) / TL;
  for (int base = 0; base < nslot; base += per) {
    if (base + wslot0 >= nslot) break;
    const int sl = base + tid / TL;
    const bool live = sl < nslot;
    const int2 info = live ? s.slot[sl] : make_int2(-1, 0);
    const bool act = live && slot_in_range(s, info);
    cpx<float> v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
      const int n2 = freq_of(pos_a<N2, TL>(t, i), N2);
      v[i] = (!a_outside(N2, TL, i) && act && iabs(n2) <= info.x) ? S1[info.y + n2 + info.x]
                                                                   : zero<float>();
    }
    fft_a2b<float, N2, TL, +1>(v, t, tws);
    if (act) {
#pragma unroll
      for (int i = 0; i < M; ++i) T2[t2_at(sl, pos_b<N2, TL>(t, i), TS)] = v[i];
    }
  }
}

template <int N2, typename TW>
__device__ __forceinline__ void y_forward(const SphereDev<float>& s, const cpx<float>* T2, cpx<float>* S1,
                                          int tid, int nthreads, const TW& tws) {
  constexpr int TL = Tpl<float, N2>::v;
  constexpr int TS = T2Stride<N2>::v;
  constexpr int M = N2 / TL;
  const int nslot = 2 * s.R3 + 1;
  const int per = nthreads / TL;
  const int t = tid & (TL - 1);
  const int wslot0 = (tid & ~31) / TL;
  for (int base = 0; base < nslot; base += per) {
    if (base + wslot0 >= nslot) break;
    const int sl = base + tid / TL;
    const bool live = sl < nslot;
    const int2 info = live ? s.slot[sl] : make_int2(-1, 0);
    const bool act = live && slot_in_range(s, info);
    cpx<float> v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = act ? T2[t2_at(sl, pos_b<N2, TL>(t, i), TS)] : zero<float>();
    fft_b2a<float, N2, TL, -1>(v, t, tws);
    if (act) {
#pragma unroll
      for (int i = 0; i < M; ++i) {
        if (a_outside(N2, TL, i)) continue;
        const int n2 = freq_of(pos_a<N2, TL>(t, i), N2);
        if (iabs(n2) <= info.x) S1[info.y + n2 + info.x] = v[i];
      }
    }
  }
}

// FP32 to FP64 on the integer pipe (an FP64 conversion of a warp takes 64 clocks
// of its pipe); subnormal and non-finite values by the conversion
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  if (e - 1u >= 254u) return (double)x;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))),
                          (int)(b << 29));
}

// one x-plane i1 of one item; DN: its density response is added to acc (this
// thread's positions of its z-line)
template <int N2, int N3, bool DN>
__device__ __forceinline__ void slab_unit(const SphereDev<float>& s, const SlabArgs<float>& a, int nl,
                                          int item, int i1, cpx<float>* S1, cpx<float>* T2,
                                          double* acc) {
  constexpr int TL3 = Tpl<float, N3>::v;
  constexpr int M3 = N3 / TL3;
  constexpr int TS = T2Stride<N2>::v;
  const int R3 = s.R3;
  const int t3 = threadIdx.x & (TL3 - 1);
  const int zper = blockDim.x / TL3;
  const long long plane = (long long)i1 * N2 * N3;

  cpx<float>* row = a.b1 + ((long long)item * s.N1 + i1) * s.n_col;
  if (a.mode != SLAB_FROM_GRID) {
    for (int j = threadIdx.x; j < s.n_col; j += blockDim.x) S1[j] = row[j];
    __syncthreads();
    y_inverse<N2>(s, S1, T2, threadIdx.x, blockDim.x, TableTw<float>{s.tw2});
    __syncthreads();
  }

  for (int base = 0; base < N2; base += zper) {
    const int i2 = base + threadIdx.x / TL3;
    const bool act = i2 < N2;
    cpx<float> v[M3];
    if (a.mode == SLAB_FROM_GRID) {
      const int grp = item / a.map.items_per_group;
      const int w = item - grp * a.map.items_per_group;
      const int va = 2 * w, vb = 2 * w + 1;
      const long long off = plane + (long long)i2 * N3;
      using T = float;
      const T* f = (act && a.src.f) ? a.src.f + (long long)grp * a.src.f_stride + off : nullptr;
      const T* ga = act ? a.src.g + (long long)va * a.src.g_stride + off : nullptr;
      const T* gb = (act && vb < a.map.vecs_per_group) ? a.src.g + (long long)vb * a.src.g_stride + off
                                                        : nullptr;
#pragma unroll
      for (int i = 0; i < M3; ++i) {
        const int i3 = pos_b<N3, TL3>(t3, i);
        const float fv = f ? *(f + i3) : 1.f;
        v[i] = act ? mk(fv * *(ga + i3), gb ? fv * *(gb + i3) : 0.f) : zero<float>();
      }
    } else {
#pragma unroll
      for (int i = 0; i < M3; ++i) {
        const int n3 = freq_of(pos_a<N3, TL3>(t3, i), N3);
        v[i] = (act && iabs(n3) <= R3) ? T2[t2_at(n3 + R3, i2, TS)] : zero<float>();
      }
      fft_a2b<float, N3, TL3, +1>(v, t3, s.tw3);
      if (a.mode == SLAB_TO_GRID) {
        if (act) {
          const int ia = a.map.vec(item, 0, nl), ib = a.map.vec(item, 1, nl);
          const long long off = plane + (long long)i2 * N3;
          float* oa = ia >= 0 ? a.out + (long long)ia * a.out_stride + off : nullptr;
          float* ob = ib >= 0 ? a.out + (long long)ib * a.out_stride + off : nullptr;
#pragma unroll
          for (int i = 0; i < M3; ++i) {
            const int i3 = pos_b<N3, TL3>(t3, i);
            if (oa) oa[i3] = (v[i].x * (float)a.out_scale);
            if (ob) ob[i3] = (v[i].y * (float)a.out_scale);
          }
        }
        continue;
      }
      if (DN && act) {
        // density response of the two vectors of the item on this z-line
        // (Eq. deltani), summed over the items of one perturbation
        const int ia = a.map.vec(item, 0, nl), ib = a.map.vec(item, 1, nl);
        const long long off = plane + (long long)i2 * N3;
        const int ja = ia / a.dn_nocc, jb = ib >= 0 ? ib / a.dn_nocc : -1;
        const double* ua = a.u + (long long)(ia - ja * a.dn_nocc) * a.dn_stride + off;
        const double* ub = ib >= 0 ? a.u + (long long)(ib - jb * a.dn_nocc) * a.dn_stride + off : ua;
        const bool same = jb == ja;
#pragma unroll
        for (int i = 0; i < M3; ++i) {
          const int i3 = pos_b<N3, TL3>(t3, i);
          acc[i] = fma(widen(v[i].x), ua[i3], acc[i]);
          const double xb = widen(v[i].y);
          if (same)
            acc[i] = fma(xb, ub[i3], acc[i]);
          else if (ib >= 0)
            atomicAdd(*a.dn_at + (long long)jb * a.dn_stride + off + i3, a.dn_scale * (xb * ub[i3]));
        }
      }
      // SLAB_HPSI: multiply by the local potential on the grid
      const float* vr = a.v + plane + (long long)i2 * N3;
#pragma unroll
      for (int i = 0; i < M3; ++i) v[i] = scale(v[i], act ? vr[pos_b<N3, TL3>(t3, i)] : 0.f);
    }
    fft_b2a<float, N3, TL3, -1>(v, t3, s.tw3);
    if (act) {
#pragma unroll
      for (int i = 0; i < M3; ++i) {
        const int n3 = freq_of(pos_a<N3, TL3>(t3, i), N3);
        if (iabs(n3) <= R3) T2[t2_at(n3 + R3, i2, TS)] = v[i];
      }
    }
  }
  if (a.mode == SLAB_TO_GRID) return;
  __syncthreads();
  y_forward<N2>(s, T2, S1, threadIdx.x, blockDim.x, TableTw<float>{s.tw2});
  __syncthreads();
  for (int j = threadIdx.x; j < s.n_col; j += blockDim.x) row[j] = S1[j];
}

// A persistent grid of the resident blocks strides over the (item, plane)
// units, so a launch sized for a whole batch whose device count has shrunk
// costs no empty blocks.  DN: a unit is 'group' items of one plane, whose
// density response stays in registers until the perturbation changes: the FP64
// pipe's conversions and products and an atomic per point bound this form (the
// slab passes of one application to 128 perturbations on 48^3: 8.0 ms with two
// conversions, four operations and an atomic per point and item, 5.4 ms with
// two multiply-adds).
template <int N2, int N3, bool DN>
__global__ void __launch_bounds__(SlabThreads<N2, N3>::v, (SlabMinBlocks<N2, N3>::v))
    k_slab(SphereDev<float> s, SlabArgs<float> a, int group) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* S1 = reinterpret_cast<cpx<float>*>(smem_raw);
  cpx<float>* T2 = S1 + s.n_col;
  const int nl = listed_count(a.map);
  const int n_items = items_of(a.map, a.n_items, nl);
  if constexpr (!DN) {
    const int units = n_items * s.N1;
#pragma unroll 1
    for (int w = blockIdx.x; w < units; w += gridDim.x) {
      const int item = w / s.N1;
      __syncthreads();  // the previous unit's shared-memory reads are done
      slab_unit<N2, N3, false>(s, a, nl, item, w - item * s.N1, S1, T2, nullptr);
    }
  } else {
    constexpr int TL3 = Tpl<float, N3>::v, M3 = N3 / TL3;
    const int t3 = threadIdx.x & (TL3 - 1), i2 = threadIdx.x / TL3;
    const int units = (n_items + group - 1) / group * s.N1;
    double acc[M3];
#pragma unroll
    for (int i = 0; i < M3; ++i) acc[i] = 0.0;
#pragma unroll 1
    for (int w = blockIdx.x; w < units; w += gridDim.x) {
      const int g0 = w / s.N1 * group, i1 = w % s.N1;
      auto flush = [&](int j) {
        if (i2 >= N2) return;
        double* dn = *a.dn_at + (long long)j * a.dn_stride + ((long long)i1 * N2 + i2) * N3;
#pragma unroll
        for (int i = 0; i < M3; ++i) {
          atomicAdd(dn + pos_b<N3, TL3>(t3, i), a.dn_scale * acc[i]);
          acc[i] = 0.0;
        }
      };
      int cur = -1;
#pragma unroll 1
      for (int item = g0; item < min(n_items, g0 + group); ++item) {
        const int j = a.map.vec(item, 0, nl) / a.dn_nocc;
        if (cur >= 0 && j != cur) flush(cur);
        cur = j;
        __syncthreads();
        slab_unit<N2, N3, true>(s, a, nl, item, i1, S1, T2, acc);
      }
      if (cur >= 0) flush(cur);
    }
  }
}

// ---------------------------------------------------------------------------
// fused FP32 H x: the whole transform of one item in one block
// ---------------------------------------------------------------------------
// For cubic grids whose column scratch of one item (N x n_col complex) fits
// in shared memory (24^3 .. 48^3), one block runs, per item: the x-line inverse
// FFTs of every column into shared memory, then the y and z passes of the
// x-planes (the potential multiplied between the z inverse and forward FFTs),
// then the x-line forward FFTs and the epilogue.  The column scratch never
// leaves the SM: per item the HBM traffic is the two input vectors (read for
// the transform and for the diagonal term) and the two outputs.  Blocks are
// persistent over the items.
//
// Every line is transformed by one thread, in registers: with a line on four
// lanes the shuffles, selects, swizzled addresses and predicates outnumbered
// the arithmetic two to one (443 thousand warp instructions per item of 48^3,
// 57% of them floating point, and the kernel is bound by the issue slots).  In
// one thread the positions are compile-time constants: offsets are immediate,
// twiddles constant-bank operands, quarter turns free, and the zero half of a
// sphere's line costs nothing.  Three warps form a group that takes as many
// planes as its lanes cover z-lines (4, 3, 2, 2 planes of 24, 32, 40, 48 lines);
// the groups share nothing but B1 and synchronise by named barriers.  168
// registers (96 hold a line of 48) leave 12 warps.  Measured against four lanes
// per line: 264 thousand instructions per item; 56 launches of up to 4096 items on
// 48^3 87.0 -> 55.6 ms (68.1 ms with a group's planes beside the whole column
// scratch, three groups; 74.3 ms with the three steps' code apart), 37 launches
// on 32^3 3.22 -> 2.24 ms.  Error of H x against FP64 5.4e-8 -> 5.1e-8 on 48^3.
// What is left is latency: the potential comes from L2 (48 loads a line), and two
// of three warps have y-lines.
constexpr int FG_THREADS = 96;  // threads of a group
// PLANES: x-planes of a group at a time.  GROUPS: of a block, as many as the
// registers leave (24: two blocks per SM).  OVER: 48^3 does not fit its planes'
// (n3, i2) values beside the column scratch; a plane in work keeps some n3 rows
// in its own row of the column scratch, which is dead meanwhile.
template <int N>
struct Fused {
  static constexpr int PLANES = FG_THREADS / N;
  static constexpr int GROUPS = N == 32 ? 6 : N == 40 ? 5 : 4;
  static constexpr bool OVER = N > 40;
};
// n3 rows a plane keeps in the column scratch, and beside it: (i2, n3) with odd
// strides, so that neither y-lines (lanes along n3) nor z-lines (along i2)
// conflict in the banks
struct FusedRows {
  int in, out;
};
__host__ __device__ __forceinline__ FusedRows fused_rows(bool over, int n_col, int R3, int N) {
  const int nslot = 2 * R3 + 1;
  int k = over ? (n_col / N < nslot ? n_col / N : nslot) : 0;
  if (k % 2 == 0 && k > 0) --k;
  return {k, (nslot - k) | 1};
}

template <int N>
__global__ void __launch_bounds__(FG_THREADS * Fused<N>::GROUPS, (N <= 24 ? 2 : 1))
    k_hpsi_fused(SphereDev<float> s, const float* __restrict__ x, long long ldx, ItemMap map,
                 int n_items, const float* __restrict__ vt, Epilogue<float> ep,
                 DevTimer* timer, double item_flops, double item_bytes) {
  const unsigned long long t0 = dev_clock_ns();
  constexpr unsigned long long BAND = band_mask(N), ALL = all_live(N);
  constexpr int PG = Fused<N>::PLANES;
  constexpr bool OVER = Fused<N>::OVER;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* B1 = reinterpret_cast<cpx<float>*>(smem_raw);
  cpx<float>* T = B1 + (size_t)N * s.n_col;
  // between the passes T holds the item's members, (a, b) per half index, and
  // the real G = 0 components last
  float4* st = reinterpret_cast<float4*>(T);
  float* stf = reinterpret_cast<float*>(T);
  const int tid = threadIdx.x;
  const int nslot = 2 * s.R3 + 1;
  const int nl = listed_count(map);
  const int items = items_of(map, n_items, nl);
  const int grp = tid / FG_THREADS, gt = tid - grp * FG_THREADS;
  const int groups = blockDim.x / FG_THREADS;
  const FusedRows rows = fused_rows(OVER, s.n_col, s.R3, N);
  cpx<float>* T2 = T + (size_t)grp * PG * N * rows.out;
  // this thread's y-line (plane yp of the group's, n3 slot, columns ymid - yR ..
  // ymid + yR of the plane) and z-line (plane zp, i2)
  // (threads without a line keep to the first line's addresses)
  const bool yon = gt < PG * nslot, zon = gt < PG * N;
  const int yp = yon ? gt / nslot : 0, ysl = yon ? gt - yp * nslot : 0;
  const int2 info = s.slot[ysl];
  const bool yact = yon && slot_in_range(s, info);
  const int yR = info.x, ymid = info.y + info.x;
  const bool yin = ysl < rows.in;
  const int zp = zon ? gt / N : 0, i2 = zon ? gt - zp * N : 0;
  // the field is carried at sqrt(2) times its size: the members' 1/sqrt(2) in and
  // out become one exact 1/2
  const float rt2 = 1.4142135623730950488016887242097f;
  const int j0 = 2 * s.n_half;
  auto group_sync = [&] {
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(FG_THREADS) : "memory");
  };
#pragma unroll 1
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    const int ia = map.vec(item, 0, nl), ib = map.vec(item, 1, nl);
    const float* xa = x + (long long)ia * ldx;
    const float* xb = ib >= 0 ? x + (long long)ib * ldx : nullptr;
    __syncthreads();  // the previous item's reads of T are done
#pragma unroll 8
    for (int j = tid; j < j0; j += blockDim.x) {
      float* d = stf + (j >> 1) * 4 + (j & 1);
      d[0] = xa[j];
      d[2] = xb ? xb[j] : 0.f;
    }
    __syncthreads();
    // x-lines of the columns (which = 0) and of their mirror columns (1):
    // A + i B at n1, conj(A) + i conj(B) at -n1
#pragma unroll 1
    for (int u = tid; u < 2 * s.n_ucol; u += blockDim.x) {
      const int which = u >= s.n_ucol;
      const UCol c = s.ucol[u - which * s.n_ucol];
      const bool self = c.col == c.mcol;
      if ((self && which) || !ucol_in_range(s, c)) continue;
      // member of n1: fp/fn + sp/sn n1 for positive and negative n1; the sign
      // is also that of the conjugation
      const int sp = which ? -1 : 1, sn = self ? -1 : sp;
      const int fp = self ? c.h0 - 1 : c.h0 + c.R1;
      const float gp = (float)sp, gn = (float)sn;
      cpx<float> v[N];
#pragma unroll
      for (int p = 0; p < N; ++p) {
        v[p] = zero<float>();
        if (!in_sphere_band(p, N)) continue;
        const int n1 = freq_of(p, N);
        if (n1 == 0) {
          if (self) {
            v[p] = mk(rt2 * xa[j0], xb ? rt2 * xb[j0] : 0.f);
          } else {
            const float4 f = st[fp];
            v[p] = mk(f.x - gp * f.w, gp * f.y + f.z);
          }
        } else if (iabs(n1) <= c.R1) {
          const float4 f = st[fp + (n1 > 0 ? sp : sn) * n1];
          const float g = n1 > 0 ? gp : gn;
          v[p] = mk(f.x - g * f.w, g * f.y + f.z);
        }
      }
      LineDFT<float, N, +1, BAND>::run(v);
      cpx<float>* o = B1 + (which ? c.mcol : c.col);
#pragma unroll
      for (int p = 0; p < N; ++p) o[(long long)p * s.n_col] = v[p];
    }
    __syncthreads();
    // planes of this thread's group, PG at a time: y-lines (plane, n3), z-lines
    // (plane, i2) with the potential, y-lines back, a line per thread.  A thread's
    // y-lines there and back are the same.  One loop body for the three keeps
    // the code of one transform each way in the instruction cache.
#pragma unroll 1
    for (int p0 = grp * PG; p0 < N; p0 += groups * PG) {
#pragma unroll 1
      for (int step = 0; step < 3; ++step) {
        const bool z = step == 1;
        const int i1 = min(p0 + (z ? zp : yp), N - 1);
        const bool act = p0 + (z ? zp : yp) < N && (z ? zon : yact);
        const int bound = act ? (z ? s.R3 : yR) : -1;
        const int col = i1 * s.n_col;
        // a y-line's columns, its (n3, i2) row, and a z-line's two parts
        auto line = [&] { return B1 + (col + ymid); };
        auto yt = [&] { return yin ? B1 + (col + ysl) : T2 + (yp * N * rows.out + ysl - rows.in); };
        auto zin = [&] { return B1 + (col + i2 * rows.in + s.R3); };
        auto zout = [&] { return T2 + ((zp * N + i2) * rows.out + s.R3 - rows.in); };
        // OVER: a plane's y-lines overwrite what others read, so a barrier follows
        // their loads.  The body is the warp's, with the lines' loads and stores
        // predicated: a branch per line around the barrier spilled its registers.
        if (__any_sync(0xffffffffu, act)) {
          cpx<float> v[N];
          if (step < 2) {
            if (z) {
              const cpx<float>*zi = zin(), *zo = zout();
#pragma unroll
              for (int p = 0; p < N; ++p) {
                const int n = freq_of(p, N);
                v[p] = in_sphere_band(p, N) && iabs(n) <= bound
                           ? (OVER && n + s.R3 < rows.in ? zi : zo)[n]
                           : zero<float>();
              }
            } else {
              const cpx<float>* l = line();
#pragma unroll
              for (int p = 0; p < N; ++p) {
                const int n = freq_of(p, N);
                v[p] = in_sphere_band(p, N) && iabs(n) <= bound ? l[n] : zero<float>();
              }
            }
            if (OVER && !z) group_sync();
            LineDFT<float, N, +1, BAND>::run(v);
          } else {
            const cpx<float>* y = yt();
            const int ys = yin ? rows.in : rows.out;
#pragma unroll
            for (int p = 0; p < N; ++p, y += ys) v[p] = *y;
            if (OVER) group_sync();
          }
          if (step == 0) {
            cpx<float>* y = yt();
            const int ys = yin ? rows.in : rows.out;
#pragma unroll
            for (int p = 0; p < N; ++p, y += ys)
              if (act) *y = v[p];
          } else {
            if (z) {
              const float* vp = vt + i1 * (N * N) + i2;
#pragma unroll
              for (int p = 0; p < N; ++p) v[p] = scale(v[p], __ldg(vp + p * N));
            }
            LineDFT<float, N, -1, ALL>::run(v);
            if (z) {
              cpx<float>*zi = zin(), *zo = zout();
#pragma unroll
              for (int p = 0; p < N; ++p) {
                const int n = freq_of(p, N);
                if (in_sphere_band(p, N) && iabs(n) <= bound)
                  (OVER && n + s.R3 < rows.in ? zi : zo)[n] = v[p];
              }
            } else {
              cpx<float>* l = line();
#pragma unroll
              for (int p = 0; p < N; ++p) {
                const int n = freq_of(p, N);
                if (in_sphere_band(p, N) && iabs(n) <= bound) l[n] = v[p];
              }
            }
          }
        } else if (OVER && !z) {
          group_sync();
        }
        if (step < 2) group_sync();
      }
    }
    __syncthreads();
    // x-lines back.  With d the transform of a column and dm that of its
    // mirror at -n1, 2 Va = d + conj(dm) and 2 i Vb = d - conj(dm): the line of
    // a (which = 0) or b (1) is the transform of that combination of the columns
#pragma unroll 1
    for (int u = tid; u < 2 * s.n_ucol; u += blockDim.x) {
      const int which = u >= s.n_ucol;
      const UCol c = s.ucol[u - which * s.n_ucol];
      if (!ucol_in_range(s, c)) continue;
      const bool self = c.col == c.mcol;
      const float g = which ? -1.f : 1.f;
      const cpx<float>* o = B1 + c.col;
      const long long dm = c.mcol - c.col;
      cpx<float> v[N];
#pragma unroll
      for (int p = 0; p < N; ++p) {
        const cpx<float> a = o[(long long)p * s.n_col], b = o[(long long)p * s.n_col + dm];
        v[p] = mk(a.x + g * b.x, a.y - g * b.y);
      }
      LineDFT<float, N, -1, ALL>::run(v);
      // b's value is -i times the line's
      float* d = stf + 4 * (self ? c.h0 - 1 : c.h0 + c.R1) + 2 * which;
#pragma unroll
      for (int p = 0; p < N; ++p) {
        if (!in_sphere_band(p, N)) continue;
        const int n1 = freq_of(p, N);
        const float re = which ? v[p].y : v[p].x, im = which ? -v[p].x : v[p].y;
        if (n1 == 0 && self)
          stf[2 * j0 + 2 * which] = re;
        else if (iabs(n1) <= c.R1 && (!self || n1 > 0))
          *reinterpret_cast<float2*>(d + 4 * n1) = make_float2(re, im);
      }
    }
    __syncthreads();
    // four components at a time: their loads are in flight together (the
    // outputs may alias the inputs, so the compiler keeps loads behind stores)
    const OutRow<float> oa(ep, ia), ob(ep, ib);
    const bool old = ep.beta != 0;
#pragma unroll 1
    for (int jb = tid; jb <= j0; jb += 4 * blockDim.x) {
      float xi[4][2], yo[4][2], kin[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = jb + q * blockDim.x;
        const bool on = j <= j0, two = on && ib >= 0;
        xi[q][0] = on && oa.x_ ? oa.x_[j] : 0.f;
        xi[q][1] = two && ob.x_ ? ob.x_[j] : 0.f;
        yo[q][0] = on && old ? oa.y_[j] : 0.f;
        yo[q][1] = two && old ? ob.y_[j] : 0.f;
        kin[q] = j < j0 ? s.kin[j >> 1] : 0.f;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = jb + q * blockDim.x;
        if (j > j0) break;
        const bool g0 = j == j0;
        const float* d = stf + (j >> 1) * 4 + (j & 1);
        const float w = ep.scale * (g0 ? 0.25f * rt2 : 0.5f) *
                        (g0 ? (ep.coef == COEF_ONE ? 1.f : 0.f) : coef_of<float>(ep.coef, s.g2, j >> 1));
        const float dg = ep.kin * kin[q];
        // the diagonal term is the large one: its product is the fused one.
        // Without a diagonal term or an old output its value above is zero.
        oa.y_[j] = fmaf(ep.beta, yo[q][0], fmaf(dg + oa.sh_, xi[q][0], w * d[0]));
        if (ib >= 0) ob.y_[j] = fmaf(ep.beta, yo[q][1], fmaf(dg + ob.sh_, xi[q][1], w * d[2]));
      }
    }
  }
  if (tid == 0) {
    const int mine = items > (int)blockIdx.x ? (items - 1 - (int)blockIdx.x) / gridDim.x + 1 : 0;
    dev_timer_block_end(timer, t0, mine * item_flops, mine * item_bytes);
  }
}

// out (i1, i3, i2) = scale in (i1, i2, i3) on a cubic grid: a z-line per thread
// then reads the potential coalesced, and the transforms' 1 / (N1 N2 N3), which
// rounded to FP32 would be a common error of all components, is in its rounding
__global__ void k_fused_potential(const double* __restrict__ in, float* __restrict__ out, int N,
                                  double scale) {
  const int plane = blockIdx.x * N * N;
  for (int j = threadIdx.x; j < N * N; j += blockDim.x)
    out[plane + j] = (float)(scale * in[plane + (j % N) * N + j / N]);
}

// resident blocks per SM of a kernel at a block size and shared memory
// (queried once per combination)
template <typename K>
static int occupancy(K kern, int threads, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int, size_t>, int> cache;
  std::lock_guard<std::mutex> g(mu);
  const auto key = std::make_tuple((const void*)kern, threads, smem);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  int o = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, threads, smem) != cudaSuccess || o < 1) {
    cudaGetLastError();
    o = 1;
  }
  cache[key] = o;
  return o;
}

static int sm_count() {
  static const int n = [] {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 152;
  }();
  return n;
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
size_t slab_smem_bytes(int n_col, int R3, int N2, size_t elem) {
  const int ts = elem == 4 ? N2 + 8 : N2;  // T2Stride
  return (size_t)(n_col + (2 * R3 + 1) * ts) * 2 * elem;
}

template <typename R, int N>
static int threads_for(int lines) {
  int n = lines * Tpl<R, N>::v;
  return ((n + 31) / 32) * 32;
}

template <typename R, int N1>
static cudaError_t cols_fwd_impl(const SphereDev<R>& s, const R* x, long long ldx,
                                 ItemMap map,
                                 int n_items, int coef, cpx<R>* b1, cudaStream_t st) {
  const int per = 128 / Tpl<R, N1>::v;
  const long long total = (long long)n_items * s.n_ucol;
  if (total == 0) return cudaSuccess;
  const long long blocks = (total + per - 1) / per;
  // one x-line per column (n_col lines per item): 5 L log2 L flops each
  const double lines = (double)n_items * s.n_col;
  ProfScope ps(PC_COLS_F32, st,
               lines * 5.0 * N1 * log2((double)N1),
               (double)n_items * 2.0 * s.n_pw * sizeof(R) +
                   lines * N1 * 2.0 * sizeof(R),
               map.list ? map.n_dev : nullptr, map.n_list);
  count_launch();
  k_cols_fwd<R, N1><<<(unsigned)blocks, 128, 0, st>>>(s, x, ldx, map, n_items, coef, b1);
  return cudaGetLastError();
}

template <typename R, int N1>
static cudaError_t cols_bwd_impl(const SphereDev<R>& s, const cpx<R>* b1, ItemMap map,
                                 int n_items, const Epilogue<R>& ep, cudaStream_t st) {
  const int per = 128 / Tpl<R, N1>::v;
  const long long total = (long long)n_items * s.n_ucol;
  if (total == 0) return cudaSuccess;
  const long long blocks = (total + per - 1) / per;
  const double lines = (double)n_items * s.n_col;
  const double vecs = (double)n_items * 2.0 * s.n_pw * sizeof(R);
  ProfScope ps(PC_COLS_F32, st,
               lines * 5.0 * N1 * log2((double)N1),
               lines * N1 * 2.0 * sizeof(R) + vecs * (1.0 + (ep.x_in ? 1.0 : 0.0) +
                                                      (ep.beta != 0 ? 1.0 : 0.0)),
               map.list ? map.n_dev : nullptr, map.n_list);
  count_launch();
  k_cols_bwd<R, N1><<<(unsigned)blocks, 128, 0, st>>>(s, b1, map, n_items, ep);
  return cudaGetLastError();
}

template <int N2, int N3, bool DN>
static cudaError_t slab_impl_dn(const SphereDev<float>& s, const SlabArgs<float>& a,
                                cudaStream_t st) {
  int nt = threads_for<float, N3>(N2);
  int ny = threads_for<float, N2>(2 * s.R3 + 1);
  if (ny > nt) nt = ny;
  if (nt > SlabThreads<N2, N3>::v) return cudaErrorInvalidConfiguration;
  const size_t smem = slab_smem_bytes(s.n_col, s.R3, N2, sizeof(float));
  auto kern = k_slab<N2, N3, DN>;
  static OncePerDevice limit;  // per instantiation
  if (const cudaError_t e = raise_smem_limit(limit, kern, 200 * 1024)) return e;
  const int gx = a.n_items;
  if (gx == 0) return cudaSuccess;
  const long long resident = (long long)occupancy(kern, nt, smem) * sm_count();
  // as many items per unit as leave some eight units per resident block
  const int group =
      DN ? (int)std::max<long long>(1, std::min<long long>(8, (long long)gx * s.N1 / (8 * resident)))
         : 1;
  const long long units = (long long)((gx + group - 1) / group) * s.N1;
  const dim3 grid((unsigned)std::min<long long>(units, resident));
  double fl = 0, by = 0;
  slab_work(s, a, fl, by);
  ProfScope ps(PC_SLAB_F32, st, fl, by, a.map.list ? a.map.n_dev : nullptr, a.map.n_list);
  count_launch();
  kern<<<grid, nt, smem, st>>>(s, a, group);
  return cudaGetLastError();
}
template <int N2, int N3>
static cudaError_t slab_impl(const SphereDev<float>& s, const SlabArgs<float>& a, cudaStream_t st) {
  return a.mode == SLAB_HPSI && a.dn_at ? slab_impl_dn<N2, N3, true>(s, a, st)
                                     : slab_impl_dn<N2, N3, false>(s, a, st);
}

cudaError_t launch_cols_fwd(const SphereDev<float>& s, const float* x, long long ldx,
                            ItemMap map, int n_items, int coef, cpx<float>* b1, cudaStream_t st) {
  switch (s.N1) {
    case 24: return cols_fwd_impl<float, 24>(s, x, ldx, map, n_items, coef, b1, st);
    case 32: return cols_fwd_impl<float, 32>(s, x, ldx, map, n_items, coef, b1, st);
    case 40: return cols_fwd_impl<float, 40>(s, x, ldx, map, n_items, coef, b1, st);
    case 48: return cols_fwd_impl<float, 48>(s, x, ldx, map, n_items, coef, b1, st);
    case 64: return cols_fwd_impl<float, 64>(s, x, ldx, map, n_items, coef, b1, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_cols_bwd(const SphereDev<float>& s, const cpx<float>* b1, ItemMap map, int n_items,
                            const Epilogue<float>& ep, cudaStream_t st) {
  switch (s.N1) {
    case 24: return cols_bwd_impl<float, 24>(s, b1, map, n_items, ep, st);
    case 32: return cols_bwd_impl<float, 32>(s, b1, map, n_items, ep, st);
    case 40: return cols_bwd_impl<float, 40>(s, b1, map, n_items, ep, st);
    case 48: return cols_bwd_impl<float, 48>(s, b1, map, n_items, ep, st);
    case 64: return cols_bwd_impl<float, 64>(s, b1, map, n_items, ep, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_slab(const SphereDev<float>& s, const SlabArgs<float>& a, cudaStream_t st) {
  if (s.N2 == s.N3) {
    switch (s.N2) {
      case 24: return slab_impl<24, 24>(s, a, st);
      case 32: return slab_impl<32, 32>(s, a, st);
      case 40: return slab_impl<40, 40>(s, a, st);
      case 48: return slab_impl<48, 48>(s, a, st);
      case 64: return slab_impl<64, 64>(s, a, st);
    }
  } else if (s.N2 == 64 && s.N3 == 192) {
    return slab_impl<64, 192>(s, a, st);
  }
  return cudaErrorInvalidValue;
}

struct FusedShape {
  int planes, groups;
  bool over;
};
static FusedShape fused_shape(int N) {
  switch (N) {
    case 24: return {Fused<24>::PLANES, Fused<24>::GROUPS, Fused<24>::OVER};
    case 32: return {Fused<32>::PLANES, Fused<32>::GROUPS, Fused<32>::OVER};
    case 40: return {Fused<40>::PLANES, Fused<40>::GROUPS, Fused<40>::OVER};
    case 48: return {Fused<48>::PLANES, Fused<48>::GROUPS, Fused<48>::OVER};
  }
  return {0, 0, false};
}

// shared memory of a block of 'groups' groups
static size_t fused_bytes(const SphereDev<float>& s, int groups) {
  const FusedShape f = fused_shape(s.N1);
  const size_t t2 = (size_t)groups * f.planes * s.N1 * fused_rows(f.over, s.n_col, s.R3, s.N1).out;
  const size_t members = ((size_t)s.n_half + 1) * 2;  // (a, b) of a half index: two complex
  return ((size_t)s.N1 * s.n_col + std::max(t2, members)) * sizeof(cpx<float>);
}

int hpsi_fused_planes(const SphereDev<float>& s, int planes) {
  if (s.N1 != s.N2 || s.N2 != s.N3) return 0;
  const FusedShape f = fused_shape(s.N1);
  if (!f.planes) return 0;
  int groups = planes > 0 ? std::min(std::max(planes / f.planes, 1), f.groups) : f.groups;
  while (groups > 0 && fused_bytes(s, groups) > 226 * 1024) --groups;
  return groups * f.planes;
}

size_t hpsi_fused_smem(const SphereDev<float>& s, int planes) {
  const int G = hpsi_fused_planes(s, planes);
  return G > 0 ? fused_bytes(s, G / fused_shape(s.N1).planes) : 0;
}

cudaError_t fused_potential(const double* in, float* out, int N, double scale, cudaStream_t st) {
  count_launch();
  k_fused_potential<<<N, 256, 0, st>>>(in, out, N, scale);
  return cudaGetLastError();
}

template <int N>
static cudaError_t hpsi_fused_impl(const SphereDev<float>& s, const float* x, long long ldx,
                                   ItemMap map, int n_items, const float* vt,
                                   const Epilogue<float>& ep, size_t smem, int G,
                                   cudaStream_t st) {
  auto kern = k_hpsi_fused<N>;
  static OncePerDevice limit;  // per instantiation
  if (const cudaError_t e = raise_smem_limit(limit, kern, 226 * 1024)) return e;
  const int threads = G / Fused<N>::PLANES * FG_THREADS;
  const unsigned grid = (unsigned)std::min<long long>(
      n_items, (long long)occupancy(kern, threads, smem) * sm_count());
  // algorithmic work: as the three launches it replaces (x-lines both ways,
  // y- and z-lines both ways, V products); bytes: the vectors only
  const double planes = (double)n_items * s.N1;
  const double fl = (double)n_items * 2.0 * s.n_col * 5.0 * N * log2((double)N) +
                    planes * (2.0 * (2 * s.R3 + 1) * 5.0 * N * log2((double)N) +
                              2.0 * N * 5.0 * N * log2((double)N) + 2.0 * N * N);
  const double by = (double)n_items * 2.0 * s.n_pw * sizeof(float) * 3.0;
  // timed on the device (this kernel also runs inside the CG graphs): the
  // work is counted per processed item
  count_launch();
  kern<<<grid, threads, smem, st>>>(s, x, ldx, map, n_items, vt, ep, dev_timer(PC_HPSI_FUSED),
                                    fl / n_items, by / n_items);
  return cudaGetLastError();
}

cudaError_t launch_hpsi_fused(const SphereDev<float>& s, const float* x, long long ldx, ItemMap map,
                              int n_items, const float* vt, const Epilogue<float>& ep,
                              cudaStream_t st, int planes) {
  const size_t smem = hpsi_fused_smem(s, planes);
  if (smem == 0) return cudaErrorInvalidValue;
  if (n_items <= 0) return cudaSuccess;
  const int G = hpsi_fused_planes(s, planes);
  switch (s.N1) {
    case 24: return hpsi_fused_impl<24>(s, x, ldx, map, n_items, vt, ep, smem, G, st);
    case 32: return hpsi_fused_impl<32>(s, x, ldx, map, n_items, vt, ep, smem, G, st);
    case 40: return hpsi_fused_impl<40>(s, x, ldx, map, n_items, vt, ep, smem, G, st);
    case 48: return hpsi_fused_impl<48>(s, x, ldx, map, n_items, vt, ep, smem, G, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pdep
