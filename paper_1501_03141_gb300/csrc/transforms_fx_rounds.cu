// The FP64 slab pass (fx_slab.cuh) of refinement rounds inside a graph: H x with
// the density response, whose array the kernel finds through a.dn_at.
#include "fx_slab.cuh"

namespace pdep {
namespace {

template <int N2, int N3>
cudaError_t rounds_impl(const SphereDev<double>& s, const SlabArgs<double>& a, cudaStream_t st) {
  return a.digits < FX_S ? slab_fx_mode<SLAB_HPSI, true, 7, N2, N3>(s, a, st)
                         : slab_fx_mode<SLAB_HPSI, true, 8, N2, N3>(s, a, st);
}

}  // namespace

cudaError_t launch_slab_rounds(const SphereDev<double>& s, const SlabArgs<double>& a,
                               cudaStream_t st) {
  if (a.mode != SLAB_HPSI || !a.dn_at) return cudaErrorInvalidValue;
  if (s.N2 == s.N3) {
    switch (s.N2) {
      case 24: return rounds_impl<24, 24>(s, a, st);
      case 32: return rounds_impl<32, 32>(s, a, st);
      case 40: return rounds_impl<40, 40>(s, a, st);
      case 48: return rounds_impl<48, 48>(s, a, st);
      case 64: return rounds_impl<64, 64>(s, a, st);
    }
  } else if (s.N2 == 64 && s.N3 == 192) {
    return rounds_impl<64, 192>(s, a, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pdep
