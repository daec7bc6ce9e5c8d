// tm_dslash_fx.cu -- instantiation of the FP64 / 18-real hopping kernel reading FX half fields
// (tm_dslash_fx.cuh), compiled as its own unit.
#include "tm_hop_fx.cuh"

namespace tmq {
tm_status hop_launch_fx(tm_lattice lat, const HopArgs& a, cudaStream_t s) {
  return hop_fx_launch_t<true>(lat, a, s);
}
}  // namespace tmq
