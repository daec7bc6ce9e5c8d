// tm_dslash_f64_18.cu -- the hopping launches of TM_F64 spinor storage with 18-real links (the
// fixed-point kernel of tm_hop_fx.cuh, every epilogue) reading FP64 fields; those that read FX fields
// are instantiated in tm_dslash_fx.cu.
#include "tm_hop_fx.cuh"

namespace tmq {

tm_status hop_launch_fx(tm_lattice lat, const HopArgs& a, cudaStream_t s);

tm_status hop_launch_f64_18(tm_lattice lat, const HopArgs& a, cudaStream_t s) {
  return (a.fx.flags & FX_IN) ? hop_launch_fx(lat, a, s) : hop_fx_launch_t<false>(lat, a, s);
}

}  // namespace tmq
