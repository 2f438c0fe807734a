// Fixed-point FP64 hop of one direction (see hop_fx.cuh).
#include "hop_fx.cuh"

namespace dwf {
template cudaError_t hop_fx_launch<false>(const HopArgs &, cudaStream_t);
}  // namespace dwf
