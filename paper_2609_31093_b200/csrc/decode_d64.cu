// The decoding kernels for head dimension 64 (decode_kernel.cuh).
#include "decode_kernel.cuh"

namespace pisa {

int launch_decode_d64(const Geometry& g, const DecArgs& a, cudaStream_t s) { return launch_decode_dim<64>(g, a, s); }

}  // namespace pisa
