// The decoding kernels for head dimension 128 (decode_kernel.cuh).
#include "decode_kernel.cuh"

namespace pisa {

int launch_decode_d128(const Geometry& g, const DecArgs& a, cudaStream_t s) { return launch_decode_dim<128>(g, a, s); }

}  // namespace pisa
