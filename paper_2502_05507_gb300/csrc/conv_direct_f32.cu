// The direct i pass for float32.
#include "conv_direct.cuh"

namespace bae {

template void direct_configure<float>();
template void launch_direct_i<float>(const ConvArgs<float>&, cudaStream_t);

}  // namespace bae
