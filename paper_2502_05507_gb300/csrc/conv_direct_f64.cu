// The direct i pass for float64.
#include "conv_direct.cuh"

namespace bae {

template void direct_configure<double>();
template void launch_direct_i<double>(const ConvArgs<double>&, cudaStream_t);

}  // namespace bae
