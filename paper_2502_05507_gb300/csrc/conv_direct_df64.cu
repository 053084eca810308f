// The direct i pass for double-float.
#include "conv_direct.cuh"

namespace bae {

template void direct_configure<dsf>();
template void launch_direct_i<dsf>(const ConvArgs<dsf>&, cudaStream_t);

}  // namespace bae
