// The even-odd schedule for float32, transform length 256.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<float, 256>(const ConvArgs<float>&);
template bool eo_apply<float, 256>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 256>();

}  // namespace bae
