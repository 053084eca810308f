// The even-odd schedule for float32, transform length 512.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<float, 512>(const ConvArgs<float>&);
template bool eo_apply<float, 512>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 512>();

}  // namespace bae
