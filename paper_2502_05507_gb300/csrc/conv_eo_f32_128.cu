// The even-odd schedule for float32, transform length 128.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<float, 128>(const ConvArgs<float>&);
template bool eo_apply<float, 128>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 128>();

}  // namespace bae
