// The even-odd schedule for float32, transform lengths 16, 32, 64.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<float, 16>(const ConvArgs<float>&);
template bool eo_apply<float, 16>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 16>();
template bool eo_runs<float, 32>(const ConvArgs<float>&);
template bool eo_apply<float, 32>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 32>();
template bool eo_runs<float, 64>(const ConvArgs<float>&);
template bool eo_apply<float, 64>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 64>();

}  // namespace bae
