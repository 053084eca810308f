// The even-odd schedule for float64, transform lengths 16, 32, 64.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<double, 16>(const ConvArgs<double>&);
template bool eo_apply<double, 16>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 16>();
template bool eo_runs<double, 32>(const ConvArgs<double>&);
template bool eo_apply<double, 32>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 32>();
template bool eo_runs<double, 64>(const ConvArgs<double>&);
template bool eo_apply<double, 64>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 64>();

}  // namespace bae
