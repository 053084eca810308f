// The even-odd schedule for double-float, transform lengths 16, 32, 64.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<dsf, 16>(const ConvArgs<dsf>&);
template bool eo_apply<dsf, 16>(const ConvArgs<dsf>&, cudaStream_t);
template void eo_configure<dsf, 16>();
template bool eo_runs<dsf, 32>(const ConvArgs<dsf>&);
template bool eo_apply<dsf, 32>(const ConvArgs<dsf>&, cudaStream_t);
template void eo_configure<dsf, 32>();
template bool eo_runs<dsf, 64>(const ConvArgs<dsf>&);
template bool eo_apply<dsf, 64>(const ConvArgs<dsf>&, cudaStream_t);
template void eo_configure<dsf, 64>();

}  // namespace bae
