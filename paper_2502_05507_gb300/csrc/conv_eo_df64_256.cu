// The even-odd schedule for double-float, transform length 256.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<dsf, 256>(const ConvArgs<dsf>&);
template bool eo_apply<dsf, 256>(const ConvArgs<dsf>&, cudaStream_t);
template void eo_configure<dsf, 256>();

}  // namespace bae
