// The even-odd schedule for float64, transform length 256.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<double, 256>(const ConvArgs<double>&);
template bool eo_apply<double, 256>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 256>();

}  // namespace bae
