// The even-odd schedule for float64, transform length 512.
#include "conv_eo.cuh"

namespace bae {

template bool eo_runs<double, 512>(const ConvArgs<double>&);
template bool eo_apply<double, 512>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 512>();

}  // namespace bae
