// The applies on windows of 96 nodes for float64 (transform length 192).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<double, 192>(const ConvArgs<double>&);
template bool eo_apply<double, 192>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 192>();
template void run_window<double, 192>(const ConvArgs<double>&, cudaStream_t);
template void conv_configure<double, 192>();

}  // namespace bae
