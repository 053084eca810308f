// The applies on windows of 192 nodes for float64 (transform length 384).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<double, 384>(const ConvArgs<double>&);
template bool eo_apply<double, 384>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 384>();
template void run_window<double, 384>(const ConvArgs<double>&, cudaStream_t);
template void conv_configure<double, 384>();

}  // namespace bae
