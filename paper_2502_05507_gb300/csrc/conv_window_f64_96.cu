// The applies on windows of 48 nodes for float64 (transform length 96).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<double, 96>(const ConvArgs<double>&);
template bool eo_apply<double, 96>(const ConvArgs<double>&, cudaStream_t);
template void eo_configure<double, 96>();
template void run_window<double, 96>(const ConvArgs<double>&, cudaStream_t);
template void conv_configure<double, 96>();

}  // namespace bae
