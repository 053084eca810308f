// The applies on windows of 48 nodes for float32 (transform length 96).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<float, 96>(const ConvArgs<float>&);
template bool eo_apply<float, 96>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 96>();
template void run_window<float, 96>(const ConvArgs<float>&, cudaStream_t);
template void conv_configure<float, 96>();

}  // namespace bae
