// The applies on windows of 96 nodes for float32 (transform length 192).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<float, 192>(const ConvArgs<float>&);
template bool eo_apply<float, 192>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 192>();
template void run_window<float, 192>(const ConvArgs<float>&, cudaStream_t);
template void conv_configure<float, 192>();

}  // namespace bae
