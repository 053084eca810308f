// The applies on windows of 192 nodes for float32 (transform length 384).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<float, 384>(const ConvArgs<float>&);
template bool eo_apply<float, 384>(const ConvArgs<float>&, cudaStream_t);
template void eo_configure<float, 384>();
template void run_window<float, 384>(const ConvArgs<float>&, cudaStream_t);
template void conv_configure<float, 384>();

}  // namespace bae
