// The applies on windows of 192 nodes for double-float (transform length 384).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<dsf, 384>(const ConvArgs<dsf>&);
template bool eo_apply<dsf, 384>(const ConvArgs<dsf>&, cudaStream_t);
template void eo_configure<dsf, 384>();
template void run_window<dsf, 384>(const ConvArgs<dsf>&, cudaStream_t);
template void conv_configure<dsf, 384>();

}  // namespace bae
