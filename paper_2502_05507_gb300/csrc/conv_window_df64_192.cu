// The applies on windows of 96 nodes for double-float (transform length 192).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<dsf, 192>(const ConvArgs<dsf>&);
template bool eo_apply<dsf, 192>(const ConvArgs<dsf>&, cudaStream_t);
template void eo_configure<dsf, 192>();
template void run_window<dsf, 192>(const ConvArgs<dsf>&, cudaStream_t);
template void conv_configure<dsf, 192>();

}  // namespace bae
