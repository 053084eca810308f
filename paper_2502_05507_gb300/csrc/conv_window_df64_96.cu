// The applies on windows of 48 nodes for double-float (transform length 96).
#include "conv_eo.cuh"
#include "conv_impl.cuh"

namespace bae {

template bool eo_runs<dsf, 96>(const ConvArgs<dsf>&);
template bool eo_apply<dsf, 96>(const ConvArgs<dsf>&, cudaStream_t);
template void eo_configure<dsf, 96>();
template void run_window<dsf, 96>(const ConvArgs<dsf>&, cudaStream_t);
template void conv_configure<dsf, 96>();

}  // namespace bae
