// Segmented reduction behind the gradient of the GATv2 logits.
#include "reduce_rows.cuh"

namespace gnn {
template <typename T>
void launch_gatv2_rows(const PropParams& P, cudaStream_t st) { launch_reduce<T, MODE_V2>(P, true, st); }
template void launch_gatv2_rows<float>(const PropParams&, cudaStream_t);
template void launch_gatv2_rows<__nv_bfloat16>(const PropParams&, cudaStream_t);
}  // namespace gnn
