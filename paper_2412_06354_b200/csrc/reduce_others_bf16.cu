// Segmented reductions over bf16 rows: max, min, the routing of their backward pass and per-feature factors.
#include "reduce_rows.cuh"

namespace gnn {
template void launch_reduce_others<__nv_bfloat16>(const PropParams&, int, bool, cudaStream_t);
}  // namespace gnn
