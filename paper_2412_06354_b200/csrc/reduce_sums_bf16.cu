// Segmented reductions over bf16 rows: sums (plain, one factor per position, one per position and head).
#include "reduce_rows.cuh"

namespace gnn {
template void launch_reduce_sums<__nv_bfloat16>(const PropParams&, int, bool, cudaStream_t);
}  // namespace gnn
