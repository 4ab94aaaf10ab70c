// Column march (k_col.cuh) of BF16 stacks.
#include "k_col.cuh"

namespace fitrig {

template cudaError_t launch_col<bf16_t, false>(const CUtensorMap*, const StackArgs&, cudaStream_t);
template cudaError_t launch_col<bf16_t, true>(const CUtensorMap*, const StackArgs&, cudaStream_t);

}  // namespace fitrig
