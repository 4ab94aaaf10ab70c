// Column march (k_col.cuh) of F16 stacks.
#include "k_col.cuh"

namespace fitrig {

template cudaError_t launch_col<f16_t, false>(const CUtensorMap*, const StackArgs&, cudaStream_t);
template cudaError_t launch_col<f16_t, true>(const CUtensorMap*, const StackArgs&, cudaStream_t);

}  // namespace fitrig
