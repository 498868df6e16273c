// Grid product in complex64 arithmetic: several contexts in one persistent launch, 16 elements per thread.
#include "matvec_kernels.cuh"

namespace aim {

template aim_status launch_multi_groups<float2, 1, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);
template aim_status launch_multi_groups<float2, 2, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);

}  // namespace aim
