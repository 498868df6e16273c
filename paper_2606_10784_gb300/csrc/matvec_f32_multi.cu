// Grid product in complex64 arithmetic: several contexts in one persistent launch (the 16-element passes are in matvec_f32_multi_e16.cu).
#include "matvec_kernels.cuh"

namespace aim {

extern template aim_status launch_multi_groups<float2, 1, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);
extern template aim_status launch_multi_groups<float2, 2, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);
template aim_status grid_pass_multi<float2>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);

}  // namespace aim
