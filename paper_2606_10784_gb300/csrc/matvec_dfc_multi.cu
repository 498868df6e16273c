// Grid product in double-float arithmetic: several contexts in one persistent launch (the 16-element passes are in matvec_dfc_multi_e16.cu).
#include "matvec_kernels.cuh"

namespace aim {

extern template aim_status launch_multi_groups<dfc, 1, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);
extern template aim_status launch_multi_groups<dfc, 2, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);
template aim_status grid_pass_multi<dfc>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);

}  // namespace aim
