// Grid product in double-float arithmetic: several contexts in one persistent launch, 16 elements per thread.
#include "matvec_kernels.cuh"

namespace aim {

template aim_status launch_multi_groups<dfc, 1, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);
template aim_status launch_multi_groups<dfc, 2, 4>(const MultiPassSpec*, int, unsigned*, int*, cudaStream_t);

}  // namespace aim
