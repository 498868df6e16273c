// Grid product in double-float arithmetic: single-context launches with 16 elements per thread (compiled apart from the rest, in parallel).
#include "matvec_kernels.cuh"

namespace aim {

template aim_status launch_tpt<dfc, 1, 4>(aim_ctx*, int, bool, RowFwdArgs, RowInvArgs, void*, const Schedule&, cudaStream_t);
template aim_status launch_tpt<dfc, 2, 4>(aim_ctx*, int, bool, RowFwdArgs, RowInvArgs, void*, const Schedule&, cudaStream_t);

}  // namespace aim
