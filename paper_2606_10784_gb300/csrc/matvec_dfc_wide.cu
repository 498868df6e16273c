// Grid product in double-float arithmetic: the wide variants of the passes with one transform of 8 elements per thread.
#include "matvec_kernels.cuh"

namespace aim {

template aim_status launch_row_fwd<dfc, 1, 3, true>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
template aim_status launch_col_conv<dfc, 1, 3, true>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
template aim_status launch_row_inv<dfc, 1, 3, true>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);

}  // namespace aim
