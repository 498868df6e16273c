// Grid product in double-float arithmetic: single-context launches with 16 elements per thread (compiled apart from the rest, in parallel).
#include "matvec_kernels.cuh"

namespace aim {

template aim_status launch_row_fwd<dfc, 1, 4, false>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
template aim_status launch_row_fwd<dfc, 2, 4, false>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
template aim_status launch_col_conv<dfc, 1, 4, false>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
template aim_status launch_col_conv<dfc, 2, 4, false>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
template aim_status launch_row_inv<dfc, 1, 4, false>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);
template aim_status launch_row_inv<dfc, 2, 4, false>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);

}  // namespace aim
