// Grid product in complex64 arithmetic: single-context launches (the 16-element passes are in matvec_f32_e16.cu).
#include "matvec_kernels.cuh"

namespace aim {

extern template aim_status launch_row_fwd<float2, 1, 4, false>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_fwd<float2, 2, 4, false>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_col_conv<float2, 1, 4, false>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_col_conv<float2, 2, 4, false>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_inv<float2, 1, 4, false>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_inv<float2, 2, 4, false>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);
template aim_status grid_pass<float2>(aim_ctx*, const PassSpec&, int, const double2*, double2*, cudaStream_t);
template aim_status grid_product_dense<float2>(aim_ctx*, bool, int, const double2*, double2*, void*, size_t, cudaStream_t);

}  // namespace aim
