// Grid product in double-float arithmetic: single-context launches (the 16-element passes are in matvec_dfc_e16.cu).
#include "matvec_kernels.cuh"

namespace aim {

extern template aim_status launch_row_fwd<dfc, 1, 4, false>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_fwd<dfc, 2, 4, false>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_col_conv<dfc, 1, 4, false>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_col_conv<dfc, 2, 4, false>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_inv<dfc, 1, 4, false>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_inv<dfc, 2, 4, false>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_fwd<dfc, 1, 3, true>(aim_ctx*, int, RowFwdArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_col_conv<dfc, 1, 3, true>(aim_ctx*, int, ColArgs, const Schedule&, cudaStream_t);
extern template aim_status launch_row_inv<dfc, 1, 3, true>(aim_ctx*, int, RowInvArgs, const Schedule&, cudaStream_t);
template aim_status grid_pass<dfc>(aim_ctx*, const PassSpec&, int, const double2*, double2*, cudaStream_t);
template aim_status grid_product_dense<dfc>(aim_ctx*, bool, int, const double2*, double2*, void*, size_t, cudaStream_t);

}  // namespace aim
