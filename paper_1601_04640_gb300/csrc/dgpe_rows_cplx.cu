// dgpe_rows_cplx.cu -- x-row pass of the FP32 bulk in real time; the
// exponential alone (ends of a second-order run) and the solve alone (reverse
// step).
#include "dgpe_rows_back.cuh"

namespace dgpe {

cudaError_t rows_back_launch(const RowArgs &A, const CUtensorMap &tm, const CnConst<float2> &K, int grid, cudaStream_t s) {
  switch (A.mode) {
    case ROWS_STEP: return back_launch<float2, ROWS_STEP>(A, tm, K, grid, s);
    case ROWS_CN: return back_launch<float2, ROWS_CN>(A, tm, K, grid, s);
    case ROWS_EXP: return back_launch<float2, ROWS_EXP>(A, tm, K, grid, s);
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t rows_back_grid_cplx(int n, int nrows, int mode, int nsm, int *grid) {
  switch (mode) {
    case ROWS_STEP: return back_grid<float2, ROWS_STEP>(n, nrows, nsm, grid);
    case ROWS_CN: return back_grid<float2, ROWS_CN>(n, nrows, nsm, grid);
    case ROWS_EXP: return back_grid<float2, ROWS_EXP>(n, nrows, nsm, grid);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dgpe
