// dgpe_rows_real.cu -- x-row pass of the FP32 bulk in imaginary time (complex
// and real state), and Phi_d alone.
#include "dgpe_rows_back.cuh"

namespace dgpe {

cudaError_t rows_back_launch(const RowArgs &A, const CUtensorMap &tm, const CnConst<float> &K, int grid, cudaStream_t s) {
  switch (A.mode) {
    case ROWS_STEP: return back_launch<float, ROWS_STEP>(A, tm, K, grid, s);
    case ROWS_PHI: return back_launch<float, ROWS_PHI>(A, tm, K, grid, s);
    case ROWS_REAL: return back_launch<float, ROWS_REAL>(A, tm, K, grid, s);
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t rows_back_grid_real(int n, int nrows, int mode, int nsm, int *grid) {
  switch (mode) {
    case ROWS_STEP: return back_grid<float, ROWS_STEP>(n, nrows, nsm, grid);
    case ROWS_PHI: return back_grid<float, ROWS_PHI>(n, nrows, nsm, grid);
    case ROWS_REAL: return back_grid<float, ROWS_REAL>(n, nrows, nsm, grid);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dgpe
