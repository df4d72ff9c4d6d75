// dgpe_fine.h -- passes of the FP64 form on grids too small to fill the GPU
// (dgpe_fine.cu): arguments and launchers.
#pragma once

#include <cuda_runtime.h>

namespace dgpe {

// Constant-coefficient Crank-Nicolson solve of one axis in FP64 (the
// factorisation is derived in dgpe_lines.cuh): alpha, -2 kt m, alpha^1 ..
// alpha^CL, alpha^(CL 2^k) for the scan over chunks, the chunks dl an inflow
// reaches (0: all, by a scan), and the exact correction of the first row,
// table E_a = (alpha^(a+2) - alpha^(2n-a+2)) / (1 - alpha^(2n+2)) of which the
// first nE chunks are not negligible.
enum { FINE_CL = 16, FINE_LOG = 5, FINE_DL = 4 };
template <typename Coef> struct FineCn {
  Coef al, m2, pw[FINE_CL], pc[FINE_LOG];
  const Coef *E;
  int dl, nE;
};
struct FineArgs {
  double2 *psi;  // complex state (src 2, real: nx reals per row)
  double2 *spec;
  double *phi_out;
  const double *dens_in, *U;
  double *prm, *partial;
  long long *step;
  unsigned *counter;
  const double2 *tw;  // exp(-2 pi i t / n) of the axis
  const double *vx, *vy, *vz;
  int nx, ny, nrows, px;
  int n, ncols, outer;  // strided passes: line length, columns, outer index count
  long long es, os;
  int has_dip, final_pass, norm, nsm, early;
};
// radix of a transform's stage with `left` points to go
constexpr int fine_radix(int left) { return left % 4 == 0 ? 4 : left % 5 == 0 ? 5 : left % 3 == 0 ? 3 : 2; }
// points per lane of the solve (n / that is a power of two <= 32)
int fine_chunk(int n);
// density (src 0: sc^2 |psi|^2, 1: dens_in, 2: of a real state) + R2C along x
cudaError_t fine_dens(const FineArgs &A, int src, cudaStream_t s);
// FFT along a strided axis of the half spectrum: mode 0 forward, 1 inverse, 2 forward . U . inverse
cudaError_t fine_fft(const FineArgs &A, int mode, cudaStream_t s);
// C2R along x, exponential, Crank-Nicolson along x (real: of a real state); Phi_d alone
cudaError_t fine_back(const FineArgs &A, const FineCn<double> &K, bool real, cudaStream_t s);
cudaError_t fine_back(const FineArgs &A, const FineCn<double2> &K, cudaStream_t s);
cudaError_t fine_phi(const FineArgs &A, cudaStream_t s);
// Crank-Nicolson along a strided axis; at most fine_cn_blocks norm partials
int fine_cn_blocks(int n, int tot, int nsm);
cudaError_t fine_cn(const FineArgs &A, const FineCn<double> &K, cudaStream_t s);
cudaError_t fine_cn(const FineArgs &A, const FineCn<double2> &K, cudaStream_t s);

}  // namespace dgpe
