// dgpe_lines.h -- arguments and launchers of the register-resident line
// passes of the FP32 bulk (dgpe_rows*.cu: x-rows; dgpe_cols.cu: the strided
// Crank-Nicolson solves along y and z).  Each kernel is compiled once, in
// those units; the solver (and dgpe_noalloc.cu, the row passes) calls the launchers.
#pragma once

#include <cuda.h>  // CUtensorMap
#include <cuda_runtime.h>

namespace dgpe {

// Launch of a pass that begins with pdl_wait (dgpe_device.cuh).  early: its
// blocks may start before the kernel ahead of it in the stream has ended.
template <class... P, class... A>
inline cudaError_t launch_pdl(bool early, void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                              const A &...args) {
  cudaLaunchConfig_t c{};
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &a;
  c.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&c, k, static_cast<P>(args)...);
}

// Constant-coefficient form of one Crank-Nicolson substep along a line
// (dgpe_lines.cuh): alpha, -2 kt m, alpha^CL and alpha^1 .. alpha^CL, the
// reach dl of the chunk inflow (1..4 chunks; 0: the coefficients decay too
// slowly for this form) and the number J <= CL of sites of a chunk that an
// inflow still changes.
enum { CN_PW = 20, CN_DL = 4 };
template <typename Coef> struct CnConst {
  Coef al, m2, pc, pw[CN_PW];
  int dl, J;
};

// Strided CN pass: `tot` columns (column c starts at
// (c / ncols) os + c % ncols) of n points es apart.
struct ColArgs {
  float2 *psi;
  const void *cntab;  // m, alpha, P, Q (n each): the table form's coefficients
  double *prm;
  double *partial;
  unsigned *counter;
  long long *step;
  long long es, os;
  unsigned tot, ncols;
  int n, cl;       // points; points per chunk (16, 12 or 10)
  int back;        // tiles from the last to the first
  int nsm;         // SMs, as in cols_grid
  int final_pass, norm;
  int early;       // launch_pdl
  int dlim;        // chunk reach of the table form (0: all chunks)
  double tau;      // kt = tau (imaginary time) or i tau (real time)
};
// Persistent grid of the pass over `tot` columns (real_coef: imaginary time;
// tab: the table form), at most one block per tile; then the launch.
int cols_grid(int n, int cl, unsigned tot, int nsm, bool real_coef, bool tab);
cudaError_t cols_launch(const ColArgs &A, const CnConst<float> &K, int grid, cudaStream_t s);
cudaError_t cols_launch(const ColArgs &A, const CnConst<float2> &K, int grid, cudaStream_t s);

// x-row passes (dgpe_rows*.cu).  psi: [nrows][n] complex (src 2 / ROWS_REAL:
// real), 16-byte aligned; spec: the half spectrum, rows of n / 2 + 2 elements.
struct RowArgs {
  float2 *psi;
  float2 *spec;
  float *phi_out;
  const float *dens_in;
  const double *prm;
  const long long *step;
  const float2 *tw;  // exp(-2 pi i t / n)
  const float *vx, *vy, *vz;
  int n, ny, nrows;
  int has_dip;
  int early;   // launch_pdl
  int src;     // forward: 0 sc^2 |psi|^2, 1 the real field dens_in, 2 sc^2 psi^2 of a real state
  int mode;    // backward: ROWS_*
  double dtf;  // fraction of dt of the exponential substep
};
// C2R along x, exponential, Crank-Nicolson along x (STEP; REAL: of a real
// state), or one of them alone (PHI: Phi_d into phi_out; CN; EXP)
enum { ROWS_STEP = 0, ROWS_PHI = 1, ROWS_CN = 2, ROWS_EXP = 3, ROWS_REAL = 4, ROWS_MODES = 5 };
// points of a row that one lane solves: the chunk length of the constant form
int rows_chunk(int n);
// rows of a warp's tile
int rows_per_tile(int n);
// The grids raise the kernels' shared-memory limits: once before a launch.
cudaError_t rows_fwd_grid(int n, int nrows, int src, int nsm, int *grid);
cudaError_t rows_fwd_launch(const RowArgs &A, int grid, cudaStream_t s);
// tm: the state as rows of 16 elements (2^k lengths; see rows_back.cuh)
cudaError_t rows_back_grid_real(int n, int nrows, int mode, int nsm, int *grid);
cudaError_t rows_back_grid_cplx(int n, int nrows, int mode, int nsm, int *grid);
cudaError_t rows_back_launch(const RowArgs &A, const CUtensorMap &tm, const CnConst<float> &K, int grid, cudaStream_t s);
cudaError_t rows_back_launch(const RowArgs &A, const CUtensorMap &tm, const CnConst<float2> &K, int grid, cudaStream_t s);

}  // namespace dgpe
