// dgpe_noalloc.cu -- dgpe_dipolar_potential_noalloc: the dipolar-potential
// chain (density + R2C along x, transforms along y / z with the kernel
// multiply, C2R along x) on caller-owned device buffers, with every piece of
// scratch (half spectrum, U(k)/N table, FFT roots, parameter block) placed in
// one file-scope device array instead of memory from cudaMalloc.
//
// Who needs it: code that may not allocate device memory while it runs --
// work recorded into a stream capture by a host framework that owns every
// allocation, callers running under a fixed device-memory budget or a caching
// allocator that must see all allocations, and real-time loops where an
// allocation's latency and possible failure are not acceptable.
//
// The array below stays resident on every GPU that loads this library until
// the process exits.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "dgpe.h"
#include "dgpe_kernels.cuh"
#include "dgpe_fine.h"
#include "dgpe_lines.h"

namespace dgpe {
namespace {

constexpr size_t kScratchBytes = size_t(4) << 20;     // 4 MiB per device
constexpr size_t kMaxSites = size_t(1) << 18;         // largest grid accepted
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

std::mutex g_mu;
void *g_scratch_ptr[kMaxDevices];      // device address of g_scratch, per device
bool g_ready[kMaxDevices];
thread_local char g_err[256];  // fixed buffer: no allocation on error paths either

void set_err(const char *msg, const char *detail = nullptr) {
  if (detail) snprintf(g_err, sizeof(g_err), "%s: %s", msg, detail);
  else snprintf(g_err, sizeof(g_err), "%s", msg);
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Roots w[t] = exp(-2 pi i t / n) per axis, U(k)/N on the half spectrum
// [z][y][kx] (pitch px), and the parameter block (sc = 1, everything else 0).
// FP64 work at 64 cycles per warp instruction and scheduler is what this costs:
// U depends on |ky| and |kz| alone, so each value is computed once and written
// to its two (2D) or four (3D) places (64^3: the whole call 104 -> 60 us), from wavenumber steps dq = 2 pi / (n h)
// and the factor 1 / N that the host forms; one division (3D) is left.
template <typename R>
__global__ void k_noalloc_tables(cx<R> *tw0, cx<R> *tw1, cx<R> *tw2, R *U, double *prm,
                                 long long *step, int dim, int nx, int ny, int nz, int px,
                                 double dqx, double dqy, double dqz, int kernel, double qd, double pref, double rN) {
  const unsigned gid = blockIdx.x * blockDim.x + threadIdx.x, gs = gridDim.x * blockDim.x;
  const int ns[3] = {nx, ny, nz};
  cx<R> *tw[3] = {tw0, tw1, tw2};
  for (int a = 0; a < dim; ++a)
    for (unsigned t = gs - 1 - gid; t < (unsigned)ns[a]; t += gs) {  // the threads with the fewest U values
      double s, c;
      sincospi(-2.0 * (double)t / (double)ns[a], &s, &c);
      tw[a][t] = mk<R>((R)c, (R)s);
    }
  const unsigned nxh = nx / 2 + 1, nyh = ny / 2 + 1, nzh = nz / 2 + 1, cnt = nxh * nyh * nzh;
  for (unsigned i = gid; i < cnt; i += gs) {
    const unsigned kx = i % nxh, r = i / nxh, ky = r % nyh, kz = r / nyh;
    const double qx = (double)kx * dqx, qy = (double)ky * dqy;
    double u = 0.0;
    if (kernel == DGPE_KERNEL_DIPOLAR_3D) {
      const double qz = (double)kz * dqz, z2 = qz * qz, k2 = fma(qx, qx, fma(qy, qy, z2));
      u = (k2 == 0.0) ? 0.0 : pref * fma(3.0, z2 / k2, -1.0);
    } else if (kernel == DGPE_KERNEL_QUASI2D_XY) {
      const double q = sqrt(qx * qx + qy * qy) * qd, v = q * 0.70710678118654752440;
      double ex;
      if (v < 25.0) {
        ex = exp(v * v) * erfc(v);
      } else {  // asymptotic series of exp(v^2) erfc(v)
        double term = 1.0, sum = 1.0;
        for (int m = 1; m < 8; ++m) { term *= -(2.0 * m - 1.0) / (2.0 * v * v); sum += term; }
        ex = sum / (v * sqrt(M_PI));
      }
      u = pref * (2.0 - 3.0 * sqrt(M_PI / 2.0) * q * ex);
    }
    const R ur = (R)(u * rN);
    const unsigned my = ky ? ny - ky : 0, mz = kz ? nz - kz : 0;
    U[((size_t)kz * ny + ky) * px + kx] = ur;
    U[((size_t)kz * ny + my) * px + kx] = ur;
    U[((size_t)mz * ny + ky) * px + kx] = ur;
    U[((size_t)mz * ny + my) * px + kx] = ur;
  }
  if (gid < PRM_COUNT) prm[gid] = (gid == PRM_SC) ? 1.0 : 0.0;
  if (gid == 0) *step = 0;
}

bool pow2_in_range(int n) { return n >= 32 && n <= 512 && (n & (n - 1)) == 0; }

// The chain behind the table kernel: density + R2C along x, the transforms
// along y and z, C2R along x.
struct Chain {
  int dim, nx, ny, nz, nrows, px, ncols, nsm;
  const void *psi;
  void *phi, *spec, *U, *tw[3];
  double *prm;
  long long *step;
};

// FP32: the solver's warp-per-tile row passes and length-specialised strided
// transforms (64^3: 60 -> 27 us against runtime lengths, one launch after the
// other).  The row kernels' grids (blocks that fit times SMs, and the
// shared-memory limit that goes with them) depend on the device and the
// length alone and are found once per device.
template <int MODE> cudaError_t strided32(const Chain &c, int n, long long es, long long os, int outer, const void *tw,
                                          cudaStream_t s) {
  constexpr int E = 16;
  SArgs<float> A{};
  A.spec = (float2 *)c.spec; A.U = (float *)c.U; A.tw = (const float2 *)tw; A.estride = es; A.ostride = os;
  A.n = n; A.ncols = c.ncols; A.nxh = c.nx / 2;
  auto go = [&](auto Nc) {
    constexpr int N = decltype(Nc)::value, W = N == 512 ? 8 : 16;
    return launch_pdl(true, k_fft_strided_ct<E, MODE, N, W>, dim3((c.ncols + W - 1) / W, outer), W * N / E,
                      sizeof(float2) * N * W, s, A);
  };
  switch (n) {
    case 32: return go(std::integral_constant<int, 32>{});
    case 64: return go(std::integral_constant<int, 64>{});
    case 128: return go(std::integral_constant<int, 128>{});
    case 256: return go(std::integral_constant<int, 256>{});
    default: return go(std::integral_constant<int, 512>{});
  }
}
// The density pass of a state that bulk copies cannot start at.
cudaError_t dens_any(const Chain &c, cudaStream_t s) {
  constexpr int EPT = 8, CL = 16, PW = 128 / (int)sizeof(float2);
  XArgs<float> X{};
  X.psi = (float2 *)c.psi; X.spec = (float2 *)c.spec; X.prm = c.prm; X.tw = (const float2 *)c.tw[0];
  X.nx = c.nx; X.ny = c.ny; X.nrows = c.nrows; X.px = c.px; X.TPL = c.nx / CL; X.C = CL;
  X.LP = DGPE_MAXT / 2 / X.TPL;
  X.pitchz = c.nx + c.nx / PW + 1;
  X.pl.n = c.nx;
  for (int m = c.nx; m > 1; m /= X.pl.rad[X.pl.ns++]) X.pl.rad[X.pl.ns] = m % 8 == 0 ? 8 : m % 4 == 0 ? 4 : 2;
  const int npairs = (c.nrows + 1) / 2;
  const size_t sm = sizeof(float2) * (size_t)X.LP * X.pitchz;  // at most 18 KB
  k_dens_r2c_x<float, EPT><<<(npairs + X.LP - 1) / X.LP, 2 * X.LP * X.TPL, sm, s>>>(X);
  return cudaGetLastError();
}
cudaError_t chain32(const Chain &c, int dev, cudaStream_t s) {
  static std::atomic<int> fwd[kMaxDevices][5], back[kMaxDevices][5];  // largest grids, 0: not yet known
  int k = 0;
  while ((32 << k) < c.nx) ++k;
  cudaError_t e;
  const int all = 1 << 30;
  int gf = fwd[dev][k].load(), gb = back[dev][k].load();
  if (!gf) {
    if ((e = rows_fwd_grid(c.nx, all, 0, c.nsm, &gf)) != cudaSuccess) return e;
    fwd[dev][k].store(gf);
  }
  if (!gb) {
    if ((e = rows_back_grid_real(c.nx, all, ROWS_PHI, c.nsm, &gb)) != cudaSuccess) return e;
    back[dev][k].store(gb);
  }
  RowArgs A{};
  A.psi = (float2 *)c.psi; A.spec = (float2 *)c.spec; A.phi_out = (float *)c.phi; A.prm = c.prm; A.step = c.step;
  A.tw = (const float2 *)c.tw[0]; A.n = c.nx; A.ny = c.ny; A.nrows = c.nrows; A.has_dip = 1;
  const int tiles = (c.nrows + rows_per_tile(c.nx) - 1) / rows_per_tile(c.nx);
  if (((uintptr_t)c.psi & 15) == 0) {
    if ((e = rows_fwd_launch(A, std::min(gf, tiles), s)) != cudaSuccess) return e;
  } else if ((e = dens_any(c, s)) != cudaSuccess) {
    return e;
  }
  const long long py = c.px, pz = (long long)c.ny * c.px;
  if (c.dim == 3) {
    if ((e = strided32<0>(c, c.ny, py, pz, c.nz, c.tw[1], s)) != cudaSuccess) return e;
    if ((e = strided32<2>(c, c.nz, pz, py, c.ny, c.tw[2], s)) != cudaSuccess) return e;
    if ((e = strided32<1>(c, c.ny, py, pz, c.nz, c.tw[1], s)) != cudaSuccess) return e;
  } else if ((e = strided32<2>(c, c.ny, py, pz, 1, c.tw[1], s)) != cudaSuccess) {
    return e;
  }
  A.mode = ROWS_PHI;
  A.early = 1;
  return rows_back_launch(A, CUtensorMap{}, CnConst<float>{}, std::min(gb, tiles), s);
}

// FP64: the solver's passes for small grids.
cudaError_t chain64(const Chain &c, cudaStream_t s) {
  FineArgs A{};
  A.psi = (double2 *)c.psi; A.spec = (double2 *)c.spec; A.phi_out = (double *)c.phi; A.U = (double *)c.U;
  A.prm = c.prm; A.step = c.step; A.tw = (const double2 *)c.tw[0];
  A.nx = c.nx; A.ny = c.ny; A.nrows = c.nrows; A.px = c.px; A.ncols = c.ncols; A.has_dip = 1; A.nsm = c.nsm;
  cudaError_t e = fine_dens(A, 0, s);  // reads what the table kernel wrote: not early
  A.early = 1;
  auto strided = [&](int mode, int axis) {
    if (e != cudaSuccess) return;
    FineArgs B = A;
    const long long py = c.px, pz = (long long)c.ny * c.px;
    B.tw = (const double2 *)c.tw[axis];
    B.n = axis == 1 ? c.ny : c.nz; B.es = axis == 1 ? py : pz; B.os = axis == 1 ? pz : py; B.outer = axis == 1 ? c.nz : c.ny;
    e = fine_fft(B, mode, s);
  };
  if (c.dim == 3) {
    strided(0, 1);
    strided(2, 2);
    strided(1, 1);
  } else {
    strided(2, 1);
  }
  return e == cudaSuccess ? fine_phi(A, s) : e;
}

template <typename R>
int run(const void *psi, void *phi, int dim, const int *n, const double *h, int kernel, double qd,
        cudaStream_t s, int dev, unsigned char *base) {
  typedef cx<R> Cx;
  Chain c{};
  c.dim = dim; c.psi = psi; c.phi = phi;
  c.nx = n[0]; c.ny = n[1]; c.nz = (dim == 3) ? n[2] : 1;
  c.nrows = c.ny * c.nz;
  c.px = c.nx / 2 + 1;
  if (sizeof(Cx) == 8) c.px = (c.px + 1) & ~1;
  c.ncols = c.nx / 2 + 1;
  // carve the scratch array
  size_t off = 0;
  auto carve = [&](size_t bytes) { void *p = base + off; off = align256(off + bytes); return p; };
  const size_t nspec = (size_t)c.px * c.nrows;
  c.spec = carve(nspec * sizeof(Cx));
  c.U = carve(nspec * sizeof(R));
  for (int a = 0; a < 3; ++a) c.tw[a] = carve(512 * sizeof(Cx));
  c.prm = (double *)carve(PRM_COUNT * sizeof(double));
  c.step = (long long *)carve(sizeof(long long));
  if (off > kScratchBytes) { set_err("grid too large for the static scratch array"); return DGPE_EUNSUPPORTED; }
  cudaError_t e = cudaDeviceGetAttribute(&c.nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) {
    const double twopi = 6.283185307179586476925286766559, hz = dim == 3 ? h[2] : 1.0;
    const double pref = kernel == DGPE_KERNEL_DIPOLAR_3D ? 4.0 * M_PI / 3.0 : (4.0 * M_PI / 3.0) / (sqrt(2.0 * M_PI) * qd);
    const int cnt = (c.nx / 2 + 1) * (c.ny / 2 + 1) * (c.nz / 2 + 1);
    k_noalloc_tables<R><<<std::min((cnt + 63) / 64, c.nsm * 8), 64, 0, s>>>(
        (Cx *)c.tw[0], (Cx *)c.tw[1], (Cx *)c.tw[2], (R *)c.U, c.prm, c.step, dim, c.nx, c.ny, c.nz, c.px,
        twopi / (c.nx * h[0]), twopi / (c.ny * h[1]), twopi / (c.nz * hz), kernel, qd, pref,
        1.0 / ((double)c.nx * c.ny * c.nz));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    if constexpr (sizeof(R) == 4) e = chain32(c, dev, s);
    else e = chain64(c, s);
  }
  if (e != cudaSuccess) {
    set_err("launch", cudaGetErrorString(e));
    return DGPE_ECUDA;
  }
  return DGPE_OK;
}

}  // namespace
}  // namespace dgpe

// Phi_d of |psi|^2 for a caller's state, without allocating device memory.
extern "C" int dgpe_dipolar_potential_noalloc(const void *psi, void *phi, int fp64, int dim,
                                              const int n[3], const double h[3], int kernel,
                                              double qd, void *cuda_stream) {
  using namespace dgpe;
  if (!psi || !phi || !n || !h) { set_err("NULL argument"); return DGPE_EINVAL; }
  if (dim != 2 && dim != 3) { set_err("dim must be 2 or 3"); return DGPE_EINVAL; }
  if (kernel == DGPE_KERNEL_QUASI2D_XZ) {
    set_err("the quasi-2D XZ kernel is not supported by this entry point");
    return DGPE_EUNSUPPORTED;
  }
  if ((kernel == DGPE_KERNEL_DIPOLAR_3D && dim != 3) ||
      (kernel == DGPE_KERNEL_QUASI2D_XY && (dim != 2 || !(qd > 0.0))) ||
      (kernel != DGPE_KERNEL_DIPOLAR_3D && kernel != DGPE_KERNEL_QUASI2D_XY)) {
    set_err("kernel does not match the dimension");
    return DGPE_EINVAL;
  }
  size_t sites = 1;
  for (int a = 0; a < dim; ++a) {
    if (!pow2_in_range(n[a])) { set_err("each n must be a power of two in [32, 512]"); return DGPE_EUNSUPPORTED; }
    if (!(h[a] > 0.0) || !std::isfinite(h[a])) { set_err("spacing must be > 0"); return DGPE_EINVAL; }
    sites *= (size_t)n[a];
  }
  if (sites > kMaxSites) {
    set_err("grid has more than 262144 sites, the limit of the static scratch array");
    return DGPE_EUNSUPPORTED;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    set_err("cudaGetDevice", cudaGetErrorString(e));
    return DGPE_ECUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) {
    set_err("device index above 63: this entry point serves devices 0..63");
    return DGPE_EUNSUPPORTED;
  }
  void *base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_ready[dev]) {
      // first call on this device: look up where the array lives
      e = cudaGetSymbolAddress(&g_scratch_ptr[dev], g_scratch);
      if (e != cudaSuccess) {
        set_err("cudaGetSymbolAddress", cudaGetErrorString(e));
        return DGPE_ECUDA;
      }
      g_ready[dev] = true;
    }
    base = g_scratch_ptr[dev];
  }
  cudaStream_t s = (cudaStream_t)cuda_stream;
  return fp64 ? run<double>(psi, phi, dim, n, h, kernel, qd, s, dev, (unsigned char *)base)
              : run<float>(psi, phi, dim, n, h, kernel, qd, s, dev, (unsigned char *)base);
}

extern "C" const char *dgpe_noalloc_last_error(void) { return dgpe::g_err; }
