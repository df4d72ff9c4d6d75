// dgpe_fine.cu -- the passes of one step in FP64 on grids of up to some 10^6
// sites (the paper's calcpsidd2, calcnu, calclux/y/z, calcnorm).
//
// The smaller ones have fewer warps than the GPU has schedulers, so a pass takes
// what one warp executes: every instruction of a lone warp costs some 10 cycles,
// an FP64 one 64 (2 FMA per SM and clock), and code that runs once is fetched as
// it runs.  So a thread holds few points (one radix-4 or -5 butterfly, chunks of
// 3 to 5 points of a line), lengths are compile-time constants, the state goes
// from global memory to registers and back, and the solve needs no tables.
// A step of 32^3 in imaginary time went from 123 to 43 us, of a 96 x 160 plane
// from 156 to 37, of 256^2 from 129 to 56, of 64^3 from 143 to 118 (real time 183
// to 143) and of 64 x 80 x 64 in real time from 250 to 174; what is left on the
// smallest is some 6 us per pass: launch, a cold start and one warp's chain of
// FP64 instructions.
#include <algorithm>

#include "dgpe_kernels.cuh"
#include "dgpe_fine.h"
#include "dgpe_lines.h"

namespace dgpe {
namespace {

constexpr int fine_cl(int n) {
  int cl = n % 3 == 0 ? 3 : n % 5 == 0 ? 5 : 4;
  while (n / cl > 32) cl *= 2;
  return cl;
}

// Stockham stages over NL lines of a tile in shared memory, T threads.  Lines
// along the threads (COLS: element a of line l at a NL + l, NL = 2^ll) or one
// after the other (l SL + a + a / 8).  The first stage reads through load, the
// last writes through store.
template <int N> constexpr int fine_sl() { return N + N / 8 + 1; }
template <int N, bool COLS> __device__ __forceinline__ int fine_at(int l, int a, int ll) {
  return COLS ? (a << ll) + l : l * fine_sl<N>() + a + a / 8;
}
template <int N, int NS, bool INV, bool COLS, class Load, class Store>
__device__ __forceinline__ void fine_stages(double2 *z, const double2 *tw, int NL, int ll, Load &load, Store &store) {
  if constexpr (NS < N) {
    constexpr int RAD = fine_radix(N / NS), NBL = N / RAD, STR = N / (NS * RAD);
    constexpr bool FIRST = NS == 1, LAST = NS * RAD == N;
    const int B = NBL * NL, T = blockDim.x;
    // at most two butterflies per thread (radix 2 behind a block of n / 4 threads)
    double2 v[2][RAD];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int b = threadIdx.x + i * T;
      if (b >= B) break;
      const int l = COLS ? b & (NL - 1) : b / NBL, j = COLS ? b >> ll : b % NBL, k = j % NS;
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        v[i][r] = FIRST ? load(l, j + r * NBL) : z[fine_at<N, COLS>(l, j + r * NBL, ll)];
        if (!FIRST && r > 0) v[i][r] = INV ? cmulconj(v[i][r], tw[k * r * STR]) : cmul(v[i][r], tw[k * r * STR]);
      }
      dft<RAD, INV>(v[i]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int b = threadIdx.x + i * T;
      if (b >= B) break;
      const int l = COLS ? b & (NL - 1) : b / NBL, j = COLS ? b >> ll : b % NBL, base = (j / NS) * NS * RAD + j % NS;
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        if (LAST) store(l, base + r * NS, v[i][r]);
        else z[fine_at<N, COLS>(l, base + r * NS, ll)] = v[i][r];
      }
    }
    __syncthreads();
    fine_stages<N, NS * RAD, INV, COLS>(z, tw, NL, ll, load, store);
  }
}
// threads for NL lines: one per radix-4 butterfly, two radix-2 (or a radix-3
// and a part) ones at most
inline int fine_threads(int n, int nl) {
  const int per = n % 3 == 0 ? n / 3 : n / 4;
  return (std::max(per * nl, 1) + 31) / 32 * 32;
}

template <int N, int SRC> __global__ void __launch_bounds__(256) k_fine_dens(const __grid_constant__ FineArgs A, int LP) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ __align__(16) double2 tw[N];
  double2 *const z = reinterpret_cast<double2 *>(smraw);
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = A.tw[i];
  pdl_wait();
  const int p0 = blockIdx.x * LP;
  const double sc = SRC == 1 ? 1.0 : A.prm[PRM_SC], sc2 = sc * sc;
  __syncthreads();
  auto load = [&](int l, int a) -> double2 {
    const int r0 = 2 * (p0 + l);
    if (r0 >= A.nrows) return make_double2(0.0, 0.0);
    const size_t i = (size_t)r0 * N + a;
    if constexpr (SRC == 0) {
      const double2 x = A.psi[i], y = A.psi[i + N];
      return make_double2(sc2 * (x.x * x.x + x.y * x.y), sc2 * (y.x * y.x + y.y * y.y));
    } else if constexpr (SRC == 1) {
      return make_double2(A.dens_in[i], A.dens_in[i + N]);
    } else {
      const double *const pr = reinterpret_cast<const double *>(A.psi);
      return make_double2(sc2 * (pr[i] * pr[i]), sc2 * (pr[i + N] * pr[i + N]));
    }
  };
  auto store = [&](int l, int a, double2 v) { z[fine_at<N, false>(l, a, 0)] = v; };
  fine_stages<N, 1, false, false>(z, tw, LP, 0, load, store);
  // two real lines were packed as Z = n0 + i n1
  constexpr int NH = N / 2 + 1;
  for (int idx = threadIdx.x; idx < LP * NH; idx += blockDim.x) {
    const int l = idx / NH, k = idx % NH, r0 = 2 * (p0 + l);
    if (r0 >= A.nrows) break;
    const double2 Zk = z[fine_at<N, false>(l, k, 0)], Zm = z[fine_at<N, false>(l, k ? N - k : 0, 0)];
    double2 *const o = A.spec + (size_t)r0 * A.px + k;
    o[0] = make_double2(0.5 * (Zk.x + Zm.x), 0.5 * (Zk.y - Zm.y));
    o[A.px] = make_double2(0.5 * (Zk.y + Zm.y), 0.5 * (Zm.x - Zk.x));
  }
}

template <int N, int MODE> __global__ void __launch_bounds__(256) k_fine_fft(const __grid_constant__ FineArgs A, int lw) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ __align__(16) double2 tw[N];
  double2 *const z = reinterpret_cast<double2 *>(smraw);
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = A.tw[i];
  pdl_wait();
  __syncthreads();
  const int W = 1 << lw, c0 = blockIdx.x << lw;
  double2 *const p = A.spec + (size_t)blockIdx.y * A.os + c0;
  auto gload = [&](int l, int a) -> double2 { return c0 + l < A.ncols ? p[a * A.es + l] : make_double2(0.0, 0.0); };
  auto gstore = [&](int l, int a, double2 v) {
    if (c0 + l < A.ncols) p[a * A.es + l] = v;
  };
  if constexpr (MODE != 2) {
    fine_stages<N, 1, MODE == 1, true>(z, tw, W, lw, gload, gstore);
  } else {
    const double *const u = A.U + (size_t)blockIdx.y * A.os + c0;
    auto mstore = [&](int l, int a, double2 v) {
      z[(a << lw) + l] = cscale(v, c0 + l < A.ncols ? u[a * A.es + l] : 0.0);
    };
    auto sload = [&](int l, int a) -> double2 { return z[(a << lw) + l]; };
    fine_stages<N, 1, false, true>(z, tw, W, lw, gload, mstore);
    fine_stages<N, 1, true, true>(z, tw, W, lw, sload, gstore);
  }
}

// CL consecutive points of a line per lane, TPL lanes per line
template <typename Coef, int CL, int TPL>
__device__ __forceinline__ void fine_solve(double2 (&v)[CL], int q, const FineCn<Coef> &K) {
  double2 y[CL], prev = shfl_up(v[CL - 1], 1, TPL), next = shfl_down(v[0], 1, TPL);
  if (q == 0) prev = make_double2(0.0, 0.0);
  if (q == TPL - 1) next = make_double2(0.0, 0.0);
  double2 acc = make_double2(0.0, 0.0);
#pragma unroll
  for (int i = 0; i < CL; ++i) {
    // (2 psi_a - psi_{a-1}) - psi_{a+1}, one after the other: where psi is smooth both differences are exact, while a
    // rounded psi_{a-1} + psi_{a+1} leaves 2^-53 psi, which -2 kt m and the two recurrences amplify (two solves of
    // 32 to 256 points at kt between 1 and 10, relative L2: 1.9e-16 instead of 5.2e-16 in real time)
    // psi_{a+1} first at the chunk's first point, whose psi_{a-1} comes by a shuffle (96 x 160: 2014 -> 1999 us for
    // 50 steps and the observables).
    const double2 l = i ? v[i - 1] : prev, r = i + 1 < CL ? v[i + 1 < CL ? i + 1 : i] : next, f = i ? l : r, g = i ? r : l;
    acc = coef_fma(K.al, acc, make_double2(fma(2.0, v[i].x, -f.x) - g.x, fma(2.0, v[i].y, -f.y) - g.y));
    y[i] = acc;
  }
  double2 in = make_double2(0.0, 0.0);
  if (K.dl) {
    for (int d = K.dl; d > 0; --d) {
      const double2 t = shfl_up(acc, d, TPL);
      if (q >= d) in = coef_fma(K.pc[0], in, t);
    }
  } else {
#pragma unroll
    for (int k = 0; (1 << k) < TPL; ++k) {
      const double2 t = shfl_up(acc, 1 << k, TPL);
      if (q >= 1 << k) acc = coef_fma(K.pc[k], t, acc);
    }
    in = shfl_up(acc, 1, TPL);
    if (q == 0) in = make_double2(0.0, 0.0);
  }
  acc = make_double2(0.0, 0.0);
#pragma unroll
  for (int i = 0; i < CL; ++i) y[i] = coef_fma(K.pw[i], in, y[i]);
#pragma unroll
  for (int i = CL - 1; i >= 0; --i) {
    acc = coef_fma(K.al, acc, y[i]);
    y[i] = acc;
  }
  in = make_double2(0.0, 0.0);
  if (K.dl) {
    for (int d = K.dl; d > 0; --d) {
      const double2 t = shfl_down(acc, d, TPL);
      if (q + d < TPL) in = coef_fma(K.pc[0], in, t);
    }
  } else {
#pragma unroll
    for (int k = 0; (1 << k) < TPL; ++k) {
      const double2 t = shfl_down(acc, 1 << k, TPL);
      if (q + (1 << k) < TPL) acc = coef_fma(K.pc[k], t, acc);
    }
    in = shfl_down(acc, 1, TPL);
    if (q == TPL - 1) in = make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int i = 0; i < CL; ++i) y[CL - 1 - i] = coef_fma(K.pw[i], in, y[CL - 1 - i]);
  const double2 u0 = make_double2(-__shfl_sync(0xffffffffu, y[0].x, 0, TPL), -__shfl_sync(0xffffffffu, y[0].y, 0, TPL));
  if (q < K.nE) {
#pragma unroll
    for (int i = 0; i < CL; ++i) y[i] = coef_fma(K.E[q * CL + i], u0, y[i]);
  }
#pragma unroll
  for (int i = 0; i < CL; ++i) v[i] = v[i] + coef_mul(K.m2, y[i]);
}

enum { FB_STEP, FB_REAL, FB_PHI };
// LP pairs of rows: the transform by pairs, then one lane per chunk of a row
// (FB_REAL: of a pair, its rows the parts of one complex line).
template <typename Coef, int N, int MODE>
__global__ void __launch_bounds__(256)
    k_fine_back(const __grid_constant__ FineArgs A, const __grid_constant__ FineCn<Coef> K, int LP) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ __align__(16) double2 tw[N];
  __shared__ double s_k[4];
  constexpr int CL = fine_cl(N), TPL = N / CL;
  constexpr bool RT = std::is_same<Coef, double2>::value;
  double2 *const z = reinterpret_cast<double2 *>(smraw);
  const int p0 = blockIdx.x * LP, L = threadIdx.x / TPL, q = threadIdx.x % TPL;
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = A.tw[i];
  const int row = MODE == FB_REAL ? 2 * (p0 + L) : 2 * p0 + L;
  const bool on = MODE != FB_PHI && row < A.nrows && L < (MODE == FB_REAL ? LP : 2 * LP);
  double vx[CL], vr = 0.0, vb = 0.0;
  if (on) {
#pragma unroll
    for (int i = 0; i < CL; ++i) vx[i] = A.vx[q * CL + i];
    vr = A.vy[row % A.ny] + A.vz[row / A.ny];
    if (MODE == FB_REAL) vb = A.vy[(row + 1) % A.ny] + A.vz[(row + 1) / A.ny];
  }
  pdl_wait();
  double2 v[CL];
#pragma unroll
  for (int i = 0; i < CL; ++i) {
    v[i] = make_double2(0.0, 0.0);
    if (on) {
      const size_t at = (size_t)row * N + q * CL + i;
      if constexpr (MODE == FB_REAL) {
        const double *const pr = reinterpret_cast<const double *>(A.psi);
        v[i] = make_double2(pr[at], pr[at + N]);
      } else {
        v[i] = A.psi[at];
      }
    }
  }
  if (MODE != FB_PHI && threadIdx.x == 0) {
    s_k[0] = trap_dts(A.prm, *A.step);
    s_k[1] = A.prm[PRM_DT] * A.prm[PRM_G];
    s_k[2] = A.prm[PRM_DT] * A.prm[PRM_GDD];
    s_k[3] = A.prm[PRM_SC];
  }
  __syncthreads();
  if (A.has_dip) {
    auto load = [&](int l, int a) -> double2 {
      const int r0 = 2 * (p0 + l);
      if (r0 >= A.nrows) return make_double2(0.0, 0.0);
      const double2 *const o = A.spec + (size_t)r0 * A.px + (a <= N / 2 ? a : N - a);
      double2 x = o[0], y = o[A.px];
      if (a > N / 2) { x.y = -x.y; y.y = -y.y; }                 // Hermitian extension
      if (a == 0 || a == N / 2) { x.y = 0.0; y.y = 0.0; }        // real ends
      return make_double2(x.x - y.y, x.y + y.x);
    };
    auto store = [&](int l, int a, double2 f) {
      if constexpr (MODE == FB_PHI) {
        const int r0 = 2 * (p0 + l);
        if (r0 < A.nrows) {
          A.phi_out[(size_t)r0 * N + a] = f.x;
          A.phi_out[(size_t)(r0 + 1) * N + a] = f.y;
        }
      } else {
        z[fine_at<N, false>(l, a, 0)] = f;
      }
    };
    fine_stages<N, 1, true, false>(z, tw, LP, 0, load, store);
  }
  if constexpr (MODE != FB_PHI) {
    const double dts = s_k[0], gdt = s_k[1], gdddt = s_k[2], sc = RT ? 1.0 : s_k[3];
    const int l = MODE == FB_REAL ? L : L >> 1;
    if (on) {
#pragma unroll
      for (int i = 0; i < CL; ++i) {
        const double2 f = A.has_dip ? z[fine_at<N, false>(l, q * CL + i, 0)] : make_double2(0.0, 0.0);
        if constexpr (MODE == FB_REAL) {
          const double s = v[i].x * sc, t = v[i].y * sc;
          const double fa = fexpm1(-(dts * (vx[i] + vr) + gdt * (s * s) + gdddt * f.x));
          const double fb = fexpm1(-(dts * (vx[i] + vb) + gdt * (t * t) + gdddt * f.y));
          v[i] = make_double2(s + s * fa, t + t * fb);
        } else {
          const double2 u = RT ? v[i] : cscale(v[i], sc);
          const double phi = (L & 1) ? f.y : f.x;
          const double th = dts * (vx[i] + vr) + gdt * (u.x * u.x + u.y * u.y) + gdddt * phi;
          v[i] = nonlinear_factor<double>(u, th, RT ? 0 : 1);
        }
      }
    }
    fine_solve<Coef, CL, TPL>(v, q, K);
    if (on) {
#pragma unroll
      for (int i = 0; i < CL; ++i) {
        const size_t at = (size_t)row * N + q * CL + i;
        if constexpr (MODE == FB_REAL) {
          double *const pr = reinterpret_cast<double *>(A.psi);
          pr[at] = v[i].x;
          pr[at + N] = v[i].y;
        } else {
          A.psi[at] = v[i];
        }
      }
    }
  }
}

// Columns one after the other, TPL lanes each.
template <typename Coef, int N, bool NORM>
__global__ void __launch_bounds__(128)
    k_fine_cn(const __grid_constant__ FineArgs A, const __grid_constant__ FineCn<Coef> K) {
  __shared__ double red[32];
  __shared__ int am_last;
  constexpr int CL = fine_cl(N), TPL = N / CL;
  const unsigned g = blockIdx.x * blockDim.x + threadIdx.x, c = g / TPL, q = g % TPL;
  const unsigned o = c / A.ncols, tot = (unsigned)A.ncols * A.outer;
  double2 *const p = A.psi + (size_t)o * A.os + (c - o * A.ncols) + (size_t)(q * CL) * A.es;
  pdl_wait();
  double2 v[CL];
#pragma unroll
  for (int i = 0; i < CL; ++i) v[i] = c < tot ? p[i * A.es] : make_double2(0.0, 0.0);
  fine_solve<Coef, CL, TPL>(v, (int)q, K);
  double acc = 0.0;
  if (c < tot) {
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      p[i * A.es] = v[i];
      if (NORM) acc += v[i].x * v[i].x + v[i].y * v[i].y;
    }
  }
  if (!A.final_pass) return;
  // last pass of the step: the norm's partials (imaginary time) and, in the
  // last block to finish, their total in a fixed order, the new scale and the
  // step counter
  if (NORM) {
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) A.partial[blockIdx.x] = s;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    am_last = atomicAdd(A.counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  if (NORM) {
    double s = 0.0;
    for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) s += __ldcg(A.partial + i);
    s = block_sum(s, red);
    if (threadIdx.x == 0) {
      const double norm = A.prm[PRM_CELL] * s;
      if (norm > 0.0 && isfinite(norm)) A.prm[PRM_SC] = 1.0 / sqrt(norm);
      else A.prm[PRM_NONFINITE] = 1.0;
    }
  }
  if (threadIdx.x == 0) {
    *A.step += 1;
    *A.counter = 0u;
  }
}

template <class F> cudaError_t with_length(int n, F &&f) {
  switch (n) {
#define DGPE_FINE(N) case N: return f(std::integral_constant<int, N>{});
    DGPE_FINE(32) DGPE_FINE(64) DGPE_FINE(128) DGPE_FINE(256) DGPE_FINE(512)
    DGPE_FINE(48) DGPE_FINE(96) DGPE_FINE(192) DGPE_FINE(384)
    DGPE_FINE(40) DGPE_FINE(80) DGPE_FINE(160) DGPE_FINE(320)
#undef DGPE_FINE
    default: return cudaErrorInvalidValue;
  }
}
// one warp per block while that spreads the work over more SMs
inline int cn_threads(int n, int tot, int nsm) {
  const long long warps = ((long long)tot * (n / fine_cl(n)) + 31) / 32;
  return warps <= 8ll * nsm ? 32 : 128;
}
template <typename Coef, int MODE> cudaError_t back(const FineArgs &A, const FineCn<Coef> &K, cudaStream_t s) {
  return with_length(A.nx, [&](auto Nc) {
    constexpr int N = decltype(Nc)::value, TPL = N / fine_cl(N), R = MODE == FB_STEP ? 2 : 1;  // lanes per pair: R TPL
    const int LP = std::max(1, 32 / (R * TPL)), npairs = A.nrows / 2;
    const int T = MODE == FB_PHI ? fine_threads(N, LP) : std::max(R * LP * TPL, fine_threads(N, LP));
    return launch_pdl(A.early != 0, k_fine_back<Coef, N, MODE>, dim3((npairs + LP - 1) / LP), (T + 31) / 32 * 32,
                      sizeof(double2) * (size_t)LP * fine_sl<N>(), s, A, K, LP);
  });
}
template <typename Coef> cudaError_t cn(const FineArgs &A, const FineCn<Coef> &K, cudaStream_t s) {
  return with_length(A.n, [&](auto Nc) {
    constexpr int N = decltype(Nc)::value;
    const int tot = A.ncols * A.outer, T = cn_threads(N, tot, A.nsm), grid = fine_cn_blocks(N, tot, A.nsm);
    if constexpr (std::is_same<Coef, double>::value)
      if (A.norm) return launch_pdl(A.early != 0, k_fine_cn<Coef, N, true>, dim3(grid), T, 0, s, A, K);
    return launch_pdl(A.early != 0, k_fine_cn<Coef, N, false>, dim3(grid), T, 0, s, A, K);
  });
}

}  // namespace

int fine_chunk(int n) { return fine_cl(n); }
int fine_cn_blocks(int n, int tot, int nsm) {
  const long long threads = (long long)tot * (n / fine_cl(n));
  const int T = cn_threads(n, tot, nsm);
  return (int)((threads + T - 1) / T);
}
cudaError_t fine_dens(const FineArgs &A, int src, cudaStream_t s) {
  return with_length(A.nx, [&](auto Nc) {
    constexpr int N = decltype(Nc)::value;
    const int LP = std::max(1, 128 / N), npairs = A.nrows / 2, T = fine_threads(N, LP);
    const dim3 grid((npairs + LP - 1) / LP);
    const size_t sm = sizeof(double2) * (size_t)LP * fine_sl<N>();
    if (src == 0) return launch_pdl(A.early != 0, k_fine_dens<N, 0>, grid, T, sm, s, A, LP);
    if (src == 1) return launch_pdl(A.early != 0, k_fine_dens<N, 1>, grid, T, sm, s, A, LP);
    return launch_pdl(A.early != 0, k_fine_dens<N, 2>, grid, T, sm, s, A, LP);
  });
}
cudaError_t fine_fft(const FineArgs &A, int mode, cudaStream_t s) {
  return with_length(A.n, [&](auto Nc) {
    constexpr int N = decltype(Nc)::value;
    // eight columns (128-byte rows), halved to one warp while SMs are left without a block
    int lw = 3;
    while (lw > 0 && ((N << lw) / 4 > 256 || ((N << lw) / 4 > 32 && ((A.ncols >> lw) + 1) * A.outer < A.nsm))) --lw;
    const dim3 grid((A.ncols + (1 << lw) - 1) >> lw, A.outer);
    const int T = fine_threads(N, 1 << lw);
    const size_t sm = sizeof(double2) * (size_t)N << lw;
    if (mode == 0) return launch_pdl(A.early != 0, k_fine_fft<N, 0>, grid, T, sm, s, A, lw);
    if (mode == 1) return launch_pdl(A.early != 0, k_fine_fft<N, 1>, grid, T, sm, s, A, lw);
    return launch_pdl(A.early != 0, k_fine_fft<N, 2>, grid, T, sm, s, A, lw);
  });
}
cudaError_t fine_back(const FineArgs &A, const FineCn<double> &K, bool real, cudaStream_t s) {
  return real ? back<double, FB_REAL>(A, K, s) : back<double, FB_STEP>(A, K, s);
}
cudaError_t fine_back(const FineArgs &A, const FineCn<double2> &K, cudaStream_t s) { return back<double2, FB_STEP>(A, K, s); }
cudaError_t fine_phi(const FineArgs &A, cudaStream_t s) { return back<double, FB_PHI>(A, FineCn<double>{}, s); }
cudaError_t fine_cn(const FineArgs &A, const FineCn<double> &K, cudaStream_t s) { return cn(A, K, s); }
cudaError_t fine_cn(const FineArgs &A, const FineCn<double2> &K, cudaStream_t s) { return cn(A, K, s); }

}  // namespace dgpe
