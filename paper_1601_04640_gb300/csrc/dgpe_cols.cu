// dgpe_cols.cu -- Crank-Nicolson along y and z for the FP32 bulk: strided
// lines solved from registers (the paper's calcluy, calcluz, "Summary of
// revisions").
#include <algorithm>

#include "dgpe_lines.cuh"

namespace dgpe {
namespace {

// Columns per block of 256 threads: 8 (32 chunks) to 128 (2 chunks), halved
// while a grid leaves SMs without a block, to blocks of one warp or segments of
// two columns; the table form to 128 threads, because every block brings in the
// whole of the tables (512 x 512 in real time: two columns per block 14.3 us,
// four 10.2).
constexpr int kColsThreads = 256;
inline int cols_lw(int n, int cl, unsigned tot, int nsm, bool tab) {
  const int tpl = n / cl, least = tab ? 128 : 32;
  int lw = 0;
  while ((2 << lw) * tpl <= kColsThreads) ++lw;
  while (lw > 1 && (1 << lw) * tpl > least && (tot >> lw) < (unsigned)nsm) --lw;
  return lw;
}

// One thread holds CL consecutive points of one column in registers; the n /
// CL chunks of a column are threads of the same block, and a warp is 32 (8,
// 16) neighbouring columns of one (4, 2) chunks, so every load and store of
// psi is a contiguous segment and a table read is one address for the lanes of
// a chunk.  Chunks exchange their end values through shared memory, twice per
// solve.  TAB: coefficients from the tables m, alpha, P, Q (slowly decaying
// coefficients, K.dl = 0) instead of the constant form.
//
// Bound by HBM: 51 us per pass at 256^3 complex (5.2 TB/s of the 6.7 measured
// by a copy), 198 / 187 us (y / z) at 512 x 512 x 256; the same solve from a
// shared tile with four shared tables, two blocks per SM, took 81 us and 368 /
// 300 us.  256 threads at three blocks per SM (80 registers) was the fastest
// shape: two blocks 57 us, four blocks (64 registers, spills) 61 us, 512
// threads of 32 columns 62 us, chunks of 8 points 57 us.
template <typename Coef, int CL, bool NORM, bool TAB>
__global__ void __launch_bounds__(kColsThreads, 3)
    k_cn_cols(const __grid_constant__ ColArgs A, const __grid_constant__ CnConst<Coef> K, int lw, int ntiles) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double red[32];
  __shared__ int am_last;
  const int T = blockDim.x, t = threadIdx.x;
  const int lc = t & ((1 << lw) - 1), q = t >> lw, tpl = A.n / CL, n = A.n;
  float2 *const se = reinterpret_cast<float2 *>(smraw);  // chunk ends: forward, backward
  Coef *const tm = reinterpret_cast<Coef *>(se + 2 * T);  // TAB: -2 kt m, alpha, P, Q
  const Coef *const ta = tm + n, *const tp = ta + n, *const tq = tp + n;
  pdl_wait();
  if (TAB) {
    const Coef *g = reinterpret_cast<const Coef *>(A.cntab);
    const Coef m2kt = coef_scale(make_kt<Coef>(A.tau), -2.0f);
    for (int i = t; i < n; i += T) {
      tm[i] = coef_prod(m2kt, g[i]);
      for (int k = 1; k < 4; ++k) tm[k * n + i] = g[k * n + i];
    }
    __syncthreads();
  }
  const int a0 = q * CL;
  double acc = 0.0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const unsigned c = ((unsigned)(A.back ? ntiles - 1 - tile : tile) << lw) + (unsigned)lc;
    const bool ok = c < A.tot;
    const unsigned o = c / A.ncols;
    float2 *const p = A.psi + (size_t)o * A.os + (c - o * A.ncols) + (size_t)a0 * A.es;
    float2 v[CL], y[CL], prev = make_float2(0.0f, 0.0f), next = prev;
#pragma unroll
    for (int i = 0; i < CL; ++i) v[i] = prev;
    if (ok) {
      if (q > 0) prev = *(p - A.es);
#pragma unroll
      for (int i = 0; i < CL; ++i) v[i] = p[(size_t)i * A.es];
      if (q < tpl - 1) next = p[(size_t)CL * A.es];
    }
    if constexpr (!TAB) {
      col_solve<Coef, CL>(v, y, prev, next, q, tpl, lw, lc, se, K);
    } else {
      float2 e = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int i = 0; i < CL; ++i) {
        const float2 l = second_diff(i ? v[i - 1] : prev, v[i], i + 1 < CL ? v[i + 1] : next);
        e = coef_fma(ta[a0 + i], e, coef_mul(tm[a0 + i], l));
        y[i] = e;
      }
      se[t] = e;
      __syncthreads();
      const int dl = A.dlim > 0 ? A.dlim : tpl;
      float2 in = make_float2(0.0f, 0.0f);
      for (int j = max(0, q - dl); j < q; ++j) in = coef_fma(tp[j * CL + CL - 1], in, se[(j << lw) + lc]);
#pragma unroll
      for (int i = 0; i < CL; ++i) y[i] = coef_fma(tp[a0 + i], in, y[i]);
      e = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int i = CL - 1; i >= 0; --i) {
        e = coef_fma(ta[a0 + i], e, y[i]);
        y[i] = e;
      }
      float2 *const sb = se + T;
      sb[t] = e;
      __syncthreads();
      in = make_float2(0.0f, 0.0f);
      for (int j = min(tpl - 1, q + dl); j > q; --j) in = coef_fma(tq[j * CL], in, sb[(j << lw) + lc]);
#pragma unroll
      for (int i = 0; i < CL; ++i) v[i] = v[i] + coef_fma(tq[a0 + i], in, y[i]);
    }
    if (ok) {
      // |x|^2 of the thread's CL points in FP32, FP64 above them
      float ts = 0.0f;
#pragma unroll
      for (int i = 0; i < CL; ++i) {
        p[(size_t)i * A.es] = v[i];
        if (NORM) ts += v[i].x * v[i].x + v[i].y * v[i].y;
      }
      if (NORM) acc += (double)ts;
    }
  }
  if (!A.final_pass) return;
  // last pass of the step: the norm's partials (imaginary time) and, in the
  // last block to finish, their total in a fixed order, the new scale and
  // the step counter
  if (NORM) {
    const double s = block_sum(acc, red);
    if (t == 0) A.partial[blockIdx.x] = s;
  }
  if (t == 0) {
    __threadfence();
    am_last = (atomicAdd(A.counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  if (NORM) {
    double s = 0.0;
    for (unsigned i = t; i < gridDim.x; i += T) s += __ldcg(A.partial + i);
    s = block_sum(s, red);
    if (t == 0) {
      const double norm = A.prm[PRM_CELL] * s;
      if (norm > 0.0 && isfinite(norm)) A.prm[PRM_SC] = 1.0 / sqrt(norm);
      else A.prm[PRM_NONFINITE] = 1.0;
    }
  }
  if (t == 0) {
    *A.step += 1;
    *A.counter = 0u;
  }
}

template <class F> cudaError_t with_chunk(int cl, F &&f) {
  switch (cl) {
    case 16: return f(std::integral_constant<int, 16>{});
    case 12: return f(std::integral_constant<int, 12>{});
    case 10: return f(std::integral_constant<int, 10>{});
    default: return cudaErrorInvalidValue;
  }
}

template <typename Coef> size_t cols_smem(int n, int T, bool tab) {
  return sizeof(float2) * 2 * (size_t)T + (tab ? sizeof(Coef) * 4 * (size_t)n : 0);
}
// f(kernel) of the variant: the norm's code only in the pass that takes it
// (imaginary time)
template <typename Coef, class F> cudaError_t with_kernel(int cl, bool norm, bool tab, F &&f) {
  return with_chunk(cl, [&](auto CLc) -> cudaError_t {
    constexpr int CL = decltype(CLc)::value;
    if constexpr (std::is_same<Coef, float>::value) {
      if (norm) return tab ? f(k_cn_cols<Coef, CL, true, true>) : f(k_cn_cols<Coef, CL, true, false>);
    }
    return tab ? f(k_cn_cols<Coef, CL, false, true>) : f(k_cn_cols<Coef, CL, false, false>);
  });
}
template <typename Coef> int grid_of(int n, int cl, unsigned tot, int nsm, bool tab) {
  const int w = 1 << cols_lw(n, cl, tot, nsm, tab), T = w * (n / cl), ntiles = (int)((tot + (unsigned)w - 1) / (unsigned)w);
  int occ = 0;
  with_kernel<Coef>(cl, true, tab, [&](auto k) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, T, cols_smem<Coef>(n, T, tab));
  });
  return std::max(1, std::min(ntiles, nsm * std::max(occ, 1)));
}
template <typename Coef> cudaError_t launch(const ColArgs &A, const CnConst<Coef> &K, int grid, cudaStream_t s) {
  const bool tab = K.dl == 0;
  const int lw = cols_lw(A.n, A.cl, A.tot, A.nsm, tab), w = 1 << lw, T = w * (A.n / A.cl);
  const int ntiles = (int)((A.tot + (unsigned)w - 1) / (unsigned)w);
  return with_kernel<Coef>(A.cl, A.norm != 0, tab, [&](auto k) {
    return launch_pdl(A.early != 0, k, dim3(grid), T, cols_smem<Coef>(A.n, T, tab), s, A, K, lw, ntiles);
  });
}

}  // namespace

int cols_grid(int n, int cl, unsigned tot, int nsm, bool real_coef, bool tab) {
  return real_coef ? grid_of<float>(n, cl, tot, nsm, tab) : grid_of<float2>(n, cl, tot, nsm, tab);
}
cudaError_t cols_launch(const ColArgs &A, const CnConst<float> &K, int grid, cudaStream_t s) {
  return launch<float>(A, K, grid, s);
}
cudaError_t cols_launch(const ColArgs &A, const CnConst<float2> &K, int grid, cudaStream_t s) {
  return launch<float2>(A, K, grid, s);
}
}  // namespace dgpe
