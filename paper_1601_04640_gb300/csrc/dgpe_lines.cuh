// dgpe_lines.cuh -- device code of the register-resident line passes of the
// FP32 bulk: a Crank-Nicolson solve of CL consecutive points per thread whose
// chunks exchange only their end values.
//
// Constant-coefficient Crank-Nicolson solve.  Along a line of n points the
// substep is x = psi + w, A w = -2 kt T psi, A = I + kt T = tridiag(-kt,
// b, -kt), b = 1 + 2 kt, T = tridiag(-1, 2, -1).  The LU pivots m_a = 1 /
// (b - kt^2 m_{a-1}) converge to the fixed point m = 1 / (b - kt^2 m) =
// 2 / (b + sqrt(1 + 4 kt)) (b^2 - 4 kt^2 = 1 + 4 kt), and with alpha = kt m,
//   A = (1/m) [ (I - alpha S)(I - alpha S^T) + alpha^2 e_0 e_0^T ]
// exactly (S the shift; the product has 1 instead of 1 + alpha^2 in its first
// row).  So with
//   y_a = alpha y_{a-1} + (T psi)_a,   u_a = y_a + alpha u_{a+1},
// the solution is w_a = -2 kt m (u_a - alpha^{a+2} u_0): the correction is the
// image of the line in its first ghost point (up to factors 1 - alpha^{2n};
// the form is taken only where alpha^{4 CL} and so alpha^n are below 2^-32).
// No table is read: alpha, alpha^k and -2 kt m are kernel parameters, so the
// multiplies take them from the constant bank.  A chunk's inflow is the
// neighbouring chunk's end value; dl chunks reach further than 2^-32, and an
// inflow changes only the first J sites of a chunk by more than that.
#pragma once

#include <type_traits>

#include "dgpe_kernels.cuh"
#include "dgpe_lines.h"

namespace dgpe {
namespace {

// (T psi)_a = 2 psi_a - psi_{a-1} - psi_{a+1}
__device__ __forceinline__ float2 second_diff(float2 prev, float2 cur, float2 next) {
  const float2 s = prev + next;
  return make_float2(fmaf(2.0f, cur.x, -s.x), fmaf(2.0f, cur.y, -s.y));
}
// forward recurrence of a chunk with zero inflow; returns the end value
template <typename Coef, int CL>
__device__ __forceinline__ float2 cn_chunk_forward(const float2 (&v)[CL], float2 prev, float2 next,
                                                   const CnConst<Coef> &K, float2 (&y)[CL]) {
  float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int i = 0; i < CL; ++i) {
    acc = coef_fma(K.al, acc, second_diff(i ? v[i - 1] : prev, v[i], i + 1 < CL ? v[i + 1] : next));
    y[i] = acc;
  }
  return acc;
}
// add the forward inflow, then the backward recurrence with zero inflow;
// returns its end value (at the chunk's first site)
template <typename Coef, int CL>
__device__ __forceinline__ float2 cn_chunk_backward(float2 yin, const CnConst<Coef> &K, float2 (&y)[CL]) {
#pragma unroll
  for (int i = 0; i < CL; ++i) {
    if (i >= K.J) break;
    y[i] = coef_fma(K.pw[i], yin, y[i]);
  }
  float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int i = CL - 1; i >= 0; --i) {
    acc = coef_fma(K.al, acc, y[i]);
    y[i] = acc;
  }
  return acc;
}
// add the backward inflow
template <typename Coef, int CL>
__device__ __forceinline__ void cn_chunk_inflow(float2 win, const CnConst<Coef> &K, float2 (&y)[CL]) {
#pragma unroll
  for (int i = 0; i < CL; ++i) {
    if (i >= K.J) break;
    y[CL - 1 - i] = coef_fma(K.pw[i], win, y[CL - 1 - i]);
  }
}
// subtract the image, img = alpha^{a0 + 1} u_0 for the chunk that starts at
// a0 (0 where it has died out), and form x = psi - 2 kt m u
template <typename Coef, int CL>
__device__ __forceinline__ void cn_chunk_finish(float2 img, const CnConst<Coef> &K, float2 (&y)[CL], float2 (&v)[CL]) {
  img = make_float2(-img.x, -img.y);
#pragma unroll
  for (int i = 0; i < CL; ++i) {
    if (i >= K.J) break;
    y[i] = coef_fma(K.pw[i], img, y[i]);
  }
  // the product first: one rounding at the size of psi, not two
#pragma unroll
  for (int i = 0; i < CL; ++i) v[i] = v[i] + coef_mul(K.m2, y[i]);
}


// Solve of strided columns by a block: thread t holds chunk q = t >> lw of
// column lc, the chunks exchange their ends through se (2 blockDim.x elements).
template <typename Coef, int CL>
__device__ __forceinline__ void col_solve(float2 (&v)[CL], float2 (&y)[CL], float2 prev, float2 next, int q, int tpl, int lw,
                                          int lc, float2 *se, const CnConst<Coef> &K) {
  const int t = threadIdx.x;
  se[t] = cn_chunk_forward<Coef, CL>(v, prev, next, K, y);
  __syncthreads();
  float2 in = make_float2(0.0f, 0.0f);
  for (int j = max(0, q - K.dl); j < q; ++j) in = coef_fma(K.pc, in, se[(j << lw) + lc]);
  float2 *const sb = se + blockDim.x;
  sb[t] = cn_chunk_backward<Coef, CL>(in, K, y);
  __syncthreads();
  in = make_float2(0.0f, 0.0f);
  for (int j = min(tpl - 1, q + K.dl); j > q; --j) in = coef_fma(K.pc, in, sb[(j << lw) + lc]);
  cn_chunk_inflow<Coef, CL>(in, K, y);
  // u_0 of the column is the first chunk's y[0]
  float2 img = make_float2(0.0f, 0.0f);
  if (K.dl == 1) {
    if (q == 0) img = coef_mul(K.al, y[0]);
  } else {
    __syncthreads();  // the forward ends have been read
    if (q == 0) se[lc] = y[0];
    __syncthreads();
    if (q < K.dl) {
      img = coef_mul(K.al, se[lc]);
      for (int j = 0; j < q; ++j) img = coef_mul(K.pc, img);
    }
    __syncthreads();  // before the next tile's forward ends
  }
  cn_chunk_finish<Coef, CL>(img, K, y, v);
}

}  // namespace
}  // namespace dgpe
