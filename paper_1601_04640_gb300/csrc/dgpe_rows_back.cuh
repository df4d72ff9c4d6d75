// dgpe_rows_back.cuh -- C2R transform, exponential and Crank-Nicolson solve
// along x of the FP32 bulk (compiled in dgpe_rows_real.cu for the real
// coefficients of imaginary time, in dgpe_rows_cplx.cu for real time).
#pragma once

#include "dgpe_rows.cuh"

namespace dgpe {
namespace {

// Staged state of a warp: chunk i (CL points of one row) at i CL EB bytes, in
// pieces of 16 bytes.  Chunks of 128 and 64 bytes (power-of-two lengths) are
// copied through a tensor map whose swizzle spreads the pieces of eight
// neighbouring chunks over the banks; the other lengths' strides (96, 160, 48,
// 80 bytes) need no more than two wavefronts per access and are copied as
// they are.
template <int CL, bool REAL> struct RowStage {
  static constexpr int EB = REAL ? 4 : 8, CB = CL * EB, NP = CB / 16;
  static constexpr bool SWZ = CL == 16;
  static __device__ __forceinline__ int off(int i, int c) {
    if constexpr (SWZ && !REAL) return i * CB + ((c ^ (i & 7)) << 4);
    else if constexpr (SWZ) return i * CB + ((c ^ ((i >> 1) & 3)) << 4);
    else return i * CB + (c << 4);
  }
};

// The exponential of a lane's CL sites.  A lane whose exponents all lie within
// 1/8 takes the short Taylor series (sin_cosm1, fexpm1), within 2 (1) the
// series below, whose first omitted terms are below 2e-10 (3e-9) relative;
// beyond that the library functions, out of line.
__device__ __forceinline__ float2 phase_update(float2 v, float sn, float cm1) {  // v e^{-i th}, as in nonlinear_factor
  return make_float2(v.x + (v.x * cm1 + v.y * sn), v.y + (v.y * cm1 - v.x * sn));
}
template <int CL> __device__ __forceinline__ void exp_real_time(float2 (&v)[CL], const float (&th)[CL]) {
  float m = 0.0f;
#pragma unroll
  for (int i = 0; i < CL; ++i) m = fabsf(th[i]) <= m ? m : fabsf(th[i]);  // a NaN gives NaN on any path
  if (m <= 0.125f) {
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      const float x = th[i], x2 = x * x;
      const float ps = (1.0f / 120.0f) * x2 + (-1.0f / 6.0f), pc = ((-1.0f / 720.0f) * x2 + (1.0f / 24.0f)) * x2 - 0.5f;
      v[i] = phase_update(v[i], x + (x * x2) * ps, x2 * pc);
    }
  } else if (m <= 2.0f) {
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      const float x = th[i], x2 = x * x;
      float ps = -1.0f / 1307674368000.0f, pc = 1.0f / 20922789888000.0f;  // 15!, 16!
      ps = fmaf(ps, x2, 1.0f / 6227020800.0f);
      ps = fmaf(ps, x2, -1.0f / 39916800.0f);
      ps = fmaf(ps, x2, 1.0f / 362880.0f);
      ps = fmaf(ps, x2, -1.0f / 5040.0f);
      ps = fmaf(ps, x2, 1.0f / 120.0f);
      ps = fmaf(ps, x2, -1.0f / 6.0f);
      pc = fmaf(pc, x2, -1.0f / 87178291200.0f);
      pc = fmaf(pc, x2, 1.0f / 479001600.0f);
      pc = fmaf(pc, x2, -1.0f / 3628800.0f);
      pc = fmaf(pc, x2, 1.0f / 40320.0f);
      pc = fmaf(pc, x2, -1.0f / 720.0f);
      pc = fmaf(pc, x2, 1.0f / 24.0f);
      pc = fmaf(pc, x2, -0.5f);
      v[i] = phase_update(v[i], fmaf(x * x2, ps, x), x2 * pc);
    }
  } else {
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      const float2 e = sincos_call(th[i] * 0.5f);
      v[i] = phase_update(v[i], 2.0f * e.x * e.y, -2.0f * e.x * e.x);
    }
  }
}
// f = e^{-th} - 1 in place of th
template <int CL> __device__ __forceinline__ void exp_imag_time(float (&th)[CL]) {
  float m = 0.0f;
#pragma unroll
  for (int i = 0; i < CL; ++i) m = fabsf(th[i]) <= m ? m : fabsf(th[i]);
  if (m <= 0.125f) {
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      const float a = -th[i];
      float p = 1.0f / 720.0f;
      p = fmaf(p, a, 1.0f / 120.0f);
      p = fmaf(p, a, 1.0f / 24.0f);
      p = fmaf(p, a, 1.0f / 6.0f);
      p = fmaf(p, a, 0.5f);
      th[i] = fmaf(a * a, p, a);
    }
  } else if (m <= 1.0f) {
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      const float a = -th[i];
      float p = 1.0f / 39916800.0f;
      p = fmaf(p, a, 1.0f / 3628800.0f);
      p = fmaf(p, a, 1.0f / 362880.0f);
      p = fmaf(p, a, 1.0f / 40320.0f);
      p = fmaf(p, a, 1.0f / 5040.0f);
      p = fmaf(p, a, 1.0f / 720.0f);
      p = fmaf(p, a, 1.0f / 120.0f);
      p = fmaf(p, a, 1.0f / 24.0f);
      p = fmaf(p, a, 1.0f / 6.0f);
      p = fmaf(p, a, 0.5f);
      th[i] = fmaf(a * a, p, a);
    }
  } else {
#pragma unroll
    for (int i = 0; i < CL; ++i) th[i] = expm1_call(-th[i]);
  }
}

// Crank-Nicolson along x: CL consecutive points of a row per lane, TPL lanes
// per row.
template <typename Coef, int CL, int TPL>
__device__ __forceinline__ void row_solve(float2 (&v)[CL], int q, const CnConst<Coef> &K) {
  float2 y[CL];
  float2 prev = shfl_up(v[CL - 1], 1, TPL), next = shfl_down(v[0], 1, TPL);
  if (q == 0) prev = make_float2(0.0f, 0.0f);
  if (q == TPL - 1) next = make_float2(0.0f, 0.0f);
  const float2 e = cn_chunk_forward<Coef, CL>(v, prev, next, K, y);
  float2 in = make_float2(0.0f, 0.0f);
  for (int d = K.dl; d > 0; --d) {
    const float2 t = shfl_up(e, d, TPL);
    if (q >= d) in = coef_fma(K.pc, in, t);
  }
  const float2 g = cn_chunk_backward<Coef, CL>(in, K, y);
  in = make_float2(0.0f, 0.0f);
  for (int d = K.dl; d > 0; --d) {
    const float2 t = shfl_down(g, d, TPL);
    if (q + d < TPL) in = coef_fma(K.pc, in, t);
  }
  cn_chunk_inflow<Coef, CL>(in, K, y);
  // u_0 of the line is the first chunk's y[0]
  float2 img = make_float2(__shfl_sync(0xffffffffu, y[0].x, 0, TPL), __shfl_sync(0xffffffffu, y[0].y, 0, TPL));
  img = coef_mul(K.al, img);
  for (int d = 0; d < K.dl; ++d)
    if (d < q) img = coef_mul(K.pc, img);
  if (q >= K.dl) img = make_float2(0.0f, 0.0f);
  cn_chunk_finish<Coef, CL>(img, K, y, v);
}
// C2R of a pair of rows from their staged half spectra: Phi_d of both at the
// lane's CL consecutive points.  xa, xb: the rows' spectra (in z or elsewhere).
template <int N> __device__ __forceinline__ void row_c2r(float2 *z, const float2 *xa, const float2 *xb, int q) {
  constexpr int CL = Row<N>::CL, TPL = Row<N>::TPL;
  float2 v[CL];
#pragma unroll
  for (int r = 0; r < CL; ++r) {
    // Z = X0 + i X1 of the two rows, extended by X(N - k) = conj X(k)
    const int a = q + r * TPL;
    const bool up = r > CL / 2 || (r == CL / 2 && q > 0);  // a > N / 2
    float2 x = xa[up ? N - a : a], y = xb[up ? N - a : a];
    if (up) { x.y = -x.y; y.y = -y.y; }
    if ((r == 0 || r == CL / 2) && q == 0) { x.y = 0.0f; y.y = 0.0f; }  // real ends
    v[r] = make_float2(x.x - y.y, x.y + y.x);
  }
  row_first<N, true>(z, v);
}

template <int N, int MODE> struct BackCfg {
  typedef Row<N> C;
  static constexpr bool REAL = MODE == ROWS_REAL, PSI = MODE != ROWS_PHI;
  typedef RowStage<C::CL, REAL> G;
  // 2 NL rows = 64 chunks
  typedef RowSmem<N, PSI ? 64 * G::CB : 0> S;
};

// Bound by HBM and latency: 66 us at 256^3 complex (5.0 TB/s of the 6.7 of a
// copy; the block-wide form with shared tables took 110), 243 us at 512 x 512 x
// 256 (410), 47 us at 256^3 with a real state (159), 27 us at 192 x 160 x 128
// (78).  A lane holds CL points of a row: the transform is then two or three
// stages, the solve needs no table, and 16 warps per SM are what the staged
// tiles (12.5 KB a warp) and 128 registers leave.  The two rows share one copy
// of the code: unrolled twice, with the library's sincosf inlined at every site,
// the warps waited for instructions (98 us).
template <typename Coef, int N, int MODE>
__global__ void __launch_bounds__(32 * kRowWarps, Row<N>::BLOCKS)
    k_rows_back(const __grid_constant__ CUtensorMap tm, const __grid_constant__ RowArgs A,
                const __grid_constant__ CnConst<Coef> K, int ntiles) {
  typedef Row<N> C;
  typedef BackCfg<N, MODE> B;
  typedef typename B::S S;
  typedef typename B::G G;
  extern __shared__ __align__(1024) unsigned char smrows[];
  constexpr int CL = C::CL, TPL = C::TPL, NL = C::NL;
  constexpr bool EXP = MODE == ROWS_STEP || MODE == ROWS_EXP || MODE == ROWS_REAL;
  constexpr bool CN = MODE == ROWS_STEP || MODE == ROWS_CN || MODE == ROWS_REAL;
  constexpr bool RT = std::is_same<Coef, float2>::value;  // real time
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane / TPL, q = lane % TPL;
  unsigned char *const stage = smrows + w * S::psi;
  float2 *const z = reinterpret_cast<float2 *>(smrows + S::off_z + w * S::z);
  float2 *const tws = reinterpret_cast<float2 *>(smrows + S::off_tw);
  float4 *const vxs = reinterpret_cast<float4 *>(smrows + S::off_vx);  // V_x of lane q: [CL / 4][TPL]
  unsigned long long *const bz = reinterpret_cast<unsigned long long *>(smrows + S::off_bar) + 2 * w, *const bp = bz + 1;
  const bool dip = MODE != ROWS_CN && A.has_dip != 0;

  // lane i copies row i of the spectrum (even rows, then odd rows)
  auto issue_spec = [&](int tile) {
    const int r0 = tile * C::ROWS, nr = min(C::ROWS, A.nrows - r0);
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_expect_tx(bz, (unsigned)(nr * C::PX * 8));
    __syncwarp();
    if (lane < nr)
      bulk_g2s(z + ((lane >> 1) + (lane & 1) * NL) * C::PS, A.spec + (size_t)(r0 + lane) * C::PX, C::PX * 8, bz);
  };
  auto issue_psi = [&](int tile) {  // lane 0
    const int r0 = tile * C::ROWS, nr = min(C::ROWS, A.nrows - r0);
    if constexpr (G::SWZ) {
      mbar_expect_tx(bp, 64 * G::CB);  // rows beyond the last load as zeros
      tma_load_2d(stage, &tm, 0, r0 * TPL, bp);
    } else {
      mbar_expect_tx(bp, (unsigned)(nr * N * G::EB));
      bulk_g2s(stage, reinterpret_cast<const unsigned char *>(A.psi) + (size_t)r0 * N * G::EB, nr * N * G::EB, bp);
    }
  };
  auto store_psi = [&](int tile) {  // lane 0
    const int r0 = tile * C::ROWS, nr = min(C::ROWS, A.nrows - r0);
    if constexpr (G::SWZ) tma_store_2d(&tm, 0, r0 * TPL, stage);
    else bulk_s2g(reinterpret_cast<unsigned char *>(A.psi) + (size_t)r0 * N * G::EB, stage, nr * N * G::EB);
    bulk_commit();
  };

  if (lane == 0) {
    mbar_init(bz, 1);
    mbar_init(bp, 1);
  }
  __syncwarp();
  // tiles are dealt out block by block, so few tiles spread over the SMs
  int tile = w * gridDim.x + blockIdx.x;
  const int nw = gridDim.x * kRowWarps;
  row_twiddles<N>(tws, A.tw);
  if constexpr (EXP)
    for (int i = threadIdx.x; i < N; i += blockDim.x)
      reinterpret_cast<float *>(vxs)[((i % CL) / 4 * TPL + i / CL) * 4 + i % 4] = A.vx[i];
  pdl_wait();
  if (tile < ntiles) {
    if (dip) issue_spec(tile);
    if (B::PSI && lane == 0) issue_psi(tile);
  }
  float dts = 0.0f, gdt = 0.0f, gdddt = 0.0f, sc = 1.0f;
  if constexpr (EXP) {
    float *const s_k = reinterpret_cast<float *>(smrows + S::off_k);
    if (threadIdx.x == 0) {
      s_k[0] = (float)(trap_dts(A.prm, *A.step) * A.dtf);
      s_k[1] = (float)(A.prm[PRM_DT] * A.dtf * A.prm[PRM_G]);
      s_k[2] = (float)(A.prm[PRM_DT] * A.dtf * A.prm[PRM_GDD]);
      s_k[3] = (float)A.prm[PRM_SC];
    }
    __syncthreads();
    dts = s_k[0], gdt = s_k[1], gdddt = s_k[2];
    if (!RT) sc = s_k[3];  // real time: the lazy norm scale is 1
  } else {
    __syncthreads();
  }

  unsigned ph = 0;
  for (bool first = true; tile < ntiles; tile += nw, ph ^= 1u, first = false) {
    const int row0 = tile * C::ROWS;
    float2 f[CL];  // Phi_d of the lane's points, both rows
    if (dip) {
      bool ok = mbar_wait_bounded(bz, ph, DGPE_WAIT_LIMIT);
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) {
          if (B::PSI) {
            bulk_wait_all();
            if (first) mbar_wait_bounded(bp, ph, DGPE_WAIT_LIMIT);
          }
          const_cast<double *>(A.prm)[PRM_TIMEOUT] = 1.0;
        }
        return;
      }
      const float2 *const xa = z + l * C::PS, *const xb = xa + NL * C::PS;
      row_c2r<N>(z, xa, xb, q);
      // the state's next tile, once the store of its last one has been read
      if (B::PSI && !first && lane == 0) {
        bulk_wait_read_all();
        issue_psi(tile);
      }
      row_stages<N, CL, 0, true>(z, tws);
      if constexpr (MODE == ROWS_PHI) {
#pragma unroll
        for (int i = 0; i < CL; ++i) {
          const unsigned idx = lane + 32 * i, ll = idx / N, a = idx % N;
          const int ra = row0 + 2 * (int)ll;
          const float2 p = z[ll * C::SL + a + a / CL];
          if (ra < A.nrows) {
            A.phi_out[(size_t)ra * N + a] = p.x;
            A.phi_out[(size_t)(ra + 1) * N + a] = p.y;
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < CL; ++i) f[i] = z[l * C::SL + q * (CL + 1) + i];
      }
      if (tile + nw < ntiles) issue_spec(tile + nw);
    } else {
      if (B::PSI && !first && lane == 0) {
        bulk_wait_read_all();
        issue_psi(tile);
      }
#pragma unroll
      for (int i = 0; i < CL; ++i) f[i] = make_float2(0.0f, 0.0f);
    }
    if constexpr (B::PSI) {
      const bool ok = mbar_wait_bounded(bp, ph, DGPE_WAIT_LIMIT);
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) {
          if (dip && tile + nw < ntiles) mbar_wait_bounded(bz, ph ^ 1u, DGPE_WAIT_LIMIT);
          const_cast<double *>(A.prm)[PRM_TIMEOUT] = 1.0;
        }
        return;
      }
      if constexpr (MODE == ROWS_REAL) {
        // the pair's rows are the parts of one complex line: each part scaled
        // by its own row's factor, one solve with the real coefficients
        const int ia = 2 * l * TPL + q, ib = ia + TPL, ra = row0 + 2 * l;
        float2 v[CL];
#pragma unroll
        for (int c = 0; c < G::NP; ++c) {
          const float4 a = *reinterpret_cast<const float4 *>(stage + G::off(ia, c));
          const float4 b = *reinterpret_cast<const float4 *>(stage + G::off(ib, c));
          v[4 * c] = make_float2(a.x, b.x);
          v[4 * c + 1] = make_float2(a.y, b.y);
          v[4 * c + 2] = make_float2(a.z, b.z);
          v[4 * c + 3] = make_float2(a.w, b.w);
        }
        const int rc = min(ra, A.nrows - 2);
        const float va = A.vy[rc % A.ny] + A.vz[rc / A.ny], vb = A.vy[(rc + 1) % A.ny] + A.vz[(rc + 1) / A.ny];
        float ta[CL], tb[CL];
#pragma unroll
        for (int c = 0; c < CL / 4; ++c) {
          const float4 x4 = vxs[c * TPL + q];
          const float xs[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
          for (int i = 4 * c; i < 4 * c + 4; ++i) {
            v[i].x *= sc;
            v[i].y *= sc;
            ta[i] = dts * (xs[i - 4 * c] + va) + gdt * (v[i].x * v[i].x) + gdddt * f[i].x;
            tb[i] = dts * (xs[i - 4 * c] + vb) + gdt * (v[i].y * v[i].y) + gdddt * f[i].y;
          }
        }
        exp_imag_time<CL>(ta);
        exp_imag_time<CL>(tb);
#pragma unroll
        for (int i = 0; i < CL; ++i) v[i] = make_float2(v[i].x + v[i].x * ta[i], v[i].y + v[i].y * tb[i]);
        row_solve<Coef, CL, TPL>(v, q, K);
#pragma unroll
        for (int c = 0; c < G::NP; ++c) {
          *reinterpret_cast<float4 *>(stage + G::off(ia, c)) =
              make_float4(v[4 * c].x, v[4 * c + 1].x, v[4 * c + 2].x, v[4 * c + 3].x);
          *reinterpret_cast<float4 *>(stage + G::off(ib, c)) =
              make_float4(v[4 * c].y, v[4 * c + 1].y, v[4 * c + 2].y, v[4 * c + 3].y);
        }
      } else {
        // the pair's rows one after the other, one copy of the code
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const int ic = (2 * l + h) * TPL + q;
          float2 v[CL];
#pragma unroll
          for (int c = 0; c < G::NP; ++c) {
            const float4 a = *reinterpret_cast<const float4 *>(stage + G::off(ic, c));
            v[2 * c] = make_float2(a.x, a.y);
            v[2 * c + 1] = make_float2(a.z, a.w);
          }
          if constexpr (EXP) {
            const int row = min(row0 + 2 * l + h, A.nrows - 1);
            const float vr = A.vy[row % A.ny] + A.vz[row / A.ny];
            float th[CL];
#pragma unroll
            for (int c = 0; c < CL / 4; ++c) {
              const float4 x4 = vxs[c * TPL + q];
              const float xs[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
              for (int i = 4 * c; i < 4 * c + 4; ++i) {
                if (!RT) v[i] = cscale(v[i], sc);
                th[i] = dts * (xs[i - 4 * c] + vr) + gdt * (v[i].x * v[i].x + v[i].y * v[i].y) + gdddt * f[i].x;
                f[i].x = f[i].y;  // the second row's Phi_d
              }
            }
            if constexpr (RT) {
              exp_real_time<CL>(v, th);
            } else {
              exp_imag_time<CL>(th);
#pragma unroll
              for (int i = 0; i < CL; ++i) v[i] = make_float2(v[i].x + v[i].x * th[i], v[i].y + v[i].y * th[i]);
            }
          }
          if constexpr (CN) row_solve<Coef, CL, TPL>(v, q, K);
#pragma unroll
          for (int c = 0; c < G::NP; ++c)
            *reinterpret_cast<float4 *>(stage + G::off(ic, c)) =
                make_float4(v[2 * c].x, v[2 * c].y, v[2 * c + 1].x, v[2 * c + 1].y);
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) store_psi(tile);
    }
  }
  if (B::PSI && lane == 0) bulk_wait_all();
}

// f(kernel, shared bytes, rows per tile) of the length's kernel
template <typename Coef, int MODE, class F> cudaError_t with_back(int n, F &&f) {
  return with_row_length(n, [&](auto Nc) {
    constexpr int N = decltype(Nc)::value;
    return f(k_rows_back<Coef, N, MODE>, (int)BackCfg<N, MODE>::S::total, (int)Row<N>::ROWS);
  });
}
template <typename Coef, int MODE>
cudaError_t back_launch(const RowArgs &A, const CUtensorMap &tm, const CnConst<Coef> &K, int grid, cudaStream_t s) {
  return with_back<Coef, MODE>(A.n, [&](auto k, int smem, int rows) {
    return launch_pdl(A.early != 0, k, dim3(grid), 32 * kRowWarps, smem, s, tm, A, K, (A.nrows + rows - 1) / rows);
  });
}
template <typename Coef, int MODE> cudaError_t back_grid(int n, int nrows, int nsm, int *grid) {
  return with_back<Coef, MODE>(n, [&](auto k, int smem, int rows) {
    return row_grid(k, smem, (nrows + rows - 1) / rows, nsm, grid);
  });
}

}  // namespace
}  // namespace dgpe
