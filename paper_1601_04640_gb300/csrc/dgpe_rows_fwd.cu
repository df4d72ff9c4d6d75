// dgpe_rows_fwd.cu -- density and R2C transform along x of the FP32 bulk.
#include <algorithm>

#include "dgpe_rows.cuh"

namespace dgpe {
namespace {

template <int N, int SRC> struct FwdCfg {
  typedef Row<N> C;
  static constexpr int EB = SRC == 0 ? 8 : 4;                     // bytes per staged element
  static constexpr int PITCH = (SRC == 0 ? C::PR : C::PRR) * EB;  // bytes per staged row
  typedef RowSmem<N, C::ROWS * PITCH> S;
};

// Bound by HBM: 36 us at 256^3 (5.6 TB/s of the 6.7 of a copy; the block-wide
// pipelined form took 50), 140 us at 512 x 512 x 256 (187), 27 us for a real
// state (76), 15 us at 192 x 160 x 128 (42, runtime lengths).
// SRC 0: sc^2 |psi|^2, 1: the real field dens_in, 2: sc^2 psi^2 of a real
// state.  Lane i copies row i of the tile (even rows, then odd rows, at a
// pitch that spreads the lines over the banks); the rows are free again after
// the first stage, so the next tile's copies run behind the rest.
template <int N, int SRC>
__global__ void __launch_bounds__(32 * kRowWarps, Row<N>::BLOCKS) k_rows_fwd(const __grid_constant__ RowArgs A, int ntiles) {
  typedef Row<N> C;
  typedef FwdCfg<N, SRC> F;
  typedef typename F::S S;
  extern __shared__ __align__(1024) unsigned char smrows[];
  constexpr int CL = C::CL, TPL = C::TPL, NL = C::NL;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char *const rows = smrows + w * S::psi;
  float2 *const z = reinterpret_cast<float2 *>(smrows + S::off_z + w * S::z);
  float2 *const tws = reinterpret_cast<float2 *>(smrows + S::off_tw);
  unsigned long long *const bar = reinterpret_cast<unsigned long long *>(smrows + S::off_bar) + 2 * w;
  const unsigned char *const src =
      SRC == 1 ? reinterpret_cast<const unsigned char *>(A.dens_in) : reinterpret_cast<const unsigned char *>(A.psi);
  // from the last rows to the first: the y transform starts with the rows
  // written last, and so do the passes behind it (part of psi and of the
  // spectrum is then still in L2; with cn_y and the inverse y transform taken
  // backwards too a 256^3 step went from 267 to 254 us)
  auto first_row = [&](int tile) { return (ntiles - 1 - tile) * C::ROWS; };
  auto issue = [&](int tile) {
    const int r0 = first_row(tile), nr = min(C::ROWS, A.nrows - r0);
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_expect_tx(bar, (unsigned)(nr * N * F::EB));
    __syncwarp();
    if (lane < nr)
      bulk_g2s(rows + ((lane >> 1) + (lane & 1) * NL) * F::PITCH, src + (size_t)(r0 + lane) * N * F::EB, N * F::EB, bar);
  };
  if (lane == 0) mbar_init(bar, 1);
  __syncwarp();
  // tiles are dealt out block by block, so few tiles spread over the SMs
  int tile = w * gridDim.x + blockIdx.x;
  const int nw = gridDim.x * kRowWarps;
  row_twiddles<N>(tws, A.tw);
  pdl_wait();
  if (tile < ntiles) issue(tile);
  float sc2 = 1.0f;
  if (SRC != 1) {
    const float sc = (float)A.prm[PRM_SC];
    sc2 = sc * sc;
  }
  __syncthreads();
  const int l = lane / TPL, j = lane % TPL;
  for (unsigned ph = 0; tile < ntiles; tile += nw, ph ^= 1u) {
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar, ph, DGPE_WAIT_LIMIT))) {
      if (lane == 0) const_cast<double *>(A.prm)[PRM_TIMEOUT] = 1.0;
      return;
    }
    float2 v[CL];
    const unsigned char *const pa = rows + l * F::PITCH, *const pb = pa + NL * F::PITCH;
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      const int a = j + r * TPL;
      if constexpr (SRC == 0) {
        const float2 x = reinterpret_cast<const float2 *>(pa)[a], y = reinterpret_cast<const float2 *>(pb)[a];
        v[r] = make_float2(sc2 * (x.x * x.x + x.y * x.y), sc2 * (y.x * y.x + y.y * y.y));
      } else {
        const float x = reinterpret_cast<const float *>(pa)[a], y = reinterpret_cast<const float *>(pb)[a];
        v[r] = SRC == 1 ? make_float2(x, y) : make_float2(sc2 * (x * x), sc2 * (y * y));
      }
    }
    row_first<N, false>(z, v);
    if (tile + nw < ntiles) issue(tile + nw);
    row_stages<N, CL, 0, false>(z, tws);
    // two real lines were packed as Z = n0 + i n1
    const int row0 = first_row(tile);
    constexpr int NH = N / 2;
#pragma unroll
    for (int i = 0; i < NL * NH / 32; ++i) {
      const unsigned idx = lane + 32 * i, ll = idx / NH, k = idx % NH, km = k == 0 ? 0 : N - k;
      const int ra = row0 + 2 * (int)ll;
      const float2 Zk = z[ll * C::SL + k + k / CL], Zm = z[ll * C::SL + km + km / CL];
      if (ra < A.nrows) {
        float2 *const o = A.spec + (size_t)ra * C::PX + k;
        o[0] = make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y - Zm.y));
        o[C::PX] = make_float2(0.5f * (Zk.y + Zm.y), 0.5f * (Zm.x - Zk.x));
      }
    }
    if (lane < NL && row0 + 2 * lane < A.nrows) {
      const float2 Zk = z[lane * C::SL + NH + NH / CL];
      float2 *const o = A.spec + (size_t)(row0 + 2 * lane) * C::PX + NH;
      o[0] = make_float2(Zk.x, 0.0f);
      o[C::PX] = make_float2(Zk.y, 0.0f);
    }
    __syncwarp();
  }
}

template <int SRC, class F> cudaError_t with_fwd(int n, F &&f) {
  return with_row_length(n, [&](auto Nc) {
    constexpr int N = decltype(Nc)::value;
    return f(k_rows_fwd<N, SRC>, (int)FwdCfg<N, SRC>::S::total, (int)Row<N>::ROWS);
  });
}
template <class F> cudaError_t with_fwd(int n, int src, F &&f) {
  return src == 0 ? with_fwd<0>(n, f) : src == 1 ? with_fwd<1>(n, f) : with_fwd<2>(n, f);
}

}  // namespace

int rows_chunk(int n) { return rows_cl(n); }
int rows_per_tile(int n) { return 64 * rows_cl(n) / n; }
cudaError_t rows_fwd_launch(const RowArgs &A, int grid, cudaStream_t s) {
  return with_fwd(A.n, A.src, [&](auto k, int smem, int rows) {
    return launch_pdl(A.early != 0, k, dim3(grid), 32 * kRowWarps, smem, s, A, (A.nrows + rows - 1) / rows);
  });
}
cudaError_t rows_fwd_grid(int n, int nrows, int src, int nsm, int *grid) {
  return with_fwd(n, src, [&](auto k, int smem, int rows) {
    return row_grid(k, smem, (nrows + rows - 1) / rows, nsm, grid);
  });
}
}  // namespace dgpe
