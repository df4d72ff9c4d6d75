// dgpe_rows.cuh -- x-row passes of the FP32 bulk, one warp per tile: the
// density and its R2C transform along x, and the C2R transform, exponential
// and Crank-Nicolson solve along x (the paper's calcpsidd2, calcnu, calclux,
// "Summary of revisions").
//
// A warp owns NL pairs of neighbouring rows, N / CL lanes per pair and CL
// points of both rows per lane, and works through its tiles alone: the copies
// into its part of the shared memory complete on its own mbarriers, the
// exchanges of the transform go through that memory behind __syncwarp, and the
// chunks of the Crank-Nicolson solve exchange their ends by shuffles.  No
// barrier joins the warps of a block, so their waits, transforms and solves
// overlap each other.
#pragma once

#include "dgpe_lines.cuh"

namespace dgpe {
namespace {

constexpr int kRowWarps = 4;  // warps per block

constexpr int rows_cl(int n) { return n % 3 == 0 ? 12 : n % 5 == 0 ? 20 : 16; }
// Smallest even pitch >= m (units of 8 bytes) at which `lanes` consecutive
// elements of 16 / lanes neighbouring lines lie on different banks.
constexpr int row_pitch(int m, int lanes) {
  int p = (m + 1) & ~1;
  if (lanes < 16)
    while (p % (2 * lanes) != lanes) p += 2;
  return p;
}
template <int N_> struct Row {
  static constexpr int N = N_, CL = rows_cl(N), TPL = N / CL, NL = 32 / TPL, ROWS = 2 * NL;
  static constexpr int BLOCKS = CL == 20 ? 3 : 4;   // per SM, by shared memory
  static constexpr int PX = N / 2 + 2;              // the spectrum's row pitch
  static constexpr int PS = row_pitch(PX, TPL);     // ... of its staged rows
  static constexpr int SL = N + N / CL;             // transform line: one pad per CL elements
  static constexpr int PR = row_pitch(N, TPL);      // staged complex rows (density)
  static constexpr int PRR = TPL < 4 ? N + 4 : 2 * row_pitch(N / 2, TPL / 2);  // staged real rows, floats
  static constexpr int ZEL = (ROWS * PS > NL * SL ? ROWS * PS : NL * SL);
  static_assert(TPL >= 2 && TPL <= 32 && (TPL & (TPL - 1)) == 0 && N == CL * TPL, "line length");
};

// ------------------------------------------------------------- transform
// Radices: CL first (one butterfly per lane), then the largest of 16 (CL 16),
// 8, 4, 2 that divides what is left; a lane always holds CL elements.
template <int CL> constexpr int row_radix(int left) {
  if (CL == 16 && left % 16 == 0) return 16;
  if (CL == 16 && left % 8 == 0) return 8;
  return left % 4 == 0 ? 4 : 2;
}
// Twiddles of the later stages, w_{NS RAD}^{k r} at offset + (r - 1) NS + k:
// the lanes of a stage read consecutive k.  Fewer than N in all.
template <int N> __device__ __forceinline__ void row_twiddles(float2 *dst, const float2 *__restrict__ tw) {
  typedef Row<N> C;
  int off = 0, ns = C::CL;
  while (ns < N) {
    const int rad = row_radix<C::CL>(N / ns), str = N / (ns * rad), cnt = (rad - 1) * ns;
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) dst[off + i] = tw[(i % ns) * (i / ns + 1) * str];
    off += cnt;
    ns *= rad;
  }
}
template <int N, int NS, int OFF, bool INV> __device__ __forceinline__ void row_stages(float2 *z, const float2 *tws) {
  typedef Row<N> C;
  if constexpr (NS < N) {
    constexpr int RAD = row_radix<C::CL>(N / NS), NB = C::CL / RAD, NBL = N / RAD, CL = C::CL;
    static_assert(C::CL % RAD == 0 && NBL % CL == 0 && NS % CL == 0, "stage");
    const int lane = threadIdx.x & 31;
    float2 v[CL];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const unsigned b = lane + 32 * i, l = b / NBL, j = b % NBL, k = j % NS;
      const float2 *const p = z + l * C::SL + j + j / CL;
      float2 *u = v + i * RAD;
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        u[r] = p[r * (NBL + NBL / CL)];
        if (r > 0) {
          const float2 w = tws[OFF + (r - 1) * NS + k];
          u[r] = INV ? cmulconj(u[r], w) : cmul(u[r], w);
        }
      }
      dft<RAD, INV>(u);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const unsigned b = lane + 32 * i, l = b / NBL, j = b % NBL, base = (j / NS) * NS * RAD + j % NS;
      float2 *const p = z + l * C::SL + base + base / CL;
#pragma unroll
      for (int r = 0; r < RAD; ++r) p[r * (NS + NS / CL)] = v[i * RAD + r];
    }
    __syncwarp();
    row_stages<N, NS * RAD, OFF + (RAD - 1) * NS, INV>(z, tws);
  }
}
// First stage: lane (l, j) transforms elements j + r TPL of line l, v[r].
template <int N, bool INV> __device__ __forceinline__ void row_first(float2 *z, float2 *v) {
  typedef Row<N> C;
  const int lane = threadIdx.x & 31, l = lane / C::TPL, j = lane % C::TPL;
  dft<C::CL, INV>(v);
  __syncwarp();  // z may hold what the lanes read v from
  float2 *const p = z + l * C::SL + j * (C::CL + 1);
#pragma unroll
  for (int r = 0; r < C::CL; ++r) p[r] = v[r];
  __syncwarp();
}

__device__ __forceinline__ void bulk_s2g(void *dst, const void *src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void tma_load_2d(void *dst, const void *tmap, int c0, int c1, unsigned long long *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
          smem_u32(dst)),
      "l"(tmap), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_store_2d(const void *tmap, int c0, int c1, const void *src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];\n" ::"l"(tmap), "r"(c0),
               "r"(c1), "r"(smem_u32(src))
               : "memory");
}

// Shared memory of a block: the warps' psi tiles, their transform lines (also
// the staged spectrum rows), twiddles, V_x, the mbarriers, four
// scalars.
template <int N, int PSI_BYTES> struct RowSmem {
  static constexpr int psi = (PSI_BYTES + 127) & ~127, z = (Row<N>::ZEL * 8 + 15) & ~15;
  static constexpr int off_z = kRowWarps * psi, off_tw = off_z + kRowWarps * z, off_vx = off_tw + 8 * N;
  static constexpr int off_bar = off_vx + 4 * N, off_k = off_bar + kRowWarps * 16, total = off_k + 16;
};

template <class F> cudaError_t with_row_length(int n, F &&f) {
  switch (n) {
#define DGPE_ROW(N) case N: return f(std::integral_constant<int, N>{});
    DGPE_ROW(32) DGPE_ROW(64) DGPE_ROW(128) DGPE_ROW(256) DGPE_ROW(512)
    DGPE_ROW(48) DGPE_ROW(96) DGPE_ROW(192) DGPE_ROW(384)
    DGPE_ROW(40) DGPE_ROW(80) DGPE_ROW(160) DGPE_ROW(320)
#undef DGPE_ROW
    default: return cudaErrorInvalidValue;
  }
}
// Persistent grid: as many blocks as fit, at most one per tile (the tiles are
// dealt out to the blocks first, then to their warps).
template <class K> cudaError_t row_grid(K kernel, int smem, int ntiles, int nsm, int *grid) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 32 * kRowWarps, smem);
  if (e == cudaSuccess && occ < 1) e = cudaErrorLaunchOutOfResources;
  if (e == cudaSuccess) *grid = ntiles < nsm * occ ? ntiles : nsm * occ;
  return e;
}

}  // namespace
}  // namespace dgpe
