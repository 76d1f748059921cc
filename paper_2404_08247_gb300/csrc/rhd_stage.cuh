// rhd_stage.cuh -- the stage kernel of one grid and its launch, shared by
// the PLM unit (rhd_stage.cu) and the PPM unit (rhd_stage_ppm.cu), which
// compile in parallel.
#pragma once

#include <type_traits>

#include "rhd_tile.cuh"

namespace rhd {

// resident blocks per SM the kernels are compiled for: 128 registers a thread
template <class T>
constexpr int kMinBlocks = 512 / T::NT;

template <int STAGE, int NDIM, typename R, bool GEN, bool PPM, bool SMALL>
__global__ void __launch_bounds__(TileOf<NDIM, PPM, SMALL>::NT,
                                  kMinBlocks<TileOf<NDIM, PPM, SMALL>>)
    stage_kernel(const StageArgs A) {
  using T = TileOf<NDIM, PPM, SMALL>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_skip;
  if (threadIdx.x == 0) s_skip = (A.st->fail_key != ~0ull) ? 1 : 0;
  __syncthreads();
  if (s_skip) return;  // a previous launch of this batch failed
  TileStats ts;
  const int x0 = blockIdx.x * T::TX + (NDIM == 1 ? A.lo : 0);
  const int y0 = blockIdx.y * T::TY + (NDIM == 2 ? A.lo : 0);
  int k0 = 0, k1 = 1;
  if (NDIM == 3) block_planes(blockIdx.z, A.lo, A.hi, A.lz, k0, k1);
  stage_tile<STAGE, T, R, GEN>(A, x0, y0, k0, k1, smem_raw, ts);
  flush_stats<T::NT>(A.st, ts);
}

// The tile and the planes per block of a stage over a grid (launches over parts
// of it, which run side by side, take the whole grid's, and where a part's 8-plane
// rows are an odd number its last blocks march 8 planes of 16).  Both candidates
// (the large tile; the small one, whose faces take more warp rounds a cell)
// and 1 to 16 planes a block (a block adds a z face a column and its ghost
// planes' loads) are priced, and the cheapest is taken.  Prices are FP64
// instructions a warp: a face, a z face and a cell's slopes, update and solve.
// The busiest SM (of 152) issues its instructions at one in 16 cycles, slowed by
// (1 + 6/w) when w warps are resident: 73 % of the pipe with 16 warps, 50 to 57 %
// with 8, 11 to 14 % with one, as measured.  w counts the 16 warps that registers
// allow; shared memory holds the small 3-D tiles to fewer (FP64 PLM 14, PPM 10,
// mixed PPM 12), which the price leaves out.  Against the large tile with 8 planes
// a block everywhere: a 40 x 37 x 33 box, five steps, 5.3 -> 2.2 ms; a 256-cell
// row, 50 steps, 4.6 -> 3.5 ms; 256^3, where both price 8 or 16 planes alike,
// unchanged; 48 boxes of 315 cells to 128 x 96 x 110 between 1 and 7 times as
// fast, but for three that it prices wrongly (mixed precision, two steps):
// 96 x 80 x 72 takes 2.28 ms for 1.94, with PPM 2.81 for 2.15, and 64^3 with PPM
// 1.54 for 1.50.
struct TilePlan {
  bool small;
  int lz;
};

inline TilePlan plan_tiles(const Geometry& g, bool mixed, bool ppm, bool allow_small) {
  constexpr int kSMs = 152;
  const double face = mixed ? 12.0 : ppm ? 100.0 : 60.0, cell = mixed ? 190.0 : 210.0;
  TilePlan best = {false, 1};
  double tbest = 0.0;
  for (int small = 0; small < (allow_small ? 2 : 1); ++small) {
    const int tx = g.ndim == 1 ? (small ? 32 : 256) : small ? 16 : 32;
    const int ty = g.ndim == 1 ? 1 : small ? 4 : 8;
    const int nw = tx * ty / 32, resident = 16 / nw;
    const int rx = ((tx + 1) * ty + 31) / 32, ry = g.ndim >= 2 ? (tx * (ty + 1) + 31) / 32 : 0;
    for (int lz = g.ndim == 3 ? 16 : 1; lz >= 1; lz /= 2) {
      long long nb[3] = {1, 1, 1};
      for (int d = 0; d < g.ndim; ++d) {
        const int w = d == 0 ? tx : d == 1 ? ty : lz;
        nb[d] = (g.n[d] + w - 1) / w;
      }
      if (nb[1] > 65535 || nb[2] > 65535) continue;
      const double z = g.ndim == 3 ? face : 0.0;
      const double plane = face * (rx + ry) + (cell + z) * nw, start = 2.0 * z * nw;
      const long long per_sm = (nb[0] * nb[1] * nb[2] + kSMs - 1) / kSMs;
      const double warps = nw * (double)(per_sm < resident ? per_sm : resident);
      const double t = per_sm * (lz * plane + start) * (1.0 + 6.0 / warps);
      if (tbest == 0.0 || t < tbest) {
        tbest = t;
        best.small = small != 0;
        best.lz = lz;
      }
    }
  }
  return best;
}

template <int STAGE, int NDIM, typename R, bool GEN, bool PPM, bool SMALL>
static cudaError_t launch_tile(const StageArgs& A, cudaStream_t s) {
  using T = TileOf<NDIM, PPM, SMALL>;
  using S = SmemT<T, R>;
  // opt in to more than 48 KiB of dynamic shared memory (idempotent)
  cudaError_t e = cudaFuncSetAttribute(stage_kernel<STAGE, NDIM, R, GEN, PPM, SMALL>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)S::BYTES);
  if (e != cudaSuccess) return e;
  unsigned nb[3] = {1, 1, 1};
  const int w[3] = {T::TX, T::TY, A.lz};
  for (int d = 0; d < NDIM; ++d)
    nb[d] = (unsigned)(((d == NDIM - 1 ? A.hi - A.lo : A.g.n[d]) + w[d] - 1) / w[d]);
  stage_kernel<STAGE, NDIM, R, GEN, PPM, SMALL>
      <<<dim3(nb[0], nb[1], nb[2]), T::NT, S::BYTES, s>>>(A);
  return cudaGetLastError();
}

// The tile rows [b0, b1) of the slowest axis (b1 < 0: all of them).
template <int STAGE, int NDIM, typename R, bool GEN, bool PPM>
static cudaError_t launch_nd(const StageArgs& A, cudaStream_t s, int b0, int b1) {
  constexpr bool MIXED = sizeof(R) == sizeof(float);
  constexpr int W = kRowCells[NDIM];
  const int n = A.g.n[NDIM - 1], rows = (n + W - 1) / W;
  if (b1 < 0 || b1 > rows) b1 = rows;
  if (b0 < 0 || b0 >= b1) return cudaErrorInvalidValue;
  StageArgs a = A;
  a.lo = b0 * W;
  a.hi = b1 * W < n ? b1 * W : n;
  const TilePlan P = plan_tiles(A.g, MIXED, PPM, STAGE != 0);
  a.lz = P.lz;
  flux_weights(A.g, A.ph, MIXED, STAGE == 0 ? 1.0 : STAGE == 1 ? A.dt : 0.5 * A.dt, a.wE, a.wF);
  if constexpr (STAGE != 0)
    if (P.small) return launch_tile<STAGE, NDIM, R, GEN, PPM, true>(a, s);
  return launch_tile<STAGE, NDIM, R, GEN, PPM, false>(a, s);
}

template <int STAGE, typename R, bool GEN, bool PPM>
static cudaError_t launch_prec(const StageArgs& A, cudaStream_t s, int b0, int b1) {
  switch (A.g.ndim) {
    case 1: return launch_nd<STAGE, 1, R, GEN, PPM>(A, s, b0, b1);
    case 2: return launch_nd<STAGE, 2, R, GEN, PPM>(A, s, b0, b1);
    default: return launch_nd<STAGE, 3, R, GEN, PPM>(A, s, b0, b1);
  }
}

}  // namespace rhd
