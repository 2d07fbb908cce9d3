// Data term of the registration objective (Ploner et al., Eq. 2-8) and its
// gradient with respect to every A-scan displacement, fused in one kernel.
//
// For output A-scan (i, j) and each scan V in {X, Y}, the volume S^V is
// sampled along depth at (i + dx^V, j + dy^V, k + dz^V), k = 0..d-1, with
// the separable 4x4x4 Catmull-Rom interpolator (clamp-to-edge).  The
// residual R_k = I^X(k) - I^Y(k) (Eq. 2) goes through the loss (Eq. 4, or
// squared differences) and is summed over k (Eq. 3/5); the derivative of
// the sum with respect to the 6 displacement values of the A-scan is reduced
// over depth in the same pass.  The en-face angiography term (Eq. 6), the
// resampled validity (Eq. 7) and delta (Eq. 8) are per-A-scan scalars.
//
// Mapping: one warp per output A-scan; the sampling and its lane layout are
// described in sample.cuh.  A block's 4 warps take a tile of 2 x 2
// neighbouring A-scans (their 4 x 4 neighbourhoods overlap, which the L1 cache
// turns into hits).  At 64 registers 8 blocks (32 warps) run per SM: the
// kernel is bound by the L1 data pipe (80 % busy: volume loads, 5 wavefronts
// per 512 unaligned bytes, then shuffles and spills) and by the latency of its
// misses, so both more registers (fewer warps) and fewer (more spills) lose.
// 300 x 300 x 512, float32, data kernel alone: 48 / 56 / 64 / 72 / 80 registers
// 462 / 438 / 420 / 449 / 437 us, 8- and 16-warp blocks 423 and 437 us (529 us
// with depth-paired multiply-adds, spilled weights and a per-lane prologue and
// epilogue; bfloat16 535 -> 395 us; 64^3 19.2 -> 14.0 us).
//
// The per-A-scan prologue (coordinate split, 24 weight pairs, 16 offsets) is
// evaluated by a few lanes into a table in shared memory and the epilogue's 7
// sums go through one reduce-scatter: at 64 samples of depth these were 1162
// of a warp's 1958 instructions.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "data.cuh"
#include "sample.cuh"

namespace octmc {
namespace {

#ifndef OCTMC_DATA_MINB
#define OCTMC_DATA_MINB 8
#endif
#ifndef OCTMC_DTILE_X
#define OCTMC_DTILE_X 2
#endif
constexpr int kWarpsPerBlock = 4;
constexpr int kDTileX = OCTMC_DTILE_X;  // a block's A-scans as kDTileX x (kWarpsPerBlock / kDTileX)
constexpr int kDTileY = kWarpsPerBlock / kDTileX;

// A-scan of warp `warp` of direct block b: tiles of kDTileX x kDTileY.
__device__ __forceinline__ bool direct_ascan(const LevelDev& L, unsigned b, int warp, int* i, int* j) {
  const unsigned tiles_x = (unsigned)(L.w + kDTileX - 1) / kDTileX;
  *i = (int)(b % tiles_x) * kDTileX + warp % kDTileX;
  *j = (int)(b / tiles_x) * kDTileY + warp / kDTileX;
  return *i < L.w && *j < L.h;
}

__host__ __device__ inline int64_t direct_blocks(int w, int h) {
  return (int64_t)((w + kDTileX - 1) / kDTileX) * ((h + kDTileY - 1) / kDTileY);
}

template <typename T>
__global__ void __launch_bounds__(kWarpsPerBlock * kWarp, OCTMC_DATA_MINB)
data_kernel(const DataArgs A) {
  __shared__ VolTab tab[kWarpsPerBlock][2];
  const int warp = threadIdx.x >> 5;
  int i, j;
  if (!direct_ascan(A.L, blockIdx.x, warp, &i, &j)) return;  // warp-uniform
  data_ascan<T>(A, tab[warp], (int64_t)j * A.L.w + i, i, j, threadIdx.x & 31);
}

// Several problems ("slots") in one launch: grid (x, slots), block
// (x, s) takes tile x of slot s (blocks past a slot's last tile exit at
// once).  The slots' arguments travel in the kernel's parameter block and
// the slot index is uniform per block.  Each A-scan's result does not depend
// on which other slots are in the launch.
template <typename T>
__global__ void __launch_bounds__(kWarpsPerBlock * kWarp, OCTMC_DATA_MINB)
data_multi_kernel(const __grid_constant__ DataMulti M) {
  const DataArgs A = M.da[blockIdx.y];
  if ((int64_t)blockIdx.x >= direct_blocks(A.L.w, A.L.h)) return;
  __shared__ VolTab tab[kWarpsPerBlock][2];
  const int warp = threadIdx.x >> 5;
  int i, j;
  if (!direct_ascan(A.L, blockIdx.x, warp, &i, &j)) return;  // warp-uniform
  data_ascan<T>(A, tab[warp], (int64_t)j * A.L.w + i, i, j, threadIdx.x & 31);
}

// The data term of a field without transverse displacement: one warp per
// A-scan, two columns read once.  Bound by instruction issue: 115.9 M warp
// instructions fill 79 % of the issue slots of 300 x 300 x 512, float32, in
// 122 us cold (the general kernel: 420), while the 376.6 MB are 45 % of the HBM
// rate.  8-warp blocks of at most 64 registers keep 32 warps with two depth
// blocks of loads each in flight per SM.
constexpr int kColumnWarps = 8;
template <typename T>
__global__ void __launch_bounds__(kColumnWarps * kWarp, 4) column_kernel(const DataArgs A) {
  const int64_t p = (int64_t)blockIdx.x * kColumnWarps + (threadIdx.x >> 5);
  if (p >= (int64_t)A.L.w * A.L.h) return;  // warp-uniform
  data_column<T>(A, p, (int)(p % A.L.w), (int)(p / A.L.w), threadIdx.x & 31);
}

}  // namespace

cudaError_t launch_data_multi(const DataMulti& M, int dtype, cudaStream_t s) {
  if (M.nslots <= 0) return cudaSuccess;
  int64_t bx = 0;
  for (int k = 0; k < M.nslots; k++) bx = max(bx, direct_blocks(M.da[k].L.w, M.da[k].L.h));
  if (bx <= 0) return cudaSuccess;
  const dim3 g((unsigned)bx, (unsigned)M.nslots);
  if (dtype == OCTMC_BF16)
    data_multi_kernel<__nv_bfloat16><<<g, kWarpsPerBlock * kWarp, 0, s>>>(M);
  else if (dtype == OCTMC_F16)
    data_multi_kernel<__half><<<g, kWarpsPerBlock * kWarp, 0, s>>>(M);
  else
    data_multi_kernel<float><<<g, kWarpsPerBlock * kWarp, 0, s>>>(M);
  return cudaGetLastError();
}

cudaError_t launch_data(const DataArgs& a, cudaStream_t s) {
  const int64_t blocks = direct_blocks(a.L.w, a.L.h);
  if (blocks <= 0) return cudaSuccess;
  if (a.L.dtype == OCTMC_BF16)
    data_kernel<__nv_bfloat16><<<(unsigned)blocks, kWarpsPerBlock * kWarp, 0, s>>>(a);
  else if (a.L.dtype == OCTMC_F16)
    data_kernel<__half><<<(unsigned)blocks, kWarpsPerBlock * kWarp, 0, s>>>(a);
  else
    data_kernel<float><<<(unsigned)blocks, kWarpsPerBlock * kWarp, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_data_column(const DataArgs& a, cudaStream_t s) {
  const int64_t blocks = ((int64_t)a.L.w * a.L.h + kColumnWarps - 1) / kColumnWarps;
  if (blocks <= 0) return cudaSuccess;
  if (a.L.dtype == OCTMC_BF16)
    column_kernel<__nv_bfloat16><<<(unsigned)blocks, kColumnWarps * kWarp, 0, s>>>(a);
  else if (a.L.dtype == OCTMC_F16)
    column_kernel<__half><<<(unsigned)blocks, kColumnWarps * kWarp, 0, s>>>(a);
  else
    column_kernel<float><<<(unsigned)blocks, kColumnWarps * kWarp, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace octmc
