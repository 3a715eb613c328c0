// Visibility kernels (Sec. 5.1; App. A "Detecting Visible Triangles"): the launch
// wrappers of the stage bodies in raster.cuh and the launch sequence of one
// visibility pass.
#include <algorithm>

#include "raster.cuh"

namespace fa {
namespace {

using rs::RasterArgs;

template <bool DEV_M>
__global__ void __launch_bounds__(rs::kFrontThreads, 2) k_raster_front(RasterArgs A) {
  pdl_wait();
  rs::front_body<DEV_M>(A, blockIdx.x, gridDim.x);
}

enum ExactMode { kExactTwice, kExactWinners, kExactWinnersCons };

template <bool DEV_M, int MODE>
__global__ void __launch_bounds__(256, 4) k_raster_exact(RasterArgs A) {
  pdl_wait();
  if (MODE == kExactWinners) rs::exact_win_body<DEV_M, 256, false>(A, blockIdx.x, gridDim.x);
  else if (MODE == kExactWinnersCons) rs::exact_win_body<DEV_M, 256, true>(A, blockIdx.x, gridDim.x);
  else rs::exact_body<DEV_M, 256>(A, blockIdx.x, gridDim.x);
}

// (four resident blocks per SM for the winners' form: 317 us for the larger boxes of a
// 3.2M-triangle floor at 1440p, against 374 at its own 77 registers and three blocks)
template <bool WIN>
__global__ void __launch_bounds__(256, WIN ? 4 : 1) k_raster_depth_big(RasterArgs A) {
  pdl_wait();
  if (WIN) rs::depth_win_body(A, blockIdx.x, gridDim.x);
  else rs::depth_big_body(A, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(256) k_raster_zmax(RasterArgs A) {
  pdl_wait();
  rs::zmax_body(A, blockIdx.x, gridDim.x);
}

enum MarkMode { kMarkSamples, kMarkConservative, kMarkWinners };

template <int MODE>
__global__ void __launch_bounds__(256, 4) k_raster_mark(RasterArgs A) {
  pdl_wait();
  if (MODE == kMarkWinners) rs::mark_win_body<256>(A, blockIdx.x, gridDim.x);
  else rs::mark_body<MODE == kMarkConservative, 256>(A, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(256, 4) k_raster_mark_cons(RasterArgs A) {
  pdl_wait();
  rs::mark_cons_body<256>(A, blockIdx.x, gridDim.x);
  rs::mark_cons_tiles(A, blockIdx.x, gridDim.x);
}

}  // namespace

fa_status launch_visibility(fa_ctx* ctx, const fa_mesh* mesh, const Mat4& M, uint32_t W, uint32_t H,
                            uint32_t* vt, bool reset_status, cudaStream_t s, const float* Mdev, bool cons,
                            int32_t* tri_chart_init, uint32_t* partial_clear) {
  // one wave (two resident blocks per SM): half the survivor regions of two waves,
  // so the passes that look regions up scan fewer counts
  // (and enough blocks for the clears: at most 16 depth-buffer pixels per thread)
  const uint32_t fb = std::max(grid_for(mesh->T, rs::kFrontThreads, 152u * 2u),
                               grid_for((uint64_t)W * H, rs::kFrontThreads * 16u, 152u * 2u));
  const unsigned gb = 152 * 8;
  RasterArgs A = rs::make_raster_args(ctx, mesh, M, W, H, vt, reset_status, Mdev, cons, tri_chart_init, fb,
                                            rs::kFrontThreads);
  A.partial_clear = partial_clear;
  rs::set_exact_grid(A, gb, 256);
  ctx->front_blocks = A.front_blocks;
  mark(ctx, "k_raster_front", s);
  if (Mdev)
    launch_k(k_raster_front<true>, A.front_blocks, rs::kFrontThreads, 0, s, A);
  else
    launch_k(k_raster_front<false>, A.front_blocks, rs::kFrontThreads, 0, s, A);
  mark(ctx, "k_raster_exact", s);
  if (A.win && cons)
    launch_k(Mdev ? k_raster_exact<true, kExactWinnersCons> : k_raster_exact<false, kExactWinnersCons>, gb, 256, 0, s, A);
  else if (A.win)
    launch_k(Mdev ? k_raster_exact<true, kExactWinners> : k_raster_exact<false, kExactWinners>, gb, 256, 0, s, A);
  else
    launch_k(Mdev ? k_raster_exact<true, kExactTwice> : k_raster_exact<false, kExactTwice>, gb, 256, 0, s, A);
  mark(ctx, "k_raster_depth_big", s);
  launch_k(A.win ? k_raster_depth_big<true> : k_raster_depth_big<false>, gb, 256, 0, s, A);
  if (A.zmax) {
    mark(ctx, "k_raster_zmax", s);
    launch_k(k_raster_zmax, grid_for((uint64_t)A.ztx * ((H + 15) / 16) * 32, 256, 152 * 8), 256, 0, s, A);
  }
  mark(ctx, "k_raster_mark", s);
  // one wave of four resident blocks per SM: each block scans the region counts once
  if (A.win)  // (blocks of 64 x 32 pixels; enough threads for many triangles in a small window, should ties overflow)
    launch_k(k_raster_mark<kMarkWinners>,
             std::min(std::max(((W + 63) / 64) * ((H + 31) / 32), (mesh->T + 255) / 256), 152u * 8u), 256, 0, s, A);
  else
    launch_k(cons ? k_raster_mark<kMarkConservative> : k_raster_mark<kMarkSamples>, 152 * 4, 256, 0, s, A);
  if (A.win && cons) {
    mark(ctx, "k_raster_mark_cons", s);
    launch_k(k_raster_mark_cons, 152 * 4, 256, 0, s, A);  // (one wave: the shares are claimed)
  }
  FA_CUDA_TRY(cudaGetLastError());
  return FA_OK;
}

}  // namespace fa
