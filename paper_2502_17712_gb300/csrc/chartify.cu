// Chart kernels (Sec. 5.1; App. A "GPU Union Find", Alg. 1): the launch wrappers
// of the stage bodies in chartify.cuh and the launch sequence of one chart pass.
#include <algorithm>

#include "chartify.cuh"

namespace fa {
namespace {

using cf::UfArgs;
using cf::kBlock;
using cf::kPerBlock;
using cf::kTile;

template <bool LIST, int NT>
__global__ void __launch_bounds__(NT) k_uf_local(UfArgs a) {
  pdl_wait();
  cf::local_body<LIST, NT>(a, blockIdx.x, gridDim.x);
}

// The local union-find with the context's tile shape (NT threads per tile; listed
// tiles: a grid of the resident blocks, 2048 / NT per SM).
template <bool LIST>
void launch_local(uint32_t nt, uint32_t ntiles, cudaStream_t s, const UfArgs& a) {
  auto grid = [&](uint32_t per_sm) { return LIST ? std::min(ntiles, 152u * per_sm) : ntiles; };
  if (nt == 256)
    launch_k(k_uf_local<LIST, 256>, grid(8), 256, 0, s, a);
  else if (nt == 512)
    launch_k(k_uf_local<LIST, 512>, grid(4), 512, 0, s, a);
  else
    launch_k(k_uf_local<LIST, 1024>, grid(2), 1024, 0, s, a);
}

template <bool LIST>
__global__ void __launch_bounds__(128) k_uf_hook(UfArgs a) {
  pdl_wait();
  cf::hook_body<LIST>(a, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(kBlock) k_uf_hook_v(UfArgs a) {
  pdl_wait();
  cf::hook_v_body(a, blockIdx.x, gridDim.x);
}

__global__ void k_uf_hook_nm(UfArgs a, const uint32_t* nm_off, const uint32_t* nm_list, uint32_t n_nm) {
  pdl_wait();
  cf::hook_nm_body(a, nm_off, nm_list, n_nm, blockIdx.x, gridDim.x);
}

template <bool LIST>
__global__ void __launch_bounds__(kBlock) k_uf_flatten(UfArgs a, uint32_t* blockcnt, uint32_t* viscnt,
                                                       uint2* wordroots) {
  pdl_wait();
  cf::flatten_body<LIST, kBlock>(a, blockcnt, viscnt, wordroots, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(1024) k_scan_blocks(uint32_t* blockcnt, uint32_t* viscnt, uint32_t nblocks,
                                                      uint32_t* count_out, uint32_t max_charts,
                                                      DevCounters* ctr) {
  pdl_wait();
  cf::scan_blocks_body(blockcnt, viscnt, nblocks, count_out, max_charts, ctr);
}

template <bool LIST>
__global__ void __launch_bounds__(kBlock) k_tri_chart(UfArgs a, const uint32_t* blockcnt, const uint2* wordroots,
                                                      int32_t* tri_chart, uint32_t* roots, uint32_t* box_enc,
                                                      uint32_t* box_full, uint32_t max_charts,
                                                      const uint32_t* visstart, uint2* vis, uint32_t tri_blocks,
                                                      int32_t* vert_chart, int vertex_mode) {
  pdl_wait();
  // (the vertices' charts, when asked for, by the blocks past tri_blocks: they read what
  // the triangles' do, and a launch of their own costs 5 us)
  if (blockIdx.x < tri_blocks)
    cf::tri_chart_body<LIST, kBlock>(a, blockcnt, wordroots, tri_chart, roots, box_enc, box_full, max_charts,
                                     visstart, vis, blockIdx.x, tri_blocks);
  else
    cf::vert_chart_body(a, blockcnt, wordroots, vert_chart, vertex_mode, blockIdx.x - tri_blocks,
                        gridDim.x - tri_blocks);
}

}  // namespace

fa_status launch_chartify(fa_ctx* ctx, const fa_mesh* mesh, const uint32_t* vt, uint32_t mode,
                          int32_t* tri_chart, int32_t* vert_chart, const fa_charts* ch, cudaStream_t s,
                          bool tile_list, bool tri_chart_cleared) {
  UfArgs a = cf::make_uf_args(ctx, mesh, vt);
  const int vm = mode == FA_CHARTS_VERTEX;
  a.init_v = vm ? 1u : 0u;
  const unsigned gw = grid_for((uint64_t)((mesh->T + 31) / 32) * 32, kBlock, 152 * 16);
  const uint32_t ntiles = (mesh->T + kTile - 1) / kTile;
  mark(ctx, "k_uf_local", s);
  if (tile_list)
    launch_local<true>(ctx->uf_threads, ntiles, s, a);
  else
    launch_local<false>(ctx->uf_threads, ntiles, s, a);
  mark(ctx, "k_uf_hook", s);
  if (vm)
    launch_k(k_uf_hook_v, gw, kBlock, 0, s, a);
  else if (tile_list)
    launch_k(k_uf_hook<true>, ntiles < 152u * 8u ? ntiles : 152u * 8u, 128, 0, s, a);
  else
    launch_k(k_uf_hook<false>, ntiles, 128, 0, s, a);
  if (!vm && mesh->n_nm) {
    mark(ctx, "k_uf_hook_nm", s);
    launch_k(k_uf_hook_nm, grid_for(mesh->n_nm, 256), 256, 0, s, a, mesh->nm_off, mesh->nm_list, mesh->n_nm);
  }
  const uint32_t nb = (mesh->T + kPerBlock - 1) / kPerBlock;
  mark(ctx, "k_uf_flatten", s);
  if (tile_list)
    launch_k(k_uf_flatten<true>, nb < 152u * 8u ? (nb ? nb : 1u) : 152u * 8u, kBlock, 0, s, a, ctx->blockcnt,
             ctx->viscnt, ctx->wordroots);
  else
    launch_k(k_uf_flatten<false>, nb ? nb : 1, kBlock, 0, s, a, ctx->blockcnt, ctx->viscnt, ctx->wordroots);
  mark(ctx, "k_scan_blocks", s);
  launch_k(k_scan_blocks, 1, 1024, 0, s, ctx->blockcnt, ctx->viscnt, nb ? nb : 1, ch->count, ctx->cfg.max_charts,
           ctx->ctr);
  mark(ctx, "k_tri_chart", s);
  const bool listed = tile_list && tri_chart_cleared;
  const uint32_t tb = listed ? std::min(nb ? nb : 1u, 152u * 8u) : (nb ? nb : 1u);
  const uint32_t vb = vert_chart ? grid_for(mesh->V, kBlock, 152 * 8) : 0u;
  launch_k(listed ? k_tri_chart<true> : k_tri_chart<false>, tb + vb, kBlock, 0, s, a, ctx->blockcnt, ctx->wordroots,
           tri_chart, ch->root, ctx->box_enc, ctx->box_full, ctx->cfg.max_charts, ctx->viscnt, ctx->vis, tb, vert_chart,
           vm);
  FA_CUDA_TRY(cudaGetLastError());
  return FA_OK;
}

}  // namespace fa
