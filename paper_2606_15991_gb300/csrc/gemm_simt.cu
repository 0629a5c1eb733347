// FP32 GEMM on the CUDA cores (FFMA, FP32 accumulation, no TF32): one 64x64
// C tile per tile program with a K loop (§3.6, Listing 6). Plain partitions
// launch one program per tile; mapped partitions launch persistent programs
// that walk their tiles (strided slots or a device queue), slots being turned
// into tiles by the band raster shared with the tensor-core GEMM.
#include "gemm_f32.cuh"

namespace tp {

tp_status launch_gemm_simt(tp_ctx* ctx, tp_partition* c, const tp_tensor* a, const tp_tensor* b,
                           const tp_gemm_config* cfg, const tp_exec* ex, cudaStream_t stream,
                           unsigned* queue) {
  if (c->tile[0] != BM || c->tile[1] != BN)
    return fail(TP_ERR_UNSUPPORTED, "the FP32 GEMM uses 64 x 64 output tiles");
  if ((ex->write_counts == nullptr) != (ex->write_owner == nullptr))
    return fail(TP_ERR_INVALID, "write_counts and write_owner must be given together");
  SimtArgs p{};
  p.a = static_cast<const float*>(a->ptr);
  p.b = static_cast<const float*>(b->ptr);
  p.c = static_cast<float*>(c->t.ptr);
  p.M = a->shape[0];
  p.K = a->shape[1];
  p.N = b->shape[1];
  p.sam = a->strides[0];
  p.sak = a->strides[1];
  p.sbk = b->strides[0];
  p.sbn = b->strides[1];
  p.gm = c->grid[0];
  p.gn = c->grid[1];
  p.kind = c->kind;
  // a plain partition is program p -> tile p in row-major order (§3.4)
  p.group_m = (c->kind != TP_MAP_IDENTITY && cfg && cfg->group_m > 0) ? cfg->group_m : 1;
  p.queue = queue;
  p.counts = ex->write_counts;
  p.owner = ex->write_owner;
  if (p.M == 0 || p.N == 0) return TP_OK;
  const int64_t grid = c->kind == TP_MAP_IDENTITY ? c->num_tiles : c->num_programs;
  const int bk = (cfg && cfg->bk > 0) ? cfg->bk : 32;
  p.split = (cfg && cfg->split_k > 1) ? cfg->split_k : 1;
  if (cfg && (cfg->split_k < 0 || cfg->split_k > 4 || (p.split & (p.split - 1))))
    return fail(TP_ERR_INVALID, "FP32 GEMM split_k must be 0, 1, 2 or 4");
  if (p.split > 1 && c->kind == TP_MAP_QUEUE)
    return fail(TP_ERR_UNSUPPORTED, "FP32 GEMM split_k with a queue map (each CTA would dequeue its own tile)");
  if (bk != 8 && bk != 16 && bk != 32) return fail(TP_ERR_UNSUPPORTED, "FP32 GEMM bk must be 8, 16 or 32");
  p.bk = bk;
  const cudaError_t e = p.counts ? launch_f32_counted(p, grid, ctx->sm_count, stream) : launch<false>(p, grid, ctx->sm_count, stream);
  if (e != cudaSuccess) return cuda_fail(e, "FP32 GEMM launch");
  return TP_OK;
}

}  // namespace tp
