// Tensor maps of bf16 matrices for bulk-tensor loads: boxes of 64 tokens with the 128-byte swizzle the MMA's
// B descriptor expects.  The encoder lives in the driver library; it is looked up through the runtime
// so that this library has no link-time dependency on the driver.
#include <string.h>

#include "ts_internal.h"

namespace ts {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn g_encode = nullptr;

static bool encoder() {
  if (g_encode) return true;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess || !fn || q != cudaDriverEntryPointSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  g_encode = (EncodeTiledFn)fn;
  return true;
}

// tensor map of a matrix [ctx r][stride] for boxes of 64 x box_rows
static bool encode(const ts_ctx* ctx, const void* W, int stride, int box_rows, CUtensorMap* out) {
  if (!encoder()) return false;
  const cuuint64_t gdim[2] = {(cuuint64_t)stride, (cuuint64_t)ctx->cfg.r};
  const cuuint64_t gstride[1] = {(cuuint64_t)stride * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows}, estr[2] = {1u, 1u};
  return g_encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(W), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool w_tensor_map(ts_ctx* ctx, const void* W) {
  if (ctx->tma_state < 0 || ((uintptr_t)W & 15u) != 0) return false;
  if (ctx->tma_state == 1 && ctx->tmapW_ptr == W) return true;
  CUtensorMap tm;
  if (!encode(ctx, W, ctx->cfg.V, (ctx->cfg.r + 15) / 16 * 16, &tm)) { ctx->tma_state = -1; return false; }   // (r <= 256 = the most rows a box may have)
  memcpy(ctx->tmapW, &tm, sizeof(tm));
  ctx->tmapW_ptr = W;
  ctx->tma_state = 1;
  return true;
}

bool tree_tensor_map(ts_ctx* ctx, const void* W, int stride, CUtensorMap* out) {
  if (ctx->test_mode & TS_TEST_NO_TMA) return false;
  if (ctx->tmapT_ptr == W) { memcpy(out, ctx->tmapT, sizeof(*out)); return true; }
  if (!encode(ctx, W, stride, (ctx->cfg.r + 15) / 16 * 16, out)) return false;
  memcpy(ctx->tmapT, out, sizeof(*out));
  ctx->tmapT_ptr = W;
  return true;
}

bool u_tensor_map(ts_ctx* ctx, const void* U, int stride, int B, int rows, CUtensorMap* out) {
  if (ctx->test_mode & TS_TEST_NO_TMA) return false;
  if (ctx->tmapU_ptr == U && ctx->tmapU_B == B) { memcpy(out, ctx->tmapU, sizeof(*out)); return true; }
  if (!encoder()) return false;
  const cuuint64_t gdim[3] = {(cuuint64_t)stride, (cuuint64_t)ctx->cfg.D, (cuuint64_t)B};
  const cuuint64_t gstride[2] = {(cuuint64_t)stride * 2, (cuuint64_t)stride * 2 * (cuuint64_t)ctx->cfg.D};
  const cuuint32_t box[3] = {64u, 1u, (cuuint32_t)rows}, estr[3] = {1u, 1u, 1u};
  if (g_encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(U), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return false;
  memcpy(ctx->tmapU, out, sizeof(*out));
  ctx->tmapU_ptr = U; ctx->tmapU_B = B;
  return true;
}

}  // namespace ts
